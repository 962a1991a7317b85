"""A step graph that cannot be uploaded is released: the network's set-up fails with an error
and leaves no instantiated graph behind.  The failure is an error code from a stand-in for
cudaGraphUpload, preloaded into a process of its own."""

import os
import subprocess
import sys
import textwrap

import pytest

from conftest import ROOT

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no GPU", allow_module_level=True)

STAND_IN = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
static int live, uploads;
static void *next(const char *name) { return dlsym(RTLD_NEXT, name); }
int cudaGraphInstantiate(void **exec, void *graph, unsigned long long flags)
{
    int (*f)(void **, void *, unsigned long long) = next("cudaGraphInstantiate");
    const int e = f(exec, graph, flags);
    live += e == 0;
    return e;
}
int cudaGraphExecDestroy(void *exec)
{
    int (*f)(void *) = next("cudaGraphExecDestroy");
    live -= 1;
    return f(exec);
}
int cudaGraphUpload(void *exec, void *stream)
{
    int (*f)(void *, void *) = next("cudaGraphUpload");
    return ++uploads == FAIL_AT ? 2 : f(exec, stream);  /* 2: cudaErrorMemoryAllocation */
}
int graphs_live(void) { return live; }
int graphs_uploaded(void) { return uploads; }
"""

CHILD = """
    import ctypes, sys
    sys.path.insert(0, {root!r})
    import torch, workload
    import paper_2405_02019_gb300 as snn
    shim = ctypes.CDLL({shim!r})
    try:
        snn.Network(workload.microcircuit_model(), 30, 100, engine={engine})
    except snn.SnnError as e:
        print("code", e.code)
    print("uploads", shim.graphs_uploaded(), "live", shim.graphs_live())
"""


@pytest.mark.parametrize("engine", [1, 3])  # the graph and the pipelined engine
@pytest.mark.parametrize("fail_at", [1, 3])
def test_failed_upload_releases_the_graph(tmp_path, engine, fail_at):
    from paper_2405_02019_gb300 import build

    build.build()
    src, shim = tmp_path / "stand_in.c", tmp_path / "stand_in.so"
    src.write_text(STAND_IN.replace("FAIL_AT", str(fail_at)))
    subprocess.run(["gcc", "-shared", "-fPIC", "-w", "-o", str(shim), str(src), "-ldl"], check=True)
    code = textwrap.dedent(CHILD.format(root=ROOT, shim=str(shim), engine=engine))
    r = subprocess.run([sys.executable, "-c", code], env=dict(os.environ, LD_PRELOAD=str(shim)), capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.split() == ["code", "3", "uploads", str(fail_at), "live", "0"], r.stdout
