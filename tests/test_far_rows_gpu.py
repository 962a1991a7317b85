"""Rows beyond record 2^34: a step's list of rows keeps every bit of where a row starts.

A network of that size takes hours to sample, so a small one's rows are moved: its record
arrays are copied 2^34 records up, inside an arena that is large enough, zeros are left in
their place, and the device's row bounds point to the copies.  The run must not change."""

import ctypes as C

import numpy as np
import pytest

import workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no GPU", allow_module_level=True)

import paper_2405_02019_gb300 as snn  # noqa: E402

FAR = 1 << 34
RECORDS = {  # bytes per record of each array that the format keeps
    "plain": (snn.RECORD_PLAIN9, {"syn_tgt": 4, "syn_w": 4, "syn_delay": 1}),
    "int8": (snn.RECORD_PACKED_I8, {"syn_tgt": 4, "syn_w": 1}),
}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2405_02019_gb300 import build

    build.build()


def _run(custom, engine, record, arrays, far):
    """Spikes and ring of 150 steps."""
    m = workload.microcircuit_model()
    kept = snn._Spec(m, custom=custom, engine=engine, record_format=record)  # owns the arrays spec points to
    spec = kept.spec
    need = int(snn.snn_query_sizes(spec).arena_bytes)
    span = 4 * FAR + 2 * need if far else need
    arena = torch.empty(span + 256, dtype=torch.uint8, device="cuda")
    base = (arena.data_ptr() + 255) // 256 * 256
    at = base - arena.data_ptr()
    stream = torch.cuda.current_stream().cuda_stream
    h = snn.snn_build_network(spec, base, span, stream)
    try:
        lay = snn.snn_get_layout(h)
        n = len(custom["u0"])
        if far:
            rows = arena[at + lay.row_ptr: at + lay.row_ptr + 8 * (n + 1)].view(torch.int64)
            records = int(rows[n])
            for name, size in arrays.items():
                lo = at + getattr(lay, name)
                near = arena[lo: lo + size * records]
                arena[lo + size * FAR: lo + size * (FAR + records)].copy_(near)
                near.zero_()
            rows += FAR
        torch.cuda.synchronize()
        snn.snn_step_n(h, 150, stream)
        steps, neurons = snn.snn_read_spikes(h)
        npad = int(lay.n_neurons_padded)
        ring = arena[at + lay.ring: at + lay.ring + 4 * 64 * npad].cpu().numpy()
        return steps, neurons, ring
    finally:
        snn.load().snn_destroy(C.c_void_p(h))


@pytest.mark.parametrize("record", list(RECORDS))
@pytest.mark.parametrize("engine", [snn.ENGINE_GRAPH, snn.ENGINE_PIPELINED, snn.ENGINE_PERSISTENT])
def test_rows_beyond_2_34_records(engine, record):
    if torch.cuda.mem_get_info()[0] < 4 * FAR + (8 << 30):
        pytest.skip("needs 77 GB of free device memory")
    n = 1200
    rng = np.random.default_rng(7)
    pre = np.repeat(np.arange(n), rng.integers(0, 700, n))
    w = rng.integers(-40, 100, len(pre)) * 4096
    w[:2] = (127 * 4096, -127 * 4096)  # whole multiples of 1 pA: every format keeps them
    custom = {"pre": pre, "post": rng.integers(0, n, len(pre)), "w_fx": w,
              "delay": rng.integers(1, 64, len(pre)), "u0": np.zeros(n, np.float32)}
    fmt, arrays = RECORDS[record]
    want = _run(custom, engine, fmt, arrays, False)
    got = _run(custom, engine, fmt, arrays, True)
    assert len(want[0]) > 100 and len(np.unique(want[0])) > 5
    for a, b in zip(want, got):
        assert np.array_equal(a, b)
    torch.cuda.empty_cache()
