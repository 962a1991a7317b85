"""Raster reads ordered on the device: (step, neuron) order at the sizes where the host and
the device take over from each other, and with circuit groups, whose runs of steps lie one
group after another in the raster."""

import numpy as np
import pytest

import oracle
import workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no GPU", allow_module_level=True)

import paper_2405_02019_gb300 as snn  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2405_02019_gb300 import build

    build.build()
    oracle.build()


@pytest.mark.parametrize("engine", [snn.ENGINE_PIPELINED, snn.ENGINE_GRAPH, snn.ENGINE_RESIDENT])
@pytest.mark.parametrize("burst", [1, 2047, 2048, 2049, 8192, 8193, 20000])
def test_burst_of_one_step(burst, engine):
    """`burst` neurons, every third of them, start above threshold and spike at step 0 (the
    largest number of spikes of one step that the device orders is 8,192)."""
    m = workload.microcircuit_model().replace(nu_th_hz=0.0)
    n = 3 * burst + 1
    u0 = np.zeros(n, np.float32)
    u0[1::3] = 100.0
    none = np.zeros(0, np.int32)
    net = snn.Network(m, custom={"pre": none, "post": none, "w_fx": none, "delay": none, "u0": u0}, engine=engine)
    net.step(3)
    steps, neurons = net.read_spikes()
    assert np.array_equal(neurons, np.arange(1, n, 3)) and np.all(steps == 0)
    net.step(2)
    assert len(net.read_spikes()[0]) == 0


@pytest.mark.parametrize("engine", [snn.ENGINE_PIPELINED, snn.ENGINE_GRAPH])
@pytest.mark.parametrize("groups", [0, 1, 2])
def test_grouped_batch(model, groups, engine):
    circuits = [(60, 100, 3), (100, 150, 4), (45, 120, 5)]
    net = snn.Network(model, circuits=circuits, engine=engine)
    net.set_circuit_groups(groups)
    base, count = net.circuits()
    got = [[], []]
    for m in (1, 1500, 40):
        net.step(m)
        for g, r in zip(got, net.read_spikes()):
            g.append(r)
    steps, neurons = map(np.concatenate, got)
    assert np.array_equal(np.lexsort((neurons, steps)), np.arange(len(steps)))
    for c, (sn, sk, seed) in enumerate(circuits):
        onet = oracle.build_network(model, sn, sk, seed)
        ts, ns = oracle.Sim(model, onet, seed).run(1541)
        mine = (neurons >= base[c]) & (neurons < base[c] + count[c])
        assert np.array_equal(steps[mine], ts) and np.array_equal(neurons[mine] - base[c], ns)
