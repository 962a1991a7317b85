"""Steps captured into the caller's own CUDA graph: replays, reads, state views, checkpoints
and calls outside the graph, in any order, give the spikes of an uninterrupted run."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no GPU", allow_module_level=True)

import paper_2405_02019_gb300 as snn  # noqa: E402

ENGINES = [snn.ENGINE_GRAPH, snn.ENGINE_PIPELINED, snn.ENGINE_PERSISTENT, snn.ENGINE_RESIDENT]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2405_02019_gb300 import build

    build.build()


def _state(net):
    n, npad = net.n_neurons, int(net.layout().n_neurons_padded)
    return [net.device_view("U", torch.int32, n).cpu(), net.device_view("R", torch.uint8, n).cpu(),
            net.device_view("ring", torch.int32, 64 * npad).cpu()]


@pytest.mark.parametrize("engine", ENGINES)
def test_replays_and_reads(model, engine):
    ref = snn.Network(model, 100, 100, seed=5, engine=engine)
    net = snn.Network(model, 100, 100, seed=5, engine=engine)
    steps, neurons = [], []

    def read(how):
        torch.cuda.synchronize()
        for out, part in zip((steps, neurons), how()):
            out.append(part)

    def check(t):
        ref.step(t - int(ref.info().t))
        assert int(net.info().t) == t
        for a, b in zip(_state(ref), _state(net)):
            assert torch.equal(a, b)

    net.step(7)
    read(net.read_spikes)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        net.step(33)
        assert int(net.info().t) == 7  # nothing has run
    read(net.read_spikes)
    check(7)
    graph.replay()
    read(net.read_spikes)
    check(40)
    graph.replay()
    graph.replay()
    read(net.collect_spikes)
    check(106)
    net.step(70)
    graph.replay()  # after a call whose end the host knows
    torch.cuda.synchronize()
    check(209)
    rates, counts = net.read_rates(0, 209)
    graph.replay()
    torch.cuda.synchronize()
    saved = net.save_state()
    read(net.read_spikes)
    check(242)
    graph.replay()
    read(net.read_spikes)
    want_t, want_i = ref.read_spikes()
    ref.step(33)
    late = ref.read_spikes()
    want_t, want_i = np.concatenate([want_t, late[0]]), np.concatenate([want_i, late[1]])
    assert len(want_t) > 500
    assert np.array_equal(np.concatenate(steps), want_t) and np.array_equal(np.concatenate(neurons), want_i)
    assert np.array_equal(counts, np.bincount(want_i[want_t < 209], minlength=net.n_neurons))
    net.load_state(saved)
    check_t = int(net.info().t)
    graph.replay()
    torch.cuda.synchronize()
    again = net.read_spikes()
    assert check_t == 242 and np.array_equal(again[0], late[0]) and np.array_equal(again[1], late[1])


@pytest.mark.parametrize("groups", [1, 2])
def test_groups_change_after_a_replay(model, groups):
    """The pending spikes move with the queue of the device's step, which the host has not
    counted."""
    circuits = [(60, 100, 3), (100, 150, 4), (45, 120, 5)]
    ref = snn.Network(model, circuits=circuits)
    net = snn.Network(model, circuits=circuits)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        net.step(5)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    net.set_circuit_groups(groups)
    net.step(300)
    ref.step(315)
    for a, b in zip(ref.read_spikes(), net.read_spikes()):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("engine", ENGINES[:2])
def test_long_captured_call_is_refused(model, engine):
    ref = snn.Network(model, 100, 100, seed=6, engine=engine, steps_per_graph=128)
    net = snn.Network(model, 100, 100, seed=6, engine=engine, steps_per_graph=128)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        with pytest.raises(snn.SnnError) as e:
            net.step(128)
        assert e.value.code == snn._abi.SNN_ENOTSUP
        net.step(127)  # the capture and the network are as they were
    graph.replay()
    torch.cuda.synchronize()
    ref.step(127)
    assert int(net.info().t) == 127
    for a, b in zip(ref.read_spikes(), net.read_spikes()):
        assert np.array_equal(a, b)
