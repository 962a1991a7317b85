"""Lists delivered by slices of delays, at the sizes where their layout changes: two delays of
all targets in shared memory at a time up to 20,480 neurons, one up to 40,960, one of half the
targets up to 81,920, and rows beyond; and on a batch, whose gaps are rows without synapses.

A list goes by slices where a cost rule finds them faster.  With m synapses in a mean row, G
groups of delays and P target ranges that is the case from 12 / (5.8e-6 m - 1.42e-6 P (m + 20 G))
senders on: about 33,000 for m = 257, G = 7 and P = 2 below, 3,500 for the batch."""

import numpy as np
import pytest

import workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no GPU", allow_module_level=True)

import paper_2405_02019_gb300 as snn  # noqa: E402

RECORDS = {"plain": snn.RECORD_PLAIN9, "int8": snn.RECORD_PACKED_I8, "bf16": snn.RECORD_PACKED_BF16}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2405_02019_gb300 import build

    build.build()


def _ring(net, senders, t):
    npad = int(net.layout().n_neurons_padded)
    ring = net.device_view("ring", torch.int32, 64 * npad)
    ring.zero_()
    net.deliver_spikes(torch.from_numpy(senders.astype(np.int32)).cuda(), t)
    return ring.cpu().numpy().reshape(64, npad)


def _want(npad, t, times, post, delay, w):
    """The ring after every sender's synapses were added `times` of the sender (float64 sums of
    integers below 2^53: exact)."""
    at = ((t + delay.astype(np.int64)) % 64) * npad + post
    total = np.bincount(at, weights=w.astype(np.float64) * times, minlength=64 * npad)
    assert np.abs(total).max() < 1 << 31
    return total.astype(np.int64).reshape(64, npad)


@pytest.fixture(scope="module")
def edges():
    """Rows of 0 to 600 synapses; delays with empty groups and a few long ones; weights that
    every format keeps exactly (multiples of 1 pA up to 127, both ends in every pair)."""
    made = {}

    def get(n):
        if n not in made:
            made.clear()
            rng = np.random.default_rng(n)
            length = rng.integers(0, 601, n)
            length[::7] = 0
            length[0] = 5000
            pre = np.repeat(np.arange(n, dtype=np.int32), length)
            k = len(pre)
            delay = rng.choice(np.array([1, 2, 3, 6], np.uint8), k, p=[0.3, 0.3, 0.2, 0.2])
            long = rng.random(k) < 0.02
            delay[long] = rng.integers(40, 64, int(long.sum()))
            w = (rng.integers(1, 128, k) * rng.choice([-4096, 4096], k)).astype(np.int32)
            made[n] = {"pre": pre, "post": rng.integers(0, n, k, dtype=np.int32), "w_fx": w, "delay": delay,
                       "u0": np.zeros(n, np.float32),
                       "pop_offsets": [0, n // 3, n // 2] + [n] * 6}
        return made[n]

    return get


@pytest.mark.parametrize("n", [20480, 20481, 40960, 40961, 81920, 81921])
def test_ring_where_the_layout_changes(edges, n):
    e = edges(n)
    m = workload.microcircuit_model().replace(nu_th_hz=0.0)
    rng = np.random.default_rng(3)
    senders = rng.integers(0, n, 60000)
    senders[:3] = (0, n - 1, n - 2)
    t = 59
    want = None
    for record in RECORDS.values():
        net = snn.Network(m, custom=e, record_format=record)
        got = _ring(net, senders, t)
        if want is None:
            times = np.bincount(senders, minlength=n)[e["pre"]]
            want = _want(got.shape[1], t, times, e["post"], e["delay"], e["w_fx"])
        assert np.array_equal(got, want), record
        net.close()


@pytest.mark.parametrize("record", ["plain", "int8"])
def test_ring_of_a_batch(model, record):
    """Three uneven circuits of 15,822 neurons in all, with the packed weights as they are read
    back."""
    circuits = [(60, 300, 3), (100, 300, 4), (45, 300, 5)]
    net = snn.Network(model, circuits=circuits, record_format=RECORDS[record])
    kept = snn._Spec(model, circuits=circuits, record_format=RECORDS[record])
    rows = snn.snn_export_network(kept.spec)
    n = net.n_neurons
    t, senders = 3, np.random.default_rng(4).integers(0, n, 8000)
    pre = np.repeat(np.arange(n), np.diff(rows["row_ptr"]))
    got = _ring(net, senders, t)
    times = np.bincount(senders, minlength=n)[pre]
    assert np.array_equal(got, _want(got.shape[1], t, times, rows["post"], rows["delay"], rows["w_fx"]))
