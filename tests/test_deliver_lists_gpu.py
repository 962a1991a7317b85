"""Phase 2 alone on every record layout, at the list lengths and row shapes where the
kernels change course: fewer and more senders than warps, batches and summing start at,
empty rows, segments longer than a batch's round, delays that are summed and delays that
are not, and lists long enough for the slices of delays."""

import numpy as np
import pytest

import workload

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no GPU", allow_module_level=True)

import paper_2405_02019_gb300 as snn  # noqa: E402

FORMS = {"plain": (snn.RECORD_PLAIN9, 0), "int8": (snn.RECORD_PACKED_I8, 0), "bf16": (snn.RECORD_PACKED_BF16, 0),
         "blocked4": (snn.RECORD_BLOCKED4, 0), "blocked6": (snn.RECORD_BLOCKED6, 0),
         "blocked8": (snn.RECORD_BLOCKED8, 0), "resident": (snn.RECORD_PLAIN9, snn.ENGINE_RESIDENT)}


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2405_02019_gb300 import build

    build.build()


def _edges(n, mean_row, long_delays):
    """Rows of very different lengths, every seventh empty; weights that every format keeps
    exactly (whole multiples of 1 pA up to 127)."""
    rng = np.random.default_rng(n + mean_row)
    length = rng.integers(0, 2 * mean_row, n)
    length[::7] = 0
    pre = np.repeat(np.arange(n), length)
    # one sender reaches few targets often (long segments)
    post = np.where(pre == 5, rng.integers(0, 40, len(pre)), rng.integers(0, n, len(pre)))
    d = np.clip(np.rint(rng.normal(15, 7.5, len(pre))), 1, 63)
    if long_delays:
        some = rng.random(len(pre)) < 0.05
        d[some] = rng.integers(28, 64, some.sum())
    w = rng.integers(1, 128, len(pre)) * np.where(rng.random(len(pre)) < 0.5, -1, 1) * 4096
    w[:2] = (127 * 4096, -127 * 4096)
    return {"pre": pre, "post": post, "w_fx": w, "delay": d, "u0": np.zeros(n, np.float32)}


@pytest.fixture(scope="module")
def nets():
    made = {}

    def get(form, n, mean_row, long_delays):
        key = (form, n, mean_row, long_delays)
        if key not in made:
            m = workload.microcircuit_model().replace(nu_th_hz=0.0)
            e = _edges(n, mean_row, long_delays)
            record, engine = FORMS[form]
            made[key] = (e, snn.Network(m, custom=e, record_format=record, engine=engine))
        return made[key]

    yield get
    for _, net in made.values():
        net.close()


@pytest.mark.parametrize("count", [1, 31, 64, 65, 1025, 5003])
@pytest.mark.parametrize("shape", [(1733, 1500, True), (4100, 300, False)])
@pytest.mark.parametrize("form", list(FORMS))
def test_ring_after_list(nets, form, shape, count):
    e, net = nets(form, *shape)
    n = shape[0]
    rng = np.random.default_rng(count)
    senders = rng.integers(0, n, count)
    senders[0] = 5
    t = 61
    npad = int(net.layout().n_neurons_padded)
    ring = net.device_view("ring", torch.int32, 64 * npad)
    ring.zero_()
    net.deliver_spikes(torch.from_numpy(senders.astype(np.int32)).cuda(), t)
    times = np.bincount(senders, minlength=n)[e["pre"]]
    want = np.zeros((64, npad), np.int64)
    np.add.at(want, ((t + e["delay"].astype(np.int64)) % 64, e["post"]), e["w_fx"].astype(np.int64) * times)
    assert np.abs(want).max() < 1 << 31
    assert np.array_equal(ring.cpu().numpy().reshape(64, npad), want)


@pytest.mark.parametrize("form", ["plain", "blocked4", "blocked6", "blocked8"])
def test_ring_after_burst_step(form):
    """Every neuron spikes at step 0: the graph engine's phase 2 on a step with more events
    than it reduces row by row."""
    n = 1733
    e = dict(_edges(n, 1500, True), u0=np.full(n, 100.0, np.float32))
    m = workload.microcircuit_model().replace(nu_th_hz=0.0)
    net = snn.Network(m, custom=e, record_format=FORMS[form][0], engine=snn.ENGINE_GRAPH)
    net.step(1)
    assert len(net.read_spikes()[0]) == n
    npad = int(net.layout().n_neurons_padded)
    want = np.zeros((64, npad), np.int64)
    np.add.at(want, (e["delay"].astype(np.int64) % 64, e["post"]), e["w_fx"].astype(np.int64))
    ring = net.device_view("ring", torch.int32, 64 * npad).cpu().numpy().reshape(64, npad)
    assert np.array_equal(ring, want)
