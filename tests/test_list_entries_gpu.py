"""Sender lists on block-major records: entries outside [0, n) deliver nothing, whatever
their low bits are."""

import numpy as np
import pytest

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


@pytest.mark.parametrize("count", [7, 64, 1025])
def test_entries_outside_the_network_deliver_nothing(count):
    n = 700
    rng = np.random.default_rng(count)
    pre = np.repeat(np.arange(n), 90)
    e = {"pre": pre, "post": rng.integers(0, n, len(pre)), "delay": rng.integers(1, 64, len(pre)),
         "w_fx": rng.integers(-4096, 4097, len(pre)), "u0": np.zeros(n, np.float32)}
    m = workload.microcircuit_model().replace(nu_th_hz=0.0)
    net = snn.Network(m, custom=e, engine=snn.ENGINE_RESIDENT)
    senders = rng.integers(0, n, count)
    outside = np.array([-1, n, 2**31 - 1, -2**31, -2**31 + 5, -2**31 + n - 1])
    at = rng.permutation(count)[: len(outside)]
    senders[at] = outside
    t = 9
    npad = int(net.layout().n_neurons_padded)
    ring = net.device_view("ring", torch.int32, 64 * npad)
    ring.zero_()
    net.deliver_spikes(torch.from_numpy(senders.astype(np.int32)).cuda(), t)
    times = np.bincount(np.delete(senders, at), minlength=n)[pre]
    want = np.zeros((64, npad), np.int64)
    np.add.at(want, ((t + e["delay"]) % 64, e["post"]), e["w_fx"] * times)
    assert np.array_equal(ring.cpu().numpy().reshape(64, npad), want)
    net.close()
