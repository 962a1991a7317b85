"""Arena sizes that snn_query_sizes reports (host only)."""

import numpy as np
import pytest

import paper_2405_02019_gb300 as snn


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2405_02019_gb300 import build

    build.build()


def _arena(model, n=0, **kw):
    if n:
        none = np.zeros(0, np.int32)
        kw["custom"] = {"pre": none, "post": none, "w_fx": none, "delay": none, "u0": np.zeros(n, np.float32)}
    spec = snn._Spec(model, raster_capacity=1024, **kw)
    return int(snn.snn_query_sizes(spec.spec).arena_bytes)


@pytest.mark.parametrize("record", [snn.RECORD_PLAIN9, snn.RECORD_PACKED_I8, snn.RECORD_PACKED_BF16])
def test_delay_table_only_where_lists_read_it(model, record):
    """Lists go by slices of delays up to 81,920 neurons; the table of 128 bytes a neuron that
    they read is not part of a larger network's arena."""
    slices = _arena(model, 81920, record_format=record)
    rows = _arena(model, 81921, record_format=record)
    assert slices - rows > 120 * 81920
    assert _arena(model, 81793, record_format=record) > rows


def test_delay_table_of_a_batch(model):
    """A batch is one network: its circuits' neurons count together (77,169 at full scale)."""
    one, two, three = (_arena(model, circuits=[(1000, 0, 1 + c) for c in range(k)]) for k in (1, 2, 3))
    assert (three - two) - (two - one) > 120 * 77169  # the second circuit takes the first one's table out
