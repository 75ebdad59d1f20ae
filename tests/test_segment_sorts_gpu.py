"""Segmented sorts of few, long segments: exact against the oracle where every
class of segment lengths has several segments to a block or a block to itself,
and as fast as with many short segments beside them."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _netlist(cells, sizes, seed):
    from paper_2511_10073_gb300 import netgen
    rng = np.random.default_rng(seed)
    ptr = np.r_[0, np.cumsum(sizes)].astype(np.int64)
    pins = rng.integers(0, cells, int(ptr[-1])).astype(np.int32)
    z, one = np.zeros(len(pins), np.float32), np.ones(cells, np.float32)
    kind, pos = np.zeros(cells, np.uint8), np.zeros(cells, np.float32)
    return netgen.Netlist(ptr, pins, z, z, one, one, kind, pos, pos, (0.0, 0.0, 100.0, 100.0))


@pytest.mark.parametrize("sizes", [[1000] * 70, [4096] * 3 + [513] * 5 + [300] * 9 + [5] * 3,
                                   [100] * 200 + [9] * 5 + [4097], [2000], [40] * 65])
def test_few_long_nets(sizes):
    from test_gpu_parity import Side
    s = Side(_netlist(3000, sizes, 3), nbx=16, nby=16)
    ge, oe = s.g.export_static(), s.o.static_csr()
    for a, b in (("rp", "rp"), ("col", "col"), ("w", "w_store"), ("base_w", "base_w")):
        assert np.array_equal(ge[a], oe[b])


def test_long_nets_alone_take_no_longer():
    """A netlist of 600 nets of 1000 pins builds no slower than one that holds
    the same nets and 40,000 two-pin nets more."""
    import paper_2511_10073_gb300 as pl

    def build_time(sizes):
        dnl = pl.DeviceNetlist(_netlist(30000, sizes, 1))
        prm = pl.params(nbx=16, nby=16)
        g = pl.pl_build_graph(dnl, prm)
        best = np.inf
        for _ in range(12):
            torch.cuda.synchronize()
            t = time.perf_counter()
            pl.pl_build_graph(dnl, prm, graph=g)
            best = min(best, time.perf_counter() - t)
        return best

    assert build_time([1000] * 600) <= 1.1 * build_time([1000] * 600 + [2] * 40000)
