"""pl_hpwl with more long nets than a warp's list holds, in one batch and over
several of the warp's batches, against the oracle (1e-5 relative, the bar of the
other HPWL tests); the time of long nets, which is that of their number, and of
nets just above what a lane spans alone."""
import time

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _nl(sizes, seed):
    from paper_2511_10073_gb300 import netgen
    rng = np.random.default_rng(seed)
    C = 5000
    ptr = np.r_[0, np.cumsum(sizes)].astype(np.int64)
    pins = rng.integers(0, C, ptr[-1]).astype(np.int32)
    one, z = np.ones(C, np.float32), np.zeros(C, np.float32)
    return netgen.Netlist(ptr, pins, None, None, one, one, np.zeros(C, np.uint8), z, z,
                          (0.0, 0.0, 100.0, 100.0)), rng.uniform(0, 100, (C, 2)).astype(np.float32)


BATCHES = np.ones(320000, np.int64)
BATCHES[:40] = 1100            # the first warp's batches: of 608 blocks of 8 warps of 32 nets
BATCHES[155648:155680] = 1030
BATCHES[311296:311299] = 1500
BATCHES[-1] = 2000


@pytest.mark.parametrize("sizes", [[1025] * 31, [1025] * 32, [1025] * 33 + [3] * 40 + [1024, 1100],
                                   [1, 1500] * 60, BATCHES], ids=["31", "32", "33", "every_other", "batches"])
def test_more_long_nets_than_a_list(sizes):
    import paper_2511_10073_gb300 as pl
    nl, xy = _nl(sizes, 3)
    ws, out = pl.hpwl_workspace(nl.num_nets), torch.zeros(1, dtype=torch.float64, device="cuda")
    dnl, t = pl.DeviceNetlist(nl), torch.tensor(xy, device="cuda")
    pl.pl_hpwl(dnl, t, out, ws)
    ref = oracle.hpwl(nl, xy[:, 0].astype(np.float64), xy[:, 1].astype(np.float64))
    assert float(out) == pytest.approx(ref, rel=1e-5)
    dnl.pin_cell[nl.net_ptr[-2]] = -1  # a bad pin in the last net
    pl.pl_hpwl(dnl, t, out, ws)
    assert np.isnan(float(out))


def _time(sizes):
    import paper_2511_10073_gb300 as pl
    nl, xy = _nl(sizes, 5)
    ws, out = pl.hpwl_workspace(nl.num_nets), torch.zeros(1, dtype=torch.float64, device="cuda")
    dnl, t, best = pl.DeviceNetlist(nl), torch.tensor(xy, device="cuda"), np.inf
    for _ in range(12):
        torch.cuda.synchronize()
        a = time.perf_counter()
        pl.pl_hpwl(dnl, t, out, ws)
        torch.cuda.synchronize()
        best = min(best, time.perf_counter() - a)
    return best


def test_time_of_long_nets_is_linear():
    assert _time([200000] * 24) <= 1.25 * 3 * _time([200000] * 8)


def test_nets_of_17_pins_take_little_longer_than_of_16():
    assert _time([17] * 400000) <= 1.25 * _time([16] * 400000)
