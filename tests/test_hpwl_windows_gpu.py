"""pl_hpwl where its windows and lists end: nets around the window, lane and
block sizes at every offset, more long nets in one batch than a warp keeps for
its block, empty nets between them, and bad pins at both ends; against the
oracle (1e-5 relative, the bar of the other HPWL tests)."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = {
    "windows": [1, 255, 1, 256, 2, 257, 16, 17, 0, 240, 15, 1, 511, 513, 33] * 9,
    "long_batch": [1500] * 12 + [3] * 5 + [1025, 1024, 1026] * 6 + [0, 2, 0],
    "one_long": [20000],
    "long_ends": [1200] + [2] * 30 + [1300] + [1100, 0, 1, 1400],
    "short": [2, 3] * 500 + [0] * 40 + [1] * 70,
}


def _nl(sizes, seed, offsets):
    from paper_2511_10073_gb300 import netgen
    rng = np.random.default_rng(seed)
    C = 700
    ptr = np.r_[0, np.cumsum(sizes)].astype(np.int64)
    pins = rng.integers(0, C, ptr[-1]).astype(np.int32)
    d = [rng.uniform(-2, 2, ptr[-1]).astype(np.float32) if offsets else None for _ in range(2)]
    one, z = np.ones(C, np.float32), np.zeros(C, np.float32)
    return netgen.Netlist(ptr, pins, d[0], d[1], one, one, np.zeros(C, np.uint8), z, z, (0.0, 0.0, 100.0, 100.0)), \
        rng.uniform(0, 100, (C, 2)).astype(np.float32)


@pytest.mark.parametrize("offsets", [True, False])
@pytest.mark.parametrize("name", sorted(SIZES))
def test_hpwl_sizes(name, offsets):
    import paper_2511_10073_gb300 as pl
    nl, xy = _nl(SIZES[name], 3, offsets)
    dnl = pl.DeviceNetlist(nl)
    ws = pl.hpwl_workspace(nl.num_nets)
    ws.zero_()
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    for _ in range(2):  # the workspace is left ready for the next call
        pl.pl_hpwl(dnl, torch.tensor(xy, device="cuda"), out, ws)
        ref = oracle.hpwl(nl, xy[:, 0].astype(np.float64), xy[:, 1].astype(np.float64))
        assert float(out) == pytest.approx(ref, rel=1e-5)
    for at in (0, -1):
        bad = dnl.pin_cell.clone()
        dnl.pin_cell[at] = 700
        pl.pl_hpwl(dnl, torch.tensor(xy, device="cuda"), out, ws)
        assert np.isnan(float(out))
        dnl.pin_cell.copy_(bad)


def test_hpwl_nan_net():
    import paper_2511_10073_gb300 as pl
    nl, xy = _nl([5, 4, 1500], 5, False)
    ws = pl.hpwl_workspace(nl.num_nets)
    ws.zero_()
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    xy[nl.pin_cell[:5]] = np.nan  # every pin of the first net
    pl.pl_hpwl(pl.DeviceNetlist(nl), torch.tensor(xy, device="cuda"), out, ws)
    assert np.isnan(float(out))
