"""Hint build on grids of one to six bins whose buckets hold more chunks than one
lane numbers (64 of 256 cells), and just as many: the graph against the oracle's as
in the other parity tests, one filter step within 1e-4 of the die."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _netlist(cells):
    from paper_2511_10073_gb300 import netgen
    rng = np.random.default_rng(6)
    pins = rng.permutation(cells)[:cells // 3 * 3].astype(np.int32)
    ptr = np.arange(0, pins.size + 1, 3).astype(np.int64)
    one, z = np.ones(cells, np.float32), np.zeros(cells, np.float32)
    kind = np.zeros(cells, np.uint8)
    kind[-1] = 2
    return netgen.Netlist(ptr, pins, np.zeros(pins.size, np.float32), np.zeros(pins.size, np.float32), one,
                          one, kind, z + 3.0, z + 4.0, (0.0, 0.0, 300.0, 300.0))


@pytest.mark.parametrize("wd", [1, 2])
@pytest.mark.parametrize("cells,nbx,nby", [(16384, 1, 1), (16400, 1, 1), (40000, 2, 1), (60001, 3, 2)])
def test_buckets_of_many_chunks(cells, nbx, nby, wd):
    import paper_2511_10073_gb300 as pl
    from test_gpu_parity import Side, _compare_hints, to_np
    s = Side(_netlist(cells), nbx=nbx, nby=nby, det_ratio=1.0, wdtype=wd)
    xy = torch.empty((s.N, 2), dtype=torch.float32, device="cuda")
    p = np.random.default_rng(7).normal(0.0, 60.0, (cells, 2)).clip(0.0, 300.0)  # most in the first bin
    pl.pl_init_signal(s.g, 1, torch.tensor(p.astype(np.float32), device="cuda"), xy)
    pl.pl_build_hints(s.g, s.prm, xy)
    a = to_np(xy)
    s.o.build_hints(a[:, 0], a[:, 1])
    _compare_hints(s, s.g.export(), s.o.merged())
    out = torch.empty_like(xy)
    pl.pl_filter_apply(s.g, s.prm, xy, out)
    ref = np.stack(s.o.filter(a[:, 0], a[:, 1]), 1)
    assert np.abs(to_np(out) - ref).max() <= 1e-4 * s.die
