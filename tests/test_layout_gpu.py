"""The hint matrix' layout on both of its routes: with hub rows and chunks bounded
(no read of sizes by the host) and, where a bound does not hold or does not fit
the workspace, with their exact counts.  Many cells have static rows just below
the hub threshold, so that whether a row is a hub row depends on its hints."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
CELLS = 3120


def _netlist(extra_macros):
    from paper_2511_10073_gb300 import netgen
    rng = np.random.default_rng(4)
    cells, mac = CELLS, extra_macros
    # every cell in seven cliques of 16 and one of 13: 117 static entries, fewer where cliques share
    nets = [n for size in [16] * 7 + [13] for n in rng.permutation(cells).reshape(-1, size)]
    nets += [np.r_[cells + k, rng.choice(cells, 3, replace=False)] for k in range(mac)]
    ptr = np.r_[0, np.cumsum([len(n) for n in nets])].astype(np.int64)
    pins = np.concatenate(nets).astype(np.int32)
    z = np.zeros(len(pins), np.float32)
    C = cells + mac
    w = np.ones(C, np.float32)
    w[cells:] = 30.0  # macros over one another: a cell overlaps all of them or none
    kind = np.r_[np.zeros(cells), np.ones(mac)].astype(np.uint8)
    pos = np.full(C, 50.0, np.float32)
    return netgen.Netlist(ptr, pins, z, z, w, w.copy(), kind, pos, pos.copy(), (0.0, 0.0, 100.0, 100.0))


@pytest.mark.parametrize("macros", [3, 12])
@pytest.mark.parametrize("wd", [1, 2])
def test_bounded_and_exact_layout(macros, wd):
    import paper_2511_10073_gb300 as pl
    from test_gpu_parity import Side, _compare_hints, to_np
    s = Side(_netlist(macros), nbx=32, nby=32, wdtype=wd)
    _, xy = s.oracle_signal(1)
    rng = np.random.default_rng(1)
    a = xy.view(-1, 2)
    a[:CELLS] = torch.tensor(rng.uniform(1.0, 99.0, (CELLS, 2)).astype(np.float32), device="cuda")
    pl.pl_build_hints(s.g, s.prm, xy)
    b = to_np(xy)
    s.o.build_hints(b[:, 0], b[:, 1])
    ge, oe = s.g.export(), s.o.merged()
    _compare_hints(s, ge, oe)
    lens = np.diff(oe["rp"])[:CELLS]
    assert (lens > 128).sum() > 20 and (lens <= 128).sum() > 100
    want = torch.empty_like(xy)
    pl.pl_filter_apply(s.g, s.prm, xy, want)
    # a workspace that the exact counts fit and the bounds do not (with more
    # macros over a cell than the bounds assume, the first build was exact already)
    need = s.g.info()["ws_peak"] - (40_000 if macros == 3 else 0)
    ws = pl.workspace(need)
    g = pl.pl_build_graph(s.dnl, s.prm, xy, ws=ws)
    got = torch.empty_like(xy)
    pl.pl_filter_apply(g, s.prm, xy, got)
    assert torch.equal(got, want)
    with pytest.raises(pl.PlError) as e:
        pl.pl_build_graph(s.dnl, s.prm, xy, ws=pl.workspace(need // 2))
    assert e.value.code == pl.PL_ERR_WORKSPACE
