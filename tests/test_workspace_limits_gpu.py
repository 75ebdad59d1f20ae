"""Builds at the limits of the workspace: a build that runs out of it leaves no
kernel behind that the given stream does not cover, and the graph can be built
again."""
import numpy as np
import pytest

from paper_2511_10073_gb300 import netgen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _build(pl, dnl, prm, **kw):
    """Whether a build fits its workspace."""
    try:
        return pl.pl_build_graph(dnl, prm, **kw)
    except pl.PlError as e:
        assert e.code == pl.PL_ERR_WORKSPACE and "workspace too small" in str(e)
        return None


@pytest.mark.parametrize("own_stream", [False, True])
def test_a_failed_build_is_covered_by_its_stream(own_stream):
    import paper_2511_10073_gb300 as pl
    dnl = pl.DeviceNetlist(netgen.make_netlist("medium", 1))
    prm = pl.params(nbx=32, nby=32)
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream() if own_stream else torch.cuda.default_stream()):
        g = pl.pl_build_graph(dnl, prm)
        xy = torch.empty(g.info()["N"] * 2, dtype=torch.float32, device="cuda")
        pl.pl_init_signal(g, 1, None, xy)
        pl.pl_build_hints(g, prm, xy)
        want, out = torch.empty_like(xy), torch.empty_like(xy)
        pl.pl_filter_apply(g, prm, xy, want)
        static, peak = g.info()["ws_static"], g.info()["ws_peak"]

        def nothing_writes(ws):  # what the stream does next is not written over
            ws.fill_(0xA5)
            torch.cuda.synchronize()
            assert bool((ws == 0xA5).all())

        failed = 0
        for size in np.linspace(0.4 * static, static, 13)[:-1]:
            ws = pl.workspace(int(size))
            if _build(pl, dnl, prm, graph=g, ws=ws) is None:
                nothing_writes(ws)
                failed += 1
        assert failed >= 8
        failed = 0
        for size in np.linspace(static, peak, 25)[:-1]:
            ws = pl.workspace(int(size))
            h = _build(pl, dnl, prm, ws=ws)
            assert h is not None
            try:
                pl.pl_build_hints(h, prm, xy)
            except pl.PlError as e:
                assert e.code == pl.PL_ERR_WORKSPACE
                failed += 1
                nothing_writes(ws)
                pl.pl_build_graph(dnl, prm, graph=h)
                pl.pl_build_hints(h, prm, xy)
            pl.pl_filter_apply(h, prm, xy, out)
            assert torch.equal(out, want)
            h.destroy()
        assert failed >= 8
        pl.pl_build_graph(dnl, prm, graph=g)
        pl.pl_build_hints(g, prm, xy)
        pl.pl_filter_apply(g, prm, xy, out)
        assert torch.equal(out, want)


def test_a_rebuild_waits_for_what_was_queued_on_the_default_stream():
    """A call that does not synchronize, queued on the default stream (NULL) behind
    other work, reads the graph's workspace after a rebuild of the graph on
    another stream was asked for."""
    import paper_2511_10073_gb300 as pl
    dnl = pl.DeviceNetlist(netgen.make_netlist("medium", 1))
    other = pl.DeviceNetlist(netgen.make_netlist("medium", 2))
    prm = pl.params(nbx=32, nby=32)
    ws = pl.workspace(max(pl.pl_workspace_size(d, prm) for d in (dnl, other)))
    with torch.cuda.stream(torch.cuda.default_stream()):
        g = pl.pl_build_graph(dnl, prm, ws=ws)
        want = torch.empty(g.info()["N"] * 2, dtype=torch.float32, device="cuda")
        out = torch.zeros_like(want)
        pl.pl_init_signal(g, 1, None, want)
        a = torch.ones((8192, 8192), device="cuda")
        torch.cuda.synchronize()
        for _ in range(4):
            a @ a
        pl.pl_init_signal(g, 1, None, out)
    with torch.cuda.stream(torch.cuda.Stream()):
        pl.pl_build_graph(other, prm, graph=g, ws=ws)
    torch.cuda.synchronize()
    assert torch.equal(out, want)


@pytest.mark.parametrize("wd", [1, 2])
def test_small_tiles_do_not_cost_a_workspace(wd):
    """A design whose counting sorts take tiles of 1024 cells where there is room:
    workspaces that hold the build only with tiles of 4096 cells (12 bytes for
    each tile and bucket or macro) suffice too, and a size that suffices is not
    followed by a larger one that does not."""
    import paper_2511_10073_gb300 as pl
    nl = netgen.make_netlist("medium", 1)
    dnl = pl.DeviceNetlist(nl)
    prm = pl.params(nbx=10, nby=10, det_ratio=0.5, wdtype=wd)
    g = pl.pl_build_graph(dnl, prm)
    xy = torch.empty(g.info()["N"] * 2, dtype=torch.float32, device="cuda")
    pl.pl_init_signal(g, 1, None, xy)
    pl.pl_build_hints(g, prm, xy)
    want, out = torch.empty_like(xy), torch.empty_like(xy)
    pl.pl_filter_apply(g, prm, xy, want)
    info = g.info()
    counts = lambda tile: -(-nl.num_cells // tile) * (info["macros"] + 2 * info["bins"]) * 12
    extra = counts(1024) - counts(4096)
    assert counts(1024) * 16 + 4 * extra < info["ws_peak"] - info["ws_static"]  # small tiles are taken
    fits = []
    for less in [4 * extra, 2 * extra, extra - (1 << 16), extra // 2, 1 << 16, 4096, 0]:
        h = _build(pl, dnl, prm, ws=pl.workspace(info["ws_peak"] - less))
        if h is None:
            fits.append(False)
            continue
        try:
            pl.pl_build_hints(h, prm, xy)
        except pl.PlError as e:
            assert e.code == pl.PL_ERR_WORKSPACE
            fits.append(False)
            continue
        pl.pl_filter_apply(h, prm, xy, out)
        assert torch.equal(out, want)
        fits.append(True)
    assert all(fits[2:])
    assert fits == sorted(fits)
