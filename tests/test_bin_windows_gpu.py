"""Hint build and refinement filter for window sizes with every remainder of the
bin rows' slot groups (1, 3, 21, 27, 63 and 65 slots), on bins that hold a few
cells and on bins that hold more than a chunk: the graph against the oracle's as
in the other parity tests, one filter step within 1e-4 of the die."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wd", [1, 2])
@pytest.mark.parametrize("nbx,nby", [(3, 2), (6, 2), (14, 6), (18, 6), (18, 14), (26, 10)])
def test_windows(nbx, nby, wd):
    from paper_2511_10073_gb300 import netgen
    import paper_2511_10073_gb300 as pl
    from test_gpu_parity import Side, _compare_hints, to_np
    s = Side(netgen.make_netlist("tiny", 9), nbx=nbx, nby=nby, det_ratio=0.5, wdtype=wd)
    _, xy = s.oracle_signal(2)
    pl.pl_build_hints(s.g, s.prm, xy)
    a = to_np(xy)
    s.o.build_hints(a[:, 0], a[:, 1])
    _compare_hints(s, s.g.export(), s.o.merged())
    out = torch.empty_like(xy)
    pl.pl_filter_apply(s.g, s.prm, xy, out)
    got = to_np(out)
    ref = np.stack(s.o.filter(a[:, 0], a[:, 1]), 1)
    assert np.abs(got - ref).max() <= 1e-4 * s.die
