"""FP32 hint weights bit-exact against the oracle where their double-float form
decides least: a region far from the origin, windows of one to seven columns, bin
counts that are no power of two, and cells far outside the region (long
exponentials, which take the FP64 value)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [(0.0, 0.0), (1e4, -3e5)])
@pytest.mark.parametrize("kw", [dict(nbx=7, nby=9), dict(nbx=33, nby=31), dict(nbx=61, nby=20, det_ratio=0.12)])
def test_fp32_weights_bitexact(kw, shift):
    from paper_2511_10073_gb300 import netgen
    import paper_2511_10073_gb300 as pl
    from test_gpu_parity import Side, _compare_hints, to_np
    nl = netgen.make_netlist("tiny", 5).translated(*shift)
    s = Side(nl, wdtype=1, **kw)
    _, xy = s.oracle_signal(3)
    a = xy.view(-1, 2)
    rng = np.random.default_rng(2)
    far = torch.tensor(rng.choice(2000, 300, replace=False), device="cuda")  # std cells come first
    a[far] += torch.tensor(rng.normal(0.0, 8.0 * s.die, (300, 2)).astype(np.float32), device="cuda")
    pl.pl_build_hints(s.g, s.prm, xy)
    b = to_np(xy)
    s.o.build_hints(b[:, 0], b[:, 1])
    _compare_hints(s, s.g.export(), s.o.merged())
