"""GPU parity of pl_macro_density where its tiles and lists end: bin grids that
no tile size divides, both tile sizes, more macros over one tile than a list or
a batch holds, macros larger than the grid's tiles or partly outside the region,
and quadrature rules on either side of the half-warp's width.  Tolerances as for
the other parity tests: 1e-11 for the FP64 models, 1e-6 for the two whose point
values are FP32 (about 1e-7 relative each)."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = {
    # bins, macros, side range, region origin
    "one_bin": ((1, 1), 7, (1.0, 30.0), 0.0),
    "ragged_small": ((33, 17), 90, (2.0, 25.0), -40.0),
    "large_tiles": ((325, 259), 60, (1.0, 40.0), 0.0),
    "long_list": ((5, 3), 4500, (0.2, 3.0), 1000.0),
    "wide_macros": ((70, 41), 70, (60.0, 150.0), 0.0),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("model,rule", [(0, {}), (1, {}), (2, {}), (3, {}), (3, dict(panels=9, nodes=3)),
                                        (2, dict(panels=1, nodes=5))])
def test_tiles_match_oracle(name, model, rule):
    import paper_2511_10073_gb300 as pl
    (nbx, nby), nm, (lo, hi), org = CASES[name]
    rng = np.random.default_rng(nm + model)
    side = 200.0
    geo = [org + rng.uniform(-5.0, side + 5.0, nm), org + rng.uniform(-5.0, side + 5.0, nm),
           rng.uniform(lo, hi, nm), rng.uniform(lo, hi, nm)]
    geo[2][nm // 2] = 0.0  # a macro without width charges nothing
    geo = [a.astype(np.float32) for a in geo]
    region = (org, org, org + side, org + side)
    out = torch.full((nbx * nby,), -1.0, dtype=torch.float64, device="cuda")
    pl.pl_macro_density(pl.rho_params(model=model, **rule), 120,
                        *[torch.tensor(a, device="cuda") for a in geo], region, nbx, nby, out)
    keep = (geo[2] > 0) & (geo[3] > 0)
    ref = oracle.macro_density(oracle.rho_params(model=model, **rule), 120,
                               *(a[keep].astype(np.float64) for a in geo), region, nbx, nby)
    got = out.cpu().numpy()
    tol = 1e-11 if model in (0, 1) else 1e-6
    assert np.allclose(got, ref, rtol=tol, atol=tol * side * side / (nbx * nby)), np.abs(got - ref).max()
