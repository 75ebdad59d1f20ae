"""Refinement powers as one launch of independent units: designs without macros
(bin rows only, no stored hub entry at all), with one movable cell, and with long
static rows, each round against the oracle's (1e-4 of the die)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _plain(cells, nets, seed):
    from paper_2511_10073_gb300 import netgen
    rng = np.random.default_rng(seed)
    ns = [rng.choice(cells, int(k), replace=False) for k in nets]
    ptr = np.r_[0, np.cumsum([len(n) for n in ns])].astype(np.int64)
    pins = np.concatenate(ns).astype(np.int32)
    one, z = np.ones(cells, np.float32), np.zeros(cells, np.float32)
    d = np.zeros(len(pins), np.float32)
    kind = np.zeros(cells, np.uint8)
    kind[-1] = 2  # one fixed I/O
    return netgen.Netlist(ptr, pins, d, d, one, one, kind, z + 40.0, z + 50.0, (0.0, 0.0, 100.0, 100.0))


CASES = {
    "no_macros": (500, [2] * 400 + [5] * 60, dict(nbx=16, nby=16)),
    "one_cell": (2, [2], dict(nbx=5, nby=3)),
    "long_rows": (600, [16] * 350 + [40] * 3 + [300], dict(nbx=32, nby=32)),
    # more bins than one block numbers the chunks of
    "bins_18000": (300, [3] * 250, dict(nbx=150, nby=120)),
    "many_bins": (900, [3] * 800, dict(nbx=64, nby=64)),
}


@pytest.mark.parametrize("pin", [0, 1])
@pytest.mark.parametrize("wd", [1, 2])
@pytest.mark.parametrize("name", sorted(CASES))
def test_rounds(name, wd, pin):
    import paper_2511_10073_gb300 as pl
    from test_gpu_parity import Side, to_np
    cells, nets, kw = CASES[name]
    s = Side(_plain(cells, nets, 7), wdtype=wd, pin_every_step=pin, ntaps=2, tap_k=(3, 5, 0, 0),
             tap_alpha=(0.4, 0.6, 0, 0), **kw)
    _, xy = s.oracle_signal(4)
    for _ in range(2):
        a = to_np(xy)
        s.o.build_hints(a[:, 0], a[:, 1])
        ref = np.stack(s.o.filter(a[:, 0], a[:, 1]), 1)
        out = torch.empty_like(xy)
        pl.pl_build_hints(s.g, s.prm, xy)
        pl.pl_filter_apply(s.g, s.prm, xy, out)
        assert np.abs(to_np(out) - ref).max() <= 1e-4 * s.die
        xy = torch.tensor(ref.astype(np.float32).reshape(-1), device="cuda")
