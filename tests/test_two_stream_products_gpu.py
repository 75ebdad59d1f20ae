"""Refinement rounds of designs just beyond the size up to which a power is one
launch of independent units: short rows beside hub, bin and macro rows on the
second stream, for both weight types, windows of 9 and 25 slots and re-pinning
after every power, against the oracle (graph as in the other parity tests, the
round within 1e-4 of the die), and against the batch's union form (same bits)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
CELLS, MACROS = 330_003, 12


def _netlist():
    from paper_2511_10073_gb300 import netgen
    rng = np.random.default_rng(8)
    near = np.minimum(np.arange(CELLS) + rng.integers(1, 200, CELLS), CELLS - 1)
    nets = [np.stack([np.arange(CELLS), near], 1)]            # a two-pin net per cell
    nets.append(rng.integers(0, CELLS, (2_000, 5)))
    nets.append(np.stack([rng.integers(0, CELLS, 4 * MACROS), CELLS + np.arange(4 * MACROS) % MACROS], 1))
    flat = [a.reshape(-1) for a in nets] + [rng.choice(CELLS, k, replace=False) for k in (700, 1500)]
    flat += [np.r_[17, rng.choice(CELLS, 15, replace=False)] for _ in range(12)]  # a long static row
    sizes = np.r_[np.full(CELLS, 2), np.full(2_000, 5), np.full(4 * MACROS, 2), 700, 1500, np.full(12, 16)]
    pins = np.concatenate(flat).astype(np.int32)
    C = CELLS + MACROS
    w, z = np.ones(C, np.float32), np.zeros(len(pins), np.float32)
    w[CELLS:] = 60.0
    kind = np.r_[np.zeros(CELLS), np.ones(MACROS)].astype(np.uint8)
    fx, fy = np.zeros(C, np.float32), np.zeros(C, np.float32)
    fx[CELLS:] = 100.0 + 70.0 * (np.arange(MACROS) % 4)
    fy[CELLS:] = 150.0 + 130.0 * (np.arange(MACROS) // 4)
    return netgen.Netlist(np.r_[0, np.cumsum(sizes)].astype(np.int64), pins, z, z, w, w.copy(), kind, fx, fy,
                          (0.0, 0.0, 640.0, 640.0))


@pytest.mark.parametrize("pin", [0, 1])
@pytest.mark.parametrize("nb", [32, 64])
@pytest.mark.parametrize("wd", [1, 2])
def test_rounds(wd, nb, pin):
    import paper_2511_10073_gb300 as pl
    from test_gpu_parity import Side, _compare_hints, to_np
    s = Side(_netlist(), nbx=nb, nby=nb, wdtype=wd, pin_every_step=pin, ntaps=2, tap_k=(1, 3, 0, 0),
             tap_alpha=(0.4, 0.6, 0, 0))
    assert s.N / 128 > 16 * torch.cuda.get_device_properties(0).multi_processor_count
    _, xy = s.oracle_signal(4)
    a = to_np(xy)
    pl.pl_build_hints(s.g, s.prm, xy)
    s.o.build_hints(a[:, 0], a[:, 1])
    _compare_hints(s, s.g.export(), s.o.merged())
    out = torch.empty_like(xy)
    pl.pl_filter_apply(s.g, s.prm, xy, out)
    ref = np.stack(s.o.filter(a[:, 0], a[:, 1]), 1)
    assert np.abs(to_np(out) - ref).max() <= 1e-4 * s.die


@pytest.mark.parametrize("nb", [32, 64])
@pytest.mark.parametrize("wd", [1, 2])
def test_same_bits_as_the_union_form(wd, nb):
    import paper_2511_10073_gb300 as pl
    nl = _netlist()
    prm = pl.params(nbx=nb, nby=nb, wdtype=wd, ntaps=2, tap_k=(1, 3, 0, 0), tap_alpha=(0.4, 0.6, 0, 0))
    g = pl.pl_build_graph(pl.DeviceNetlist(nl), prm)
    want = torch.empty(nl.num_cells * 2, dtype=torch.float32, device="cuda")
    got = torch.empty_like(want)
    pl.pl_filter_init(g, prm, 5, None, want)
    torch.cuda.synchronize()
    pl.pl_filter_init_batch([g], prm, [5], [got], [torch.cuda.Stream()], pl.batch_opts(union_products=1),
                            pl.batch_workspace(1, prm))
    torch.cuda.synchronize()
    assert torch.equal(got, want)
