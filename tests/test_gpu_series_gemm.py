"""The products with the embedding series on the tensor cores, for boxes where
they run apart (2^22 atoms x terms x features): term counts and widths off the
16- and 32-column chunks, one to three types, D rows as short as the four
components, rows beyond the series.  Against the oracle, with the FP64
bar of the other parity tests (1e-10 of the largest entry), and bit-repeatable."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10


def rel(a, b):
    a, b = np.asarray(a, dtype=np.float64), np.asarray(b, dtype=np.float64)
    return float(np.abs(a - b).max() / max(np.abs(b).max(), 1e-300))


@pytest.fixture(scope="module")
def dp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2004_11658_gb300 import dp as _dp
    _dp.lib()
    return _dp


def check(dp, oracle, desc, P, c, t, box):
    o = oracle.evaluate(desc, P, c, t, box)
    ctx = dp.Context(dp.Model(desc, P), len(c))
    x = torch.tensor(c, dtype=torch.float64, device="cuda")
    ty = torch.tensor(t, dtype=torch.int32, device="cuda")
    dp.dp_build_nlist(ctx, x, ty, box, 0.0)
    g = dp.dp_eval(ctx, x, ty, box, want_atom_energy=True)
    assert rel(g["atom_energy"].cpu(), o["atom_energy"]) < TOL
    assert rel(g["force"].cpu(), o["force"]) < TOL
    assert rel(g["virial"].cpu().reshape(3, 3), o["virial"]) < TOL
    g2 = dp.dp_eval(ctx, x, ty, box)
    assert torch.equal(g["force"], g2["force"])


@pytest.mark.parametrize("emb,m2,fit", [((25, 50, 100), 16, (48, 48)), ((16, 32, 64), 4, (48, 48)),
                                        ((32, 64, 128), 128, (24,)), ((20, 40, 41), 5, (17, 17))])
def test_water(dp, oracle, synth, emb, m2, fit):
    c, t, b = synth.water_box(10, 10 * 49.7 / 16, seed=3)
    desc = dict(synth.WATER_MODEL, emb=emb, m2=m2, fit=fit)
    check(dp, oracle, desc, synth.model_params(desc, 4, fit_in_gain=1.0, out_scale=1.0), c, t, b)


@pytest.mark.parametrize("ntypes,emb,side", [(1, (10, 20, 40), 11), (3, (32, 64, 128), 6)])
def test_copper(dp, oracle, synth, ntypes, emb, side):
    c, _, b = synth.copper_fcc(side, seed=2)
    t = np.random.default_rng(5).integers(0, ntypes, len(c)).astype(np.int32)
    desc = dict(synth.CU_MODEL, ntypes=ntypes, sel=(400,) if ntypes == 1 else (120, 120, 120), emb=emb, fit=(32, 32))
    check(dp, oracle, desc, synth.model_params(desc, 1, fit_in_gain=1.0, out_scale=1.0), c, t, b)


def test_rows_beyond_the_series(dp, oracle, synth):
    c, t, b = synth.water_box(10, 10 * 49.7 / 16, seed=3)
    for k, r in enumerate((0.05, 0.3, 0.5, 0.7499999, 0.7500001, 0.8)):
        c[30 * k + 4] = np.mod(c[30 * k] + r * np.array([0.6, 0.0, 0.8]), b[0])
    desc = synth.WATER_MODEL
    check(dp, oracle, desc, synth.model_params(desc, 0), c, t, b)
