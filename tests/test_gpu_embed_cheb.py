"""The FP64 embedding kernels with the nets as Chebyshev series in s: net
shapes, row counts around the CTA's 128 rows, rows beyond the series' domain
(r < 0.75 A), and nets the series does not resolve (which take the kernels that
evaluate the net), against the oracle.

Tolerance: the FP64 bar of the other parity tests, 1e-10 of the largest entry.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.fixture(scope="module")
def dp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2004_11658_gb300 import dp as _dp
    _dp.lib()
    return _dp


def rel(a, b):
    a, b = np.asarray(a, dtype=np.float64), np.asarray(b, dtype=np.float64)
    return float(np.abs(a - b).max() / max(np.abs(b).max(), 1e-300))


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
    return ctx


@pytest.mark.parametrize("emb,m2,sel", [((24,), 24, (60, 120)), ((20, 20), 3, (46, 92)), ((25, 50, 100), 16, (46, 92)),
                                        ((32, 64, 128), 128, (46, 92)), ((8, 16, 16, 33), 5, (300, 700))])
def test_net_shapes(dp, oracle, synth, emb, m2, sel):
    c, t, b = synth.water_box(5, 5 * 49.7 / 16, seed=3)
    desc = dict(synth.WATER_MODEL, emb=emb, m2=m2, sel=sel, fit=(48, 48))
    check(dp, oracle, desc, synth.model_params(desc, 4, fit_in_gain=1.0, out_scale=1.0), c, t, b)


@pytest.mark.parametrize("rcut", [5.2, 7.16, 8.0])
def test_row_counts(dp, oracle, synth, rcut):
    """~50, ~128 (the CTA's rows, shells on both sides) and ~180 rows, three types."""
    c, _, b = synth.copper_fcc(5, seed=2)
    t = np.random.default_rng(5).integers(0, 3, len(c)).astype(np.int32)
    desc = dict(synth.CU_MODEL, ntypes=3, sel=(120, 120, 120), rcut=rcut, emb=(8, 16, 32), fit=(32, 32))
    check(dp, oracle, desc, synth.model_params(desc, 1, fit_in_gain=1.0, out_scale=1.0), c, t, b)


def test_rows_beyond_the_series(dp, oracle, synth):
    """Pairs at 0.05 to 0.8 A, on both sides of s = 4/3 (r = 0.75 A)."""
    c, t, b = synth.water_box(5, 5 * 49.7 / 16, seed=3)
    for k, r in enumerate((0.05, 0.3, 0.5, 0.7499999, 0.7500001, 0.8)):
        c[30 * k + 4] = np.mod(c[30 * k] + r * np.array([0.6, 0.0, 0.8]), b[0])
    desc = synth.WATER_MODEL
    check(dp, oracle, desc, synth.model_params(desc, 0), c, t, b)


@pytest.mark.parametrize("emb", [(25, 50, 100), (20, 40, 80)])
def test_steep_nets_take_the_net_kernels(dp, oracle, synth, emb):
    """A first layer 100 times steeper needs more terms than are kept."""
    c, t, b = synth.water_box(5, 5 * 49.7 / 16, seed=3)
    desc = dict(synth.WATER_MODEL, emb=emb)
    P = synth.model_params(desc, 0)
    off = 0
    for name, shape in synth.layer_shapes(desc):
        n = int(np.prod(shape))
        if name.endswith(".W0"):
            P[off:off + n] *= 100.0
        off += n
    check(dp, oracle, desc, P, c, t, b)


def test_new_parameters_make_new_series(dp, oracle, synth):
    c, t, b = synth.water_box(5, 5 * 49.7 / 16, seed=3)
    desc = synth.WATER_STUDENT
    P0, P1 = synth.model_params(desc, 0), synth.model_params(desc, 1)
    model = dp.Model(desc, P0)
    ctx = dp.Context(model, len(c))
    x = torch.tensor(c, device="cuda")
    ty = torch.tensor(t, device="cuda")
    for P in (P0, P1, P0):
        model.set_params(P)
        dp.dp_build_nlist(ctx, x, ty, b, 0.0)
        f = dp.dp_eval(ctx, x, ty, b)["force"]
        assert rel(f.cpu(), oracle.evaluate(desc, P, c, t, b)["force"]) < TOL


def check_grad(dp, oracle, desc, P, c, t, box):
    rng = np.random.default_rng(8)
    lam = rng.standard_normal((len(c), 3))
    ref = oracle.param_grad(desc, P, c, t, box, 0.37, lam)
    ctx = dp.Context(dp.Model(desc, P), len(c))
    x = torch.tensor(c, dtype=torch.float64, device="cuda")
    ty = torch.tensor(t, dtype=torch.int32, device="cuda")
    dp.dp_build_nlist(ctx, x, ty, box, 0.0)
    g = dp.dp_param_grad(ctx, x, ty, box, 0.37, torch.tensor(lam, device="cuda"))
    # embedding and fitting parameters apart: each block has its own scale
    ne = sum(int(np.prod(s)) for n, s in synth_shapes(desc) if n.startswith("emb"))
    assert rel(g[:ne].cpu(), ref[:ne]) < TOL
    assert rel(g[ne:].cpu(), ref[ne:]) < TOL
    g2 = dp.dp_param_grad(ctx, x, ty, box, 0.37, torch.tensor(lam, device="cuda"))
    assert torch.equal(g, g2)


def synth_shapes(desc):
    from paper_2004_11658_gb300 import synth
    return synth.layer_shapes(desc)


@pytest.mark.parametrize("emb,m2,fit", [((24,), 24, (48, 48)), ((20, 20), 3, (17, 17)), ((8, 16, 16, 33), 5, (33,)),
                                        ((25, 50, 100), 16, (64, 64, 64)), ((32, 64, 128), 16, (240, 240))])
def test_gradient_shapes(dp, oracle, synth, emb, m2, fit):
    c, t, b = synth.water_box(5, 5 * 49.7 / 16, seed=3)
    desc = dict(synth.WATER_MODEL, emb=emb, m2=m2, fit=fit)
    check_grad(dp, oracle, desc, synth.model_params(desc, 4, fit_in_gain=30.0, out_scale=1.0), c, t, b)


def test_gradient_three_types_many_rows(dp, oracle, synth):
    c, _, b = synth.copper_fcc(5, seed=2)
    t = np.random.default_rng(5).integers(0, 3, len(c)).astype(np.int32)
    desc = dict(synth.CU_MODEL, ntypes=3, sel=(120, 120, 120), emb=(8, 16, 32), fit=(32, 32))
    check_grad(dp, oracle, desc, synth.model_params(desc, 1, fit_in_gain=30.0, out_scale=1.0), c, t, b)


@pytest.mark.parametrize("case", ["rows beyond the series", "steep nets"])
def test_gradient_through_the_nets(dp, oracle, synth, case):
    """Frames and nets the series does not cover take the kernels that work
    through the net."""
    c, t, b = synth.water_box(5, 5 * 49.7 / 16, seed=3)
    desc = synth.WATER_STUDENT
    P = synth.model_params(desc, 0)
    if case == "steep nets":
        off = 0
        for name, shape in synth.layer_shapes(desc):
            n = int(np.prod(shape))
            if name.endswith(".W0"):
                P[off:off + n] *= 100.0
            off += n
    else:
        c[34] = np.mod(c[30] + 0.4 * np.array([0.6, 0.0, 0.8]), b[0])
    check_grad(dp, oracle, desc, P, c, t, b)
