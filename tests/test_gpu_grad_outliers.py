"""Weight gradients of the fitting net on columns with outliers, and on types
whose atoms end at, before and after the 16-atom chunks and 256-atom segments of
the contraction, against the oracle.

Outliers: a pair at 1e-3 and 1e-4 A gives its two atoms descriptors up to 1e5
times the others', and one atom far from it a lambda 1e4 and 1e6 times the
others', so that the two factors of X^T Z have their outliers at different
atoms and the products of all the other atoms with them matter.  Tolerance: both
sides sum 648 atoms in float64, 648 2^-53 = 7.2e-14 each of a block's largest entry.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 2 * 648 * 2.0 ** -53


def check(oracle, synth, desc, P, c, t, b, lam):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2004_11658_gb300 import dp
    ref = oracle.param_grad(desc, P, c, t, b, 0.37, lam)
    ctx = dp.Context(dp.Model(desc, P), len(c))
    x = torch.tensor(c, dtype=torch.float64, device="cuda")
    ty = torch.tensor(t, device="cuda")
    lm = torch.tensor(lam, device="cuda")
    dp.dp_build_nlist(ctx, x, ty, b, 0.0)
    g = dp.dp_param_grad(ctx, x, ty, b, 0.37, lm)
    assert torch.equal(g, dp.dp_param_grad(ctx, x, ty, b, 0.37, lm))
    g, k = g.cpu().numpy(), 0
    for name, shape in synth.layer_shapes(desc):
        n = int(np.prod(shape))
        if name.startswith("fit"):
            r = ref[k:k + n]
            assert np.abs(g[k:k + n] - r).max() <= TOL * np.abs(r).max(), name
        k += n


def system(synth, ntypes, fit):
    c, t, b = synth.water_box(6, 6 * 49.7 / 16, seed=3)
    desc = dict(synth.WATER_MODEL, ntypes=ntypes, sel=(200,) * ntypes, emb=(8, 16, 32), m2=8, fit=fit)
    return desc, synth.model_params(desc, 0, fit_in_gain=30.0, out_scale=1.0), np.array(c), np.array(t), b


@pytest.mark.parametrize("r,scale", [(1e-3, 1e4), (1e-4, 1e6)])
@pytest.mark.parametrize("fit", [(64, 64), (33,)])
def test_outliers_at_different_atoms(oracle, synth, r, scale, fit):
    desc, P, c, t, b = system(synth, 2, fit)
    lam = np.random.default_rng(7).standard_normal((len(c), 3))
    c[34] = np.mod(c[30] + r * np.array([0.6, 0.0, 0.8]), b)
    d = c - c[30]
    d -= np.asarray(b) * np.rint(d / np.asarray(b))
    lam[np.argmax((d * d).sum(1))] *= scale
    check(oracle, synth, desc, P, c, t, b, lam)


@pytest.mark.parametrize("n0", [1, 15, 16, 17, 128, 255, 256, 257, 391])
def test_ends_of_segments(oracle, synth, n0):
    desc, P, c, _, b = system(synth, 2, (17, 17))
    t = (np.random.default_rng(n0).permutation(len(c)) >= n0).astype(np.int32)
    lam = np.random.default_rng(7).standard_normal((len(c), 3))
    check(oracle, synth, desc, P, c, t, b, lam)
