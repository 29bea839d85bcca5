"""Parameter gradient of a frame in which a type of the model has no atom: the
absent type's parameters have gradient exactly 0 and the others the oracle's.

The frame is worked on in a context whose scratch holds the exponents that a
frame with NaN adjoints has left there, and in fresh contexts."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10   # of the largest entry, the bar of the other gradient tests


def blocks(synth, desc, g):
    out, k = {}, 0
    for name, shape in synth.layer_shapes(desc):
        n = int(np.prod(shape))
        out[name] = g[k:k + n]
        k += n
    return out


@pytest.mark.parametrize("ntypes,absent", [(2, (0,)), (2, (1,)), (3, (1,)), (3, (0, 2))])
@pytest.mark.parametrize("fit", [(64, 64), (240,)])
def test_absent_type_has_no_gradient(oracle, synth, ntypes, absent, fit):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2004_11658_gb300 import dp
    c, t, b = synth.water_box(6, 6 * 49.7 / 16, seed=3)
    desc = dict(synth.WATER_MODEL, ntypes=ntypes, sel=(200,) * ntypes, emb=(8, 16, 32), m2=8, fit=fit)
    P = synth.model_params(desc, 0, fit_in_gain=30.0, out_scale=1.0)
    rng = np.random.default_rng(3)
    lam = rng.standard_normal((len(c), 3))
    present = [a for a in range(ntypes) if a not in absent]
    t_all = np.arange(len(c), dtype=np.int32) % ntypes
    t_some = np.array(present, dtype=np.int32)[np.arange(len(c)) % len(present)]
    ref = blocks(synth, desc, oracle.param_grad(desc, P, c, t_some, b, 0.37, lam))
    model = dp.Model(desc, P)
    x = torch.tensor(c, dtype=torch.float64, device="cuda")

    def grad(ctx, types, lm):
        ty = torch.tensor(types, device="cuda")
        dp.dp_build_nlist(ctx, x, ty, b, 0.0)
        return dp.dp_param_grad(ctx, x, ty, b, 0.37, torch.tensor(lm, device="cuda"))

    used = dp.Context(model, len(c))
    spoilt = blocks(synth, desc, grad(used, t_all, lam * np.nan).cpu().numpy())
    assert all(np.isnan(spoilt[f"fit{a}.W1"]).any() for a in range(ntypes))
    for ctx in (used, dp.Context(model, len(c))):
        got = blocks(synth, desc, grad(ctx, t_some, lam).cpu().numpy())
        for name, g in got.items():
            a = int(name[3])
            if a in absent:
                assert np.array_equal(g, np.zeros_like(g)), name
            else:
                assert np.abs(g - ref[name]).max() <= TOL * np.abs(ref[name]).max() if np.any(ref[name]) \
                    else not np.any(g), name
