"""Weight gradients of the fitting net whose contraction over the atoms several
CTAs share: one and two types, atoms that fill neither a 16-atom chunk nor the
last part.  Against the oracle, with the bar of the other gradient tests (1e-10
of the largest entry), and bit-repeatable."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.mark.parametrize("ntypes,fit", [(1, (48, 48)), (2, (17, 17)), (2, (240,))])
def test_shared_weight_gradients(oracle, synth, ntypes, fit):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2004_11658_gb300 import dp
    c, t, b = synth.water_box(7, 7 * 49.7 / 16, seed=3)
    desc = dict(synth.WATER_STUDENT, fit=fit)
    if ntypes == 1:
        t = np.zeros_like(t)
        desc = dict(desc, ntypes=1, sel=(138,))
    P = synth.model_params(desc, 4, fit_in_gain=30.0, out_scale=1.0)
    lam = np.random.default_rng(8).standard_normal((len(c), 3))
    ref = oracle.param_grad(desc, P, c, t, b, 0.37, lam)
    ctx = dp.Context(dp.Model(desc, P), len(c))
    x = torch.tensor(c, device="cuda")
    ty = torch.tensor(t, device="cuda")
    lm = torch.tensor(lam, device="cuda")
    dp.dp_build_nlist(ctx, x, ty, b, 0.0)
    g = dp.dp_param_grad(ctx, x, ty, b, 0.37, lm)
    ne = sum(int(np.prod(s)) for n, s in synth.layer_shapes(desc) if n.startswith("emb"))
    for got, want in ((g[:ne].cpu().numpy(), ref[:ne]), (g[ne:].cpu().numpy(), ref[ne:])):
        assert np.abs(got - want).max() / np.abs(want).max() < TOL
    assert torch.equal(g, dp.dp_param_grad(ctx, x, ty, b, 0.37, lm))
