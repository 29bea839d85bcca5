"""Mixed fitting kernel on tiles whose last warp holds fewer than 32 atoms of the
type (125, 250, 343 and 686 of them): its lanes without an atom take other branches
around the warp-wide loads of the accumulators.  Against the FP64 oracle with the
mixed mode's bar (relative force RMSE 1e-2 for the water model), and bit-repeatable."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side", [5, 7])
def test_partial_warps(oracle, synth, side):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2004_11658_gb300 import dp
    c, t, b = synth.water_box(side, side * 49.7 / 16, seed=3)
    desc = synth.WATER_MODEL
    P = synth.model_params(desc, 0)
    ref = oracle.evaluate(desc, P, c, t, b)["force"]
    ctx = dp.Context(dp.Model(desc, P), len(c), precision=dp.DP_PREC_MIXED)
    x = torch.tensor(c, dtype=torch.float64, device="cuda")
    ty = torch.tensor(t, dtype=torch.int32, device="cuda")
    dp.dp_build_nlist(ctx, x, ty, b, 0.0)
    runs = [dp.dp_eval(ctx, x, ty, b, want_atom_energy=True) for _ in range(3)]
    f = runs[0]["force"].cpu().numpy()
    assert np.sqrt(((f - ref) ** 2).mean() / (ref ** 2).mean()) < 1e-2
    for g in runs[1:]:
        assert torch.equal(g["force"], runs[0]["force"])
        assert torch.equal(g["atom_energy"], runs[0]["atom_energy"])
