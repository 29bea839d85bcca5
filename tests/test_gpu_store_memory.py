"""The FP64 store of G and dG/ds takes device memory only when an evaluation's nets
need it (they are not resolved as series) or when it is switched on."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NMAX = 20000
STORE = NMAX * 138 * 2 * 100 * 8          # 4.4 GB of rows for the water model


def used(dp, before):
    torch.cuda.synchronize()
    return before - torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("steep", [False, True])
def test_memory_of_the_store(oracle, synth, steep):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2004_11658_gb300 import dp
    c, t, b = synth.water_box(5, 5 * 49.7 / 16, seed=3)
    desc = synth.WATER_MODEL
    P = synth.model_params(desc, 0)
    off = 0
    for name, shape in synth.layer_shapes(desc):
        n = int(np.prod(shape))
        if steep and name.endswith(".W0"):
            P[off:off + n] *= 100.0
        off += n
    x = torch.tensor(c, dtype=torch.float64, device="cuda")
    ty = torch.tensor(t, dtype=torch.int32, device="cuda")
    model = dp.Model(desc, P)
    dp.Context(model, 64).close()         # what the process takes once
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    ctx = dp.Context(model, NMAX)
    assert ctx.embed_store
    assert used(dp, before) < STORE // 2

    def force():
        dp.dp_build_nlist(ctx, x, ty, b, 0.0)
        return dp.dp_eval(ctx, x, ty, b)["force"].cpu().numpy()

    kept = force()
    assert ctx.embed_store
    assert (used(dp, before) >= STORE) == steep
    ref = oracle.evaluate(desc, P, c, t, b)["force"]
    assert np.abs(kept - ref).max() < 1e-10 * np.abs(ref).max()
    ctx.set_embed_store(True)
    assert ctx.embed_store and used(dp, before) >= STORE
    np.testing.assert_array_equal(force(), kept)
    ctx.set_embed_store(False)
    assert not ctx.embed_store and used(dp, before) < STORE
    assert np.abs(force() - kept).max() < 1e-13 * np.abs(kept).max()
    assert used(dp, before) < STORE and not ctx.embed_store
    ctx.close()
