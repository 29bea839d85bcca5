"""The FP64 fitting net's GEMMs on the tensor cores over the shapes where their
tiling can go wrong: contraction lengths of one chunk, around a segment of the
group accumulators (400 columns) and of 41 segments, output widths off the
32-column units, rows that do not start on 16 bytes, skip kinds, one layer, and
types of 125 and 250 atoms (tiles of 128).  Against the oracle, with the FP64
bar of the other parity tests (1e-10 of the largest entry)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10


def rel(a, b):
    a, b = np.asarray(a, dtype=np.float64), np.asarray(b, dtype=np.float64)
    return float(np.abs(a - b).max() / max(np.abs(b).max(), 1e-300))


@pytest.mark.parametrize("M,m2,fit", [(4, 1, (1,)), (16, 1, (48, 48)), (33, 7, (17, 17, 34)), (25, 16, (31, 62)),
                                      (40, 10, (240, 240)), (51, 8, (33, 33, 33)), (100, 16, (240, 240, 240)),
                                      (128, 128, (8,)), (128, 16, (256, 256))])
def test_fit_shapes(oracle, synth, M, m2, fit):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2004_11658_gb300 import dp
    c, t, b = synth.water_box(5, 5 * 49.7 / 16, seed=7)
    desc = dict(synth.WATER_MODEL, emb=(M,), m2=m2, fit=fit)
    P = synth.model_params(desc, 2, fit_in_gain=30.0, out_scale=1.0)
    o = oracle.evaluate(desc, P, c, t, b)
    ctx = dp.Context(dp.Model(desc, P), len(c))
    x = torch.tensor(c, device="cuda")
    ty = torch.tensor(t, device="cuda")
    dp.dp_build_nlist(ctx, x, ty, b, 0.0)
    g = dp.dp_eval(ctx, x, ty, b, want_atom_energy=True)
    assert rel(g["atom_energy"].cpu(), o["atom_energy"]) < TOL
    assert rel(g["force"].cpu(), o["force"]) < TOL
    assert rel(g["virial"].cpu().reshape(3, 3), o["virial"]) < TOL
    g2 = dp.dp_eval(ctx, x, ty, b)
    assert torch.equal(g["force"], g2["force"])
