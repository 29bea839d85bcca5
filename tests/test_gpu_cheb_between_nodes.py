"""Nets with one unit that turns between two nodes of the embedding series: its
coefficients look resolved, and the net itself has to be evaluated.  Parity with
the oracle, 1e-10 of the largest entry as in the other parity tests.

The first node is at s = S / 3734 = 3.6e-4; tanh(1e5 s) is 1 at every node and turns
below it, where the rows near the cut-off are.  At s = 0.7103, half way between
two nodes in angle, two units of slope 4,000 make a bump 0.002 wide, e^-170 at the
nodes beside it; O-H pairs are stretched onto it, and where the next layer has no
skip connection (the second shape) the net is smooth at every node."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.mark.parametrize("emb", [(16, 32, 64), (12, 20)])
@pytest.mark.parametrize("where", ["end", "between"])
def test_units_between_the_nodes(oracle, synth, emb, where):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2004_11658_gb300 import dp
    c, t, b = synth.water_box(5, 5 * 49.7 / 16, seed=3)
    desc = dict(synth.WATER_STUDENT, emb=emb, fit=(48, 48), rcut_smth=2.0)   # s = 1/r up to 2 A
    P = synth.model_params(desc, 0, fit_in_gain=30.0, out_scale=1.0)
    if where == "between":
        o = c[0::3].copy()
        for h in (1, 2):
            d = c[h::3] - o
            d -= np.asarray(b) * np.rint(d / np.asarray(b))
            r = 1.0 / np.linspace(0.7090, 0.7116, len(o))
            c[h::3] = np.mod(o + d * (r / np.linalg.norm(d, axis=1))[:, None], b)
    k = 0
    for name, shape in synth.layer_shapes(desc):
        n = int(np.prod(shape))
        v = P[k:k + n].reshape(shape)
        if name.startswith("emb"):
            if where == "end":
                if name.endswith(".W0"):
                    v[3] = 1e5
                elif name.endswith(".b0"):
                    v[3] = 0.0
            else:
                if name.endswith(".W0"):
                    v[3:5] = 4000.0
                elif name.endswith(".b0"):
                    v[3:5] = -4000.0 * 0.7093, -4000.0 * 0.7113
                elif name.endswith(".W1"):
                    v[4] = -v[3]
        k += n
    want = oracle.evaluate(desc, P, c, t, b)
    ctx = dp.Context(dp.Model(desc, P), len(c))
    x = torch.tensor(c, dtype=torch.float64, device="cuda")
    ty = torch.tensor(t, dtype=torch.int32, device="cuda")
    dp.dp_build_nlist(ctx, x, ty, b, 0.0)
    got = dp.dp_eval(ctx, x, ty, b, want_atom_energy=True)
    for q in ("atom_energy", "force", "virial"):
        g, w = got[q].cpu().numpy().ravel(), np.asarray(want[q]).ravel()
        assert np.abs(g - w).max() <= TOL * np.abs(w).max(), (q, np.abs(g - w).max() / np.abs(w).max())
