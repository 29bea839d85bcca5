"""The same model and box in A and in nm: the embedding nets' series covers the
same part of the rows (no cut-off makes every row a near one), and energies,
forces, virial and gradients match the oracle in both.

Tolerance: the FP64 bar of the other parity tests, 1e-10 of the largest entry."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TOL = 1e-10


def test_domain_scales_with_the_cutoff(tmp_path):
    src, so = tmp_path / "t.cpp", tmp_path / "t.so"
    src.write_text('#include "cheb_domain.h"\nextern "C" double t_dom(double r) { return dp_cheb_domain(r); }\n')
    subprocess.run(["g++", "-O2", "-fPIC", "-shared", "-I", os.path.join(ROOT, "paper_2004_11658_gb300", "csrc"),
                    str(src), "-o", str(so)], check=True)
    f = ctypes.CDLL(str(so)).t_dom
    f.restype, f.argtypes = ctypes.c_double, [ctypes.c_double]
    for rcut in (3.0, 6.0, 8.0, 15.0):      # A, Bohr: r = 0.75
        assert f(rcut) == 4.0 / 3.0
    for rcut in (6.0, 8.0):                 # nm, m: an eighth of the cut-off, 0.75 A for 6 A
        for unit in (0.1, 1e-10):
            assert 1.0 / f(rcut * unit) == pytest.approx(rcut * unit / 8, rel=1e-14)


@pytest.mark.gpu
@pytest.mark.parametrize("unit", [1.0, 0.1])
def test_parity_in_other_units(oracle, synth, unit):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2004_11658_gb300 import dp
    c, t, b = synth.water_box(5, 5 * 49.7 / 16, seed=3)
    c[34] = np.mod(c[30] + 0.5 * np.array([0.6, 0.0, 0.8]), b[0])   # one pair nearer than rcut / 8
    c, b = c * unit, np.asarray(b) * unit
    desc = dict(synth.WATER_STUDENT, rcut=6.0 * unit, rcut_smth=0.5 * unit)
    P = synth.model_params(desc, 0)
    off = 0
    for name, shape in synth.layer_shapes(desc):   # the same nets of s
        n = int(np.prod(shape))
        if name.endswith(".W0"):
            P[off:off + n] *= unit
        off += n
    o = oracle.evaluate(desc, P, c, t, b)
    lam = np.random.default_rng(8).standard_normal((len(c), 3))
    ref = oracle.param_grad(desc, P, c, t, b, 0.37, lam)
    ctx = dp.Context(dp.Model(desc, P), len(c))
    x = torch.tensor(c, dtype=torch.float64, device="cuda")
    ty = torch.tensor(t, dtype=torch.int32, device="cuda")
    dp.dp_build_nlist(ctx, x, ty, b, 0.0)
    g = dp.dp_eval(ctx, x, ty, b, want_atom_energy=True)
    for k in ("atom_energy", "force", "virial"):
        got, want = g[k].cpu().numpy().ravel(), np.asarray(o[k]).ravel()
        assert np.abs(got - want).max() <= TOL * np.abs(want).max(), k
    gp = dp.dp_param_grad(ctx, x, ty, b, 0.37, torch.tensor(lam, device="cuda")).cpu().numpy()
    ne = sum(int(np.prod(s)) for n, s in synth.layer_shapes(desc) if n.startswith("emb"))
    for got, want in ((gp[:ne], ref[:ne]), (gp[ne:], ref[ne:])):
        assert np.abs(got - want).max() <= TOL * np.abs(want).max()
