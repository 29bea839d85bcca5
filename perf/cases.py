"""The work that is timed: Deep Potential evaluation, MD, training and
neighbour lists as a user's program calls them, over the sizes of this
repository's workloads (192 to ~140,000 water atoms, copper crystals).

A case is a dict of plain values:
  kind   "eval"  neighbour list + energy, forces, virial of new coordinates
         "local" the same for one slab of a decomposed box (ghost atoms)
         "md"    a velocity-Verlet run of `steps` steps from given coordinates
         "fast"  MD on the trained student with the FP64 model as its judge
         "train" one step of training on `frames` frames (energy + forces)
         "nlist" candidates + formatted list alone
  model  "water" (25-50-100, sel 46/92), "student" (16-32-64), "copper"
         (32-64-128, sel 512)
  prec   "fp64", "mixed" (BF16 GEMMs) or "split" (split-BF16 GEMMs)
  side   molecules (water) or unit cells (copper) along an edge of the box
  dt, skin  step (fs) and list buffer (A) where they are not the usual ones
"""
import math
import os

import numpy as np
import torch

from paper_2004_11658_gb300 import domain, dp, student, synth

MODELS = {"water": synth.WATER_MODEL, "student": synth.WATER_STUDENT, "copper": synth.CU_MODEL}
PRECS = {"fp64": dp.DP_PREC_FP64, "mixed": dp.DP_PREC_MIXED, "split": dp.DP_PREC_MIXED_SPLIT}
WATER_EDGE = 49.7 / 16   # edge of one molecule's share of a water box at 1 g/cm^3
SLABS = 2                # sub-regions of a "local" case; its slab is the first
PE, PF = 1.0, 100.0      # training loss: pe ((E - E_ref)/N)^2 + pf |F - F_ref|^2 / (3 N)
LR = 1e-6                # of the plain gradient step a "train" pass ends with


def listed():
    return [
        # one evaluation of a 64-molecule box: fitting a model against reference
        # data, geometry scans; every launch and every tail counts
        dict(name="eval_water192_fp64", kind="eval", model="water", prec="fp64", side=4),
        # a short run of a small, odd-sized box (343 molecules): replicas, ensembles
        dict(name="md_water1029_fp64", kind="md", model="water", prec="fp64", side=7, steps=10),
        # the production size of the water model in the reference precision
        dict(name="md_water12288_fp64", kind="md", model="water", prec="fp64", side=16, steps=5),
        # a large box (139,968 atoms), memory- and throughput-bound
        dict(name="md_water139968_fp64", kind="md", model="water", prec="fp64", side=36, steps=1),
        # a crystal with the wide single-type model, long neighbour lists
        dict(name="md_copper32000_fp64", kind="md", model="copper", prec="fp64", side=20, steps=1),
        # one rank's share of a decomposed box (centres and ghosts)
        dict(name="local_water52728_fp64", kind="local", model="water", prec="fp64", side=26),
        # mixed-precision production MD
        dict(name="md_water98304_mixed", kind="md", model="water", prec="mixed", side=32, steps=4),
        # the mixed mode that a nearly symmetric crystal needs
        dict(name="md_copper13500_split", kind="md", model="copper", prec="split", side=15, steps=4),
        # the student as fast path, checked by the full model at the run's end
        dict(name="fast_water12288", kind="fast", model="student", prec="mixed", side=16, steps=10),
        # one training step of the student at the size of its training frames
        dict(name="train_student12288", kind="train", model="student", prec="fp64", side=16, frames=1),
        # training of the full-width model on small frames, a batch of 4
        dict(name="train_water648", kind="train", model="water", prec="fp64", side=6, frames=4),
        # neighbour lists alone, for analysis or another engine
        dict(name="nlist_water98304", kind="nlist", model="water", prec="fp64", side=32),
    ]


def _logint(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["eval", "eval", "md", "md", "md", "local", "fast", "train", "nlist"])
    if kind == "fast":
        return dict(kind=kind, model="student", prec="mixed", side=_logint(rng, 6, 20), steps=10,
                    dt=round(rng.uniform(0.25, 0.75), 2))
    if kind == "train":
        return dict(kind=kind, model=rng.choice(["student", "water"]), prec="fp64", side=_logint(rng, 4, 10),
                    frames=rng.randint(1, 3))
    if kind == "nlist":
        return dict(kind=kind, model="water", prec="fp64", side=_logint(rng, 6, 32), skin=round(rng.uniform(0.0, 2.0), 2))
    if kind == "local":
        return dict(kind=kind, model=rng.choice(["water", "student"]), prec=rng.choice(["fp64", "fp64", "mixed", "split"]),
                    side=_logint(rng, 14, 28))
    model = rng.choice(["water", "water", "student", "copper"])
    prec = rng.choice(["fp64", "fp64", "mixed", "split"])
    if model == "copper" and prec == "mixed":
        prec = "fp64"   # plain BF16 is not the mode for a crystal
    side = _logint(rng, 6, 16) if model == "copper" else _logint(rng, 6 if kind == "md" else 4, 30)
    if kind == "eval":
        return dict(kind=kind, model=model, prec=prec, side=side)
    return dict(kind=kind, model=model, prec=prec, side=side, steps=rng.randint(1, 4), dt=round(rng.uniform(0.25, 1.0), 2))


def _system(case, seed):
    """(coords [N, 3], types [N], box [3], masses per type), numpy."""
    if case["model"] == "copper":
        c, t, b = synth.copper_fcc(case["side"], seed=seed)
        return c, t, b, (synth.MASS["Cu"],)
    c, t, b = synth.water_box(case["side"], case["side"] * WATER_EDGE, seed=seed)
    return c, t, b, (synth.MASS["O"], synth.MASS["H"])


def _student_params():
    path = os.path.join(os.path.dirname(synth.__file__), "data", "student_water12288.npy")
    return np.load(path).astype(np.float64)


def _dt(case):
    return case.get("dt", 1.0 if case["model"] == "copper" else 0.5)


def _skin(desc, box):
    return max(0.0, min(2.0, 0.999 * (0.5 * float(min(box)) - desc["rcut"])))


def _out_slices(desc):
    """Flat-vector slices of every type's output weights and bias."""
    return [slice(student.param_offset(desc, f"fit{a}.wo"),
                  student.param_offset(desc, f"fit{a}.wo") + desc["fit"][-1] + 1) for a in range(desc["ntypes"])]


def _slab(case, seed):
    """The first slab of a decomposed box: coordinates, types, cell, number of
    centres (atoms it owns), the atoms' indices in the whole box and its size."""
    c, t, b, _ = _system(case, seed)
    rc = MODELS[case["model"]]["rcut"]
    plan = domain.make_plan(c, b, SLABS, rc + 2.0, rc + 2.0)
    own, src, pos = plan.owned[0], plan.ghost_src[0], plan.ghost_pos[0]
    gid = np.array([plan.owned[s][p] for s, p in zip(src, pos)], dtype=np.int64)
    x = np.concatenate([c[own], c[gid] + np.outer(plan.ghost_shift[0], [b[0], 0.0, 0.0])])
    x[:, 0] -= plan.origin(0)
    ids = np.concatenate([own, gid])
    return np.ascontiguousarray(x), t[ids], plan.sub_box(), len(own), ids, len(t)


def _train_data(case, seed):
    """Frames (geometry), their reference energies and forces in units of the
    RMS force, the box, types, and the parameters that the step starts from.
    A teacher's labels are forces of RMS 1 in these units; the seeded ones
    have that distribution, and an energy per atom of order 1."""
    desc = MODELS[case["model"]]
    frames = [_system(case, 100 * seed + f) for f in range(case["frames"])]
    N = len(frames[0][1])
    rng = np.random.default_rng(seed)
    F = rng.standard_normal((len(frames), N, 3))
    E = N * (1.0 + 0.1 * rng.standard_normal(len(frames)))
    if case["model"] == "student":
        P = _student_params()
        P = P * (1.0 + 1e-3 * rng.standard_normal(len(P)))
    else:
        P = dp.dp_model_params_from_seed(desc, seed)
    for sl in _out_slices(desc):
        P[sl] /= 1e-2   # the output layer in units of an RMS force of 1e-2 eV/A
    coords = np.stack([f[0] for f in frames])
    return coords, frames[0][1], frames[0][2], E, F, P


def prepare(case, seed):
    kind, desc, prec = case["kind"], MODELS[case["model"]], PRECS[case["prec"]]
    dev = "cuda"
    s = dict(kind=kind)
    if kind == "train":
        coords, types, box, E, F, P = _train_data(case, seed)
        model = dp.Model(desc, P)
        s.update(model=model, ctx=dp.Context(model, len(types)), box=box,
                 frames=dict(coords=torch.tensor(coords, device=dev), types=torch.tensor(types, device=dev), box=box),
                 E=torch.tensor(E, device=dev), F=torch.tensor(F, device=dev), n=case["frames"],
                 params=torch.tensor(P, dtype=torch.float64, requires_grad=True))
        return s
    if kind == "local":
        c, t, box, nloc, ids, total = _slab(case, seed)
        masses = None
        s.update(nloc=nloc, ids=torch.tensor(ids, device=dev),
                 whole=torch.empty((total, 3), dtype=torch.float64, device=dev))
    else:
        c, t, box, masses = _system(case, seed)
    x = torch.tensor(c, device=dev)
    types = torch.tensor(t, device=dev)
    s.update(x=x, types=types, box=box, masses=masses, skin=case.get("skin", _skin(desc, box)),
             steps=case.get("steps", 0))
    if kind in ("md", "fast"):
        T0 = 330.0 if case["model"] == "copper" else 300.0
        v = synth.maxwell_velocities(np.array(masses)[t], T0, seed=seed + 1)
        s.update(v=torch.tensor(v, device=dev), dt=_dt(case), xw=torch.empty_like(x), vw=torch.empty_like(x),
                 thermo=torch.empty((s["steps"], 4), dtype=torch.float64, device=dev))
    if kind == "fast":
        s["full"] = dp.Model.from_seed(synth.WATER_MODEL, 0)
        s["small"] = dp.Model(synth.WATER_STUDENT, _student_params())
        s["fast"] = student.FastPathMD(s["full"], s["small"], len(t))
    else:
        s["model"] = dp.Model.from_seed(desc, seed)
        s["ctx"] = dp.Context(s["model"], len(t), precision=prec)
    return s


def run(s):
    kind = s["kind"]
    if kind == "train":
        p = s["params"]
        p.grad = None
        loss = student.batch_loss(p, s["ctx"], s["frames"], s["E"], s["F"], range(s["n"]), PE, PF, backward=True)
        with torch.no_grad():
            p -= LR * p.grad
        return dict(loss=loss, grad=p.grad, params=p.detach())
    x, t, box = s["x"], s["types"], s["box"]
    if kind == "nlist":
        dp.dp_build_nlist(s["ctx"], x, t, box, s["skin"])
        nlist, nreal, _ = dp.dp_format_nlist(s["ctx"], x, t, box)
        return dict(nlist=nlist, nreal=nreal)
    if kind == "eval":
        dp.dp_build_nlist(s["ctx"], x, t, box, 0.0)
        o = dp.dp_eval(s["ctx"], x, t, box, want_atom_energy=True)
        return {k: o[k] for k in ("energy", "force", "virial", "atom_energy")}
    if kind == "local":
        dp.dp_build_nlist(s["ctx"], x, t, box, 0.0)
        o = dp.dp_eval_local(s["ctx"], x, t, box, s["nloc"])
        # the increments go back to the atoms' owners
        s["whole"].zero_().index_add_(0, s["ids"], o["force"])
        return dict(energy=o["energy"], force=s["whole"], virial=o["virial"])
    # MD runs start from the given coordinates and velocities
    xw, vw = s["xw"], s["vw"]
    xw.copy_(x)
    vw.copy_(s["v"])
    if kind == "fast":
        f = s["fast"]
        dp.dp_md_reset(f.fast)
        checks, switched = f.run(xw, vw, t, box, s["masses"], s["dt"], s["steps"], skin=s["skin"])
        return dict(coords=xw, vel=vw, force_rms_full=checks[-1]["force_rms_full"],
                    force=dp.dp_md_get_force(f.fast, len(t)))
    dp.dp_md_reset(s["ctx"])
    dp.dp_md_step(s["ctx"], xw, vw, t, box, s["masses"], s["dt"], s["steps"], skin=s["skin"], thermo=s["thermo"])
    return dict(coords=xw, vel=vw, thermo=s["thermo"], force=dp.dp_md_get_force(s["ctx"], len(t)))


def _rows(desc):
    """Expected neighbours within rcut at the model's density."""
    rho = 4 / 3.634 ** 3 if desc["ntypes"] == 1 else 3 / WATER_EDGE ** 3
    return rho * 4.0 / 3.0 * math.pi * desc["rcut"] ** 3


def _eval_flops(desc):
    """Per atom: the embedding net with its s-derivative and the contractions
    of its rows, the descriptor, and the fitting net forward and backward."""
    e1, e2, M = desc["emb"]
    row = 2 * 2 * (e1 + e1 * e2 + e2 * M) + 3 * 8 * M
    m2, fit = desc["m2"], [desc["m2"] * M] + list(desc["fit"]) + [1]
    return _rows(desc) * row + 3 * 8 * m2 * M + 4 * sum(a * b for a, b in zip(fit[:-1], fit[1:]))


def work(case):
    desc = MODELS[case["model"]]
    N = case["side"] ** 3 * (4 if case["model"] == "copper" else 3)
    kind = case["kind"]
    npar = synth.n_params(desc)
    if kind == "nlist":
        return dict(bytes=N * (24 + 4) + N * 4 * (sum(desc["sel"]) + desc["ntypes"]),
                    flops=10.0 * N * _rows(desc) * (1 + 2 / desc["rcut"]) ** 3)
    if kind == "train":
        nf = case["frames"]
        return dict(bytes=nf * (N * (24 + 4 + 24) + 8) + 4 * 8 * npar, flops=nf * N * 4.0 * _eval_flops(desc))
    if kind == "eval":
        return dict(bytes=N * (24 + 4 + 24 + 8) + 8 * npar, flops=N * _eval_flops(desc))
    if kind == "local":
        return dict(bytes=N * (24 + 4 + 24) // SLABS + 8 * npar, flops=N * _eval_flops(desc) / SLABS)
    evals = (case["steps"] + 1) * _eval_flops(desc) + (_eval_flops(synth.WATER_MODEL) if kind == "fast" else 0)
    return dict(bytes=N * (2 * 24 + 4 + 3 * 24) + 8 * npar, flops=N * evals)


# ------------------------------------------------------------------- exact --
# The same quantities in plain torch, float64: neighbours by a distance search,
# the nets as written in the method, forces by reverse-mode differentiation.

_KB, _ACC = 8.617333262e-5, 9.648533212e-3


def _neighbours(x, box, rc, i0, i1):
    """Pairs (i, j), i in [i0, i1), within rc: a float32 search with a margin,
    then the float64 minimum-image distance."""
    L = torch.as_tensor(box, dtype=torch.float64, device=x.device)
    xf, Lf = (x / L).float(), L.float()
    out_i, out_j = [], []
    step = max(1, int(3e8) // len(x))
    for a in range(i0, i1, step):
        b = min(i1, a + step)
        r2 = torch.zeros((b - a, len(x)), device=x.device)
        for c in range(3):
            d = xf[None, :, c] - xf[a:b, None, c]
            r2 += ((d - torch.round(d)) * Lf[c]) ** 2
        i, j = torch.nonzero(r2 < (rc + 0.01) ** 2, as_tuple=True)
        i += a
        d = x[j] - x[i]
        d -= L * torch.round(d / L)
        keep = ((d * d).sum(1) < rc * rc) & (i != j)
        out_i.append(i[keep])
        out_j.append(j[keep])
    return torch.cat(out_i), torch.cat(out_j)


def _views(desc, p):
    out, k = {}, 0
    for name, shape in synth.layer_shapes(desc):
        m = int(np.prod(shape))
        out[name] = p[k:k + m].reshape(shape)
        k += m
    return out


def _atom_energies(desc, W, d, ic, tj, ti):
    """E_i of the centres of one chunk.  d [rows, 3]: r_ij; ic: chunk-local
    centre of each row; tj: neighbour type; ti: type of each centre."""
    rs, rc = desc["rcut_smth"], desc["rcut"]
    r = (d * d).sum(1).sqrt()
    u = (r - rs) / (rc - rs)
    w = torch.where(r < rs, torch.ones_like(r), u ** 3 * (-6 * u * u + 15 * u - 10) + 1)
    s = w / r
    R = torch.cat([s[:, None], s[:, None] * d / r[:, None]], 1)
    M, m2 = desc["emb"][-1], desc["m2"]
    T = torch.zeros((len(ti) * 4, M), dtype=torch.float64, device=d.device)
    nm = float(sum(desc["sel"])) if desc.get("desc_scale_nm", 1) else 1.0
    tc = ti[ic]
    for a in range(desc["ntypes"]):
        for b in range(desc["ntypes"]):
            q = torch.nonzero((tc == a) & (tj == b))[:, 0]
            h = torch.tanh(s[q, None] * W[f"emb{a}{b}.W0"] + W[f"emb{a}{b}.b0"])
            for l in range(1, len(desc["emb"])):
                y = torch.tanh(h @ W[f"emb{a}{b}.W{l}"] + W[f"emb{a}{b}.b{l}"])
                h = y + (torch.cat([h, h], 1) if y.shape[1] == 2 * h.shape[1] else h if y.shape == h.shape else 0.0)
            for c in range(4):
                T = T.index_add(0, ic[q] * 4 + c, R[q, c:c + 1] * h)
    T = (T / nm).reshape(-1, 4, M)
    D = torch.einsum("ncx,ncm->nxm", T[:, :, :m2], T).reshape(len(ti), m2 * M)
    E = torch.zeros(len(ti), dtype=torch.float64, device=d.device)
    for a in range(desc["ntypes"]):
        q = torch.nonzero(ti == a)[:, 0]
        h = D[q]
        for l in range(len(desc["fit"])):
            y = torch.tanh(h @ W[f"fit{a}.W{l + 1}"] + W[f"fit{a}.b{l + 1}"])
            h = y + h if l > 0 and y.shape == h.shape else y
        E = E.index_add(0, q, h @ W[f"fit{a}.wo"] + W[f"fit{a}.bo"][0])
    return E


def _chunks(desc, n):
    """Centres per chunk: the rows' activations of a chunk stay below ~10 GB."""
    step = max(1, int(1.2e6 / _rows(desc)))
    return [(a, min(n, a + step)) for a in range(0, n, step)]


def _evaluate(desc, p, x, types, box, nloc=None):
    n = len(x) if nloc is None else nloc
    W = _views(desc, p)
    L = torch.as_tensor(box, dtype=torch.float64, device=x.device)
    F = torch.zeros_like(x)
    V = torch.zeros((3, 3), dtype=torch.float64, device=x.device)
    Es = []
    for a, b in _chunks(desc, n):
        i, j = _neighbours(x, box, desc["rcut"], a, b)
        d = x[j] - x[i]
        d = (d - L * torch.round(d / L)).requires_grad_(True)
        E = _atom_energies(desc, W, d, i - a, types[j], types[a:b])
        g, = torch.autograd.grad(E.sum(), d)
        Es.append(E.detach())
        F.index_add_(0, i, g)
        F.index_add_(0, j, -g)
        V -= d.detach().T @ g
    E = torch.cat(Es)
    return E.sum().reshape(1), F, V.reshape(9), E


def _exact_train(case, seed, dev):
    desc = MODELS[case["model"]]
    coords, t, box, E_ref, F_ref, P = _train_data(case, seed)
    types = torch.tensor(t, device=dev).long()
    p = torch.tensor(P, device=dev)
    L = torch.as_tensor(box, device=dev)
    grad, total = torch.zeros_like(p), 0.0
    N, nf = len(t), case["frames"]
    for f in range(nf):
        x = torch.tensor(coords[f], device=dev)
        Fr = torch.tensor(F_ref[f], device=dev)
        E, F, _, _ = _evaluate(desc, p, x, types, box)
        total += float(PE * ((E[0] - E_ref[f]) / N) ** 2 + PF * ((F - Fr) ** 2).sum() / (3 * N))
        cE = 2 * PE * (E[0] - E_ref[f]) / N ** 2 / nf
        lam = 2 * PF * (F - Fr) / (3 * N) / nf
        # d/dW of cE E + sum lam . F, centre by centre (F is a sum over centres)
        for a, b in _chunks(desc, N):
            i, j = _neighbours(x, box, desc["rcut"], a, b)
            d = x[j] - x[i]
            d = (d - L * torch.round(d / L)).requires_grad_(True)
            q = p.clone().requires_grad_(True)
            Ei = _atom_energies(desc, _views(desc, q), d, i - a, types[j], types[a:b])
            g, = torch.autograd.grad(Ei.sum(), d, create_graph=True)
            phi = cE * Ei.sum() + ((lam[i] - lam[j]) * g).sum()
            grad += torch.autograd.grad(phi, q)[0]
    return dict(loss=total / nf, grad=grad.cpu(), params=(p - LR * grad).cpu())


def exact(case, seed):
    kind, desc = case["kind"], MODELS[case["model"]]
    if kind == "nlist":
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if kind == "train":
        return _exact_train(case, seed, dev)
    if kind == "local":
        c, t, box, nloc, ids, total = _slab(case, seed)
    else:
        c, t, box, masses = _system(case, seed)
        nloc = None
    if kind == "fast":
        P = _student_params()
    else:
        P = synth.model_params(desc, seed)
    p, x = torch.tensor(P, device=dev), torch.tensor(c, device=dev)
    types = torch.tensor(t, device=dev).long()
    if kind in ("eval", "local"):
        E, F, V, Ei = _evaluate(desc, p, x, types, box, nloc)
        if kind == "local":
            F = torch.zeros((total, 3), dtype=torch.float64, device=dev).index_add(0, torch.tensor(ids, device=dev), F)
        o = dict(energy=E, force=F, virial=V)
        if kind == "eval":
            o["atom_energy"] = Ei
        return o
    m = torch.tensor(np.array(masses), device=dev)[types]
    T0 = 330.0 if case["model"] == "copper" else 300.0
    v = torch.tensor(synth.maxwell_velocities(np.array(masses)[t], T0, seed=seed + 1), device=dev)
    dt = _dt(case)
    L = torch.as_tensor(box, dtype=torch.float64, device=dev)
    vol, N = float(np.prod(box)), len(t)
    _, F, _, _ = _evaluate(desc, p, x, types, box)
    thermo = []
    for _ in range(case["steps"]):
        v = v + F * (_ACC / m)[:, None] * (0.5 * dt)
        x = x + v * dt
        x = x - L * torch.floor(x / L)
        E, F, V, _ = _evaluate(desc, p, x, types, box)
        v = v + F * (_ACC / m)[:, None] * (0.5 * dt)
        ke = float((0.5 * m[:, None] * v * v).sum()) / _ACC
        tr = float(V[0] + V[4] + V[8])
        thermo.append([float(E), ke, 2 * ke / ((3 * N - 3) * _KB), (2 * ke + tr) / (3 * vol)])
    o = dict(coords=x, vel=v, force=F)
    if kind == "fast":
        full = torch.tensor(synth.model_params(synth.WATER_MODEL, 0), device=dev)
        f = _evaluate(synth.WATER_MODEL, full, x, types, box)[1]
        o["force_rms_full"] = float((f * f).mean().sqrt())
    else:
        o["thermo"] = torch.tensor(thermo, dtype=torch.float64)
    return o
