"""The calls whose time this framework is judged by.

Each case is one call that a program using the package makes, through the
public entry points of `paper_2602_14975_gb300.core`: the force evaluations of
both models, the neighbour build, one distillation step, an outer step of
molecular dynamics and the serving loop. Models, integrator settings and
system recipes are those of `synth.WORKLOADS` and of the serving workload;
`draw` spreads the same calls over the whole range of sizes, system kinds and
precisions they are used with.

Fields of a case
  call       cons | nc | nbr | distill | md | serve
  system     water (periodic box) | chain (solvated bead chain) | droplets
             (open small-molecule droplets, many replicas in one batch)
  n_mol      water: molecules per box; chain: beads, with water in the ratio
             of the 23,558-atom system
  n_rep      replicas in the batch (frames for distill, requests for serve)
  lo, hi     droplets: smallest and largest solute, log-spaced over the batch
  model      small (the 192-atom configuration's models) | full (those of the
             larger configurations)
  bf16       contractions in split-bf16 on the tensor cores, or plain fp32
"""
import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_2602_14975_gb300 import core
from paper_2602_14975_gb300 import synth as S

SKIN = 0.5
WATER_EDGE = 12.42 / 64 ** (1.0 / 3.0)       # box edge per molecule^(1/3) of the water configurations
CHAIN_EDGE = 62.2 / 2489 ** (1.0 / 3.0)      # and per bead^(1/3) of the solvated chain
CHAIN_WATER = 7023 / 2489                    # waters per bead


def _case(name, call, system, n_mol=0, n_rep=1, lo=0, hi=0, model="full", bf16=True, mode="respa"):
    return dict(name=name, call=call, system=system, n_mol=n_mol, n_rep=n_rep, lo=lo, hi=hi, model=model, bf16=bf16,
                mode=mode)


def listed():
    return [
        # conservative energy and forces of the smallest configuration: a call that launches and latency bound
        _case("cons_water_192_fp32", "cons", "water", 64, model="small", bf16=False),
        # the same call on the 12,288-atom water box with the tensor-core contractions
        _case("cons_water_12288", "cons", "water", 4096),
        # the single-time-step baseline's force call on the solvated chain, plain fp32 models
        _case("cons_chain_23558_fp32", "cons", "chain", 2489, bf16=False),
        # the largest box of the roofline sweep
        _case("cons_water_100000", "cons", "water", 33333),
        # the inner-step force of a lone small solute in its droplet
        _case("nc_droplet_80", "nc", "droplets", n_rep=1, lo=20, hi=20),
        # the inner-step force of the solvated chain: evaluated five times per outer step
        _case("nc_chain_23558", "nc", "chain", 2489),
        # the inner-step force of a ragged batch of resident serving replicas
        _case("nc_droplets_64", "nc", "droplets", n_rep=64, lo=20, hi=400),
        # a neighbour list at model cutoff + skin, as an analysis or a new system needs it
        _case("nbr_water_12288", "nbr", "water", 4096),
        # one training step (loss and gradient of every fitted weight) on four frames of the 12,288-atom box
        _case("distill_4x12288", "distill", "water", 4096, n_rep=4),
        # one outer step of the smallest configuration, read back after each step by the caller
        _case("md_water_192", "md", "water", 64, model="small", bf16=False),
        # one outer step (one conservative and five inner evaluations) of the solvated chain
        _case("md_chain_23558", "md", "chain", 2489),
        # a burst of short requests of uneven size through the serving loop, host buffers in and out
        _case("serve_24", "serve", "droplets", n_rep=24, lo=20, hi=400),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["cons", "cons", "cons", "nc", "nc", "md", "md", "nbr", "distill", "serve"])
    model = "full" if rng.random() < 0.75 else "small"
    bf16 = model == "full" and rng.random() < 0.7       # the small models are fp32 ones
    if call == "serve":
        lo = _log(rng, 20, 100)
        c = _case("", call, "droplets", n_rep=rng.randint(4, 24), lo=lo, hi=max(lo, _log(rng, 100, 400)), model=model,
                  bf16=bf16)
    elif call == "distill":
        n = _log(rng, 64, 4096)
        c = _case("", call, "water", n, n_rep=rng.randint(1, max(1, min(10, 16384 // n))), model=model, bf16=bf16)
    else:
        system = rng.choice(["water", "water", "chain", "droplets"])
        top = 8000 if call == "md" else 33333
        if system == "water":
            c = _case("", call, system, _log(rng, 65, top), model=model, bf16=bf16)
        elif system == "chain":
            c = _case("", call, system, _log(rng, 100, 2489), model=model, bf16=bf16)
        else:
            lo = _log(rng, 20, 150)
            c = _case("", call, system, n_rep=_log(rng, 1, 64), lo=lo, hi=max(lo, _log(rng, 60, 400)), model=model,
                      bf16=bf16)
        if call == "md" and rng.random() < 0.3:
            c["mode"] = "sts"
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
def _sizes(case):
    """Solute atoms of each droplet: log-spaced, the quantiles of the serving workload's distribution."""
    n = case["n_rep"]
    if n == 1:
        return [case["lo"]]
    a, b = math.log(case["lo"]), math.log(case["hi"])
    return [int(round(math.exp(a + (b - a) * k / (n - 1)))) for k in range(n)]


def _systems(case, seed):
    if case["system"] == "water":
        n = case["n_mol"]
        return [S.water_box(n, WATER_EDGE * n ** (1.0 / 3.0), 1000 * seed + r) for r in range(case["n_rep"])]
    if case["system"] == "chain":
        n = case["n_mol"]
        return [S.solvated_chain(n, int(CHAIN_WATER * n), CHAIN_EDGE * n ** (1.0 / 3.0), seed)]
    return [S.capped_molecule_in_droplet(n, 1000 * seed + k) for k, n in enumerate(_sizes(case))]


def _reordered(s, seed):
    """The system with its molecules in another order: other inputs with the same number of pairs."""
    rng = np.random.default_rng(seed)
    order = np.argsort(rng.permutation(int(s.mol_id.max()) + 1)[s.mol_id], kind="stable")
    back = np.empty_like(order)
    back[order] = np.arange(order.size)
    return S.System(s.name, s.x[order], s.species[order], s.mol_id[order], back[s.bonds].astype(np.int32), s.bond_r0,
                    s.box)


def _specs(case):
    if case["model"] == "small":
        cs, ns = S.cons_spec(2, 64, 1, bf16=case["bf16"]), S.nc_spec(32, rc=3.5, bf16=case["bf16"])
    else:
        cs, ns = S.cons_spec(3, 128, 2, bf16=case["bf16"]), S.nc_spec(64, rc=4.0, bf16=case["bf16"])
    return cs, ns


def _models(case, seed):
    cs, ns = _specs(case)
    return (cs, S.cons_weights(cs, seed + 1)), (ns, S.nc_weights(ns, seed + 2))


def _target(n_atoms, seed):
    """Stand-in for the large model's forces that a distillation frame is labelled with."""
    return np.random.default_rng(seed + 5).normal(0.0, 10.0, (n_atoms, 3)).astype(np.float32)


def _integrator(case):
    """Settings of the configurations: the small models' run, the others' DMTS-NC run, and the 1 fs baseline."""
    if case["mode"] == "sts":
        return (1.0, 1, (1.0,) * 5, 0.0)
    if case["model"] == "small":
        return (4.0, 4, (1.0,) * 5, 0.0)
    return (10.0, 5, (20.0, 1.0, 1.0, 1.0, 1.0), 3.0)


class _Release:
    """Frees a state's device lists with the state, as a program does when it is done with a trajectory."""

    def __init__(self, state):
        self.state = state

    def __del__(self):
        self.state.release()


def prepare(case, seed):
    cons, nc = _models(case, seed)
    call = case["call"]
    if call == "nbr":                               # lists of one length whatever the seed
        systems = [_reordered(s, seed) for s in _systems(case, 17)]
    else:
        systems = _systems(case, seed)
    st = dict(call=call)
    if call == "serve":
        dt, n_in, gamma, hmr = _integrator(case)
        rng = np.random.default_rng(seed + 3)
        reqs = []
        for k, s in enumerate(systems):
            m = core.masses_hmr(s.species, s.mol_id, s.element_masses(), hmr)
            reqs.append(core.ReplicaRequest(s, S.maxwell_boltzmann(m, 300.0, seed + 10 + k), m.astype(np.float32),
                                            int(rng.integers(2, 5)), seed=seed, replica_id=k))
        st.update(ctx=core.Context(cons=cons, nc=nc), reqs=reqs, integ=core.integrator(dt, n_in, 300.0, gamma, skin=SKIN))
        return st
    st["ctx"] = ctx = core.Context(cons=cons, nc=nc)
    st["sys"] = d = core.DeviceSystem(systems)
    if call == "md":
        dt, n_in, gamma, hmr = _integrator(case)
        m = np.concatenate([core.masses_hmr(s.species, s.mol_id, s.element_masses(), hmr) for s in systems])
        v = np.concatenate([S.maxwell_boltzmann(m[a:b], 300.0, seed + 10 + k) for k, (a, b) in
                            enumerate(zip(d.rep_off_host[:-1], d.rep_off_host[1:]))])
        st["state"] = core.MDState(d, v, m.astype(np.float32), seeds=seed)
        st["release"] = _Release(st["state"])
        mode = core.L.MODE_STS if case["mode"] == "sts" else core.L.MODE_RESPA
        st["integ"] = core.integrator(dt, n_in, 300.0, gamma, mode=mode, skin=SKIN)
    elif call == "nbr":
        st["r_list"] = cons[0].rc + SKIN
    elif call == "cons":
        st["list"] = core.nbr_build(ctx, d, cons[0].rc + SKIN)
    else:
        st["list"] = core.nbr_build(ctx, d, nc[0].rc + SKIN)
        if call == "distill":
            st["target"] = torch.from_numpy(_target(d.n_atoms, seed)).cuda()
    return st


# -------------------------------------------------------------------- run
# Per-replica energies and losses are 64-bit sums of terms formed in fp32;
# they are handed on in single precision, the accuracy they have.
def run(st):
    call = st["call"]
    if call == "cons":
        E, F = core.energy_forces_cons(st["ctx"], st["sys"], st["list"], with_prior=True)
        return {"energy": E.float(), "forces": F}
    if call == "nc":
        F, net = core.forces_nc(st["ctx"], st["sys"], st["list"], with_bonds=True)
        return {"forces": F, "net": net}
    if call == "nbr":
        nb = core.nbr_build(st["ctx"], st["sys"], st["r_list"])
        return {"row_ptr": nb.row_ptr, "col": nb.col}
    if call == "distill":
        loss, grad = core.nc_distill_step(st["ctx"], st["sys"], st["list"], st["target"], lr=0.0, with_grad=True)
        return {"loss": loss.float(), "grad": grad}
    if call == "md":
        s = st["state"]
        core.respa_step(st["ctx"], s, st["integ"], 1)
        return {"x": s.dsys.x, "v": s.v, "f_nc": s.f_nc, "f_cons": s.f_cons, "energy": s.energy.float()}
    out, _ = core.run_replicas(st["ctx"], st["reqs"], st["integ"], tick_cap=1024)
    return {"x": [o["x"] for o in out], "v": [o["v"] for o in out],
            "energy": np.array([o["energy"] for o in out], np.float32)}


# ------------------------------------------------------------------- work
def work(case):
    """Inputs read once, outputs written once, and the model's own sums: per layer the radial sums and messages of
    every neighbour (a layer on the species embedding needs only the basis sums per species), the node contractions,
    and twice that where forces are their adjoint."""
    if case["system"] == "water":
        n, dens = 3 * case["n_mol"] * case["n_rep"], 1.0
    elif case["system"] == "chain":
        n, dens = case["n_mol"] + 3 * int(CHAIN_WATER * case["n_mol"]), 1.0
    else:
        n, dens = 4 * sum(_sizes(case)), 0.6       # an open droplet has fewer neighbours
    cs, ns = _specs(case)
    ec, en = dens * n * S.expected_neighbours(cs.rc), dens * n * S.expected_neighbours(ns.rc)
    state = 3 * 4 + 1 + 4 + 8                       # position, species, molecule, bonds

    def layer(m, e, first):
        lm, k = (m.lmax + 1) ** 2, m.K
        edge = 2 * k * lm if first else 2 * (k * (m.lmax + 1) + lm) * m.C
        return e * edge + n * (2 * k * lm * m.C * 2 if first else 0) + 2 * n * m.C * m.C * (m.lmax + 2)

    H = ns.K + ns.n_l
    f_cons = 2 * (sum(layer(cs, ec, t == 0) for t in range(cs.L)) + 2 * n * cs.C * cs.C)
    f_nc = layer(ns, en, True) + 2 * n * ns.C * 2 * H * ns.n_c + en / 2 * (4 * H * ns.n_c + 60)
    w_cons, w_nc = 4 * S.cons_blob_len(cs), 4 * S.nc_blob_len(ns)
    call = case["call"]
    if call == "cons":
        return {"bytes": n * (state + 12) + 4 * ec + w_cons, "flops": f_cons}
    if call == "nc":
        return {"bytes": n * (state + 12) + 4 * en + w_nc, "flops": f_nc}
    if call == "nbr":
        return {"bytes": n * 16 + 4 * ec * (1 + SKIN / cs.rc) ** 3, "flops": 8 * ec}
    if call == "distill":
        return {"bytes": n * (state + 12) + 4 * en + 2 * w_nc, "flops": 3 * f_nc}
    steps = 3 if call == "serve" else 1             # outer steps; a served request runs two to four
    inner = _integrator(case)[1] if case["mode"] != "sts" else 0
    return {"bytes": n * (state + 4 + 4 * 24) + 4 * (ec + en) + w_cons + w_nc, "flops": steps * (f_cons + inner * f_nc)}


# ------------------------------------------------------------------ exact
# The two models and the analytic terms in 64-bit torch, written from their
# definitions: brute-force neighbours, autograd for the gradients.
K_BOND, LJ_EPS, LJ_SIG, LJ_RC, REP_RC, P_PRIOR = 450.0, 0.15, 3.15, 5.0, 3.5, 6
CHUNK = 150_000                                     # edges per step of a layer


def _envelope(u, p):
    return 1 - (p + 1) * (p + 2) / 2 * u ** p + p * (p + 2) * u ** (p + 1) - p * (p + 1) / 2 * u ** (p + 2)


def _bessel(r, rc, K):
    k = torch.arange(1, K + 1, device=r.device, dtype=r.dtype)
    return math.sqrt(2.0 / rc) * torch.sin(k * math.pi * r[:, None] / rc) / r[:, None]


def _harmonics(n, lmax):
    x, y, z = n.unbind(1)
    Y = [torch.ones_like(x)]
    if lmax >= 1:
        Y += [math.sqrt(3) * x, math.sqrt(3) * y, math.sqrt(3) * z]
    if lmax >= 2:
        s15, s5 = math.sqrt(15), math.sqrt(5)
        Y += [s15 * x * y, s15 * y * z, s5 / 2 * (3 * z * z - 1), s15 * x * z, s15 / 2 * (x * x - y * y)]
    return torch.stack(Y, 1)


class _Batch:
    """All replicas of a case in 64 bits, with the directed edges within `cut`."""

    def __init__(self, systems, cut):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        t = lambda a, dt=torch.float64: torch.as_tensor(np.asarray(a), dtype=dt, device=dev)  # noqa: E731
        off = np.concatenate([[0], np.cumsum([s.n_atoms for s in systems])])
        self.n, self.n_rep = int(off[-1]), len(systems)
        self.x = t(np.concatenate([s.x for s in systems]))
        self.species = t(np.concatenate([s.species for s in systems]), torch.int64)
        self.mol = t(np.concatenate([s.mol_id + o for s, o in zip(systems, off)]), torch.int64)
        self.rep = t(np.repeat(np.arange(self.n_rep), np.diff(off)), torch.int64)
        self.box = t(np.stack([np.asarray(s.box, np.float32) for s in systems]))
        self.bonds = t(np.concatenate([s.bonds.reshape(-1, 2) + o for s, o in zip(systems, off)]), torch.int64)
        self.r0 = t(np.concatenate([np.asarray(s.bond_r0, np.float32) for s in systems]))
        self.wrap = torch.where(self.box > 0, self.box, torch.ones_like(self.box))
        self.periodic = (self.box > 0).double()
        ii, jj = [], []
        for a, b in zip(off[:-1], off[1:]):
            step = max(1, 40_000_000 // max(1, int(b - a)))
            r = int(self.rep[a])
            for c in range(int(a), int(b), step):
                d = self.x[None, a:b] - self.x[c:min(c + step, b), None]
                d = d - self.box[r] * torch.round(d / self.wrap[r])
                i, j = torch.nonzero((d * d).sum(2) < cut * cut, as_tuple=True)
                i, j = i + c, j + int(a)
                ii.append(i[i != j])
                jj.append(j[i != j])
        self.i, self.j = torch.cat(ii), torch.cat(jj)

    def disp(self, x, i, j):
        d = x[j] - x[i]
        b, r = self.box[self.rep[i]], self.rep[i]
        return d - b * torch.round(d.detach() / self.wrap[r])

    def within(self, rc):
        d = self.disp(self.x, self.i, self.j)
        m = (d * d).sum(1) < rc * rc
        return self.i[m], self.j[m]

    def bond_energy(self, x):
        d = self.disp(x, self.bonds[:, 0], self.bonds[:, 1])
        return 0.5 * K_BOND * (d.norm(dim=1) - self.r0) ** 2

    def repulsion(self, x):
        i, j = self.within(REP_RC)
        k = i < j
        i, j = i[k], j[k]
        if self.bonds.numel():
            key = lambda a, b: torch.minimum(a, b) * self.n + torch.maximum(a, b)  # noqa: E731
            k = ~torch.isin(key(i, j), key(self.bonds[:, 0], self.bonds[:, 1]))
            i, j = i[k], j[k]
        r = self.disp(x, i, j).norm(dim=1)
        Z = torch.tensor([1.0, 6.0, 7.0, 8.0, 16.0], dtype=x.dtype, device=x.device)
        zi, zj = Z[self.species[i]], Z[self.species[j]]
        a = 0.8854 * 0.529177210903 / (zi ** 0.23 + zj ** 0.23)
        c, dd = (0.18175, 0.50986, 0.28022, 0.02817), (3.19980, 0.94229, 0.40290, 0.20162)
        phi = sum(ck * torch.exp(-dk * r / a) for ck, dk in zip(c, dd))
        return 332.0637133 * zi * zj / r * phi * _envelope(r / REP_RC, P_PRIOR)

    def lennard_jones(self, x):
        i, j = self.within(LJ_RC)
        k = (i < j) & (self.species[i] != 0) & (self.species[j] != 0) & (self.mol[i] != self.mol[j])
        r = self.disp(x, i[k], j[k]).norm(dim=1)
        s6 = (LJ_SIG / r) ** 6
        return 4 * LJ_EPS * (s6 * s6 - s6) * _envelope(r / LJ_RC, P_PRIOR)


def _take(w, *shape):
    n = math.prod(shape)
    return w[0][:n].reshape(shape), (w[0][n:],)


def _messages(b, m, x, s, wrad, lmax):
    """A[i][lm][c] of one layer, chunk by chunk (recomputed in the backward pass)."""
    i, j = b.within(m.rc)
    cuts = [0] + (torch.searchsorted(i, i[CHUNK::CHUNK].contiguous())).tolist() + [i.numel()]

    def part(x, s, wrad, lo, hi):
        ii, jj = i[lo:hi], j[lo:hi]
        d = b.disp(x, ii, jj)
        r = d.norm(dim=1)
        fB = _envelope(r / m.rc, m.p)[:, None] * _bessel(r, m.rc, m.K)
        Y = _harmonics(d / r[:, None], lmax)
        a0 = int(ii[0])
        out = []
        for l in range(lmax + 1):
            msg = (fB @ wrad[l]) * s[jj]
            for q in range(l * l, (l + 1) * (l + 1)):
                z = torch.zeros(int(ii[-1]) - a0 + 1, s.shape[1], dtype=s.dtype, device=s.device)
                out.append(z.index_add(0, ii - a0, msg * Y[:, q:q + 1]))
        return torch.stack(out, 1)

    A = torch.zeros(b.n, (lmax + 1) ** 2, s.shape[1], dtype=s.dtype, device=s.device)
    for lo, hi in zip(cuts[:-1], cuts[1:]):
        if hi > lo:
            P = torch.utils.checkpoint.checkpoint(part, x, s, wrad, lo, hi, use_reentrant=False)
            rows = torch.arange(int(i[lo]), int(i[hi - 1]) + 1, device=s.device)
            A = A.index_add(0, rows, P)
    return float(np.float32(m.nu)) * A


def _invariants(A, lmax):
    return torch.cat([(A[:, l * l:(l + 1) ** 2] ** 2).sum(1) for l in range(lmax + 1)], 1)


def _silu(v):
    return v * torch.sigmoid(v)


def _cons_exact(b, m, blob):
    x = b.x.clone().requires_grad_(True)
    w = (torch.as_tensor(blob, device=b.x.device),)
    emb, w = _take(w, m.n_species, m.C)
    s = emb[b.species]
    for _ in range(m.L):
        wrad, w = _take(w, m.lmax + 1, m.K, m.C)
        w1, w = _take(w, m.C, (m.lmax + 1) * m.C)
        b1, w = _take(w, m.C)
        w2, w = _take(w, m.C, m.C)
        b2, w = _take(w, m.C)
        q = _invariants(_messages(b, m, x, s, wrad, m.lmax), m.lmax)
        s = s + _silu(q @ w1.T + b1) @ w2.T + b2
    wr, w = _take(w, m.C, m.C)
    br, w = _take(w, m.C)
    wo, w = _take(w, m.C)
    E = float(np.float32(m.scale)) * (_silu(s @ wr.T + br) @ wo).sum()
    E = E + b.bond_energy(x).sum() + b.repulsion(x).sum() + b.lennard_jones(x).sum()
    E.backward()
    return -x.grad


def _nc_exact(b, m, blob, want_grad=False, target=None):
    x = b.x
    blob = torch.as_tensor(blob, device=x.device).clone().requires_grad_(want_grad)
    w = (blob,)
    emb, w = _take(w, m.n_species, m.C)
    wrad, w = _take(w, 2, m.K, m.C)
    w1, w = _take(w, m.C, 2 * m.C)
    b1, w = _take(w, m.C)
    w2, w = _take(w, m.C, m.C)
    b2, w = _take(w, m.C)
    U, w = _take(w, m.n_l, m.C)
    H = m.K + m.n_l
    Wq, w = _take(w, H * m.n_c, m.C)
    Wk, w = _take(w, H * m.n_c, m.C)
    s0 = emb.detach()[b.species]                    # the species embedding is not fitted
    A = _messages(b, m, x, s0, wrad, 1)
    s = s0 + _silu(_invariants(A, 1) @ w1.T + b1) @ w2.T + b2
    V = torch.einsum("hc,nac->nha", U, A[:, 1:4])
    q, k = (s @ Wq.T).reshape(-1, H, m.n_c), (s @ Wk.T).reshape(-1, H, m.n_c)
    i, j = b.within(m.rc)
    F = torch.zeros_like(x)
    step = 1_000_000

    def part(q, k, V, lo, hi):
        ii, jj = i[lo:hi], j[lo:hi]
        d = b.disp(x, ii, jj)
        r = d.norm(dim=1)
        c = (q[ii] * k[jj]).sum(2) / math.sqrt(m.n_c)
        B = _bessel(r, m.rc, m.K)
        vec = d / r[:, None] + torch.einsum("eh,eha->ea", c[:, m.K:], V[ii])
        return (c[:, :m.K] * B).sum(1, keepdim=True) * vec * _envelope(r / m.rc, m.p)[:, None]

    for lo in range(0, i.numel(), step):
        hi = min(lo + step, i.numel())
        f = torch.utils.checkpoint.checkpoint(part, q, k, V, lo, hi, use_reentrant=False)
        F = F.index_add(0, i[lo:hi], f).index_add(0, j[lo:hi], -f)
    F = float(np.float32(m.scale)) * F
    y = x.clone().requires_grad_(True)
    e = b.bond_energy(y).sum() + b.repulsion(y).sum()
    F = F - torch.autograd.grad(e, y)[0]
    cnt = torch.zeros(b.n_rep, dtype=x.dtype, device=x.device).index_add(0, b.rep, torch.ones_like(x[:, 0]))
    mean = torch.zeros(b.n_rep, 3, dtype=x.dtype, device=x.device).index_add(0, b.rep, F) / cnt[:, None]
    F = F - mean[b.rep]
    if not want_grad:
        return F
    per = ((F - target) ** 2).sum(1)
    loss = torch.zeros(b.n_rep, dtype=x.dtype, device=x.device).index_add(0, b.rep, per)
    loss.sum().backward()
    return loss.detach(), blob.grad


def exact(case, seed):
    """The outputs in 64 bits; None for a trajectory and for integers. An energy is one number per replica, whose
    error is the luck of a single sum, and the net force is zero: neither says how exact a path is."""
    call = case["call"]
    if call not in ("cons", "nc", "distill"):
        return None
    systems = _systems(case, seed)
    (cs, cb), (ns, nb) = _models(case, seed)
    if call == "cons":
        return {"energy": None, "forces": _cons_exact(_Batch(systems, max(cs.rc, LJ_RC)), cs, cb)}
    b = _Batch(systems, max(ns.rc, REP_RC))
    if call == "nc":
        return {"forces": _nc_exact(b, ns, nb), "net": None}
    loss, grad = _nc_exact(b, ns, nb, True, torch.as_tensor(_target(b.n, seed), dtype=torch.float64, device=b.x.device))
    return {"loss": loss, "grad": grad}
