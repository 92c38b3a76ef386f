"""Timed work of the random batch Ewald force path, through its public entry points.

Each case is one thing a program does with `paper_2609_02694_gb300.binding`:

  embed  an outer integrator owns the particles: every pass hands over new positions and takes
         the forces back (`set_positions` + `forces`), on the device or through pinned host
         memory, with the energies when it logs them;
  md     the library integrates: a block of Verlet steps, then a frame and the energies
         (`step` + `state` + `energies`), over cells, a Verlet list or the random batch list;
  batch  independent replicas of uneven sizes advanced together (`Batch.step`), then each
         replica's frame.

Particles come from `synth` (jittered lattice, a neutral random charged subset). Three
compositions: "dense" (0.1 particles per cubic Angstrom, sigma 3, alpha 0.09, real units),
"salt" (the same with every particle charged and two LJ types by the sign of the charge) and
"ions" (the LJ electrolyte in reduced units, 200,000 ions per 271^3).
"""
import math

import numpy as np
import torch

from paper_2609_02694_gb300 import binding, synth

_LIST = [
    # One call on a small all-charged box from host memory: latency, launches and copies.
    dict(name="embed_small", kind="embed", comp="dense", N=3000, frac=1.0, P=100, r_c=10.0,
         precision="fp32_comp", box="cubic", host=True, energies=True),
    # The headline workload as an outer integrator drives it, everything on the device.
    dict(name="embed_1m", kind="embed", comp="dense", N=1 << 20, frac=0.1, P=200, r_c=10.0,
         precision="fp32_comp", box="cubic", host=False, energies=False),
    # A large box with many modes in the plain FP32 form (the precision sweep's composition).
    dict(name="embed_4m", kind="embed", comp="dense", N=4000001, frac=0.1, P=500, r_c=10.0,
         precision="fp32", box="cubic", host=False, energies=True),
    # A molten salt: every particle charged, two LJ types, an orthorhombic box, a ragged size.
    dict(name="embed_salt", kind="embed", comp="salt", N=50002, frac=1.0, P=300, r_c=10.0,
         precision="fp32_comp", box="ortho", host=False, energies=True),
    # The FP64 form, which reference runs take (the 65,536-particle box of the error tables).
    dict(name="embed_fp64", kind="embed", comp="dense", N=65536, frac=0.1, P=200, r_c=10.0,
         precision="fp64", box="cubic", host=False, energies=True),
    # The random batch list on a dense system (the largest run's parameters), a ragged size.
    dict(name="embed_rbl", kind="embed", comp="dense", N=1000003, frac=0.05, P=500, r_c=10.0,
         r_core=5.0, p_rbl=10, precision="fp32_comp", box="cubic", host=False, energies=True),
    # Small-box molecular dynamics: step graphs whose kernels are all short.
    dict(name="md_small", kind="md", comp="dense", N=3000, frac=1.0, P=100, r_c=10.0,
         precision="fp32_comp", box="cubic", steps=10),
    # The headline workload stepped by the library, a frame every ten steps.
    dict(name="md_1m", kind="md", comp="dense", N=1 << 20, frac=0.1, P=200, r_c=10.0,
         precision="fp32_comp", box="cubic", steps=10),
    # The LJ electrolyte with the random batch list and the thermostat, at two of its sizes.
    dict(name="md_ions", kind="md", comp="ions", N=200000, frac=1.0, P=200, r_c=8.0,
         r_core=4.0, p_rbl=30, precision="fp32_comp", box="cubic", steps=20, nvt=True),
    dict(name="md_ions_1m4", kind="md", comp="ions", N=1400000, frac=1.0, P=200, r_c=8.0,
         r_core=4.0, p_rbl=30, precision="fp32_comp", box="cubic", steps=5, nvt=True),
    # The same electrolyte over a Verlet list (the dilute system it suits).
    dict(name="md_list", kind="md", comp="ions", N=100000, frac=1.0, P=200, r_c=8.0, skin=1.0,
         precision="fp32_comp", box="cubic", steps=20, nvt=True),
    # Replicas of uneven sizes in one batch.
    dict(name="batch", kind="batch", comp="dense", lo=2000, hi=60000, n=16, frac=0.1, P=200,
         r_c=10.0, precision="fp32_comp", box="cubic", steps=5),
]


def listed():
    return [dict(c) for c in _LIST]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["embed", "embed", "salt", "fp64", "rbl", "md", "md", "ions", "list", "batch"])
    base = dict(r_c=10.0, precision="fp32_comp", box=rng.choice(["cubic", "cubic", "ortho"]))
    if what == "embed":
        frac = rng.choice([0.0, 0.05, 0.1, 0.3, 1.0]) if rng.random() < 0.5 else 0.1
        return dict(base, kind="embed", comp="dense",
                    N=_log(rng, 5000, 2000000 if frac <= 0.1 else 300000), frac=frac,
                    r_c=rng.choice([8.0, 9.0, 10.0, 12.0]), P=_log(rng, 50, 1000),
                    precision=rng.choice(["fp32_comp", "fp32_comp", "fp32"]),
                    host=rng.random() < 0.3, energies=rng.random() < 0.6)
    if what == "salt":
        return dict(base, kind="embed", comp="salt", N=_log(rng, 3000, 200000), frac=1.0,
                    P=_log(rng, 100, 1000), host=rng.random() < 0.3, energies=True)
    if what == "fp64":
        return dict(base, kind="embed", comp=rng.choice(["dense", "dense", "salt"]),
                    N=_log(rng, 3000, 100000), frac=0.1, P=_log(rng, 100, 1000),
                    precision="fp64", host=False, energies=True)
    if what == "rbl":
        return dict(base, kind="embed", comp="dense", N=_log(rng, 5000, 1000000),
                    frac=rng.choice([0.05, 0.1, 1.0]), P=_log(rng, 100, 500),
                    r_core=rng.choice([4.0, 5.0, 6.0]), p_rbl=rng.choice([5, 10, 20]),
                    host=False, energies=True)
    if what == "md":
        frac = rng.choice([0.05, 0.1, 1.0]) if rng.random() < 0.5 else 0.1
        return dict(base, kind="md", comp="dense",
                    N=_log(rng, 3000, 900000 if frac <= 0.1 else 150000), frac=frac,
                    P=_log(rng, 100, 300), steps=rng.choice([5, 10]), nvt=rng.random() < 0.4)
    if what == "ions":
        return dict(base, kind="md", comp="ions", N=_log(rng, 4000, 1400000), frac=1.0, r_c=8.0,
                    P=_log(rng, 100, 200), r_core=4.0, p_rbl=rng.choice([10, 30]), steps=5,
                    nvt=True)
    if what == "list":
        return dict(base, kind="md", comp="ions", N=_log(rng, 4000, 400000), frac=1.0, r_c=8.0,
                    P=_log(rng, 100, 200), skin=rng.choice([0.5, 1.0, 2.0]), steps=10, nvt=True)
    return dict(base, kind="batch", comp="dense", lo=2000, hi=_log(rng, 10000, 60000),
                n=rng.randint(4, 16), frac=0.1, P=_log(rng, 100, 300), steps=5, box="cubic")


# ---------------------------------------------------------------------------------------
# Inputs

def _system(case, N, seed):
    """Box, positions (exact on the 2^-32 grid), charges, types, masses, velocities, LJ table."""
    ions = case["comp"] == "ions"
    density = 200000 / 271.0 ** 3 if ions else (3000 / 32.0 ** 3 if case["frac"] == 1.0 else 0.1)
    L = (N / density) ** (1.0 / 3.0)
    box = np.array([L, L, L]) * (np.array([1.1, 1.0, 1.0 / 1.1]) if case["box"] == "ortho" else 1.0)
    rng = np.random.default_rng(seed)
    s = synth.jittered_lattice(N, box, rng, 0.1)
    nq = int(math.floor(case["frac"] * N / 2.0))
    charged = rng.permutation(N)[: 2 * nq]
    q = np.zeros(N)
    q[charged[:nq]], q[charged[nq:]] = 1.0, -1.0
    mass = np.full(N, 1.0 if ions else 20.0)
    v = synth.maxwell_velocities(mass, 1.0, rng, 1.0, 1.0) if ions else \
        synth.maxwell_velocities(mass, 300.0, rng)
    types = np.zeros(N, np.int32)
    eps, sig = np.array([1.0 if ions else 0.1]), np.array([1.0 if ions else 3.0])
    if case["comp"] == "salt":
        types = (q < 0).astype(np.int32)
        eps, sig = np.array([0.1, 0.1, 0.1, 0.1]), np.array([2.6, 3.0, 3.0, 3.4])
    return dict(box=box, s=s, pos=s.astype(np.float64) * (box / synth.TWO32), q=q, types=types,
                mass=mass, v=v, eps=eps, sig=sig)


def _units(case):
    if case["comp"] == "ions":
        e = synth.LJ_ELECTROLYTE
        return dict(alpha=e["alpha"], C=e["coulomb_C"], dt=e["dt"], kappa=e["kappa"], kB=e["kB"],
                    T=e["T"], tau=e["tau"])
    # sqrt(alpha) r_c = 3 (alpha = 0.09 at r_c = 10)
    return dict(alpha=9.0 / case["r_c"] ** 2, C=synth.COULOMB_C, dt=1.0, kappa=synth.ACCEL_KAPPA,
                kB=synth.BOLTZMANN_KB, T=300.0, tau=100.0)


def _handle(case, sy, seed, replica=0):
    u = _units(case)
    h = binding.RBE(sy["box"], sy["pos"], sy["q"], sy["types"], sy["mass"], sy["v"],
                    alpha=u["alpha"], r_c=case["r_c"], P=case["P"], eps=sy["eps"], sigma=sy["sig"],
                    seed=1 + seed, replica=replica, precision=case["precision"], coulomb_C=u["C"],
                    dt=u["dt"], kappa=u["kappa"], r_core=case.get("r_core", 0.0),
                    p_rbl=case.get("p_rbl", 10))
    if case.get("skin"):
        h.set_neighbor_list(case["skin"])
    if case.get("nvt"):
        h.set_thermostat(u["T"], u["tau"], u["kB"])
    return h


def _batch_sizes(case):
    """Sizes spread over [lo, hi] in the logarithm, none of them round."""
    e = np.exp(np.linspace(math.log(case["lo"]), math.log(case["hi"]), case["n"]))
    return [int(round(x)) + (5 * r) % 8 for r, x in enumerate(e)]


def prepare(case, seed):
    if case["kind"] == "batch":
        hs = [_handle(case, _system(case, N, [seed, r]), seed, r)
              for r, N in enumerate(_batch_sizes(case))]
        return dict(case=case, handles=hs, batch=binding.Batch(hs))
    sy = _system(case, case["N"], seed)
    st = dict(case=case, h=_handle(case, sy, seed))
    if case["kind"] == "embed":
        pos = torch.from_numpy(sy["pos"])
        if case["host"]:
            st["pos"] = pos.pin_memory()
            st["F"] = torch.empty(case["N"], 3, dtype=torch.float32).pin_memory()
        else:
            st["pos"] = pos.cuda()
            st["F"] = torch.empty(case["N"], 3, dtype=torch.float32, device="cuda")
    return st


def _log_line(case, e, w):
    """Energies and virials as one vector: FP64 in the FP64 form, else the form's FP32."""
    return torch.tensor([*e.values(), *w.values()],
                        dtype=torch.float64 if case["precision"] == "fp64" else torch.float32)


def _frame(h):
    """Positions and velocities in single precision, as trajectory files hold them."""
    pos, vel, _ = h.state()
    return torch.from_numpy(pos).float(), torch.from_numpy(vel).float()


def run(state):
    case = state["case"]
    if case["kind"] == "embed":
        h = state["h"]
        h.set_positions(state["pos"])
        if not case["energies"]:
            return {"F": h.forces(0, out=state["F"], energies=False)}
        F, e, w = h.forces(0, out=state["F"], energies=True)
        return {"F": F, "e": _log_line(case, e, w)}
    if case["kind"] == "md":
        h = state["h"]
        h.step(case["steps"])
        pos, vel = _frame(h)
        return {"pos": pos, "vel": vel, "e": _log_line(case, *h.energies())}
    state["batch"].step(case["steps"])
    torch.cuda.current_stream().synchronize()
    return [_frame(h) for h in state["handles"]]


def _work(case, N):
    """One force evaluation: pairs within the cutoff once (LJ 20 flops, erfc-Coulomb 40) or the
    random batch list's directed core and drawn pairs, and two k-space passes (a phase, a sincos
    and the sums: 20 flops each); positions in, forces out."""
    ions = case["comp"] == "ions"
    rho = 200000 / 271.0 ** 3 if ions else (3000 / 32.0 ** 3 if case["frac"] == 1.0 else 0.1)
    sph = 4.0 / 3.0 * math.pi * rho
    Nq = case["frac"] * N
    per = 20.0 + 40.0 * case["frac"] ** 2
    if case.get("r_core"):
        core = sph * case["r_core"] ** 3
        shell = min(sph * case["r_c"] ** 3 - core, case["p_rbl"])
        fl = N * (core + shell) * per
    else:
        fl = 0.5 * N * sph * case["r_c"] ** 3 * per
    return fl + 40.0 * Nq * case["P"]


def work(case):
    if case["kind"] == "embed":
        N = case["N"]
        return {"bytes": N * (24 + 12), "flops": _work(case, N)}
    if case["kind"] == "md":
        N, k = case["N"], case["steps"]
        # each step reads and writes positions, velocities and forces; the frame leaves once
        return {"bytes": k * N * 72 + N * 60, "flops": k * _work(case, N)}
    b, f = 0.0, 0.0
    for N in _batch_sizes(case):
        b += case["steps"] * N * 72 + N * 60
        f += case["steps"] * _work(case, N)
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------------------
# The same results in 64 bits, in plain torch and numpy

def _philox(c, k0, k1):
    """Philox4x32-10 (Salmon et al. 2011) over uint64 arrays holding 32-bit words."""
    M = np.uint64(0xFFFFFFFF)
    a, b, d, e = c
    for r in range(10):
        p0, p1 = a * np.uint64(0xD2511F53), d * np.uint64(0xCD9E8D57)
        x0 = np.uint64((k0 + r * 0x9E3779B9) & 0xFFFFFFFF)
        x1 = np.uint64((k1 + r * 0xBB67AE85) & 0xFFFFFFFF)
        a, b, d, e = ((p1 >> np.uint64(32)) ^ b ^ x0, p1 & M, (p0 >> np.uint64(32)) ^ e ^ x1, p0 & M)
    return a, b, d, e


def _modes(box, alpha, P, seed, replica, step):
    """P modes of exp(-k^2 / 4 alpha), k != 0, by inverse CDF per axis; sum of the weights."""
    T, Ms, Z = [], [], 1.0
    for L in box:
        M = int(math.ceil(L * math.sqrt(4.0 * alpha * 53.0 * math.log(2.0)) / (2.0 * math.pi)))
        w = [math.exp(-((2.0 * math.pi * m / L) ** 2) / (4.0 * alpha)) for m in range(-M, M + 1)]
        z, acc, t = sum(w), 0.0, []
        for x in w:
            acc += x
            t.append(math.floor(acc / z * 2.0 ** 32))
        t[-1] = 1 << 32
        T.append(np.array(t, np.uint64))
        Ms.append(M)
        Z *= z
    m = np.zeros((P, 3), np.int64)
    left = np.arange(P)
    for attempt in range(64):
        z = np.zeros(left.size, np.uint64)
        w = _philox((left.astype(np.uint64), z + np.uint64(attempt), z + np.uint64(step), z),
                    seed & 0xFFFFFFFF, (seed >> 32) ^ replica)
        for d in range(3):
            m[left, d] = np.searchsorted(T[d], w[d], side="right") - Ms[d]
        left = left[(m[left] == 0).all(axis=1)]
        if left.size == 0:
            break
    return m, Z - 1.0


def _candidates(s, box, r):
    """Index pairs (i, j), i != j, in chunks that cover every pair within r (cells, or all)."""
    N, dev = s.shape[0], s.device
    n = [int(math.floor(L / r)) for L in box]
    if min(n) < 3 or N < 2000:
        for a in range(0, N, 4096):
            i = torch.arange(a, min(N, a + 4096), device=dev)
            yield i[:, None], torch.arange(N, device=dev)[None, :]
        return
    c = torch.stack([(s[:, d] * n[d]) >> 32 for d in range(3)], 1)
    key = c[:, 0] + n[0] * (c[:, 1] + n[1] * c[:, 2])
    order = torch.argsort(key)
    nc = n[0] * n[1] * n[2]
    cnt = torch.bincount(key, minlength=nc)
    mx = int(cnt.max())
    start = torch.cumsum(cnt, 0) - cnt
    slot = torch.arange(N, device=dev) - start[key[order]]
    tab = torch.full((nc, mx), -1, dtype=torch.int64, device=dev)
    tab[key[order], slot] = order
    step = max(1, int(1.5e8 / (27 * mx * mx)))
    for a in range(0, nc, step):
        k = torch.arange(a, min(nc, a + step), device=dev)
        x, y, z = k % n[0], (k // n[0]) % n[1], k // (n[0] * n[1])
        near = torch.cat([tab[(x + dx) % n[0] + n[0] * ((y + dy) % n[1] + n[1] * ((z + dz) % n[2]))]
                          for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)], 1)
        yield tab[k][:, :, None], near[:, None, :]


def _wrap32(x):
    return ((x + (1 << 31)) & 0xFFFFFFFF) - (1 << 31)


def _real_pairs(s, box, r):
    """Directed pairs within r, chunk by chunk: i, j, displacement and r^2 (FP64)."""
    h = torch.tensor(box / 2.0 ** 32, dtype=torch.float64, device=s.device)
    for i, j in _candidates(s, box, r):
        i, j = torch.broadcast_tensors(i, j)
        ok = (i >= 0) & (j >= 0) & (i != j)
        i0, j0 = i.clamp(min=0), j.clamp(min=0)
        r2 = torch.zeros(i.shape, dtype=torch.float64, device=s.device)
        for d in range(3):
            r2 += (_wrap32(s[:, d][i0] - s[:, d][j0]).double() * h[d]) ** 2
        at = (ok & (r2 <= r * r)).nonzero(as_tuple=True)
        i, j, r2 = i[at], j[at], r2[at]
        yield i, j, _wrap32(s[i] - s[j]).double() * h, r2


def _pair_terms(sy, u, i, j, d, r2):
    t = sy["types"][i] * sy["nt"] + sy["types"][j]
    e, sg = sy["eps"][t], sy["sig"][t]
    x = (sg * sg / r2) ** 3
    ulj, wlj = 4 * e * (x * x - x), 24 * e * (2 * x * x - x)
    r = r2.sqrt()
    qq = u["C"] * sy["q"][i] * sy["q"][j]
    er = torch.erfc(math.sqrt(u["alpha"]) * r) / r
    uc = qq * er
    wc = qq * (er + 2 * math.sqrt(u["alpha"] / math.pi) * torch.exp(-u["alpha"] * r2))
    return ((wlj + wc) / r2)[:, None] * d, torch.stack([uc, ulj, wc, wlj], 1)


def _canonical(sy, s, box, r, i, j):
    """The random batch list's shell order: i, then the offset cell (dz, dy, dx), (s_x, id)."""
    n = [int(math.floor(L / r)) for L in box]
    off = torch.zeros_like(i)
    for d in (2, 1, 0):
        c = (s[:, d] * n[d]) >> 32
        off = off * 3 + (c[j] - c[i] + 1) % n[d]
    order = torch.argsort(j, stable=True)
    order = order[torch.argsort(s[j[order], 0], stable=True)]
    return order[torch.argsort((i * 27 + off)[order], stable=True)]


def _forces(case, sy, s, seed, replica, step):
    """Forces (N, 3) and the energy and virial sums, in FP64, of one evaluation."""
    u, box, N, dev = _units(case), sy["box"], s.shape[0], s.device
    F = torch.zeros(N, 3, dtype=torch.float64, device=dev)
    en = torch.zeros(4, dtype=torch.float64, device=dev)
    shells = []
    for i, j, d, r2 in _real_pairs(s, box, case["r_c"]):
        if case.get("r_core"):
            sh = r2 > case["r_core"] ** 2
            shells.append((i[sh], j[sh], d[sh], r2[sh]))
            i, j, d, r2 = i[~sh], j[~sh], d[~sh], r2[~sh]
        f, t = _pair_terms(sy, u, i, j, d, r2)
        F.index_add_(0, i, f)
        en += 0.5 * t.sum(0)
    if case.get("r_core"):
        i, j, d, r2 = (torch.cat(x) for x in zip(*shells))
        o = _canonical(sy, s, box, case["r_c"], i, j)
        i, j, d, r2 = i[o], j[o], d[o], r2[o]
        cnt = torch.bincount(i, minlength=N)
        first = torch.cumsum(cnt, 0) - cnt
        p = case["p_rbl"]
        all_ = (cnt[i] <= p).nonzero()[:, 0]
        many = (cnt > p).nonzero()[:, 0]
        ids = many.cpu().numpy().astype(np.uint64)
        zero = np.zeros_like(ids)
        w = []
        for t in range(0, p, 4):
            w += _philox((ids, zero + np.uint64(t // 4), zero + np.uint64(step), zero + np.uint64(1)),
                         seed & 0xFFFFFFFF, (seed >> 32) ^ replica)
        w = torch.from_numpy(np.stack(w[:p], 1).astype(np.int64)).to(dev)
        pick = (first[many][:, None] + ((w * cnt[many][:, None]) >> 32)).reshape(-1)
        at = torch.cat([all_, pick])
        wt = torch.cat([torch.ones(all_.numel(), dtype=torch.float64, device=dev),
                        (cnt[many].double() / p).repeat_interleave(p)])
        f, t = _pair_terms(sy, u, i[at], j[at], d[at], r2[at])
        F.index_add_(0, i[at], f * wt[:, None])
        en += 0.5 * (t * wt[:, None]).sum(0)
        F -= F.mean(0)
    m, S = _modes(box, u["alpha"], case["P"], seed, replica, step)
    k = torch.from_numpy(2 * math.pi * m / box).to(dev)
    k2 = (k * k).sum(1)
    cl = 4 * math.pi * u["C"] * S / (case["P"] * float(np.prod(box)) * k2)
    ch = (sy["q"] != 0).nonzero()[:, 0]
    q, sc, mt = sy["q"][ch], s[ch], torch.from_numpy(m).to(dev)
    at = range(0, ch.numel(), max(1, int(3e7 / case["P"])))

    def phase(a):
        x = (sc[a:a + at.step, None, :] * mt[None]).sum(2) & 0xFFFFFFFF
        return x.double() * (2 * math.pi / 2.0 ** 32)

    re = torch.zeros(case["P"], dtype=torch.float64, device=dev)
    im = torch.zeros_like(re)
    for a in at:
        t = phase(a)
        re += (q[a:a + at.step, None] * torch.cos(t)).sum(0)
        im += (q[a:a + at.step, None] * torch.sin(t)).sum(0)
    for a in at:
        t = phase(a)
        g = cl * (im * torch.cos(t) - re * torch.sin(t))
        F[ch[a:a + at.step]] -= q[a:a + at.step, None] * (g @ k)
    E = 0.5 * cl * (re * re + im * im)
    W = (E * (1 - k2 / (2 * u["alpha"]))).sum()
    self_ = u["C"] * math.sqrt(u["alpha"] / math.pi) * (sy["q"] ** 2).sum()
    real, lj, wr, wl = en
    return F, [real, lj, E.sum(), self_, real + lj + E.sum() - self_], [wr, wl, W, wr + wl + W]


def _on_gpu(sy):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    out = {k: torch.from_numpy(np.ascontiguousarray(sy[k])).to(dev)
           for k in ("q", "mass", "v", "eps", "sig")}
    out["types"] = torch.from_numpy(sy["types"].astype(np.int64)).to(dev)
    return dict(out, box=sy["box"], nt=int(round(math.sqrt(sy["eps"].size)))), \
        torch.from_numpy(sy["s"].astype(np.int64)).to(dev)


def _trajectory(case, sy, seed, replica=0):
    """The frame and log line after case["steps"] Verlet steps on the 2^-32 grid."""
    u = _units(case)
    sy, s = _on_gpu(sy)
    v, im = sy["v"].clone(), (1.0 / sy["mass"])[:, None]
    N, dt = s.shape[0], u["dt"]
    grid = torch.tensor(dt * 2.0 ** 32 / sy["box"], dtype=torch.float64, device=s.device)
    Nf, kT = 3.0 * N - 3.0, u["kB"] * u["T"]
    Q = Nf * kT * u["tau"] ** 2
    xi = 0.0

    def half(x, K2):
        x += 0.25 * dt * (K2 - Nf * kT) / Q
        sc = math.exp(-x * 0.5 * dt)
        return x + 0.25 * dt * (K2 * sc * sc - Nf * kT) / Q, sc

    def kinetic():
        return float(0.5 * (sy["mass"][:, None] * v * v).sum() / u["kappa"])

    F, en, w = _forces(case, sy, s, seed, replica, 0)
    for k in range(case["steps"]):
        if case.get("nvt"):
            xi, sc = half(xi, 2 * kinetic())
            v *= sc
        v += F * im * (0.5 * dt * u["kappa"])
        s = (s + torch.round(v * grid).to(torch.int64)) & 0xFFFFFFFF
        F, en, w = _forces(case, sy, s, seed, replica, k + 1)
        v += F * im * (0.5 * dt * u["kappa"])
        if case.get("nvt"):
            xi, sc = half(xi, 2 * kinetic())
            v *= sc
    pos = s.double() * torch.tensor(sy["box"] / 2.0 ** 32, dtype=torch.float64, device=s.device)
    e = [float(x) for x in en] + [kinetic()] + [float(x) for x in w]
    return pos.cpu(), v.cpu(), torch.tensor(e, dtype=torch.float64)


def exact(case, seed):
    if case["kind"] == "batch":
        if case["n"] * case["hi"] * case["steps"] > 6e6:
            return None
        return [_trajectory(case, _system(case, N, [seed, r]), 1 + seed, r)[:2]
                for r, N in enumerate(_batch_sizes(case))]
    N, box = case["N"], case["box"]
    evaluations = case["steps"] + 1 if case["kind"] == "md" else 1
    # (about 20 seconds of FP64 pairs and phases)
    if N * evaluations * (420 + 2 * case["frac"] * case["P"]) > 8e9:
        return None
    sy = _system(case, N, seed)
    if case["kind"] == "md":
        pos, v, e = _trajectory(case, sy, 1 + seed)
        return {"pos": pos, "vel": v, "e": e}
    v = float(0.5 * (sy["mass"][:, None] * sy["v"] ** 2).sum() / _units(case)["kappa"])
    g, s = _on_gpu(sy)
    F, en, w = _forces(case, g, s, 1 + seed, 0, 0)
    out = {"F": F.cpu()}
    if case["energies"]:
        out["e"] = torch.tensor([float(x) for x in en] + [v] + [float(x) for x in w],
                                dtype=torch.float64)
    return out
