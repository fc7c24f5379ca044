"""Performance cases: the calls a user of the SPME library makes, over the sizes it accepts.

A case is one call (or the short chain of calls one time step makes) through the ctypes binding:

  compute   pme_compute: synchronous evaluation on device arrays (a program that needs E after every call)
  enqueue   pme_enqueue: asynchronous evaluation, energy and virial into device memory (an MD loop)
  stream    pme_enqueue_host on page-locked arrays, several steps in flight (host-side integrator)
  batch     pme_batch_enqueue: many uneven systems per call (replica / ensemble work)
  real      pme_real_compute: synchronous real-space and self terms
  ewald     pme_enqueue + pme_real_enqueue(accumulate): one step's full electrostatics, host-driven
  steps     pme_run_steps with the real-space term: a chunk of device-resident MD steps
  noalloc   pme_compute_noalloc: one small system, no device allocation, no plan

Reciprocal-only cases use the repository's benchmark inputs (molecules placed uniformly at random); cases with
the real-space term use a simulation-like box (molecules on a jittered lattice), since random placement has
overlapping atoms whose pair forces would be all that a comparison sees.
"""
import math
import weakref

import torch

from paper_2009_12617_gb300 import pme

BETA = 0.34
DENSITY = 0.1  # atoms / A^3, liquid water
DEV = "cuda:0"
SMOOTH = [8, 10, 12, 16, 18, 20, 24, 30, 32, 36, 40, 48, 50, 54, 60, 64, 72, 80, 90, 96, 100, 108, 120, 128]


def _case(name, kind, n, K, p, **more):
    c = {"kind": kind, "n": n, "K1": K[0], "K2": K[1], "K3": K[2], "p": p, "skew": False}
    if name:
        c["name"] = name
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: 2048 atoms, 32^3, one evaluation per host round trip; latency is everything
        _case("compute_2k_32", "compute", 2048, (32, 32, 32), 4),
        # the benchmark's headline: 65536 atoms, 64^3, p = 4, evaluations back to back
        _case("enqueue_65k_64", "enqueue", 65536, (64, 64, 64), 4),
        # the largest configured system: 262144 atoms, 128^3, p = 6
        _case("enqueue_262k_128", "enqueue", 262144, (128, 128, 128), 6),
        # a ragged mid-size system: triclinic cell, mesh edges that are no powers of two, odd order
        _case("enqueue_24k_tri_p5", "enqueue", 23901, (54, 60, 72), 5, skew=True),
        # a fine mesh at the highest order (accuracy runs): mixed edges, p = 8
        _case("enqueue_80k_fine_p8", "enqueue", 80001, (90, 96, 100), 8),
        # positions from and forces to page-locked host memory, the headline system
        _case("stream_65k_64", "stream", 65536, (64, 64, 64), 4),
        # 64 uneven systems of 1k-33k atoms, meshes 32^3-64^3, one graph per call
        _case("batch_64_uneven", "batch", 0, (0, 0, 0), 4, count=64, lo=1024, hi=32768),
        # real-space and self terms of the small system, one host round trip per call
        _case("real_2k", "real", 2048, (0, 0, 0), 0, rcut=9.0),
        # one time step's full electrostatics of the headline system, driven by the host
        _case("ewald_65k", "ewald", 65536, (64, 64, 64), 4, rcut=9.0),
        # the same at high order and a long cutoff, an odd atom count and a triclinic cell
        _case("ewald_151k_tri_p6", "ewald", 151009, (96, 90, 108), 6, rcut=12.0, skew=True),
        # a chunk of device-resident MD of a small protein-sized box: reciprocal + real space + leapfrog
        _case("steps_8k_x32", "steps", 8190, (40, 40, 40), 4, rcut=9.0, steps=32),
        # allocation-free evaluation of the small system
        _case("noalloc_2k_32", "noalloc", 2048, (32, 32, 32), 4),
    ]


def _edge(rng, length, p, most=128):
    """A mesh edge of 0.95-1.45 A spacing for a cell width, at least p and 8 points."""
    want = length / rng.uniform(0.95, 1.45)
    fit = [k for k in SMOOTH if k <= most and k >= max(8, p)]
    return min(fit, key=lambda k: abs(math.log(k / want)))


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["compute", "enqueue", "enqueue", "enqueue", "stream", "batch", "real", "real", "ewald", "ewald", "steps",
                       "noalloc"])
    skew = rng.random() < 0.3 and kind not in ("batch",)
    if kind == "batch":
        lo = _logint(rng, 700, 2500)
        return _case(None, kind, 0, (0, 0, 0), 4, count=rng.randint(5, 60), lo=lo, hi=_logint(rng, 2 * lo, 30000))
    p = rng.choice([4, 4, 5, 6, 8])
    if kind == "noalloc":
        p = rng.choice([4, 4, 6, 8])
        n = _logint(rng, 300, 5000)
        lim = 32
    else:
        n = _logint(rng, 600, {"real": 100000, "ewald": 100000, "steps": 20000, "compute": 120000}.get(kind, 200000 if p < 8 else 80000))
        lim = 128
    if n % 3 == 1 and n < 7:
        n += 1
    L = (n / DENSITY) ** (1.0 / 3.0)
    K = (0, 0, 0) if kind == "real" else tuple(_edge(rng, L, p, lim) for _ in range(3))
    more = {"skew": skew}
    if kind in ("real", "ewald", "steps"):
        more["rcut"] = round(min(rng.uniform(7.0, 12.0), 0.8 * L), 3)
    if kind == "steps":
        more["steps"] = rng.randint(3, 40)
    return _case(None, kind, n, K, 0 if kind == "real" else p, **more)


# ---------------------------------------------------------------------------------------------------------
# inputs


def _box(case, n):
    """Cell rows a, b, c (float64) of volume n / DENSITY; a triclinic one keeps the volume."""
    L = (n / DENSITY) ** (1.0 / 3.0)
    if not case.get("skew"):
        return torch.diag(torch.full((3,), L, dtype=torch.float64))
    return torch.tensor([[1.05 * L, 0.0, 0.0], [0.12 * L, L / 1.05, 0.0], [-0.08 * L, 0.15 * L, L]], dtype=torch.float64)


def _molecules(n, box, g, lattice):
    """Positions (n, 3) and charges (n) of a neutral water-like box: triplets O -0.834, H +0.417 (0.9572 A,
    104.52 degrees, random orientation) and +-1 ion pairs that make up the count. Positions are not wrapped."""
    t, pairs = {0: (n // 3, 0), 2: (n // 3, 1), 1: (n // 3 - 1, 2)}[n % 3]
    sites = t + 2 * pairs
    o = dict(device=DEV, dtype=torch.float64)
    if lattice:
        m = math.ceil(sites ** (1.0 / 3.0))
        at = torch.randperm(m ** 3, generator=g, device=DEV)[:sites]
        cell = torch.stack([at // (m * m), (at // m) % m, at % m], 1).double()
        frac = (cell + 0.5 + 0.16 * (torch.rand(sites, 3, generator=g, **o) - 0.5)) / m
    else:
        frac = torch.rand(sites, 3, generator=g, **o)
    base = frac @ box.to(DEV)
    h = math.radians(104.52) / 2
    local = 0.9572 * torch.tensor([[0, 0, 0], [math.sin(h), 0, math.cos(h)], [-math.sin(h), 0, math.cos(h)]], **o)
    w = torch.randn(t, 4, generator=g, **o)
    w = w / w.norm(dim=1, keepdim=True)
    a, b, c, d = w.unbind(1)
    R = torch.stack([1 - 2 * (c * c + d * d), 2 * (b * c - d * a), 2 * (b * d + c * a), 2 * (b * c + d * a), 1 - 2 * (b * b + d * d),
                     2 * (c * d - b * a), 2 * (b * d - c * a), 2 * (c * d + b * a), 1 - 2 * (b * b + c * c)], 1).view(t, 3, 3)
    pos = torch.cat([(base[:t, None] + torch.einsum("tij,aj->tai", R, local)).reshape(-1, 3), base[t:]])
    q = torch.cat([torch.tensor([-0.834, 0.417, 0.417], **o).repeat(t), torch.tensor([1.0, -1.0], **o).repeat(pairs)])
    return pos.float().contiguous(), q.float().contiguous()


def _systems(case, seed):
    """[(pos, q, box, K, p)] of the case, on the GPU."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 13)
    if case["kind"] != "batch":
        n = case["n"]
        box = _box(case, n)
        return [(*_molecules(n, box, g, case["kind"] in ("real", "ewald", "steps")), box, (case["K1"], case["K2"], case["K3"]), case["p"])]
    # the sizes belong to the case, the atoms to the seed
    r = torch.Generator()
    r.manual_seed(case["count"] * 1000003 + case["lo"])
    u = torch.rand(case["count"], generator=r, dtype=torch.float64).tolist()
    out = []
    for x in u:
        n = int(round(case["lo"] * (case["hi"] / case["lo"]) ** x))
        box = _box(case, n)
        L = float(box[0, 0])
        K = next((k for k in (32, 40, 48, 64, 80) if L / k <= 1.4), 80)
        out.append((*_molecules(n, box, g, False), box, (K, K, K), case["p"]))
    return out


def _motion(case, seed, n):
    """Velocities and inverse masses of a steps case: thermal speeds, a step of about a femtosecond."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 104729 + 7)
    vel = 0.5 * torch.randn(n, 3, generator=g, device=DEV)
    inv_mass = torch.full((n,), 1.0 / 16.0, device=DEV)
    return vel.contiguous(), inv_mass


DT = 0.01


# ---------------------------------------------------------------------------------------------------------
# what a program keeps, and one pass


class _Real:
    def __init__(self, box, rcut, stream):
        self.handle = pme.pme_real_create(box, BETA, rcut, stream)
        weakref.finalize(self, pme.pme_real_destroy, self.handle)


class _Batch:
    def __init__(self, plans, n, stream):
        self.plans = plans  # they outlive the batch
        self.handle = pme.pme_batch_create([p.handle for p in plans], n, stream)

    def __del__(self):
        pme.pme_batch_destroy(self.handle)


def _pinned(shape, dtype):
    return torch.empty(shape, dtype=dtype).pin_memory().numpy()


def prepare(case, seed):
    kind = case["kind"]
    systems = _systems(case, seed)
    stream = torch.cuda.current_stream()
    s = {"kind": kind}
    if kind == "batch":
        plans = [pme.Plan(K, p, BETA, box.numpy(), stream) for _, _, box, K, p in systems]
        s["batch"] = _Batch(plans, [x[1].shape[0] for x in systems], stream)
        s["pos"] = torch.cat([x[0] for x in systems])
        s["q"] = torch.cat([x[1] for x in systems])
        s["forces"] = torch.empty_like(s["pos"])
        s["ev"] = torch.zeros(len(systems), 7, dtype=torch.float64, device=DEV)
        return s
    pos, q, box, K, p = systems[0]
    s.update(pos=pos, q=q, forces=torch.empty_like(pos), box=box.numpy(), K=K, p=p)
    if kind == "noalloc":
        return s
    if kind != "real":
        s["plan"] = pme.Plan(K, p, BETA, s["box"], stream)
        pme.pme_reserve(s["plan"].handle, q.shape[0])
        s["ev"] = torch.zeros(7, dtype=torch.float64, device=DEV)
    if kind in ("real", "ewald", "steps"):
        s["rs"] = _Real(s["box"], case["rcut"], stream)
        pme.pme_real_reserve(s["rs"].handle, q.shape[0])
        s["ev_real"] = torch.zeros(8, dtype=torch.float64, device=DEV)
    if kind == "steps":
        s["vel0"], s["inv_mass"] = _motion(case, seed, q.shape[0])
        s["start"], s["vel"], s["steps"] = pos.clone(), s["vel0"].clone(), case["steps"]
        s["ev_steps"] = torch.zeros(case["steps"], 15, dtype=torch.float64, device=DEV)
    if kind == "stream":
        n = q.shape[0]
        s["hpos"], s["hq"] = _pinned((n, 3), torch.float32), _pinned(n, torch.float32)
        s["hpos"][:], s["hq"][:] = pos.cpu().numpy(), q.cpu().numpy()
        s["hforces"], s["hresult"], s["ticket"] = _pinned((n, 3), torch.float32), _pinned(8, torch.float64), -1
    return s


def run(s):
    kind = s["kind"]
    if kind == "batch":
        pme.pme_batch_enqueue(s["batch"].handle, s["pos"], s["q"], s["forces"], s["ev"])
        return {"forces": s["forces"], "ev": s["ev"]}
    if kind == "noalloc":
        e, vir = pme.pme_compute_noalloc(s["K"], s["p"], BETA, s["box"], s["pos"], s["q"], s["forces"])
        return {"forces": s["forces"], "e": e, "virial": vir}
    if kind == "compute":
        f, e, vir = s["plan"].compute(s["pos"], s["q"], s["forces"])
        return {"forces": f, "e": e, "virial": vir}
    if kind == "enqueue":
        s["plan"].enqueue(s["pos"], s["q"], s["forces"], s["ev"])
        return {"forces": s["forces"], "ev": s["ev"]}
    if kind == "stream":  # before a set of buffers is used again, its last step has to be out
        if s["ticket"] >= 0:
            pme.pme_host_wait(s["plan"].handle, s["ticket"])
        s["ticket"] = pme.pme_enqueue_host(s["plan"].handle, s["hpos"], s["hq"], s["hforces"], s["hresult"])
        return {"forces": s["hforces"], "result": s["hresult"]}
    if kind == "real":
        e, es, vir = pme.pme_real_compute(s["rs"].handle, s["pos"], s["q"], s["forces"])
        return {"forces": s["forces"], "e": e, "self": es, "virial": vir}
    if kind == "ewald":
        s["plan"].enqueue(s["pos"], s["q"], s["forces"], s["ev"])
        pme.pme_real_enqueue(s["rs"].handle, s["pos"], s["q"], s["forces"], True, s["ev_real"])
        return {"forces": s["forces"], "ev": s["ev"], "ev_real": s["ev_real"]}
    # steps: every pass starts from the same saved state, as a rerun from a checkpoint does
    s["pos"].copy_(s["start"])
    s["vel"].copy_(s["vel0"])
    pme.pme_run_steps(s["plan"].handle, s["pos"], s["vel"], s["q"], s["forces"], DT, s["steps"], s["rs"].handle, s["inv_mass"],
                      s["ev_steps"])
    return {"pos": s["pos"], "vel": s["vel"], "forces": s["forces"], "ev_steps": s["ev_steps"]}


# ---------------------------------------------------------------------------------------------------------
# what a pass cannot do without


def work(case):
    """Bytes: positions and charges in, forces (and energies) out, and the plan's influence values read once (8
    bytes per half-spectrum point); flops: spreading and interpolation over the p^3 support, the two real
    transforms, the influence multiply, and the pairs inside the cutoff (each counted once)."""
    def recip(n, K, p):
        N = K[0] * K[1] * K[2]
        return {"bytes": 28.0 * n + 8.0 * K[0] * K[1] * (K[2] // 2 + 1) + 56,
                "flops": n * (8.0 * p ** 3 + 18.0 * p * p) + 5.0 * N * math.log2(N) + 20.0 * K[0] * K[1] * (K[2] // 2 + 1)}

    def real(n, rcut):
        pairs = 0.5 * n * DENSITY * 4.0 / 3.0 * math.pi * rcut ** 3
        return {"bytes": 28.0 * n + 64, "flops": 60.0 * pairs}

    def add(a, b, times=1):
        return {k: a[k] + times * b[k] for k in a}

    kind, zero = case["kind"], {"bytes": 0.0, "flops": 0.0}
    if kind == "batch":
        r = torch.Generator()
        r.manual_seed(case["count"] * 1000003 + case["lo"])
        total = zero
        for x in torch.rand(case["count"], generator=r, dtype=torch.float64).tolist():
            n = int(round(case["lo"] * (case["hi"] / case["lo"]) ** x))
            L = (n / DENSITY) ** (1.0 / 3.0)
            K = next((k for k in (32, 40, 48, 64, 80) if L / k <= 1.4), 80)
            total = add(total, recip(n, (K, K, K), case["p"]))
        return total
    n, K = case["n"], (case["K1"], case["K2"], case["K3"])
    if kind == "real":
        return real(n, case["rcut"])
    w = recip(n, K, case["p"])
    if kind == "ewald":
        w = add(w, real(n, case["rcut"]))
    if kind == "steps":
        w = add(zero, add(add(w, real(n, case["rcut"])), {"bytes": 48.0 * n, "flops": 12.0 * n}), case["steps"])
    return w


def tolerance(case):
    """About four times the distance of the FP32 results from the same in 64 bits: 1e-6 for one evaluation's forces;
    3e-5 for the forces at the end of a trajectory, where FP32 positions of unbonded atoms have drifted apart."""
    return {"rel": 1.2e-4 if case["kind"] == "steps" else 4e-6}


# ---------------------------------------------------------------------------------------------------------
# the same in 64 bits, plain torch


def _splines(w, p):
    """M_p(w + j) and its derivative, j < p: (n, p) each."""
    th = [w, 1.0 - w]
    for k in range(3, p + 1):
        if k == p:
            d = [th[0]] + [th[j] - th[j - 1] for j in range(1, p - 1)] + [-th[p - 2]]
        z = torch.zeros_like(w)
        up = lambda j: th[j] if 0 <= j < k - 1 else z  # noqa: E731
        th = [((w + j) * up(j) + (k - j - w) * up(j - 1)) / (k - 1) for j in range(k)]
    return torch.stack(th, 1), torch.stack(d, 1)


def _moduli(K, p):
    knots = _splines(torch.zeros(1, dtype=torch.float64, device=DEV), p)[0][0, 1:]
    m = torch.arange(K, device=DEV, dtype=torch.float64)
    k = torch.arange(p - 1, device=DEV, dtype=torch.float64)
    z = (knots * torch.exp(2j * math.pi * m[:, None] * k[None, :] / K)).sum(1).abs() ** 2
    if p % 2:  # the denominator vanishes at K/2 for odd orders: the mean of its neighbours
        z[K // 2] = 0.5 * (z[K // 2 - 1] + z[K // 2 + 1])
    return 1.0 / z


PAIRS = [(0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)]


class _Recip64:
    def __init__(self, box, K, p):
        self.K, self.p = K, p
        box = box.to(DEV)
        self.recip = torch.linalg.inv(box).T.contiguous()  # rows a*
        vol = torch.linalg.det(box).abs()
        # index m of torch's transform is frequency -m of exp(+2 pi i m k / K)
        mt = []
        for k in K:
            i = (k - torch.arange(k, device=DEV)) % k
            mt.append(torch.where(2 * i <= k, i, i - k).double())
        mv = (mt[0][:, None, None, None] * self.recip[0] + mt[1][None, :, None, None] * self.recip[1]
              + mt[2][None, None, :, None] * self.recip[2])
        m2 = mv.square().sum(-1)
        m2[0, 0, 0] = 1.0
        b = [_moduli(k, p) for k in K]
        b = [x[(k - torch.arange(k, device=DEV)) % k] for x, k in zip(b, K)]
        fac = math.pi ** 2 / BETA ** 2
        self.bc = b[0][:, None, None] * b[1][None, :, None] * b[2][None, None, :] * torch.exp(-fac * m2) / (math.pi * vol * m2)
        self.bc[0, 0, 0] = 0.0
        self.mv, self.f = mv, 2.0 * (1.0 + fac * m2) / m2

    def __call__(self, pos, q):
        K, p = self.K, self.p
        Kt = torch.tensor(K, device=DEV, dtype=torch.float64)
        pos, q = pos.double(), q.double()
        s = pos @ self.recip.T
        u = (s - s.floor()) * Kt
        base = u.floor()
        th, dth, idx = [], [], []
        for a in range(3):
            t, d = _splines(u[:, a] - base[:, a], p)
            th.append(t)
            dth.append(d)
            idx.append((base[:, a, None].long() - torch.arange(p, device=DEV)) % K[a])
        Q = torch.zeros(K[0] * K[1] * K[2], dtype=torch.float64, device=DEV)
        at = []
        for c in range(0, q.shape[0], 32768):
            x = slice(c, c + 32768)
            flat = ((idx[0][x, :, None, None] * K[1] + idx[1][x, None, :, None]) * K[2] + idx[2][x, None, None, :]).reshape(-1, p ** 3)
            w = torch.einsum("n,ni,nj,nk->nijk", q[x], th[0][x], th[1][x], th[2][x])
            Q.index_add_(0, flat.reshape(-1), w.reshape(-1))
            at.append((x, flat))
        Qh = torch.fft.fftn(Q.view(K))
        em = 0.5 * self.bc * (Qh.real ** 2 + Qh.imag ** 2)
        vir = [((em * (1.0 if a == b else 0.0)) - em * self.f * self.mv[..., a] * self.mv[..., b]).sum() for a, b in PAIRS]
        phi = (torch.fft.ifftn(self.bc * Qh).real * Q.numel()).reshape(-1)
        g = torch.empty_like(pos)
        for x, flat in at:
            ph = phi[flat].view(-1, p, p, p)
            g[x, 0] = torch.einsum("ni,nj,nk,nijk->n", dth[0][x], th[1][x], th[2][x], ph)
            g[x, 1] = torch.einsum("ni,nj,nk,nijk->n", th[0][x], dth[1][x], th[2][x], ph)
            g[x, 2] = torch.einsum("ni,nj,nk,nijk->n", th[0][x], th[1][x], dth[2][x], ph)
        return -q[:, None] * ((g * Kt) @ self.recip), torch.stack([em.sum(), *vir])


def _real64(pos, q, box, rcut):
    """All pairs, nearest image (and its neighbours where the cutoff passes half the cell): forces, (E, self, virial)."""
    box = box.to(DEV)
    inv = torch.linalg.inv(box)
    wide = bool((rcut * inv.T.norm(dim=1) > 0.5).any())
    shifts = [(i, j, k) for i in (-1, 0, 1) for j in (-1, 0, 1) for k in (-1, 0, 1)] if wide else [(0, 0, 0)]
    pos, q = pos.double(), q.double()
    n = q.shape[0]
    F = torch.zeros_like(pos)
    E = torch.zeros((), dtype=torch.float64, device=DEV)
    V = torch.zeros(6, dtype=torch.float64, device=DEV)
    rows = max(1, 24_000_000 // n)
    for c in range(0, n, rows):
        x = slice(c, min(n, c + rows))
        # candidate pairs in 32 bits with slack, then the pairs themselves in 64
        df = (pos[x, None, :] - pos[None, :, :]).float()
        fr = df @ inv.float()
        df = (fr - fr.round()) @ box.float()
        for sh in shifts:
            off = torch.tensor(sh, dtype=torch.float64, device=DEV) @ box
            near = ((df + off.float()).square().sum(-1) <= (rcut + 1e-2) ** 2).nonzero()
            i, j = near[:, 0] + c, near[:, 1]
            d = pos[i] - pos[j]
            fr64 = d @ inv
            # rounded as above, so that each image is met once
            d = (fr64 - fr[near[:, 0], near[:, 1]].round().double()) @ box + off
            r2 = d.square().sum(-1)
            keep = (r2 <= rcut * rcut) & (r2 > 0)
            i, j, d, r2 = i[keep], j[keep], d[keep], r2[keep]
            r = r2.sqrt()
            er = q[i] * q[j] * torch.special.erfc(BETA * r) / r
            f = (er + q[i] * q[j] * (2 * BETA / math.sqrt(math.pi)) * torch.exp(-BETA * BETA * r2)) / r2
            F.index_add_(0, i, f[:, None] * d)
            E += 0.5 * er.sum()
            for k, (a, b) in enumerate(PAIRS):
                V[k] += 0.5 * (f * d[:, a] * d[:, b]).sum()
    return F, E, -BETA / math.sqrt(math.pi) * q.square().sum(), V


def exact(case, seed):
    kind = case["kind"]
    if kind == "steps" and case["steps"] * case["n"] ** 2 > 4e9:
        return None
    systems = _systems(case, seed)
    if kind == "batch":
        got = [_Recip64(box, K, p)(pos, q) for pos, q, box, K, p in systems]
        return {"forces": torch.cat([f for f, _ in got]), "ev": torch.stack([ev for _, ev in got])}
    pos, q, box, K, p = systems[0]
    if kind == "real":
        F, e, es, v = _real64(pos, q, box, case["rcut"])
        return {"forces": F, "e": float(e), "self": float(es), "virial": v}
    recip = _Recip64(box, K, p)
    if kind == "steps":
        vel, inv_mass = _motion(case, seed, q.shape[0])
        pos, vel, inv_mass = pos.double(), vel.double(), inv_mass.double()
        rows = []
        for _ in range(case["steps"]):
            F, ev = recip(pos, q)
            Fr, e, es, v = _real64(pos, q, box, case["rcut"])
            F = F + Fr
            rows.append(torch.cat([ev, torch.stack([e, es]), v]))
            vel = vel + F * inv_mass[:, None] * DT
            pos = pos + vel * DT
        return {"pos": pos, "vel": vel, "forces": F, "ev_steps": torch.stack(rows)}
    F, ev = recip(pos, q)
    if kind == "ewald":
        Fr, e, es, v = _real64(pos, q, box, case["rcut"])
        return {"forces": F + Fr, "ev": ev, "ev_real": torch.cat([torch.stack([e, es]), v])}
    if kind == "stream":
        return {"forces": F, "result": torch.cat([ev, torch.zeros(1, dtype=torch.float64, device=DEV)])}
    if kind == "enqueue":
        return {"forces": F, "ev": ev}
    return {"forces": F, "e": float(ev[0]), "virial": ev[1:]}
