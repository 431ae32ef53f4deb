"""Performance cases of the Ito-KMC streamer library: what a user's program has
it do, through the C ABI (include/itokmc.h) and its ctypes binding.

Five kinds of pass:

``steps``      A run of whole time steps from a given plasma state that lies in
               device memory (a restart, a coupled code, an ensemble sweep):
               the particles, ion counts and field are handed to the handle,
               ``itokmc_step`` advances them and the densities are read back
               into pinned host memory.
``transport``  The transport stage of a running simulation (interpolation,
               push, sort, deposit): the subject of the headline metric.
``kmc``        The chemistry stage on a transported state.
``field``      The field of a charge distribution on a handle (the initial
               field of a run, or of the next member of a parameter sweep):
               two ion distributions in turn, so that every solve is a new one.
``noalloc``    The field solve on caller memory for a program that owns its
               device memory.

States are made on the GPU from the seed alone: Gaussian blobs (the small and
ensemble configurations'), discharge channels with Gaussian radial profiles
and positive heads (the streamer configuration's geometry, paper_2307_01797_gb300.synth),
the discharge tree's four electron seeds, or a uniform slab (the count-pinned sweep).
"""
import ctypes
import math

import torch

from paper_2307_01797_gb300 import itokmc, synth

Q_E = 1.602176634e-19
EPS0 = 8.8541878128e-12
FRAC_BITS = 10


def listed():
    return [
        # one step of a tiny run and its particles on the host: a unit test, a
        # first try, a diagnostic after every step; latency and launches
        dict(name="step_32_fp64_particles", kind="steps", n=32, physics="small", form="fp64", state="blob",
             particles=20000, realizations=1, steps=1, read="particles"),
        # the small configuration (64^3, ppc 8): ten FP64 steps between outputs
        dict(name="step_64_fp64", kind="steps", n=64, physics="small", form="fp64", state="blob",
             particles=160000, realizations=1, steps=10, read="densities"),
        # the same in the mixed form with replayed steps, as a launch-bound run would be set up
        dict(name="step_64_mixed_graph", kind="steps", n=64, physics="small", form="mixed", state="blob",
             particles=160000, realizations=1, steps=10, read="densities", graph=True),
        # a program with its own device memory that needs the field of a charge on 64^3
        dict(name="field_64_noalloc_fp64", kind="noalloc", n=64, physics="small", form="fp64"),
        # the chemistry of a channel with recombination, on the ensemble member's grid
        dict(name="kmc_128_recombination_fp64", kind="kmc", n=128, physics="member", form="fp64", state="tree",
             particles=6000000, realizations=1, recombination=True),
        # one semi-implicit step (the paper's own coupling) on the ensemble member's grid
        dict(name="semi_128_fp64", kind="steps", n=128, physics="member", form="fp64", state="tree",
             particles=6000000, realizations=1, steps=1, read="densities", coupling="semi"),
        # an ensemble sweep: 16 members of the ensemble configuration batched in one handle
        dict(name="ensemble_16x128_mixed", kind="steps", n=128, physics="member", form="mixed", state="blob",
             particles=400000, realizations=16, steps=2, read="densities"),
        # the field of a charge on the streamer configuration's grid, FP64
        dict(name="field_256_fp64", kind="field", n=256, physics="streamer", form="fp64", state="tree",
             particles=20000000, realizations=1),
        # the headline metric's subject on its configuration: push, sort and deposit, FP64
        dict(name="transport_256_fp64", kind="transport", n=256, physics="streamer", form="fp64", state="tree",
             particles=60000000, realizations=1),
        # the headline run, both forms: two steps of the streamer configuration between outputs
        dict(name="step_256_fp64", kind="steps", n=256, physics="streamer", form="fp64", state="tree",
             particles=60000000, realizations=1, steps=2, read="densities"),
        dict(name="step_256_mixed", kind="steps", n=256, physics="streamer", form="mixed", state="tree",
             particles=60000000, realizations=1, steps=2, read="densities"),
        # the discharge tree's grid (512^3, ppc 64) early in its life, mixed form: bound by the cells
        dict(name="tree_512_mixed", kind="steps", n=512, physics="tree", form="mixed", state="seeds",
             particles=8400000, realizations=1, steps=2, read="densities"),
    ]


# largest particle count drawn per grid size
_MOST = {32: 60000, 64: 900000, 128: 7000000, 256: 50000000}


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["steps", "steps", "steps", "transport", "transport", "kmc", "field", "noalloc"])
    form = rng.choice(["fp64", "mixed"])
    if kind == "noalloc":
        return dict(kind=kind, n=rng.choice([16, 32, 64]), physics=rng.choice(["small", "member", "streamer"]),
                    form=form, charge=round(rng.uniform(0.3, 2.0), 3))
    n = rng.choice([32, 64, 128, 256])
    physics = rng.choice(["small", "member", "streamer"])
    state = rng.choice(["blob", "tree", "slab"])
    case = dict(kind=kind, n=n, physics=physics, form=form, state=state,
                particles=_log(rng, _MOST[n] // 40, _MOST[n]), realizations=1)
    if kind == "steps":
        case["steps"] = rng.choice([1, 2, 3])
        case["read"] = "particles" if n == 32 else "densities"
        option = rng.choice(["", "", "realizations", "graph", "recombination", "mobile_ions", "semi"])
        if option == "realizations" and n <= 128:
            case["realizations"] = rng.choice([2, 3, 5, 7])
            case["particles"] = max(1000, case["particles"] // 8)
        elif option in ("graph", "recombination"):
            case[option] = True
        elif option == "mobile_ions" and n <= 128:
            case[option] = True
        elif option == "semi":
            case.update(form="fp64", coupling="semi")
    elif kind == "kmc":
        case["recombination"] = rng.random() < 0.5
        if n == 256:
            case["particles"] //= 3
    return case


# --------------------------------------------------------------------------- inputs
def _physics(case):
    ph = {"small": synth.physics_small, "member": synth.physics_ensemble_member,
          "streamer": synth.physics_streamer, "tree": synth.physics_tree}[case["physics"]](case["n"])
    if case.get("recombination"):
        ph = synth.with_recombination(ph)
    if case.get("mobile_ions"):
        ph = synth.with_mobile_ions(ph)
        ph["mobile_ions"] = True
    return ph


def _rng(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _uniform(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64).clamp_(1e-9, 1.0 - 1e-9)


def _centres(ph):
    n, h = ph["n"], synth.cell_size(ph)
    c = ph["lo"][0] + (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) * h
    return c.view(1, 1, n), c.view(1, n, 1), c.view(n, 1, 1)


def _electrons(ph, case, seed, member, g):
    """Expected electrons per cell, shape (n, n, n) [k, j, i], and the positions
    of the positive heads."""
    n, h = ph["n"], synth.cell_size(ph)
    L = n * h
    X, Y, Z = _centres(ph)
    want = case["particles"]
    if case["state"] == "blob":
        # a Gaussian ball near the anode, of a radius that holds about `want` superparticles
        peak = min((1e18 if case["physics"] == "small" else 1e19) * h ** 3, 2e8)
        r = (3.0 * want / (4.0 * math.pi * 0.9 * ph["ppc"])) ** (1.0 / 3.0) * h
        sigma = min(r / math.sqrt(2.0 * math.log(max(peak, 2.0))), 0.2 * L)
        u = torch.rand(3, generator=torch.Generator().manual_seed(seed * 1000 + member), dtype=torch.float64)
        c = [float(0.45 + 0.1 * u[0]) * L, float(0.45 + 0.1 * u[1]) * L, float(0.6 + 0.15 * u[2]) * L]
        lam = peak * torch.exp(-((X - c[0]) ** 2 + (Y - c[1]) ** 2 + (Z - c[2]) ** 2) / (2 * sigma * sigma))
        return lam, []
    if case["state"] == "seeds":
        # the discharge tree's four electron seeds
        u = torch.rand(4, 3, generator=torch.Generator().manual_seed(seed * 1000 + member), dtype=torch.float64)
        lam = torch.zeros((n, n, n), device="cuda", dtype=torch.float64)
        for k in range(4):
            c = [L / 2 + (5e-3 if k & 1 else -5e-3), L / 2 + (5e-3 if k & 2 else -5e-3), 0.9 * L]
            d2 = sum((v - (c[q] + float(u[k, q] - 0.5) * 4 * h)) ** 2 for q, v in enumerate((X, Y, Z)))
            lam += torch.exp(d2.mul_(-1.0 / (2 * 3e-4 ** 2))).mul_(5e18 * h ** 3)
        return lam, []
    n_ch = min(1e19, 2e8 / h ** 3)
    sigma_r = 0.025 * L
    segs, _ = synth.streamer_tree_geometry(ph, want, seed=int(seed) % 100000 + 7 * member, n_ch=n_ch, sigma_r=sigma_r)
    lam = torch.zeros((n, n, n), device="cuda", dtype=torch.float64)
    for a, b in segs:
        ab = [float(b[q] - a[q]) for q in range(3)]
        aa = sum(v * v for v in ab)
        t = ((X - float(a[0])) * ab[0] + (Y - float(a[1])) * ab[1] + (Z - float(a[2])) * ab[2]) / aa
        t.clamp_(0.0, 1.0)
        d2 = (X - float(a[0]) - t * ab[0]) ** 2
        d2 += (Y - float(a[1]) - t * ab[1]) ** 2
        d2 += (Z - float(a[2]) - t * ab[2]) ** 2
        torch.maximum(lam, torch.exp(d2.mul_(-1.0 / (2 * sigma_r * sigma_r))).mul_(n_ch * h ** 3), out=lam)
        del t, d2
    return lam, [(tip, sigma_r) for _, tip in segs]


def _plasma(ph, case, seed, member):
    """Particles (x, y, z FP64, w int32 sorted by cell) and positive ions per cell."""
    n, h, lo = ph["n"], synth.cell_size(ph), ph["lo"][0]
    g = _rng(seed * 64 + member)
    if case["state"] == "slab":
        N = case["particles"]
        L = n * h
        pos = _uniform(g, 3, N)
        x, y = lo + pos[0] * L, lo + pos[1] * L
        z = lo + (0.4 + 0.2 * pos[2]) * L
        w = torch.full((N,), 100, device="cuda", dtype=torch.int32)
        cell = ((z - lo) / h).floor_().long() * n * n + ((y - lo) / h).floor_().long() * n + ((x - lo) / h).floor_().long()
        ions = torch.zeros(n ** 3, device="cuda", dtype=torch.int64)
        ions.index_add_(0, cell, w.long())
        return x, y, z, w, ions
    lam, heads = _electrons(ph, case, seed, member, g)
    count = torch.poisson(lam.view(-1), generator=g).long()
    ions = count.clone()
    if case["state"] == "seeds":
        ions.zero_()                      # electrons only
    elif case["physics"] == "small":
        ions = ions * 9 // 10             # a net negative charge, as the small configuration's seed has
    if heads:
        X, Y, Z = _centres(ph)
        extra = torch.zeros_like(lam)
        for tip, s in heads:
            # a net positive head on each channel tip (peak 3e18 per m^3)
            extra += 3e18 * h ** 3 * torch.exp(-((X - float(tip[0])) ** 2 + (Y - float(tip[1])) ** 2
                                                 + (Z - float(tip[2])) ** 2) / (2 * s * s))
        ions += torch.poisson(extra.view(-1), generator=g).long()
        del extra
    del lam
    cells = count.nonzero().view(-1)
    N = count[cells]
    m = N.clamp(max=ph["ppc"])
    first = torch.repeat_interleave(m.cumsum(0) - m, m)
    slot = torch.arange(first.numel(), device="cuda") - first
    w = (torch.repeat_interleave(N // m, m) + (slot < torch.repeat_interleave(N % m, m))).int()
    del first, slot
    c = torch.repeat_interleave(cells, m)
    pos = [lo + (i + _uniform(g, c.numel())) * h for i in (c % n, (c // n) % n, c // (n * n))]
    return pos[0], pos[1], pos[2], w, ions


def _check(code, handle=None):
    if code:
        raise itokmc.ItokmcError(code, itokmc.lib().itokmc_last_error(handle).decode())


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


def _pinned(count, dtype):
    return torch.empty(count, dtype=dtype, pin_memory=True)


def _members(ph, case, seed):
    """The particles and ions of all realizations."""
    R = case["realizations"]
    parts = [_plasma(ph, case, seed, r) for r in range(R)]
    x, y, z, w = (torch.cat([p[k] for p in parts]) if R > 1 else parts[0][k] for k in range(4))
    real = torch.cat([torch.full((len(p[3]),), r, device="cuda", dtype=torch.int32) for r, p in enumerate(parts)])
    return x, y, z, w, real, torch.cat([p[4] for p in parts])


def _negative(ions, seed):
    """Negative ions: about an eighth of the positive ones, drawn per cell."""
    return torch.poisson(ions.double() / 8.0, generator=_rng(seed * 64 + 63)).long()


def _charges(ph, seed, count):
    """Ion counts of a net charge: `count` smooth random balls of up to 2e18 per m^3."""
    n, h = ph["n"], synth.cell_size(ph)
    L = n * h
    X, Y, Z = _centres(ph)
    u = torch.rand(count, 4, generator=torch.Generator().manual_seed(seed), dtype=torch.float64)
    rho = torch.zeros((n, n, n), device="cuda", dtype=torch.float64)
    for k in range(count):
        c = [float(0.2 + 0.6 * u[k, q]) * L for q in range(3)]
        s = 0.04 * L
        rho += float(0.5 + u[k, 3]) * 1e18 * h ** 3 * torch.exp(
            -((X - c[0]) ** 2 + (Y - c[1]) ** 2 + (Z - c[2]) ** 2) / (2 * s * s))
    return torch.poisson(rho.view(-1), generator=_rng(seed)).long()


def prepare(case, seed):
    ph = _physics(case)
    n3 = ph["n"] ** 3
    form = itokmc.FP64 if case["form"] == "fp64" else itokmc.MIXED
    if case["kind"] == "noalloc":
        rho = (_charges(ph, seed, 5).double() * case.get("charge", 1.0)).long() << (3 * FRAC_BITS)
        cfg = itokmc.make_config(ph, 1, precision=form, stream=torch.cuda.current_stream().cuda_stream)
        return dict(kind="noalloc", cfg=cfg, rho=rho, phi=torch.empty(n3, device="cuda", dtype=torch.float64),
                    E=torch.empty(3 * n3, device="cuda", dtype=torch.float64))
    x, y, z, w, real, ions = _members(ph, case, seed)
    R, N = case["realizations"], len(w)
    species = None
    neg = torch.zeros_like(ions) if not case.get("recombination") else _negative(ions, seed)
    if case.get("mobile_ions"):
        # an ion superparticle beside every electron superparticle
        species = torch.cat([torch.zeros(N, device="cuda", dtype=torch.int32), torch.ones(N, device="cuda", dtype=torch.int32)])
        x, y, z, w, real = (torch.cat([v, v]) for v in (x, y, z, w, real))
        N *= 2
    grow = 3 if case.get("mobile_ions") else 1.35 if case["n"] == 256 else 2
    cfg = itokmc.make_config(ph, int(grow * N) + 8 * ph["ppc"] * 4096, realizations=R, seed0=1 + seed % 1000,
                             precision=form)
    if case.get("coupling") == "semi":
        cfg.coupling = itokmc.SEMI_IMPLICIT
    if case.get("graph"):
        cfg.graph_step = 1
    H = itokmc.Handle(cfg)
    L = itokmc.lib()
    s = dict(kind=case["kind"], H=H, L=L, n3=n3, R=R, x=x, y=y, z=z, w=w, real=real, species=species, ions=ions, neg=neg,
             steps=case.get("steps", 1), read=case.get("read"), room=4 * case["particles"] * R + 65536)
    _upload(s)
    if case["kind"] == "field":
        s["other"] = ions + _charges(ph, seed + 1, 3)
        s["turn"] = 0
        s["out"] = dict(phi=_pinned(n3, torch.float64), E=_pinned(3 * n3, torch.float64))
        return s
    H.itokmc_solve_field()
    if case["kind"] == "transport":
        s["out"] = dict(ne=_pinned(R * n3, torch.int64))
    elif case["kind"] == "kmc":
        H.itokmc_run_stage(itokmc.STAGE_TRANSPORT)
        s["out"] = dict(firings=_pinned(5 * R * n3, torch.int64))
    else:
        # the field that the run starts from, kept by the program
        E = _pinned(3 * R * n3, torch.float64)
        _check(L.itokmc_read_densities(H.h, -1, itokmc.E, _p(E), E.numel() * 8), H.h)
        s["E"] = E.cuda()
        if s["read"] == "densities":
            s["out"] = dict(ne=_pinned(R * n3, torch.int64), phi=_pinned(R * n3, torch.float64))
        else:
            # host arrays with room for the particles that may come back
            s["out"] = dict({k: torch.zeros(s["room"], dtype=torch.float64) for k in "xyz"},
                            w=torch.zeros(s["room"], dtype=torch.int32), block=torch.zeros(s["room"], dtype=torch.int32),
                            cell=torch.zeros(s["room"], dtype=torch.int64), phi=_pinned(R * n3, torch.float64))
    return s


def _upload(s):
    H, L = s["H"], s["L"]
    if s["species"] is None:
        H.itokmc_set_particles(s["x"], s["y"], s["z"], s["w"], realization=s["real"], mem=itokmc.DEVICE)
        _check(L.itokmc_set_ions(H.h, _p(s["ions"]), _p(s["neg"]), itokmc.DEVICE), H.h)
    else:
        H.itokmc_set_particles_species(s["x"], s["y"], s["z"], s["w"], s["species"], realization=s["real"],
                                       mem=itokmc.DEVICE)


def _read(s, which, out):
    _check(s["L"].itokmc_read_densities(s["H"].h, -1, which, _p(out), out.numel() * 8), s["H"].h)


def run(s):
    if s["kind"] == "noalloc":
        s["phi"].zero_()
        itokmc.itokmc_field_solve_noalloc(s["cfg"], s["rho"], s["phi"], s["E"])
        return dict(phi=s["phi"], E=s["E"])
    H, L = s["H"], s["L"]
    if s["kind"] == "transport":
        H.itokmc_run_stage(itokmc.STAGE_TRANSPORT)
        H.itokmc_advance_counter()
        _read(s, itokmc.NE_FIX, s["out"]["ne"])
        return dict(s["out"])
    if s["kind"] == "kmc":
        H.itokmc_run_stage(itokmc.STAGE_KMC)
        H.itokmc_advance_counter()
        _read(s, itokmc.FIRINGS, s["out"]["firings"])
        return dict(s["out"])
    if s["kind"] == "field":
        ions = (s["ions"], s["other"])[s["turn"]]
        s["turn"] ^= 1
        _check(L.itokmc_set_ions(H.h, _p(ions), _p(s["neg"]), itokmc.DEVICE), H.h)
        H.itokmc_solve_field()
        _read(s, itokmc.PHI, s["out"]["phi"])
        _read(s, itokmc.E, s["out"]["E"])
        return dict(s["out"])
    _upload(s)
    _check(L.itokmc_set_field(H.h, _p(s["E"]), itokmc.DEVICE), H.h)
    H.itokmc_step(s["steps"])
    if s["read"] == "particles":
        o, count = s["out"], ctypes.c_int64()
        _check(L.itokmc_read_particles(H.h, _p(o["x"]), _p(o["y"]), _p(o["z"]), _p(o["w"]), _p(o["block"]),
                                       _p(o["cell"]), len(o["w"]), ctypes.byref(count), itokmc.HOST), H.h)
        _read(s, itokmc.PHI, o["phi"])
        return dict(o, count=count.value)
    _read(s, itokmc.NE_FIX, s["out"]["ne"])
    _read(s, itokmc.PHI, s["out"]["phi"])
    return dict(s["out"])


# --------------------------------------------------------------------------- work
def work(case):
    """Compulsory traffic: per step each particle record (32 B FP64, 20 B
    mixed) read and written once; per cell the density, charge and potential
    written and the field read once; the outputs written once.  Operations:
    117 (FP64) or 60 per pushed particle (interpolation and update) and 8 per
    cell and V-cycle of a field solve that takes 7 of them with 4 sweeps."""
    n3 = case["n"] ** 3
    if case["kind"] == "noalloc":
        return {"bytes": n3 * (8 + 8 + 24), "flops": n3 * 8 * 4 * 7}
    R = case["realizations"]
    N = case["particles"] * R * (2 if case.get("mobile_ions") else 1)
    cells = R * n3
    rec, fld = (32, 24) if case["form"] == "fp64" else (20, 12)
    push = 117 if case["form"] == "fp64" else 60
    solve = cells * 8 * 4 * 7
    if case["kind"] == "transport":
        return {"bytes": 2 * rec * N + cells * (8 + 8), "flops": push * N}
    if case["kind"] == "kmc":
        return {"bytes": cells * (8 + 40), "flops": 100 * N / 16}
    if case["kind"] == "field":
        return {"bytes": rec * N + cells * (16 + 8 + fld + 32), "flops": solve + 20 * N}
    k = case["steps"]
    return {"bytes": k * (2 * rec * N + cells * (8 + 8 + fld + 8)) + 28 * N + cells * (16 + 24 + 16),
            "flops": k * (push * N + solve)}


# --------------------------------------------------------------------------- the exact field
def _fixed_cic(ph, x, y, z, w):
    """Electrons per cell in units of 2^-3s: cloud-in-cell weights cut to s bits."""
    n, h = ph["n"], synth.cell_size(ph)
    one = 1 << FRAC_BITS
    ne = torch.zeros(n ** 3, device="cuda", dtype=torch.int64)
    step = 1 << 24
    for at in range(0, len(w), step):
        axes = []
        for v, lo in ((x, ph["lo"][0]), (y, ph["lo"][1]), (z, ph["lo"][2])):
            u = (v[at:at + step] - lo) / h - 0.5
            i = torch.floor(u)
            f = torch.floor((u - i) * one).long()
            i = i.long()
            axes.append(((i.clamp(0, n - 1), one - f), ((i + 1).clamp(0, n - 1), f)))
        ww = w[at:at + step].long()
        for iz, fz in axes[2]:
            for iy, fy in axes[1]:
                for ix, fx in axes[0]:
                    ne.index_add_(0, (iz * n + iy) * n + ix, ww * fx * fy * fz)
    return ne


def _exact_field(ph, rho):
    """The discrete Poisson equation solved by its eigenvectors: cosines at the
    homogeneous Neumann sides, sines between the electrodes; E by centred
    differences."""
    n, h = ph["n"], synth.cell_size(ph)
    top = ph["E0"] * (ph["hi"][2] - ph["lo"][2])
    b = -(rho.double().view(n, n, n) * (Q_E * 2.0 ** (-3 * FRAC_BITS) / h ** 3)) / EPS0
    b[n - 1] -= 2.0 * top / h ** 2
    m = torch.arange(n, device="cuda", dtype=torch.float64)
    C = torch.cos(math.pi * m.view(n, 1) * (m.view(1, n) + 0.5) / n)
    C /= C.norm(dim=1, keepdim=True)
    S = torch.sin(math.pi * (m.view(n, 1) + 1.0) * (m.view(1, n) + 0.5) / n)
    S /= S.norm(dim=1, keepdim=True)
    lc, ls = 2.0 - 2.0 * torch.cos(math.pi * m / n), 2.0 - 2.0 * torch.cos(math.pi * (m + 1.0) / n)
    t = torch.einsum("ak,kji->aji", S, b)
    t = torch.einsum("bj,aji->abi", C, t)
    t = torch.einsum("ci,abi->abc", C, t)
    t *= -h * h / (ls.view(n, 1, 1) + lc.view(1, n, 1) + lc.view(1, 1, n))
    t = torch.einsum("ak,abc->kbc", S, t)
    t = torch.einsum("bj,kbc->kjc", C, t)
    phi = torch.einsum("ci,kjc->kji", C, t)
    g = torch.empty((n + 2, n + 2, n + 2), device="cuda", dtype=torch.float64)
    g[1:-1, 1:-1, 1:-1] = phi
    g[1:-1, 1:-1, 0], g[1:-1, 1:-1, -1] = phi[:, :, 0], phi[:, :, -1]
    g[1:-1, 0, 1:-1], g[1:-1, -1, 1:-1] = phi[:, 0, :], phi[:, -1, :]
    g[0, 1:-1, 1:-1], g[-1, 1:-1, 1:-1] = -phi[0], 2.0 * top - phi[-1]
    c = slice(1, -1)
    E = torch.stack([(g[c, c, :-2] - g[c, c, 2:]), (g[c, :-2, c] - g[c, 2:, c]), (g[:-2, c, c] - g[2:, c, c])])
    return phi.reshape(-1), (E / (2.0 * h)).reshape(-1)


def exact(case, seed):
    """The field solves have a value in 64 bits: the discrete equation solved
    directly.  The other passes draw from the library's random streams: their
    whole-number densities have no rounding, and the potential that goes with
    them depends on the draws."""
    if case["kind"] not in ("field", "noalloc"):
        return None
    ph = _physics(case)
    if case["kind"] == "noalloc":
        rho = (_charges(ph, seed, 5).double() * case.get("charge", 1.0)).long() << (3 * FRAC_BITS)
    else:
        x, y, z, w, _, ions = _members(ph, case, seed)
        rho = (ions << (3 * FRAC_BITS)) - _fixed_cic(ph, x, y, z, w)
    phi, E = _exact_field(ph, rho)
    return dict(phi=phi, E=E)
