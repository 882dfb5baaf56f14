"""The calls whose time matters to a user of the library, over the sizes they are made at.

Grids are the 2,3,5-smooth sides of the batched and serving workloads (16 to 64, cubic and
orthorhombic), cells silicon-like (0.32 bohr per grid point, or the named cells' own sides),
orbitals orthonormal random combinations of the plane waves |G|^2/2 <= 10 Ha, occupations
Fermi-Dirac at a finite temperature, the kernel the erfc-screened one (mu = 0.106).  Everything is
drawn on the GPU from the seed.

listed() names the cases, draw() gives more of the same ranges, prepare() makes a case's inputs,
run() is one pass through the public entry points, work() counts the bytes and operations that a
pass cannot do without, and exact() computes the same outputs in 64 bits with plain torch.
"""
import math

import torch

from paper_2501_03061_gb300 import api, synth

MU = 0.106
ECUT = 10.0
ALPHA = 0.25
SIDES = (16, 20, 24, 30, 32, 36, 40, 48, 54, 60, 64)
SMOOTH = (16, 18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64)


def _case(kind, nx, N, M=0, prec="fp32", ny=0, nz=0, h=0.32, kT=0.02, **more):
    """A case: grid nx x ny x nz (cubic by default) at h bohr a point, N orbitals, M targets (0: the orbitals themselves)."""
    return dict(kind=kind, nx=nx, ny=ny or nx, nz=nz or nx, h=h, N=N, M=M, prec=prec, kT=kT, **more)


def listed():
    return [
        # V_x of the small FP32/FP64 cell (L = 10 bohr, 24^3, N = 16): the smallest call, launches and latency
        dict(_case("exchange", 24, 16, h=10.0 / 24, kT=0.01), name="exchange_24_N16"),
        dict(_case("exchange", 24, 16, prec="fp64", h=10.0 / 24, kT=0.01), name="exchange_24_N16_fp64"),
        # V_x of an ordinary system on other orbitals than the occupied ones (a block of trial vectors)
        dict(_case("exchange", 48, 150, M=37), name="exchange_48_N150_M37"),
        # an orthorhombic cell (a supercell that is not a cube)
        dict(_case("exchange", 36, 33, ny=50, nz=48), name="exchange_36x50x48_N33"),
        # V_x of the 128-site cell, once per ACE build of a PT-IM step: the largest exchange
        dict(_case("exchange", 64, 320, h=20.5 / 64), name="exchange_64_N320"),
        # several systems of different sizes in one call (the batched workload's first ten)
        dict(_case("batched", 0, 0, items="32:61,32:84,60:175,54:128,30:98,48:132,32:186,30:109,40:186,24:43"), name="batched_10"),
        # the ACE operator of one system built and handed out (exchange, Gram, Cholesky, xi)
        dict(_case("ace_build", 36, 75), name="ace_build_36_N75"),
        # the ACE operator applied to a block, contractions on the tensor cores (every H application of an inner loop)
        dict(_case("ace_apply", 54, 200, M=200, tc=1), name="ace_apply_54_N200"),
        # H psi with the ACE exchange (an eigensolver's or a propagator's inner operation)
        dict(_case("H", 40, 61, M=61), name="H_40_N61"),
        # density of the orbitals and the Hartree + LDA potential from it (self-consistent V_Hxc)
        dict(_case("hxc", 60, 150, tc=1), name="hxc_60_N150"),
        # a whole PT-IM-ACE step as a serving request brings it: a small system, and the 128-site benchmark cell
        dict(_case("step", 32, 48, tc=1), name="step_32_N48"),
        dict(_case("step", 64, 320, h=20.5 / 64, tc=1), name="step_64_N320"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("exchange",) * 5 + ("batched", "ace_build", "ace_apply", "H", "hxc", "step"))
    n = rng.choice(SIDES)
    most = min(320, {16: 100, 20: 190}.get(n, 320))  # orbitals that the plane-wave sphere of the cell holds with room to spare
    kT = round(rng.uniform(0.01, 0.02), 4)
    if kind == "batched":
        items = []
        for _ in range(rng.randint(3, 12)):
            side = rng.choice(SIDES[2:])
            items.append("%d:%d" % (side, _log_int(rng, 16, 256 if side < 48 else 200)))
        return _case(kind, 0, 0, items=",".join(items), kT=kT)
    if kind == "exchange":
        ny = nz = n
        if rng.random() < 0.25:
            n, ny, nz = (rng.choice(SMOOTH) for _ in range(3))
            most = min(most, max(8, n * ny * nz // 120))
        prec = "fp64" if rng.random() < 0.2 else "fp32"
        N = _log_int(rng, 4, most if prec == "fp32" else min(most, 64))
        M = 0 if rng.random() < 0.7 else _log_int(rng, 1, min(most, 64))
        if ny != n or nz != n:
            N = min(N, 120)
        return _case(kind, n, N, M, prec, ny, nz, kT=kT)
    if kind == "step":
        n = rng.choice(synth.SERVE_GRID_SIZES)
        return _case(kind, n, _log_int(rng, 32, 320 if n < 64 else 200), kT=kT, tc=1)
    N = _log_int(rng, 8, min(most, 256))
    M = 0 if kind in ("ace_build", "hxc") else _log_int(rng, 4, min(most, 256))
    return _case(kind, n, N, M, kT=kT, tc=0 if kind == "H" and rng.random() < 0.5 else 1)


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------

def _cell(n, h):
    return synth.Cell(tuple(n), tuple(h * k for k in n))


def _axes(cell):
    """G of the three axes (z, y, x order, broadcastable), m wrapped to [-n/2, n/2)."""
    out = []
    for a in range(3):
        m = torch.fft.fftfreq(cell.n[a], 1.0 / cell.n[a], dtype=torch.float64, device="cuda")
        shape = [1, 1, 1]
        shape[2 - a] = cell.n[a]
        out.append((2 * math.pi / cell.L[a] * m).reshape(shape))
    return out


def _g2(cell):
    return sum(g * g for g in _axes(cell))


def _orbitals(gen, cell, N):
    idx = torch.nonzero((0.5 * _g2(cell) <= ECUT).reshape(-1)).reshape(-1)
    c = torch.complex(*(torch.randn(2, idx.numel(), N, generator=gen, device="cuda", dtype=torch.float64)))
    q = torch.linalg.qr(c)[0] / math.sqrt(cell.volume)
    spec = torch.zeros(N, cell.ng, dtype=torch.complex128, device="cuda")
    spec[:, idx] = q.T
    return torch.fft.ifftn(spec.reshape(N, cell.n[2], cell.n[1], cell.n[0]), dim=(1, 2, 3)).mul_(cell.ng)


def _wells(gen, cell):
    """-sum_a exp(-|r - R_a|^2 / 2) over the cell's sites (128 in the benchmark cell's volume), periodic."""
    sites = max(8, int(round(128 * cell.volume / 20.5 ** 3)))
    R = torch.rand(sites, 3, generator=gen, device="cuda", dtype=torch.float64)
    axis = []
    for a in range(3):
        x = torch.arange(cell.n[a], device="cuda", dtype=torch.float64) * (cell.L[a] / cell.n[a])
        d = x[None, :] - R[:, a:a + 1] * cell.L[a]
        d = d - cell.L[a] * torch.round(d / cell.L[a])
        axis.append(torch.exp(-0.5 * d * d))
    return -torch.einsum("sz,sy,sx->zyx", axis[2], axis[1], axis[0]).contiguous()


def _system(gen, case, n, N, M):
    cell = _cell(n, case["h"])
    dt = torch.complex128 if case["prec"] == "fp64" else torch.complex64
    s = {"cell": cell, "phi": _orbitals(gen, cell, N).to(dt),
         "occ": torch.from_numpy(synth.fermi_dirac_occupations(N, case["kT"])).cuda(), "psi": None}
    if M:
        s["psi"] = _orbitals(gen, cell, M).to(dt)
    return s


def _inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if case["kind"] == "batched":
        items = [tuple(int(v) for v in t.split(":")) for t in case["items"].split(",")]
        return {"items": [_system(gen, case, (n, n, n), N, 0) for n, N in items]}
    s = _system(gen, case, (case["nx"], case["ny"], case["nz"]), case["N"], case["M"])
    if case["kind"] in ("H", "hxc", "step"):
        s["vloc"] = _wells(gen, s["cell"])
    if case["kind"] in ("hxc", "step"):
        # occupations in a basis a little off the diagonal one, as a propagated state has them
        N = case["N"]
        k = torch.complex(*torch.randn(2, N, N, generator=gen, device="cuda", dtype=torch.float64)) * (0.05 / math.sqrt(N))
        u = torch.linalg.matrix_exp(k - k.mH)
        m = (u * s["occ"]) @ u.mH
        s["sigma"] = (0.5 * (m + m.mH)).contiguous()
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    ctx = s["ctx"] = api.Context(0)
    if case.get("tc"):
        ctx.set_option("tc_gram", 1)
    kernel = s["kernel"] = {"type": 1, "mu": MU}
    if case["kind"] == "batched":  # the caller's own buffers, kept from call to call as a serving loop keeps them
        s["calls"] = [{"src": i["phi"], "occ": i["occ"], "cell": i["cell"], "kernel": kernel, "out": torch.empty_like(i["phi"])} for i in s["items"]]
    if case["kind"] in ("ace_apply", "H"):
        s["ace"] = ctx.build_ace(s["phi"], s["occ"], cell=s["cell"], kernel=kernel, precision=case["prec"])
    if case["kind"] == "step":
        s["phi_t"], s["sigma_t"] = torch.empty_like(s["phi"]), torch.empty_like(s["sigma"])
    return s


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind, prec = case["kind"], case["prec"]
    if kind == "batched":
        return ctx.apply_exchange_batched(s["calls"], precision=prec)[0]
    cell = s["cell"]
    if kind == "exchange":
        return ctx.apply_exchange(s["phi"], s["occ"], s["psi"], cell=cell, kernel=s["kernel"], precision=prec)
    if kind == "ace_build":
        ace = ctx.build_ace(s["phi"], s["occ"], cell=cell, kernel=s["kernel"], precision=prec)
        xi = ace.xi()
        ace.close()
        return xi
    if kind == "ace_apply":
        return ctx.apply_ace(s["ace"], s["psi"])
    if kind == "H":
        return ctx.apply_H(s["psi"], s["vloc"], s["ace"], ALPHA, ECUT, cell=cell, precision=prec)
    if kind == "hxc":
        rho = ctx.density(s["phi"], s["sigma"], cell=cell, precision=prec)
        return rho, ctx.hxc_potential(rho, s["vloc"], cell=cell)
    # a serving request: the state it brings is taken one step further, in place
    s["phi_t"].copy_(s["phi"])
    s["sigma_t"].copy_(s["sigma"])
    ctx.ptim_step(s["phi_t"], s["sigma_t"], s["vloc"], cell=cell, kernel=s["kernel"], precision=prec, dt=0.5, alpha=ALPHA, ecut=ECUT, tol=1e-6)
    # sigma is an FP32-form result (exchange and contractions in 32 bits): handed on in the orbitals' type
    return s["phi_t"], s["sigma_t"].to(s["phi_t"].dtype)


# ------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ------------------------------------------------------------------------------------------------

def _pair_flops(ng):
    return 10.0 * ng * math.log2(ng) + 16.0 * ng


def work(case):
    kind, es = case["kind"], 16 if case["prec"] == "fp64" else 8
    if kind == "batched":
        b = f = 0.0
        for t in case["items"].split(","):
            n, N = (int(v) for v in t.split(":"))
            b += 2.0 * N * n ** 3 * es
            f += N * (N + 1) / 2 * _pair_flops(n ** 3)
        return {"bytes": b, "flops": f}
    ng, N = case["nx"] * case["ny"] * case["nz"], case["N"]
    M = case["M"] or N
    fft = 5.0 * ng * math.log2(ng)
    pairs = N * M if case["M"] else N * (N + 1) / 2
    if kind == "exchange":
        return {"bytes": es * ng * (N + (2.0 if case["M"] else 1.0) * M), "flops": pairs * _pair_flops(ng)}
    if kind == "ace_build":
        return {"bytes": 2.0 * es * ng * N, "flops": N * (N + 1) / 2 * _pair_flops(ng) + 16.0 * N * N * ng}
    if kind == "ace_apply":
        return {"bytes": es * ng * (N + 2.0 * M), "flops": 16.0 * N * M * ng}
    if kind == "H":
        return {"bytes": es * ng * (N + 2.0 * M) + 8.0 * ng, "flops": 16.0 * N * M * ng + 3 * fft * M}
    if kind == "hxc":
        return {"bytes": es * ng * N + 16.0 * N * N + 24.0 * ng, "flops": 8.0 * N * N * ng}
    # a step: one V_x for each of three ACE operators, about twenty H applications on the sphere's plane waves
    npw = 4.0 / 3 * math.pi * (2 * ECUT) ** 1.5 * ng * case["h"] ** 3 / (2 * math.pi) ** 3
    return {"bytes": 2.0 * es * ng * N + 32.0 * N * N + 8.0 * ng,
            "flops": 3 * N * (N + 1) / 2 * _pair_flops(ng) + 20 * (2 * fft * N + 40.0 * N * N * npw)}


# ------------------------------------------------------------------------------------------------
# the same outputs in 64 bits
# ------------------------------------------------------------------------------------------------

def _kernel_table(cell):
    g2 = _g2(cell)
    g2[0, 0, 0] = 1.0
    k = 4 * math.pi / g2 * -torch.expm1(-g2 / (4 * MU * MU))
    k[0, 0, 0] = math.pi / (MU * MU)
    return k


def _vx(s, tgt=None):
    """V_x on tgt, or on the orbitals themselves (v_ji = conj(v_ij): half of the transforms)."""
    phi, K = s["phi"].to(torch.complex128), _kernel_table(s["cell"])
    sym = tgt is None
    tgt = phi if sym else tgt.to(torch.complex128)
    out = torch.zeros_like(tgt)
    occ = s["occ"].tolist()
    d = s["occ"].reshape(-1, 1, 1, 1)
    for i in range(phi.shape[0]):
        j = i if sym else 0
        v = torch.fft.ifftn(torch.fft.fftn(phi[i].conj() * tgt[j:], dim=(1, 2, 3)).mul_(K), dim=(1, 2, 3))
        out[j:] -= occ[i] * phi[i] * v
        if sym and i + 1 < phi.shape[0]:
            out[i] -= (v[1:].conj_physical_().mul_(phi[i + 1:]).mul_(d[i + 1:])).sum(0)
    return out


def _xi(s):
    phi, cell = s["phi"].to(torch.complex128), s["cell"]
    W = _vx(s)
    P, Wf = phi.reshape(phi.shape[0], -1), W.reshape(phi.shape[0], -1)
    M = cell.dV * (P.conj() @ Wf.T)
    Lc = torch.linalg.cholesky(-0.5 * (M + M.mH))
    return torch.linalg.solve_triangular(Lc.conj(), Wf, upper=False)  # rows: xi = W L^{-*}


def _ace(xi, psi, cell):
    p = psi.to(torch.complex128).reshape(psi.shape[0], -1)
    c = cell.dV * (xi.conj() @ p.T)
    return -(c.T @ xi).reshape(psi.shape)


def _xc_potential(rho):
    """LDA: Slater exchange and the Perdew-Zunger (1981) correlation of the unpolarised gas."""
    r = rho.clamp_min(1e-30)
    rs = (3 / (4 * math.pi * r)) ** (1.0 / 3)
    vx = -((3 * r / math.pi) ** (1.0 / 3))
    den = 1 + 1.0529 * rs.sqrt() + 0.3334 * rs
    hi = -0.1423 / den * (1 + 7.0 / 6 * 1.0529 * rs.sqrt() + 4.0 / 3 * 0.3334 * rs) / den
    ln = rs.log()
    lo = 0.0311 * ln - 0.048 - 0.0311 / 3 + 2.0 / 3 * 0.0020 * rs * ln + (2 * -0.0116 - 0.0020) / 3 * rs
    return torch.where(rho > 1e-30, vx + torch.where(rs >= 1, hi, lo), torch.zeros_like(rho))


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        return None  # a fixed point iterated to 1e-6: in 64 bits over about 20 seconds at the larger sizes
    s = _inputs(case, seed)
    if kind == "batched":
        return [_vx(i) for i in s["items"]]
    cell = s["cell"]
    if kind == "exchange":
        return _vx(s, s["psi"])
    if kind == "ace_build":
        return _xi(s).reshape(s["phi"].shape)
    if kind == "ace_apply":
        return _ace(_xi(s), s["psi"], cell)
    if kind == "H":
        psi, g2 = s["psi"].to(torch.complex128), _g2(cell)
        local = s["vloc"] * psi + ALPHA * _ace(_xi(s), psi, cell)
        f = torch.fft.fftn(local, dim=(1, 2, 3)) + 0.5 * g2 * torch.fft.fftn(psi, dim=(1, 2, 3))
        return torch.fft.ifftn(f * (0.5 * g2 <= ECUT), dim=(1, 2, 3))
    phi = s["phi"].to(torch.complex128)
    chi = (s["sigma"].T @ phi.reshape(phi.shape[0], -1)).reshape(phi.shape)
    rho = 2.0 * (chi.real * phi.real + chi.imag * phi.imag).sum(0)
    g2 = _g2(cell)
    g2[0, 0, 0] = 1.0
    f = torch.fft.fftn(rho) * (4 * math.pi) / g2
    f[0, 0, 0] = 0.0
    return rho, s["vloc"] + torch.fft.ifftn(f).real + _xc_potential(rho)
