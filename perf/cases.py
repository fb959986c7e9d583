"""Performance cases: what programs ask of this library, over the sizes they ask it for.

A case is one call of a public entry point: an update step (energy, forces, potentials) of one periodic or grounded
system, a batch of systems sharing a plan, the near-field Coulomb sum on its own, or the harmonic basis on its own.

Results of the reduced forms ("fp32", "fp32_tc") are kept in single precision, as a mixed-precision MD program keeps
them: these forms state 1e-6 on the energy and 1e-5 on the forces.  The FP64 form's results, and the basis in both of
its forms, are kept in double precision.

exact() is the method written out in plain torch FP64: images inside the sphere, their sums at the particles and
monitoring points, the least-squares fit, the surface images (dipole layer in its cancellation-free form) and their
sums at the particles.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1806_04801_gb300 import hsma

# Plan parameters (box, boundary, p, R, Q, Kmon) of the library's own workloads.
PLANS = {
    "periodic-p8": ((1.0, 1.0, 1.0), hsma.PERIODIC, 8, 1.5, 2000, 600),
    "periodic-p10": ((1.0, 1.0, 1.0), hsma.PERIODIC, 10, 1.5, 6000, 1500),
    "periodic-p12": ((1.0, 1.0, 1.0), hsma.PERIODIC, 12, 1.5, 8000, 2000),
    # the paper's timing configuration: alpha = 1.3, P = 25, N_o = 5928
    "periodic-p25": ((1.0, 1.0, 1.0), hsma.PERIODIC, 25, 1.3 * 0.5 * math.sqrt(3.0), 5928, 1250),
    "grounded-p10": ((1.0, 1.0, 2.0), hsma.GROUNDED, 10, math.sqrt(3.0) * 0.5 * math.sqrt(6.0), 6000, 1500),
}


def listed():
    return [
        # the reference-quality form on a small box: validation runs, fitting of force fields
        {"name": "step fp64 N1000", "kind": "step", "plan": "periodic-p8", "precision": "fp64", "n": 1000},
        # the same form at the size of a solvated molecule, odd count, potentials asked for too
        {"name": "step fp64 N9999 pot", "kind": "step", "plan": "periodic-p12", "precision": "fp64", "n": 9999,
         "potentials": True},
        # a small conducting cavity in FP64
        {"name": "grounded fp64 N3001", "kind": "step", "plan": "grounded-p10", "precision": "fp64", "n": 3001},
        # the smallest systems a serving queue sees: launches and latency
        {"name": "step fp32 N500", "kind": "step", "plan": "periodic-p10", "precision": "fp32", "n": 500},
        # an MD step of a small system
        {"name": "step fp32_tc N4000", "kind": "step", "plan": "periodic-p12", "precision": "fp32_tc", "n": 4000},
        # the large periodic box: Gaussian charges, uniform positions
        {"name": "step fp32_tc N100000", "kind": "step", "plan": "periodic-p12", "precision": "fp32_tc", "n": 100000,
         "charges": "gauss"},
        # ions in a conducting cavity
        {"name": "grounded fp32_tc N20000", "kind": "step", "plan": "grounded-p10", "precision": "fp32_tc",
         "n": 20000},
        # the paper's timing configuration: lattice sites, a high order, a tight sphere
        {"name": "lattice fp32_tc N103823 p25", "kind": "step", "plan": "periodic-p25", "precision": "fp32_tc",
         "n": 103823, "charges": "lattice"},
        # many boxes of uneven size in one call
        {"name": "batch fp32 32 boxes", "kind": "batch", "plan": "periodic-p10", "precision": "fp32", "systems": 32,
         "lo": 500, "hi": 50000},
        # the near-field sum alone, FP64, ragged counts: checking another code's forces
        {"name": "coulomb fp64 20011x3001", "kind": "coulomb", "precision": "fp64", "ns": 20011, "nt": 3001,
         "field": True},
        # the basis at many points: building fitting matrices outside a plan
        {"name": "basis fp32 p12 1000003", "kind": "basis", "precision": "fp32", "p": 12, "np": 1000003},
        # the basis in FP64, high order, ragged count
        {"name": "basis fp64 p25 30011", "kind": "basis", "precision": "fp64", "p": 25, "np": 30011},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "batch", "coulomb", "basis"])
    if kind == "step":
        precision = rng.choice(["fp64", "fp32", "fp32_tc"])
        plan = rng.choice(["periodic-p8", "periodic-p10", "periodic-p12", "periodic-p25", "grounded-p10"])
        top = 10000 if precision == "fp64" else 100000
        if plan == "grounded-p10":  # the same cost: a cavity's sphere holds 20 images of each charge, a cube's 14
            top = 8000 if precision == "fp64" else 50000
        c = {"kind": "step", "plan": plan, "precision": precision, "n": _log_int(rng, 300, top)}
        if rng.random() < 0.5:
            c["potentials"] = True
        if rng.random() < 0.25:
            c["far_field"] = "series"
        if rng.random() < 0.3:
            c["charges"] = "lattice" if plan == "periodic-p25" else "gauss"
        return c
    if kind == "batch":
        return {"kind": "batch", "plan": rng.choice(["periodic-p8", "periodic-p10"]),
                "precision": rng.choice(["fp32", "fp32_tc"]), "systems": _log_int(rng, 2, 64), "lo": 500,
                "hi": _log_int(rng, 2000, 25000)}
    if kind == "coulomb":
        precision = rng.choice(["fp64", "fp32"])
        top = 100000 if precision == "fp32" else 20000
        return {"kind": "coulomb", "precision": precision, "ns": _log_int(rng, 1000, top),
                "nt": _log_int(rng, 500, top), "field": rng.random() < 0.7}
    p = rng.randint(4, 25)
    return {"kind": "basis", "precision": rng.choice(["fp32", "fp64"]), "p": p,
            "np": _log_int(rng, 2000, 1000000 * 169 // (p + 1) ** 2)}


# ------------------------------------------------------------------ inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1806_04801 + 1000003 * seed)
    return g


def _system(n, box, charges, g):
    """Positions (n, 3) in the box and neutral charges (n,), FP64 on the device.

    "ions": a disordered salt, as an MD program holds it: distinct sites of a lattice, each displaced by up to a
    quarter of its spacing, charges +-1 alternating over the sites, as many of each (odd counts: one uncharged);
    "gauss": uniform positions, normal charges; "lattice": the sites of a lattice, charges of random sign.  Grounded
    boxes (1 x 1 x 2) keep a margin of 0.05 to the walls."""
    dev = "cuda"
    L = torch.tensor(box, dtype=torch.float64, device=dev)
    margin = 0.05 if box[2] != box[0] else 0.0
    if charges == "gauss":
        x = torch.rand((n, 3), generator=g, device=dev, dtype=torch.float64)
        q = torch.randn(n, generator=g, device=dev, dtype=torch.float64)
        return (margin + x * (L - 2 * margin)).contiguous(), q - q.mean()
    aspect = box[2] / box[0]
    m = 1
    while m * m * round(m * aspect) < n:
        m += 1
    mz = round(m * aspect)
    site = torch.randperm(m * m * mz, generator=g, device=dev)
    ix = torch.stack((site // (m * mz), site // mz % m, site % mz), 1)
    cells = torch.tensor([m, m, mz], device=dev)
    if charges == "lattice":
        ix = ix[:n]
        x = (ix + 0.5) / cells
        q = torch.ones(n, device=dev, dtype=torch.float64)
        q[: n // 2] = -1.0  # the sites are in random order
        if n % 2:
            q[-1] = 0.0
    else:
        odd = ix.sum(1) % 2 == 1
        even, odd = ix[~odd], ix[odd]
        ix = torch.cat((odd[: n // 2], even[: n - n // 2]))
        d = 0.5 * torch.rand((n, 3), generator=g, device=dev, dtype=torch.float64) - 0.25
        x = (ix + 0.5 + d) / cells
        q = torch.ones(n, device=dev, dtype=torch.float64)
        q[: n // 2] = -1.0
        if n % 2:
            q[-1] = 0.0
        order = torch.randperm(n, generator=g, device=dev)
        x, q = x[order], q[order]
    return (margin + x.double() * (L - 2 * margin)).contiguous(), q


def _sizes(case, seed):
    """Log-uniform system sizes of a batch; the sizes are the case's, so that every seed has the same work."""
    r = np.random.default_rng(1806_04801 + case["systems"])
    n = np.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"]), case["systems"]))
    return [int(v) for v in np.round(n)]


def _inputs(case, seed):
    g = _generator(seed)
    if case["kind"] == "step":
        return _system(case["n"], PLANS[case["plan"]][0], case.get("charges", "ions"), g)
    if case["kind"] == "batch":
        parts = [_system(n, PLANS[case["plan"]][0], "ions", g) for n in _sizes(case, seed)]
        return torch.cat([x for x, _ in parts]).contiguous(), torch.cat([q for _, q in parts]).contiguous()
    if case["kind"] == "coulomb":
        src = torch.rand((case["ns"], 4), generator=g, device="cuda", dtype=torch.float64)
        src[:, 3] = torch.randn(case["ns"], generator=g, device="cuda", dtype=torch.float64)
        return src, torch.rand((case["nt"], 3), generator=g, device="cuda", dtype=torch.float64)
    return (torch.rand((case["np"], 3), generator=g, device="cuda", dtype=torch.float64) - 0.5,)


def prepare(case, seed):
    s = {"case": case, "inputs": _inputs(case, seed)}
    if case["kind"] in ("step", "batch"):
        s["plan"] = hsma.Plan(*PLANS[case["plan"]], precision=case["precision"],
                              far_field=case.get("far_field", "images"))
    if case["kind"] == "batch":
        s["offsets"] = np.concatenate([[0], np.cumsum(_sizes(case, seed))]).astype(np.int64)
    return s


# --------------------------------------------------------------------- run
def run(s):
    case, inp = s["case"], s["inputs"]
    if case["kind"] == "basis":
        return hsma.basis(inp[0], case["p"], 1.5, precision=case["precision"])
    if case["kind"] == "coulomb":
        pot, field = hsma.coulomb_sum(inp[0], inp[1], field=case["field"], precision=case["precision"])
        return {"pot": _kept(case, pot), "field": _kept(case, field)}
    if case["kind"] == "batch":
        e, f, _, status = s["plan"].energy_forces_batched(inp[0], inp[1], s["offsets"])
        return {"energy": e.astype(np.float32), "forces": _kept(case, f), "status": status}
    e, f, p, n_inset = s["plan"].energy_forces(inp[0], inp[1], potentials=case.get("potentials", False))
    return {"energy": e, "forces": _kept(case, f), "potentials": _kept(case, p), "n_inset": n_inset}


def _kept(case, t):
    """A result as the caller keeps it: the reduced forms' in single precision."""
    return t if t is None or case["precision"] == "fp64" else t.float()


# -------------------------------------------------------------------- work
def _fib2(Q):
    """F2 of the Fibonacci integration whose 6 (F2 + 1) images are nearest to Q."""
    a, b, best = 1, 2, None
    while a < 10**7:
        if best is None or abs(6 * (b + 1) - Q) <= abs(6 * (best[0] + 1) - Q):
            best = (b, a)
        a, b = b, a + b
    return best


def work(case):
    """Pairs of the direct sums: 3 differences, 5 for r^2, 1 for 1/r, 2 for the potential, 8 more for the field."""
    if case["kind"] == "basis":
        nb = (case["p"] + 1) ** 2
        return {"bytes": 8.0 * case["np"] * (3 + nb), "flops": 5.0 * case["np"] * nb}
    if case["kind"] == "coulomb":
        pairs = case["ns"] * case["nt"]
        return {"bytes": 8.0 * (4 * case["ns"] + (7 if case["field"] else 4) * case["nt"]),
                "flops": (19.0 if case["field"] else 11.0) * pairs}
    box, bc, p, R, Q, K = PLANS[case["plan"]]
    kmon = 2 * K if bc == hsma.PERIODIC else K
    images = 4.0 / 3.0 * math.pi * R**3 / (box[0] * box[1] * box[2])
    flops = bytes_ = 0.0
    for n in [case["n"]] if case["kind"] == "step" else _sizes(case, 0):
        far = 19.0 * 2 * (_fib2(Q)[0] + 1) if case.get("far_field", "images") == "images" else 20.0 * (p + 1) ** 2
        flops += n * (19.0 * images * n + far) + 11.0 * images * n * kmon + 2.0 * K * (p + 1) ** 2
        bytes_ += 8.0 * n * (7 + (1 if case.get("potentials") else 0)) + 8.0 * K * (p + 1) ** 2
    return {"bytes": bytes_, "flops": flops}


# ------------------------------------------------------------------- exact
def _sums(src, q, tgt, field=True, own=False):
    """sum q / |x - y| and sum q (x - y) / |x - y|^3 at the targets; own: target i leaves out source i."""
    nt, ns = tgt.shape[0], src.shape[0]
    phi, e = torch.zeros(nt, dtype=torch.float64, device="cuda"), None
    if field:
        e = torch.zeros((nt, 3), dtype=torch.float64, device="cuda")
    step = max(1, (1 << 25) // max(1, ns))
    sx = [src[:, a].contiguous() for a in range(3)]
    for i in range(0, nt, step):
        t = tgt[i:i + step]
        d = [t[:, a, None] - sx[a] for a in range(3)]
        r2 = d[0] * d[0]
        r2.addcmul_(d[1], d[1]).addcmul_(d[2], d[2])
        if own:
            k = torch.arange(t.shape[0], device="cuda")
            r2[k, i + k] = math.inf
        ri = r2.rsqrt_()
        phi[i:i + step] = ri @ q
        if field:
            w = ri * ri * ri
            for a in range(3):
                e[i:i + step, a] = d[a].mul_(w) @ q
    return phi, e


def _basis(x, p, Rs):
    """Orthonormal real solid harmonics (|x| / Rs)^n Y_nm, column n^2 + n + m (cosines m >= 0, sines m < 0)."""
    x = x / Rs
    X, Y, Z = x[:, 0], x[:, 1], x[:, 2]
    r2 = X * X + Y * Y + Z * Z
    out = torch.empty((x.shape[0], (p + 1) ** 2), dtype=torch.float64, device=x.device)
    C, S = torch.ones_like(X), torch.zeros_like(X)
    for m in range(p + 1):
        if m:
            C, S = C * X - S * Y, S * X + C * Y
        c, q0, q1 = math.sqrt((2.0 if m else 1.0) / (4.0 * math.pi)), None, None
        for n in range(m, p + 1):
            if n == m:  # (2m - 1)!! and the norm in one constant
                for j in range(1, m + 1):
                    c *= math.sqrt((2.0 * j - 1.0) / (2.0 * j))
                q2 = torch.full_like(X, c * math.sqrt(2.0 * m + 1.0))
            elif n == m + 1:
                q2 = math.sqrt(2.0 * m + 3.0) * Z * q1
            else:
                f = math.sqrt((2.0 * n + 1.0) / (n * n - m * m))
                q2 = f * (math.sqrt(2.0 * n - 1.0) * Z * q1
                          - math.sqrt(((n - 1.0) ** 2 - m * m) / (2.0 * n - 3.0)) * r2 * q0)
            q0, q1 = q1, q2
            out[:, n * n + n + m] = q2 * C
            if m:
                out[:, n * n + n - m] = q2 * S
    return out


def _basis_gradient(x, p, Rs, A):
    x = x.clone().requires_grad_(True)
    with torch.enable_grad():
        phi = torch.zeros(x.shape[0], dtype=torch.float64, device="cuda")
        # the recurrence of _basis, summed with the coefficients instead of stored
        u = x / Rs
        X, Y, Z = u[:, 0], u[:, 1], u[:, 2]
        r2 = X * X + Y * Y + Z * Z
        C, S = torch.ones_like(X), torch.zeros_like(X)
        for m in range(p + 1):
            if m:
                C, S = C * X - S * Y, S * X + C * Y
            c, q0, q1 = math.sqrt((2.0 if m else 1.0) / (4.0 * math.pi)), None, None
            for n in range(m, p + 1):
                if n == m:
                    for j in range(1, m + 1):
                        c *= math.sqrt((2.0 * j - 1.0) / (2.0 * j))
                    q2 = torch.full_like(X, c * math.sqrt(2.0 * m + 1.0))
                elif n == m + 1:
                    q2 = math.sqrt(2.0 * m + 3.0) * Z * q1
                else:
                    f = math.sqrt((2.0 * n + 1.0) / (n * n - m * m))
                    q2 = f * (math.sqrt(2.0 * n - 1.0) * Z * q1
                              - math.sqrt(((n - 1.0) ** 2 - m * m) / (2.0 * n - 3.0)) * r2 * q0)
                q0, q1 = q1, q2
                phi = phi + q2 * (A[n * n + n + m] * C + (A[n * n + n - m] * S if m else 0.0))
        (grad,) = torch.autograd.grad(phi.sum(), x)
    return phi.detach(), -grad


def _monitors(bc, K, L):
    w = (math.sqrt(5.0) - 1.0) / 2.0
    if bc == hsma.PERIODIC:
        R0 = 0.5 * math.sqrt(sum(b * b for b in L))
        i = torch.arange(1, K + 1, dtype=torch.float64, device="cuda")
        sl = (2.0 * i - 1.0) / K - 1.0
        cl = torch.sqrt(1.0 - sl * sl)
        az = 2.0 * math.pi * i * w
        return R0 * torch.stack((cl * torch.cos(az), cl * torch.sin(az), sl), 1)
    area = [L[(f // 2 + 1) % 3] * L[(f // 2 + 2) % 3] for f in range(6)]
    quota = [K * a / sum(area) for a in area]
    count = [int(v) for v in quota]
    order = sorted(range(6), key=lambda f: (-(quota[f] - count[f]), f))
    for f in order[: K - sum(count)]:
        count[f] += 1
    pts = []
    for f in range(6):
        a = f // 2
        ua, va = (1 if a == 0 else 0), (1 if a == 2 else 2)
        i = torch.arange(count[f], dtype=torch.float64, device="cuda")
        x = torch.empty((count[f], 3), dtype=torch.float64, device="cuda")
        x[:, a] = (0.5 if f % 2 else -0.5) * L[a]
        x[:, ua] = ((i + 0.5) / count[f] - 0.5) * L[ua]
        x[:, va] = (torch.fmod(i * w + 0.5, 1.0) - 0.5) * L[va]
        pts.append(x)
    return torch.cat(pts)


def _exact_system(xyz, q, plan, far_field):
    """(energy, forces, potentials, in-set size) of one system."""
    box, bc, p, Rs, Q, K = plan
    L = torch.tensor(box, dtype=torch.float64, device="cuda")
    c = (xyz - torch.floor(xyz / L) * L if bc == hsma.PERIODIC else xyz) - 0.5 * L
    shells = [max(k for k in range(20) if k * box[a] - 0.5 * box[a] < Rs) for a in range(3)]
    sx, sq = [c], [q]
    for kx in range(-shells[0], shells[0] + 1):
        for ky in range(-shells[1], shells[1] + 1):
            for kz in range(-shells[2], shells[2] + 1):
                if not (kx or ky or kz):
                    continue
                k = torch.tensor([kx, ky, kz], dtype=torch.float64, device="cuda")
                sign = 1.0 - 2.0 * (k.abs() % 2) if bc == hsma.GROUNDED else torch.ones_like(k)
                y = sign * c + k * L
                inside = (y * y).sum(1) < Rs * Rs
                sx.append(y[inside])
                sq.append((q * sign.prod())[inside])
    sx, sq = torch.cat(sx), torch.cat(sq)
    phi, e = _sums(sx, sq, c, own=True)

    x = _monitors(bc, K, box)
    b = -_sums(sx, sq, x, field=False)[0]
    if bc == hsma.PERIODIC:
        r = x / L
        xt = x - torch.sign(r) * torch.floor(r.abs() + 0.5) * L
        b = b + _sums(sx, sq, xt, field=False)[0]
        M = (_basis(x, p, Rs) - _basis(xt, p, Rs))[:, 1:]
    else:
        M = _basis(x, p, Rs)
    scale = torch.linalg.vector_norm(M, dim=0)
    A = torch.linalg.lstsq(M / scale, b[:, None]).solution[:, 0] / scale
    if bc == hsma.PERIODIC:
        A = torch.cat((torch.zeros(1, dtype=torch.float64, device="cuda"), A))

    if far_field == "series":
        phi_out, e_out = _basis_gradient(c, p, Rs, A)
    else:
        F2, F1 = _fib2(Q)
        j = torch.arange(F2 + 1, dtype=torch.float64, device="cuda")
        z = -1.0 + 2.0 * j / F2
        ct = torch.clamp(z + torch.sin(math.pi * z) / math.pi, -1.0, 1.0)
        st = torch.sqrt(1.0 - ct * ct)
        ph = math.pi * torch.remainder(j * F1, 2 * F2) / F2
        w = 2.0 * math.pi * Rs * Rs / F2 * (1.0 + torch.cos(math.pi * z))
        d = torch.stack((st * torch.cos(ph), st * torch.sin(ph), ct), 1)
        d = torch.cat((d, d * torch.tensor([-1.0, -1.0, 1.0], dtype=torch.float64, device="cuda")))
        w = torch.cat((w, w)) / (4.0 * math.pi)
        B = _basis(Rs * d, p, Rs)
        n = torch.floor(torch.sqrt(torch.arange((p + 1) ** 2, dtype=torch.float64, device="cuda") + 0.5))
        sigma, mu = w * (B @ (n * A)) / Rs, w * (B @ A)
        dr = (1e-5 if bc == hsma.PERIODIC else 1e-4) * Rs
        phi_out, e_out = _sums(Rs * d, sigma, c)
        # dipole layer: (1/a - 1/b) / dr with a, b the distances to the spheres Rs -+ dr/2
        for i in range(0, c.shape[0], 4096):
            t = c[i:i + 4096]
            va = [t[:, k, None] - (Rs - 0.5 * dr) * d[:, k] for k in range(3)]
            vb = [t[:, k, None] - (Rs + 0.5 * dr) * d[:, k] for k in range(3)]
            ra = torch.sqrt(va[0] ** 2 + va[1] ** 2 + va[2] ** 2)
            rb = torch.sqrt(vb[0] ** 2 + vb[1] ** 2 + vb[2] ** 2)
            diff = 2.0 * (Rs - t @ d.T) / ((ra + rb) * ra * rb)
            phi_out[i:i + 4096] += diff @ mu
            cube = diff * (1.0 / ra**2 + 1.0 / (ra * rb) + 1.0 / rb**2)
            for k in range(3):
                e_out[i:i + 4096, k] += (va[k] * cube + d[:, k] / rb**3) @ mu
    pot = phi + phi_out
    return 0.5 * torch.dot(q, pot).item(), q[:, None] * (e + e_out), pot, sx.shape[0]


def exact(case, seed):
    inp = _inputs(case, seed)
    if case["kind"] == "basis":
        return _basis(inp[0], case["p"], 1.5)
    if case["kind"] == "coulomb":
        pot, field = _sums(inp[0][:, :3], inp[0][:, 3].contiguous(), inp[1], field=case["field"])
        return {"pot": pot, "field": field}
    plan, far = PLANS[case["plan"]], case.get("far_field", "images")
    if case["kind"] == "step":
        e, f, p, n_inset = _exact_system(inp[0], inp[1], plan, far)
        return {"energy": e, "forces": f, "potentials": p if case.get("potentials") else None, "n_inset": n_inset}
    off = np.concatenate([[0], np.cumsum(_sizes(case, seed))])
    parts = [_exact_system(inp[0][a:b], inp[1][a:b], plan, far) for a, b in zip(off[:-1], off[1:])]
    return {"energy": np.array([v[0] for v in parts]), "forces": torch.cat([v[1] for v in parts]),
            "status": np.zeros(len(parts), dtype=np.int32)}
