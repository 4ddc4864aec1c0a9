"""The performance cases of the mixed-basis library: what a user's program
asks of it, through its public entry points (``mb.Handle``).

A case names a cell of ``workloads`` (with its number of retained B-splines,
k-points and bands), an operation and a precision:

* ``H``       Y = H X of every k-point in one batched call;
* ``S``, ``Sinv``  the same for the overlap and its inverse;
* ``eig``     the lowest roots of H c = eps S c at every k-point to 1e-6 Ha, as a
              band structure takes them (the eigenvalues: the vectors are
              fixed only up to phases and mixes of degenerate roots);
* ``fields``  the fields of one self-consistent step: the electron density of
              given bands, its Coulomb potential and its LDA potential.

Trial blocks are seeded normal deviates, as in the parity tests; the bands of
``fields`` are smooth and localized in z like a slab's states, with
Fermi-Dirac occupations.  ``exact`` restates the operators in 64 bits from
their definitions (B-splines by the Cox-de Boor recursion, Gauss-Legendre
planes, plain FFTs), without the library."""
import dataclasses
import math

import numpy as np
import torch

from paper_1406_4960_gb300 import mb
from paper_1406_4960_gb300 import workloads as W

DEV = "cuda"


def listed():
    return [
        # the smallest call: one k-point of the two-well cell, 8 bands, FP64 (latency and launches)
        {"name": "H tiny fp64", "op": "H", "cell": "tiny", "nb": 40, "nk": 1, "bands": 8, "prec": "fp64"},
        # the benchmark's block: the C(001)-like slab at its 4 k-points, the bulk cycles' precision
        {"name": "H slab fp32", "op": "H", "cell": "slab", "nb": 120, "nk": 4, "bands": 32, "prec": "fp32"},
        # the same in FP64: every cycle of a plain FP64 solve, the finish cycles of a mixed one
        {"name": "H slab fp64", "op": "H", "cell": "slab", "nb": 120, "nk": 4, "bands": 32, "prec": "fp64"},
        # the 4 x 4 graphene cell: a wide disc (1417 G) on a 64 x 64 grid, one k-point
        {"name": "H graphene fp32", "op": "H", "cell": "graphene", "nb": 80, "nk": 1, "bands": 80, "prec": "fp32"},
        {"name": "H graphene fp64", "op": "H", "cell": "graphene", "nb": 80, "nk": 1, "bands": 80, "prec": "fp64"},
        # the largest batch: 64 k-points of the 2 x 2 graphene cell in one call
        {"name": "H kbatch fp32", "op": "H", "cell": "kbatch", "nb": 100, "nk": 64, "bands": 24, "prec": "fp32"},
        # overlap products of a Gram-Schmidt step, and S^-1 of a residual norm
        {"name": "S slab fp32", "op": "S", "cell": "slab", "nb": 120, "nk": 4, "bands": 32, "prec": "fp32"},
        {"name": "Sinv slab fp64", "op": "Sinv", "cell": "slab", "nb": 120, "nk": 4, "bands": 32, "prec": "fp64"},
        # whole solves: the smallest in FP64; the slab and the graphene supercell in mixed precision
        {"name": "eig tiny fp64", "op": "eig", "cell": "tiny", "nb": 40, "nk": 1, "bands": 8, "prec": "fp64"},
        {"name": "eig slab mixed", "op": "eig", "cell": "slab", "nb": 120, "nk": 4, "bands": 32, "prec": "fp32"},
        {"name": "eig graphene mixed", "op": "eig", "cell": "graphene", "nb": 80, "nk": 1, "bands": 80, "prec": "fp32"},
        # the device steps between two solves of the self-consistent loop
        {"name": "fields slab", "op": "fields", "cell": "slab", "nb": 120, "nk": 4, "bands": 32, "prec": "fp64"},
    ]


def draw(rng):
    """A case of the served requests' ranges: 40-160 B-splines, 1-80 bands,
    1-8 k-points (up to 64 for the k-point batches)."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["H", "H", "H", "S", "Sinv", "eig", "fields"])
    cell = rng.choice(["tiny", "slab", "graphene", "kbatch"])
    c = {"op": op, "cell": cell, "nb": rng.randint(40, 160), "nk": log_int(1, 8), "bands": log_int(1, 80),
         "prec": rng.choice(["fp32", "fp32", "fp64"])}
    if cell == "kbatch" and op in ("H", "S", "Sinv"):
        c["nk"], c["bands"], c["prec"] = log_int(1, 64), log_int(1, 24), "fp32"
    if cell == "graphene":
        c["nk"] = 1
        c["nb"] = min(c["nb"], 100)
    if op == "eig":
        c["cell"] = cell if cell in ("tiny", "slab") else "tiny"
        c["nk"] = min(c["nk"], 2)
        c["bands"] = min(c["bands"] + 3, 32)
        if c["prec"] == "fp64":
            c["cell"] = "tiny"
    if op == "fields":
        c["prec"] = "fp64"
        c["cell"] = cell if cell in ("tiny", "slab") else "slab"
        c["nk"], c["bands"] = min(c["nk"], 4), min(c["bands"], 32)
    return c


def _workload(case, seed):
    """The cell at the case's z resolution; the configurations' own k-points,
    or (for solves, and where the case wants another number of them) seeded ones."""
    nb = case["nb"]
    base = W.BY_NAME[case["cell"]]()
    n_int = nb - base.order + 3
    breaks = base.breaks
    if n_int != base.n_int:
        if case["cell"] == "slab":
            try:
                breaks = W.slab_geometric_breaks(n_int)
            except ValueError:
                breaks = W.uniform_breaks(-15.0, 15.0, n_int)
        else:
            breaks = W.uniform_breaks(float(base.breaks[0]), float(base.breaks[-1]), n_int)
    kpts = base.kpts
    if case["op"] == "eig" or case["nk"] != base.nk:
        kpts = W.random_kpoints(base.a1, base.a2, case["nk"], 1000 + seed)
    if case["cell"] in ("graphene", "kbatch"):
        # the wedge's own region: discs as the configured grid takes them
        kpts = base.kpts if case["nk"] == base.nk and case["op"] != "eig" else W.wedge_kpoints(
            base.a1, base.a2, case["nk"], 1000 + seed)
    return dataclasses.replace(base, breaks=breaks, kpts=np.asarray(kpts), nbands=case["bands"])


def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _blocks(case, seed, sizes):
    """Seeded trial blocks X[band][j][ldg] of every k-point, padding zero."""
    gen = _generator(seed)
    dt = torch.complex128 if case["prec"] == "fp64" else torch.complex64
    out = []
    for ng, nb, ldg in sizes:
        x = torch.randn((case["bands"], nb, ldg), dtype=dt, device=DEV, generator=gen)
        x[:, :, ng:] = 0
        out.append(x)
    return out


def _bands(case, seed, sizes, q2s):
    """Smooth localized bands in mb_eigsolve's layout (one flat buffer) and
    Fermi-Dirac occupations of equally weighted k-points."""
    gen = _generator(seed)
    parts = []
    for (ng, nb, ldg), q2 in zip(sizes, q2s):
        c = torch.randn((case["bands"], nb, ldg), dtype=torch.complex128, device=DEV, generator=gen)
        z = (torch.arange(nb, dtype=torch.float64, device=DEV) - 0.5 * (nb - 1)) / (0.18 * nb)
        w = torch.zeros(ldg, dtype=torch.float64, device=DEV)
        w[:ng] = torch.exp(-torch.from_numpy(q2).to(DEV) / 12.0)
        parts.append((0.3 * c * torch.exp(-z * z)[None, :, None] * w[None, None, :]).reshape(-1))
    e = np.linspace(-1.0, 0.5, case["bands"])
    occ = np.tile(2.0 / case["nk"] / (1.0 + np.exp((e - 0.1) / 0.1)), (case["nk"], 1))
    return torch.cat(parts), occ


def prepare(case, seed):
    w = _workload(case, seed)
    h = mb.Handle.from_workload(w)
    sizes = [h.sizes(ik) for ik in range(w.nk)]
    s = {"case": case, "h": h, "iks": list(range(w.nk))}
    if case["op"] in ("H", "S", "Sinv"):
        s["X"] = _blocks(case, seed, sizes)
        s["Y"] = [torch.empty_like(x) for x in s["X"]]
    elif case["op"] == "fields":
        s["evecs"], s["occ"] = _bands(case, seed, sizes, [_disc(w, ik)[2] for ik in range(w.nk)])
        nq = len(h.zplanes()[0])
        s["f"] = [torch.empty((nq,) + h.grid, dtype=torch.float64, device=DEV) for _ in range(3)]
    return s


def run(s):
    case, h = s["case"], s["h"]
    op = case["op"]
    if op == "H":
        h.apply_H_batch(s["iks"], s["X"], s["Y"], case["prec"])
        return s["Y"]
    if op == "S":
        h.apply_S_batch(s["iks"], s["X"], s["Y"], case["prec"])
        return s["Y"]
    if op == "Sinv":
        h.apply_Sinv_batch(s["iks"], s["X"], s["Y"], case["prec"])
        return s["Y"]
    if op == "eig":
        return h.eigsolve(case["bands"], 1e-6, case["prec"])[0]
    rho, vh, vxc = s["f"]
    h.density(s["evecs"], case["bands"], s["occ"], rho)
    h.hartree(rho, vh)
    h.xc_lda(rho, vxc)
    return [rho, vh, vxc]


def work(case):
    """Bytes: every block read once and written once, the tables read once.
    Operations: per B-spline row a transform to the grid and one back, the
    local potential's banded product along z there, the banded kinetic term
    and the projector sums (H); the banded products (S, S^-1).  A solve is
    counted as one Krylov space of depth 5 and one FP64 product per root."""
    w = _workload(case, 0)
    cb = 16 if case["prec"] == "fp64" else 8
    n1, n2 = w.grid
    N = n1 * n2
    nq = w.n_int * w.nquad
    nb, M, kap = w.nb_retained, case["bands"], w.order
    nproj = sum(a.nproj for a in w.atoms)
    nz = len({(a.pos[2], a.rc, p == 3) for a in w.atoms for p in range(a.nproj)})
    ngs = [len(_disc(w, ik)[0]) for ik in range(w.nk)]
    vec = float(sum(ngs)) * nb * M                       # coefficients of the block
    rows = float(w.nk) * nb * M
    band = 4.0 * (2 * kap - 1) * vec
    h_flops = rows * (10.0 * N * math.log2(N) + 4.0 * (2 * kap - 1) * N) + 1.5 * band + 8.0 * nz * vec + sum(
        16.0 * nproj * g * M for g in ngs)
    h_bytes = 2.0 * vec * cb + nq * N * cb / 2 + sum(nproj * (g + nb) * cb for g in ngs)
    if case["op"] == "H":
        return {"bytes": h_bytes, "flops": h_flops}
    if case["op"] in ("S", "Sinv"):
        return {"bytes": 2.0 * vec * cb, "flops": band}
    if case["op"] == "eig":
        return {"bytes": 6.0 * h_bytes, "flops": 6.0 * (h_flops + band)}
    return {"bytes": vec * cb + 24.0 * nq * N,
            "flops": rows * 5.0 * N * math.log2(N) + float(w.nk) * M * nq * N * (4.0 * kap + 4.0)}


# ---- the definitions in 64 bits ---------------------------------------------

def _disc(w, ik):
    """Integer G of the cutoff disc ordered by (n2, n1), k + G and |k + G|^2."""
    b1, b2 = W.reciprocal(w.a1, w.a2)
    n1, n2 = w.grid
    i1, i2 = np.meshgrid(np.arange(-n1, n1 + 1), np.arange(-n2, n2 + 1), indexing="ij")
    g = np.stack([i1.ravel(), i2.ravel()], axis=1)
    q = w.kpts[ik] + g[:, :1] * b1 + g[:, 1:] * b2
    q2 = (q * q).sum(1)
    keep = 0.5 * q2 <= w.ecut
    g, q, q2 = g[keep], q[keep], q2[keep]
    o = np.lexsort((g[:, 0], g[:, 1]))
    return g[o], q[o], q2[o]


def _zbasis(w):
    """Gauss planes and weights, the retained B-splines and their derivatives there."""
    x, wt = np.polynomial.legendre.leggauss(w.nquad)
    br = np.asarray(w.breaks, dtype=np.float64)
    hs = np.diff(br)
    zq = (br[:-1, None] + 0.5 * hs[:, None] * (x + 1.0)[None]).ravel()
    wq = (0.5 * hs[:, None] * wt[None]).ravel()
    k = w.order
    tau = np.concatenate([np.full(k - 1, br[0]), br, np.full(k - 1, br[-1])])
    B = ((tau[None, :-1] <= zq[:, None]) & (zq[:, None] < tau[None, 1:])).astype(np.float64)

    def over(a, b):
        return np.divide(a, b, out=np.zeros(np.broadcast(a, b).shape), where=b != 0)

    lower = None
    for m in range(2, k + 1):
        n = len(tau) - m
        lower = B
        B = over(zq[:, None] - tau[None, :n], np.broadcast_to(tau[m - 1:m - 1 + n] - tau[:n], (len(zq), n))) * B[:, :n] \
            + over(tau[None, m:m + n] - zq[:, None], np.broadcast_to(tau[m:m + n] - tau[1:1 + n], (len(zq), n))) * B[:, 1:n + 1]
    n = len(tau) - k
    dB = (k - 1) * (over(lower[:, :n], np.broadcast_to(tau[k - 1:k - 1 + n] - tau[:n], (len(zq), n)))
                    - over(lower[:, 1:n + 1], np.broadcast_to(tau[k:k + n] - tau[1:1 + n], (len(zq), n))))
    return zq, wq, B[:, 1:-1], dB[:, 1:-1]


def _grid_g(w):
    b1, b2 = W.reciprocal(w.a1, w.a2)
    n1, n2 = w.grid
    m1 = (np.arange(n1) + n1 // 2) % n1 - n1 // 2
    m2 = (np.arange(n2) + n2 // 2) % n2 - n2 // 2
    return m1[:, None, None] * b1 + m2[None, :, None] * b2


def _cell_area(w):
    return abs(w.a1[0] * w.a2[1] - w.a1[1] * w.a2[0])


def _potential(w, zq):
    """V(r_par, z_q) of the atoms' Gaussian wells on the grid."""
    n1, n2 = w.grid
    g = _grid_g(w)
    c = np.zeros((len(zq), n1, n2), dtype=np.complex128)
    for at in w.atoms:
        a = 0.5 / (at.w * at.w)
        f = (at.A / _cell_area(w)) * (math.pi / a) * np.exp(-(g * g).sum(-1) / (4 * a)) * np.exp(
            -1j * (g[..., 0] * at.pos[0] + g[..., 1] * at.pos[1]))
        c += np.exp(-a * (zq - at.pos[2]) ** 2)[:, None, None] * f[None]
    return n1 * n2 * np.fft.ifft2(c, axes=(1, 2)).real


def _projectors(w, q, q2, zq, wq, B):
    """z factors (nproj, nb), in-plane factors (nproj, ng) and strengths."""
    zs, qs, es = [], [], []
    for at in w.atoms:
        if not at.nproj:
            continue
        al = 0.5 / (at.rc * at.rc)
        dz = zq - at.pos[2]
        gz = np.exp(-al * dz * dz)
        z0, z1 = B.T @ (wq * gz), B.T @ (wq * dz * gz)
        f = (math.pi / al) * np.exp(-q2 / (4 * al))
        cs = (2 * al / math.pi) ** 0.75
        cp = 2 * math.sqrt(al) * cs
        ph = np.exp(-1j * (q[:, 0] * at.pos[0] + q[:, 1] * at.pos[1])) / math.sqrt(_cell_area(w))
        for z, y in ((z0, cs * f), (z0, -1j * cp * q[:, 0] / (2 * al) * f), (z0, -1j * cp * q[:, 1] / (2 * al) * f),
                     (z1, cp * f)):
            zs.append(z)
            qs.append(ph * y)
        es += list(at.E)
    return np.array(zs), np.array(qs), np.array(es)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _exact_apply(case, w, X):
    zq, wq, B, dB = _zbasis(w)
    S, D = _dev(B.T @ (wq[:, None] * B)), _dev(dB.T @ (wq[:, None] * dB))
    n1, n2 = w.grid
    V = _dev(_potential(w, zq)) if case["op"] == "H" else None
    Bd, wd = _dev(B), _dev(wq)
    out = []
    for ik, x in enumerate(X):
        g, q, q2 = _disc(w, ik)
        ng = len(g)
        y = torch.zeros(x.shape, dtype=torch.complex128, device=DEV)
        xs = x[:, :, :ng].to(torch.complex128)
        if case["op"] == "S":
            y[:, :, :ng] = torch.einsum("ij,bjg->big", S.to(xs.dtype), xs)
        elif case["op"] == "Sinv":
            f = torch.linalg.cholesky(S)
            for b in range(xs.shape[0]):
                r = torch.cat([xs[b].real, xs[b].imag], dim=1)
                r = torch.cholesky_solve(r, f)
                y[b, :, :ng] = torch.complex(r[:, :ng].contiguous(), r[:, ng:].contiguous())
        else:
            pos = _dev((g[:, 0] % n1) * n2 + g[:, 1] % n2)
            zf, qf, es = _projectors(w, q, q2, zq, wq, B)
            kin = 0.5 * _dev(q2)
            for b in range(xs.shape[0]):
                xb = xs[b]
                psi = torch.zeros((len(zq), n1 * n2), dtype=torch.complex128, device=DEV)
                psi[:, pos] = Bd.to(xb.dtype) @ xb
                psi = torch.fft.ifft2(psi.view(-1, n1, n2)) * V
                psi = torch.fft.fft2(psi).view(len(zq), -1)[:, pos]
                yb = Bd.T.to(xb.dtype) @ (wd[:, None] * psi)
                yb += 0.5 * (D.to(xb.dtype) @ xb) + kin[None] * (S.to(xb.dtype) @ xb)
                if len(es):
                    zd, qd = _dev(zf).to(xb.dtype), _dev(qf)
                    c = _dev(es) * ((zd @ xb) * qd.conj()).sum(1)
                    yb += zd.T @ (c[:, None] * qd)
                y[b, :, :ng] = yb
        out.append(y)
    return out


def _exact_eig(case, w):
    """The lowest roots of the dense generalized problem, k-point by k-point."""
    zq, wq, B, dB = _zbasis(w)
    S, D = B.T @ (wq[:, None] * B), dB.T @ (wq[:, None] * dB)
    n1, n2 = w.grid
    vg = np.fft.fft2(_potential(w, zq), axes=(1, 2)) / (n1 * n2)
    nb = B.shape[1]
    bz = B.T[:, None, :] * B.T[None, :, :] * wq                       # i, j, q
    ev = []
    for ik in range(w.nk):
        g, q, q2 = _disc(w, ik)
        ng = len(g)
        d1 = (g[:, None, 0] - g[None, :, 0]) % n1
        d2 = (g[:, None, 1] - g[None, :, 1]) % n2
        ms, inv = np.unique(d1 * n2 + d2, return_inverse=True)
        blk = _dev(bz.reshape(nb * nb, -1)).to(torch.complex128) @ _dev(vg.reshape(len(zq), -1)[:, ms])
        H = blk[:, _dev(inv.reshape(-1))].view(nb, nb, ng, ng).permute(0, 2, 1, 3).reshape(nb * ng, nb * ng).clone()
        H += torch.kron(_dev(0.5 * D), torch.eye(ng, dtype=torch.float64, device=DEV)).to(H.dtype)
        H += torch.kron(_dev(S), torch.diag(_dev(0.5 * q2))).to(H.dtype)
        zf, qf, es = _projectors(w, q, q2, zq, wq, B)
        if len(es):
            U = _dev((zf[:, :, None] * qf[:, None, :]).reshape(len(es), -1))
            H += U.T @ (_dev(es)[:, None] * U.conj())
        Li = _dev(np.linalg.inv(np.linalg.cholesky(S)))
        H = H.view(nb, ng * nb * ng)
        H = (Li.to(H.dtype) @ H).view(nb * ng, nb, ng)
        H = torch.einsum("ajg,ij->aig", H, Li.to(H.dtype)).reshape(nb * ng, nb * ng)
        ev.append(torch.linalg.eigvalsh(0.5 * (H + H.conj().T))[: case["bands"]])
    return torch.stack(ev).cpu().numpy()


def _exact_fields(case, w, evecs, occ):
    zq, wq, B, _ = _zbasis(w)
    n1, n2 = w.grid
    nb, ac = B.shape[1], _cell_area(w)
    Bd = _dev(B).to(torch.complex128)
    rho = torch.zeros((len(zq), n1, n2), dtype=torch.float64, device=DEV)
    off = 0
    for ik in range(w.nk):
        g = _disc(w, ik)[0]
        ng = len(g)
        ldg = (ng + 31) // 32 * 32
        pos = _dev((g[:, 0] % n1) * n2 + g[:, 1] % n2)
        c = evecs[off:off + case["bands"] * nb * ldg].view(case["bands"], nb, ldg)[:, :, :ng]
        off += case["bands"] * nb * ldg
        for b in range(case["bands"]):
            psi = torch.zeros((len(zq), n1 * n2), dtype=torch.complex128, device=DEV)
            psi[:, pos] = Bd @ c[b]
            psi = torch.fft.ifft2(psi.view(-1, n1, n2)) * (n1 * n2)
            rho += float(occ[ik, b]) / ac * (psi.real ** 2 + psi.imag ** 2)
    rg = (torch.fft.fft2(rho) / (n1 * n2)).view(len(zq), -1)
    gn = _dev(np.sqrt((_grid_g(w) ** 2).sum(-1)).ravel())
    dz = (_dev(zq)[:, None] - _dev(zq)[None, :]).abs()
    wr = _dev(wq)[:, None] * rg
    vg = torch.empty_like(rg)
    for m in range(n1 * n2):
        gm = float(gn[m])
        ker = -2 * math.pi * dz if gm == 0 else (2 * math.pi / gm) * torch.exp(-gm * dz)
        vg[:, m] = ker.to(wr.dtype) @ wr[:, m]
    vh = (torch.fft.ifft2(vg.view(-1, n1, n2)) * (n1 * n2)).real
    d = rho.clamp(min=1e-10)
    rs = (3.0 / (4.0 * math.pi * d)) ** (1.0 / 3.0)
    ex = -0.75 * (3.0 * d / math.pi) ** (1.0 / 3.0)
    sr, lr = rs.sqrt(), rs.log()
    den = 1.0 + 1.0529 * sr + 0.3334 * rs
    vlo = -0.1423 / den * (1.0 + 7.0 / 6.0 * 1.0529 * sr + 4.0 / 3.0 * 0.3334 * rs) / den
    vhi = 0.0311 * lr + (-0.048 - 0.0311 / 3.0) + 2.0 / 3.0 * 0.0020 * rs * lr + (2.0 * -0.0116 - 0.0020) * rs / 3.0
    return [rho, vh, 4.0 / 3.0 * ex + torch.where(rs >= 1.0, vlo, vhi)]


def exact(case, seed):
    w = _workload(case, seed)
    discs = [_disc(w, ik) for ik in range(w.nk)]
    sizes = [(len(d[0]), w.nb_retained, (len(d[0]) + 31) // 32 * 32) for d in discs]
    if case["op"] == "eig":
        # beyond a few thousand basis functions the dense problem takes too long
        return _exact_eig(case, w) if max(s[0] for s in sizes) * w.nb_retained <= 3000 else None
    if case["op"] == "fields":
        evecs, occ = _bands(case, seed, sizes, [d[2] for d in discs])
        return _exact_fields(case, w, evecs, occ)
    return _exact_apply(case, w, _blocks(case, seed, sizes))
