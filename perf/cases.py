"""Performance cases of the framework: what a multiscale SU(3) simulation has it do.

A case is a dict of plain values.  `prepare` makes the inputs on the GPU from the
case and a seed (gauge fields with the plaquette of a thermalised ensemble, in a
random gauge) with torch alone, `run` makes one pass through the public entry
points of paper_1510_04675_gb300, `work` counts what that pass cannot do without,
and `exact` computes the same outputs in 64-bit torch without the framework.

The kinds of work (key "kind"):
  update         1 heat-bath + n_or overrelaxation sweeps with the plaquette record
  batch_update   the same on many lattices of uneven extents at once
  leapfrog       one P-step and one Q-step of the HMC integrator
  hmc            a whole HMC trajectory with its Metropolis test
  flow           fixed-step Wilson flow with E(t), Q(t)
  adaptive       adaptive-step Wilson flow with E(t), Q(t)
  prolong        coarse -> fine prolongation with the device-side stopping rule
  batch_prolong  the same map for many lattices, a fixed number of smoothing steps
  gradient       a flowed clover observable and its gradient through the flow
  measure        a stored configuration imported and measured
"""
import math

import numpy as np
import torch

from paper_1510_04675_gb300 import api, autograd

# the coupling, and the noise per link whose plaquette (0.59) is that of a thermalised field there
BETA, SPREAD = 6.0, 0.22


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest production call: the 8^4, beta = 5.7 benchmark chain in FP64
        {"name": "update_8x4_f64", "kind": "update", "dims": "8 8 8 8", "prec": "f64", "n_or": 4, "sweeps": 1},
        # rethermalisation of a prolongated 16^4 lattice
        {"name": "update_16x4_f32c12", "kind": "update", "dims": "16 16 16 16", "prec": "f32c12", "n_or": 4, "sweeps": 2},
        # the headline workload: 32^4 compound sweeps in the 12-real format
        {"name": "update_32x4_f32c12", "kind": "update", "dims": "32 32 32 32", "prec": "f32c12", "n_or": 4, "sweeps": 2},
        # an ensemble of uneven lattices (12^4, 16^4, 8^3x16) rethermalised together
        {"name": "batch_update_48", "kind": "batch_update", "n": 48, "scale": 2, "prec": "f32c12", "n_or": 4, "sweeps": 1},
        # the leapfrog of the 24^4, beta = 6.0 HMC
        {"name": "leapfrog_24x4_f32c12", "kind": "leapfrog", "dims": "24 24 24 24", "prec": "f32c12"},
        # a short trajectory on a small ragged lattice in FP64 (the parity path)
        {"name": "hmc_8x12_f64", "kind": "hmc", "dims": "8 8 8 12", "prec": "f64", "steps": 10},
        # scale setting on the 16^4 lattice of the multiscale step
        {"name": "flow_16x4_f32c12", "kind": "flow", "dims": "16 16 16 16", "prec": "f32c12", "steps": 20, "every": 10},
        # the 24^3x48, beta = 5.96 flow with step control, 18-real links
        {"name": "adaptive_24x48_f32", "kind": "adaptive", "dims": "24 24 24 48", "prec": "f32", "t_end": 1.0},
        # the 8^4 -> 16^4 refinement with the 0.001 % stopping rule
        {"name": "prolong_8_16_f32c12", "kind": "prolong", "dims": "8 8 8 8", "prec": "f32c12"},
        # the uneven ensemble refined together
        {"name": "batch_prolong_48", "kind": "batch_prolong", "n": 48, "scale": 1, "prec": "f32c12", "max_iter": 20},
        # gradient of the flowed topological charge through the flow
        {"name": "gradient_q_16x4_f32c12", "kind": "gradient", "dims": "16 16 16 16", "prec": "f32c12", "obs": "Q", "steps": 4},
        # a stored 24^3x48 configuration loaded and measured
        {"name": "measure_24x48_f32c12", "kind": "measure", "dims": "24 24 24 48", "prec": "f32c12", "m": 2, "n": 3},
    ]


def _draw_dims(rng, vmin, vmax):
    """Four even extents of a volume spread over the logarithm of [vmin, vmax], ragged as often as not."""
    v = math.exp(rng.uniform(math.log(vmin), math.log(vmax)))
    skew = rng.choice([0.0, 0.35])
    d = [max(4, 2 * round(v ** 0.25 * math.exp(rng.uniform(-skew, skew)) / 2)) for _ in range(4)]
    while d[0] * d[1] * d[2] * d[3] > vmax:
        d[d.index(max(d))] -= 2
    if rng.random() < 0.5:
        d[rng.randrange(4)] += 2
        while d[0] * d[1] * d[2] * d[3] > vmax:
            d[d.index(max(d))] -= 2
    return " ".join(map(str, d))


def draw(rng):
    kind = rng.choice(["update", "update", "batch_update", "leapfrog", "hmc", "flow", "adaptive", "prolong", "batch_prolong",
                       "gradient", "measure"])
    prec = rng.choice(["f64", "f32", "f32c12", "f32c12"])
    top = 0.1 if prec == "f64" else 1.0  # FP64 runs on the smaller lattices
    if kind == "update":
        return {"kind": kind, "dims": _draw_dims(rng, 4 ** 4, top * 32 ** 4), "prec": prec, "n_or": rng.choice([1, 4]),
                "sweeps": rng.choice([1, 2])}
    if kind == "batch_update":
        return {"kind": kind, "n": rng.randint(5, 48), "scale": 1 if prec == "f64" else rng.choice([1, 2]), "prec": prec,
                "n_or": rng.choice([1, 4]), "sweeps": 1}
    if kind == "leapfrog":
        return {"kind": kind, "dims": _draw_dims(rng, 4 ** 4, top * 24 ** 4), "prec": prec}
    if kind == "hmc":
        return {"kind": kind, "dims": _draw_dims(rng, 4 ** 4, 6144), "prec": "f64", "steps": rng.choice([5, 10])}
    if kind == "flow":
        return {"kind": kind, "dims": _draw_dims(rng, 4 ** 4, top * 16 ** 4), "prec": prec, "steps": rng.choice([10, 20]),
                "every": rng.choice([1, 5, 10])}
    if kind == "adaptive":
        return {"kind": kind, "dims": _draw_dims(rng, 4 ** 4, top * 24 ** 3 * 48), "prec": prec, "t_end": rng.choice([0.5, 1.0])}
    if kind == "prolong":
        return {"kind": kind, "dims": _draw_dims(rng, 4 ** 4, 0.25 * 8 ** 4 if prec == "f64" else 8 ** 4), "prec": prec}
    if kind == "batch_prolong":
        return {"kind": kind, "n": rng.randint(4, 6 if prec == "f64" else 48), "scale": 1, "prec": prec, "max_iter": rng.choice([10, 20])}
    if kind == "gradient":
        return {"kind": kind, "dims": _draw_dims(rng, 4 ** 4, top * 16 ** 4), "prec": prec, "obs": rng.choice(["E", "Q", "S"]),
                "steps": rng.choice([2, 4])}
    return {"kind": kind, "dims": _draw_dims(rng, 4 ** 4, top * 24 ** 3 * 48), "prec": prec, "m": rng.choice([1, 2]),
            "n": rng.choice([2, 3, 4])}


# ------------------------------------------------------------------ gauge fields in plain torch
# A field is U[mu, x3, x2, x1, x0, 3, 3], complex128.
def _dims(case):
    return [int(v) for v in case["dims"].split()]


def _batch_dims(case):
    """Extents of a batch: 3/8 of 6^4, 3/8 of 8^4 and 1/4 of 4^3x8, times `scale`."""
    s = case["scale"]
    shapes = [[6, 6, 6, 6], [8, 8, 8, 8], [4, 4, 4, 8], [6, 6, 6, 6], [8, 8, 8, 8], [6, 6, 6, 6], [8, 8, 8, 8], [4, 4, 4, 8]]
    return [[s * v for v in shapes[i % 8]] for i in range(case["n"])]


def _generator(seed, device):
    return torch.Generator(device=device).manual_seed(int(seed) & 0x7FFFFFFFFFFF)


def _gauss(shape, g, device):
    return torch.view_as_complex(torch.randn(*shape, 2, generator=g, device=device, dtype=torch.float64))


def _unitary(z):
    """Rows 0 and 1 orthonormalised, row 2 = conj(row0 x row1)."""
    a = z[..., 0, :]
    a = a / torch.linalg.vector_norm(a, dim=-1, keepdim=True)
    b = z[..., 1, :]
    b = b - (b * a.conj()).sum(-1, keepdim=True) * a
    b = b / torch.linalg.vector_norm(b, dim=-1, keepdim=True)
    return torch.stack([a, b, torch.linalg.cross(a, b).conj()], dim=-2)


def _dag(a):
    return a.mH


def _mm(*factors):
    """Product of 3x3 matrices, elementwise (a batched matrix product of so small matrices is far slower)."""
    r = factors[0]
    for b in factors[1:]:
        r = r[..., :, 0:1] * b[..., 0:1, :] + r[..., :, 1:2] * b[..., 1:2, :] + r[..., :, 2:3] * b[..., 2:3, :]
    return r


def _at(f, mu, n=1):
    """f(x + n e_mu) of a site field f[x3, x2, x1, x0, ...]."""
    return torch.roll(f, -n, dims=3 - mu)


def _flux(dims, device):
    """Phases of a constant field of one flux quantum in the (0,1) and (2,3) planes (charge 2 in SU(3) on diag(1, -1, 0))."""
    x = torch.meshgrid(*[torch.arange(L, device=device, dtype=torch.float64) for L in reversed(dims)], indexing="ij")[::-1]
    theta = []
    for a, b in ((0, 1), (2, 3)):
        f = 2 * math.pi / (dims[a] * dims[b])
        theta += [torch.where(x[a] == dims[a] - 1, -f * dims[a] * x[b], torch.zeros_like(x[b])), f * x[a]]
    diag = torch.tensor([1.0, -1.0, 0.0], dtype=torch.float64, device=device)
    return [torch.exp(1j * t[..., None] * diag) for t in theta]


def make_field(dims, seed, device="cuda"):
    """Links with the plaquette of a thermalised field and a topological charge, in a random gauge."""
    g = _generator(seed, device)
    shape = tuple(reversed(dims))
    flux = _flux(dims, device)
    gauge = _unitary(_gauss(shape + (3, 3), g, device))
    eye = torch.eye(3, dtype=torch.complex128, device=device)
    U = torch.empty((4,) + shape + (3, 3), dtype=torch.complex128, device=device)
    for mu in range(4):
        near = _unitary(eye + SPREAD * _gauss(shape + (3, 3), g, device))
        U[mu] = _mm(gauge, near * flux[mu][..., None, :], _dag(_at(gauge, mu)))
    return U


def _rounded(U, prec):
    """The field the library holds after importing U."""
    if prec == "f64":
        return U
    U = U.to(torch.complex64).to(torch.complex128)
    if prec == "f32":
        return U
    return torch.cat([U[..., :2, :], torch.linalg.cross(U[..., 0, :], U[..., 1, :]).conj().unsqueeze(-2)], dim=-2)


def _canonical(U):
    """double[V][4][3][3][2], the layout of mgq_import_links."""
    V = U[0].numel() // 9
    return torch.view_as_real(U.reshape(4, V, 3, 3).transpose(0, 1).contiguous()).reshape(-1)


def _sites(dims, device):
    """Lexicographic site of each (parity, h)."""
    V = dims[0] * dims[1] * dims[2] * dims[3]
    lex = torch.arange(0, V, 2, device=device)
    r, par = lex, 0
    for L in dims:
        par = par + r % L
        r = r // L
    return torch.stack([lex + (par + p) % 2 for p in (0, 1)])


def _to_links(U, dims, prec):
    """U as the library lays it out: [mu][parity][h/32][plane][h%32] (re, im), 12-real links as plane pairs."""
    V = dims[0] * dims[1] * dims[2] * dims[3]
    S = (V // 2 + 63) // 64 * 64
    planes = 6 if prec == "f32c12" else 9
    f = torch.zeros((4, 2, S, planes), dtype=torch.complex128, device=U.device)
    f[:, :, :V // 2] = U.reshape(4, V, 9)[:, _sites(dims, U.device), :planes]
    f = f.reshape(4, 2, S // 32, 32, planes)
    if prec == "f32c12":
        f = f.reshape(4, 2, S // 32, 32, 3, 2).transpose(3, 4)
    else:
        f = f.transpose(3, 4)
    return torch.view_as_real(f.contiguous()).reshape(-1)


def _lambda(device):
    m = torch.zeros((8, 3, 3), dtype=torch.complex128, device=device)
    for a, (i, j) in zip((0, 3, 5), ((0, 1), (0, 2), (1, 2))):
        m[a, i, j] = m[a, j, i] = 1
        m[a + 1, i, j], m[a + 1, j, i] = -1j, 1j
    m[2] = torch.diag(torch.tensor([1.0, -1.0, 0.0], dtype=torch.complex128, device=device))
    m[7] = torch.diag(torch.tensor([1.0, 1.0, -2.0], dtype=torch.complex128, device=device)) / math.sqrt(3)
    return m


def _alg_matrix(c):
    """sum_a c_a i lambda_a / 2."""
    return torch.einsum("...a,aij->...ij", c.to(torch.complex128), 0.5j * _lambda(c.device))


def _coeffs(M):
    """Coefficients of the traceless antihermitian part of M."""
    return -torch.einsum("...ij,aji->...a", M, 1j * _lambda(M.device)).real


def _ta(M):
    A = (M - _dag(M)) / 2
    return A - torch.eye(3, device=M.device) * torch.diagonal(A, dim1=-2, dim2=-1).sum(-1)[..., None, None] / 3


def _to_alg(c, dims):
    """Coefficients c[mu, x..., 8] in the momentum layout."""
    V = dims[0] * dims[1] * dims[2] * dims[3]
    S = (V // 2 + 63) // 64 * 64
    f = torch.zeros((4, 2, S, 8), dtype=torch.float64, device=c.device)
    f[:, :, :V // 2] = c.reshape(4, V, 8)[:, _sites(dims, c.device)]
    return f.reshape(4, 2, S // 32, 32, 8).transpose(3, 4).reshape(-1)


def _from_alg(buf, dims):
    V = dims[0] * dims[1] * dims[2] * dims[3]
    S = (V // 2 + 63) // 64 * 64
    f = buf.double().reshape(4, 2, S // 32, 8, 32).transpose(3, 4).reshape(4, 2, S, 8)[:, :, :V // 2]
    out = torch.empty((4, V, 8), dtype=torch.float64, device=buf.device)
    out[:, _sites(dims, buf.device)] = f
    return out.reshape((4,) + tuple(reversed(dims)) + (8,))


def _exp(X):
    """exp of small antihermitian matrices: Taylor series with scaling and squaring."""
    s = max(0, math.ceil(math.log2(max(1e-30, float(torch.linalg.matrix_norm(X.detach()).max()) / 0.25)))) if X.numel() else 0
    Y = X / 2 ** s
    eye = torch.eye(3, dtype=X.dtype, device=X.device)
    E = eye + Y / 14
    for k in range(13, 0, -1):
        E = eye + _mm(Y, E) / k
    for _ in range(s):
        E = _mm(E, E)
    return E


def _staple(U, mu):
    A = 0
    for nu in range(4):
        if nu != mu:
            f = _at(U[nu], mu)
            A = A + _mm(f, _dag(_mm(U[nu], _at(U[mu], nu)))) + _at(_mm(_dag(_mm(U[mu], f)), U[nu]), nu, -1)
    return A


def _generator_field(U):
    """Z(W) = -TA(W A(W)) of every link."""
    return torch.stack([-_ta(_mm(U[mu], _staple(U, mu))) for mu in range(4)])


def _flow_step(U, eps):
    Z0 = eps * _generator_field(U)
    W = _mm(_exp(Z0 / 4), U)
    Z1 = eps * _generator_field(W)
    W = _mm(_exp(8 / 9 * Z1 - 17 / 36 * Z0), W)
    Z2 = eps * _generator_field(W)
    return _mm(_exp(0.75 * Z2 - 8 / 9 * Z1 + 17 / 36 * Z0), W), 2 * Z1 - Z0


def _line(U, mu, m):
    P = U[mu]
    for k in range(1, m):
        P = _mm(P, _at(U[mu], mu, k))
    return P


def _clover(U, mu, nu, m=1):
    """Traceless part of (Q - Q^+)/8, Q the four m x m leaves of plane (mu, nu)."""
    a, b = _line(U, mu, m), _line(U, nu, m)
    a_n, b_m = _at(a, nu, m), _at(b, mu, m)
    up, dn = _mm(a, b_m), _mm(b, a_n)  # the two ways round the loop whose corner is x
    Q = _mm(up, _dag(dn))
    Q = Q + _at(_mm(b_m, _dag(dn), a), mu, -m)
    Q = Q + _at(_at(_mm(_dag(dn), up), mu, -m), nu, -m)
    Q = Q + _at(_mm(_dag(b), up, _dag(a_n)), nu, -m)
    return _ta(Q) / 4


def _trace(M):
    return torch.diagonal(M, dim1=-2, dim2=-1).sum(-1).real


def _charge(U, m=1):
    q = 0
    for s, (p, r) in ((1, ((0, 1), (2, 3))), (-1, ((0, 2), (1, 3))), (1, ((0, 3), (1, 2)))):
        q = q - s * _trace(_mm(_clover(U, *p, m), _clover(U, *r, m))).sum() / (4 * math.pi ** 2)
    return q


def _energy(U):
    return -sum(_trace(_mm(G, G)).sum() for G in (_clover(U, p, r) for p in range(4) for r in range(p + 1, 4))) / (U[0].numel() // 9)


def _loop(U, mu, nu, m, n):
    """(1/3) Re Tr of the m x n loop of plane (mu, nu) at every site."""
    a, b = _line(U, mu, m), _line(U, nu, n)
    return _trace(_mm(a, _at(b, mu, m), _dag(_mm(b, _at(a, nu, n))))) / 3


def _planes():
    return [(mu, nu) for mu in range(4) for nu in range(mu + 1, 4)]


def _odd(dims, device):
    """odd[mu][x3, x2, x1, x0]: whether x_mu is odd."""
    return [(torch.arange(L, device=device) % 2 == 1).reshape([-1 if 3 - k == mu else 1 for k in range(4)]).expand(*reversed(dims))
            for mu, L in enumerate(dims)]


def _project(M):
    """The SU(3) matrix W maximising Re Tr(W M^+): Gram-Schmidt start, then passes over the SU(2) subgroups."""
    W = _unitary(M)
    for _ in range(8):
        for i, j in ((0, 1), (0, 2), (1, 2)):
            V = _mm(W, _dag(M))
            a = (V[..., i, i] + V[..., j, j].conj()).conj()
            b = V[..., j, i].conj() - V[..., i, j]
            n = torch.sqrt((a.abs() ** 2 + b.abs() ** 2).clamp_min(1e-300))
            a, b = a / n, b / n
            ri, rj = W[..., i, :], W[..., j, :]
            W = W.clone()
            W[..., i, :], W[..., j, :] = (a[..., None] * ri + b[..., None] * rj,
                                          -b.conj()[..., None] * ri + a.conj()[..., None] * rj)
    return W


def _prolongate(Uc, cdims, c, rel_tol, max_iter):
    """The refined field, as the library's prolongation defines it, and the final S_d of the stages."""
    dims = [2 * v for v in cdims]
    dev = Uc.device
    U = torch.eye(3, dtype=torch.complex128, device=dev).expand((4,) + tuple(reversed(dims)) + (3, 3)).clone()
    U[:, ::2, ::2, ::2, ::2] = Uc
    odd = _odd(dims, dev)
    V = dims[0] * dims[1] * dims[2] * dims[3]
    index = torch.arange(V, device=dev).reshape(*reversed(dims))
    hop = {(mu, s): _at(index, mu, s).reshape(-1) for mu in range(4) for s in (1, -1)}
    flat = U.reshape(4, V, 3, 3)
    sds, counts = [], []
    for d in range(3):
        bonds = []  # per mu: the active sites and, per nu, which of them have n_nu odd
        for mu in range(4):
            chi = sum(odd[r].int() for r in range(4) if r != mu)
            at = (chi == d + 1).reshape(-1).nonzero().squeeze(-1)
            bonds.append((at, {nu: odd[nu].reshape(-1)[at].nonzero().squeeze(-1) for nu in range(4) if nu != mu}))
        plaqs = [(mu, nu, (sum(odd[r].int() for r in range(4) if r not in (mu, nu)) == d).reshape(-1).nonzero().squeeze(-1))
                 for mu, nu in _planes()]

        def partial_action():
            s = 0
            for mu, nu, at in plaqs:
                a = _mm(flat[mu][at], flat[nu][hop[mu, 1][at]])
                s = s + (1 - _trace(_mm(a, _dag(_mm(flat[nu][at], flat[mu][hop[nu, 1][at]])))) / 3).sum()
            return float(s)

        sd, it = partial_action(), 0
        while it < max_iter:
            new, summed = flat.clone(), []
            for mu, (at, by_nu) in enumerate(bonds):
                M = flat[mu][at].clone()
                for nu, k in by_nu.items():
                    n = at[k]
                    up, dn = hop[nu, 1][n], hop[nu, -1][n]
                    T = _mm(flat[nu][n], flat[mu][up], _dag(flat[nu][hop[mu, 1][n]]))
                    T = T + _mm(_dag(flat[nu][dn]), flat[mu][dn], flat[nu][hop[mu, 1][dn]])
                    M[k] += c * T
                summed.append(M)
            for (mu, (at, _)), W in zip(enumerate(bonds), _project(torch.cat(summed)).split([len(M) for M in summed])):
                new[mu][at] = W
            flat = new
            it += 1
            prev, sd = sd, partial_action()
            if rel_tol > 0 and abs(sd - prev) <= rel_tol * abs(prev):
                break
        sds.append(sd)
        counts.append(it)
    return flat.reshape((4,) + tuple(reversed(dims)) + (3, 3)), sds, counts


# ------------------------------------------------------------------ prepare
def _real(lat):
    return lat.links.view(lat.real_dtype())


def _lattice(dims, prec, seed, lattice_id=0, with_mom=False):
    lat = api.Lattice(dims, prec, seed=seed, lattice_id=lattice_id, with_mom=with_mom)
    api.mgq_import_links(lat, _canonical(make_field(dims, seed + 7919 * lattice_id)))
    return lat


def _momenta(case, dims, seed, scale):
    """Gaussian algebra field in the momentum layout, in the precision of the case."""
    V = dims[0] * dims[1] * dims[2] * dims[3]
    n = 4 * 2 * 8 * ((V // 2 + 63) // 64 * 64)
    p = scale * torch.randn(n, generator=_generator(seed + 1, "cuda"), device="cuda", dtype=torch.float64)
    return p if case["prec"] == "f64" else p.float()


def prepare(case, seed):
    kind, prec = case["kind"], case["prec"]
    s = {"case": case, "sweep": 0}
    if kind in ("batch_update", "batch_prolong"):
        dims = _batch_dims(case)
        lats = [_lattice(d, prec, seed, i) for i, d in enumerate(dims)]
        if kind == "batch_update":
            s["batch"] = api.Batch(lats, [5.8 + 0.3 * i / len(lats) for i in range(len(lats))], max_sweeps=case["sweeps"])
            s["plaq"] = s["batch"].plaquette_buffer(case["sweeps"])
        else:
            s["batch"] = api.ProlongBatch(lats, [api.Lattice([2 * v for v in d], prec, seed=seed, lattice_id=i)
                                                 for i, d in enumerate(dims)])
        return s
    dims = _dims(case)
    if kind == "measure":
        s["canon"] = _canonical(make_field(dims, seed))
        s["lat"] = api.Lattice(dims, prec, seed=seed)
        return s
    lat = s["lat"] = _lattice(dims, prec, seed, with_mom=kind in ("leapfrog", "hmc"))
    if kind == "leapfrog":
        lat.mom.view(lat.real_dtype()).copy_(_momenta(case, dims, seed, 1.0))
    elif kind in ("flow", "adaptive"):
        s["flowed"] = api.copy_lattice(lat)
    elif kind == "prolong":
        s["fine"] = api.Lattice([2 * v for v in dims], prec, seed=seed)
    elif kind == "gradient":
        s["omega"] = _momenta(case, dims, seed, 0.05).requires_grad_()
    return s


# ------------------------------------------------------------------ run
def _floats(*v):
    """Measured averages of a field, in single precision."""
    return np.stack([np.asarray(x, dtype=np.float32) for x in v])


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "update":
        n = case["sweeps"]
        plaq = api.mgq_update_sweeps(s["lat"], BETA, s["sweep"], n, 1, case["n_or"], plaq_out=True)
        s["sweep"] += n
        return {"links": _real(s["lat"]), "plaquette": _floats(plaq)}
    if kind == "batch_update":
        n = case["sweeps"]
        api.mgq_update_sweeps_batched(s["batch"], s["sweep"], n, 1, case["n_or"], plaq_out=s["plaq"])
        s["sweep"] += n
        return {"links": [_real(lat) for lat in s["batch"].lattices], "plaquette": s["plaq"].float()}
    if kind == "leapfrog":
        lat = s["lat"]
        api.mgq_hmc_momentum_step(lat, BETA, 0.05)
        api.mgq_link_exp_update(lat, lat.mom, 0.05)
        return {"links": _real(lat), "mom": lat.mom.view(lat.real_dtype())}
    if kind == "hmc":
        lat = s["lat"]
        dH, accepted = api.mgq_hmc_trajectory(lat, BETA, 0.5, case["steps"], s["sweep"])
        s["sweep"] += 1
        return {"links": _real(lat), "mom": lat.mom.view(lat.real_dtype()), "dH": dH, "accepted": accepted}
    if kind == "flow":
        w = s["flowed"]
        w.links.copy_(s["lat"].links)
        return {"EQ": _floats(*api.mgq_wilson_flow(w, 0.05, case["steps"], case["every"])), "links": _real(w)}
    if kind == "adaptive":
        w = s["flowed"]
        w.links.copy_(s["lat"].links)
        E, Q, steps, rejects = api.mgq_wilson_flow_adaptive(w, case["t_end"], dt_meas=0.25)
        return {"EQ": _floats(E, Q), "links": _real(w), "steps": steps, "rejects": rejects}
    if kind == "prolong":
        iters, sd = api.mgq_prolongate(s["lat"], s["fine"])
        return {"links": _real(s["fine"]), "iters": np.array(iters), "sd": _floats(sd)}
    if kind == "batch_prolong":
        b = s["batch"]
        api.mgq_prolongate_batched(b, rel_tol=0.0, max_iter=case["max_iter"])
        return {"links": [_real(f) for f in b.fine], "iters": b.iters, "sd": b.sd.float()}
    if kind == "gradient":
        omega = s["omega"]
        omega.grad = None
        value = autograd.flowed_observable(omega, s["lat"], case["obs"], 0.05, case["steps"], beta=BETA)
        value.backward()
        return {"value": float(value), "grad": omega.grad}
    lat = s["lat"]
    api.mgq_import_links(lat, s["canon"])
    return {"plaquette": api.mgq_plaquette(lat), "loop": api.mgq_wilson_loop(lat, case["m"], case["n"]),
            "partial": _floats(api.mgq_partial_loops(lat)), "EQ": _floats(api.mgq_topo_charge(lat)),
            "Q": _floats(api.mgq_topo_charge_improved(lat)), "links": _real(lat)}


# ------------------------------------------------------------------ work
# floating-point operations per link: staple 2466, + U A and its traceless antihermitian part 2700, overrelaxation
# 3400, heat bath 3580, exponential and product 700; per site: six clover leaves sums 6 x 10 products of 198
STAPLE, FORCE, OR, HB, EXP, CLOVER = 2466, 2700, 3400, 3580, 700, 12000


def work(case):
    kind, prec = case["kind"], case["prec"]
    link = {"f64": 144, "f32": 72, "f32c12": 48}[prec]
    alg = 64 if prec == "f64" else 32
    if kind in ("batch_update", "batch_prolong"):
        V = sum(math.prod(d) for d in _batch_dims(case))
    else:
        V = math.prod(_dims(case))
    n = 4 * V
    if kind in ("update", "batch_update"):
        return {"bytes": 2 * link * n, "flops": n * case["sweeps"] * (HB + case["n_or"] * OR)}
    if kind == "leapfrog":
        return {"bytes": 2 * (link + alg) * n, "flops": n * (FORCE + EXP)}
    if kind == "hmc":
        return {"bytes": (2 * link + alg) * n, "flops": n * ((case["steps"] + 1) * FORCE + case["steps"] * EXP)}
    if kind == "flow":
        return {"bytes": 2 * link * n, "flops": n * case["steps"] * 3 * (FORCE + EXP) + V * CLOVER * (case["steps"] // case["every"] + 1)}
    if kind == "adaptive":  # about a step for each 0.07 of flow time
        steps = math.ceil(case["t_end"] / 0.07)
        return {"bytes": 2 * link * n, "flops": n * steps * (3 * FORCE + 4 * EXP) + V * CLOVER * 5}
    if kind in ("prolong", "batch_prolong"):
        # 16 V fine sites; the three stages step on 24, 24 and 8 of the 64 fine links per coarse site, with 2, 4, 6 terms each
        it = 20 if kind == "prolong" else case["max_iter"]
        return {"bytes": link * n + 16 * link * n, "flops": V * it * (24 * 1600 + 24 * 2400 + 8 * 3200)}
    if kind == "gradient":
        return {"bytes": (link + 2 * alg) * n, "flops": n * case["steps"] * 3 * (2 * (FORCE + EXP) + 8500) + V * CLOVER * 4}
    return {"bytes": 576 * V + link * n, "flops": V * 60000}


# ------------------------------------------------------------------ exact
def exact(case, seed):
    """The outputs in 64 bits.  Markov chains (update, hmc) have none: they are defined by their random words and amplify
    rounding from sweep to sweep."""
    kind, prec = case["kind"], case["prec"]
    if kind in ("update", "batch_update", "hmc"):
        return None
    if kind == "batch_prolong":
        links, sd = [], []
        for i, d in enumerate(_batch_dims(case)):
            if i >= 3:
                links.append(None)
                continue
            U, s, _ = _prolongate(_rounded(make_field(d, seed + 7919 * i), prec), d, 0.05, 0.0, case["max_iter"])
            links.append(_to_links(U, [2 * v for v in d], prec))
        return {"links": links, "iters": None, "sd": None}
    dims = _dims(case)
    U = _rounded(make_field(dims, seed), prec)
    if kind == "leapfrog":
        P = _from_alg(_momenta(case, dims, seed, 1.0), dims)
        F = BETA / 6 * _coeffs(_generator_field(U))
        P = P + 0.05 * F
        pad = _momenta(case, dims, seed, 1.0).double()
        mask = _to_alg(torch.ones_like(P), dims)
        return {"links": _to_links(_mm(_exp(0.05 * _alg_matrix(P)), U), dims, prec), "mom": _to_alg(P, dims) + (1 - mask) * pad}
    if kind == "flow":
        EQ = []
        for k in range(case["steps"] + 1):
            if k % case["every"] == 0:
                EQ.append((float(_energy(U)), float(_charge(U))))
            if k < case["steps"]:
                U, _ = _flow_step(U, 0.05)
        return {"EQ": np.array(EQ).T.copy(), "links": _to_links(U, dims, prec)}
    if kind == "adaptive":
        t, eps, m, EQ, t_end, dt = 0.0, 0.01, 1, [(float(_energy(U)), float(_charge(U)))], case["t_end"], 0.25
        while t < t_end - 1e-12:
            stop = min(dt * m, t_end)
            h = min(eps, 0.2)
            hits = t + h >= stop - 1e-12
            h = stop - t if hits else h
            W, Y = _flow_step(U, h)
            d = float(torch.linalg.matrix_norm(W - _mm(_exp(Y), U)).max()) / 3
            fac = min(2.0, 0.95 * (0.01 / d) ** (1 / 3))
            if d > 0.01:
                eps = h * fac
                continue
            U, t = W, stop if hits else t + h
            if hits:
                EQ.append((float(_energy(U)), float(_charge(U))))
                m += 1
            else:
                eps = h * fac
        return {"EQ": np.array(EQ).T.copy(), "links": _to_links(U, dims, prec), "steps": None, "rejects": None}
    if kind == "prolong":
        F, sd, _ = _prolongate(U, dims, 0.05, 1e-5, 10000)
        return {"links": _to_links(F, [2 * v for v in dims], prec), "iters": None, "sd": np.array([sd])}
    if kind == "gradient":
        if math.prod(dims) * case["steps"] > 4 * 16 ** 4:
            return None
        buf = _momenta(case, dims, seed, 0.05)
        omega = _from_alg(buf, dims).requires_grad_()
        W = _mm(_exp(_alg_matrix(omega)), U)
        for _ in range(case["steps"]):
            W, _ = _flow_step(W, 0.05)
        if case["obs"] == "S":
            value = BETA * sum((1 - _loop(W, mu, nu, 1, 1)).sum() for mu, nu in _planes())
        else:
            value = _energy(W) if case["obs"] == "E" else _charge(W)
        value.backward()
        # the padding of the layout carries no gradient
        return {"value": float(value.detach()), "grad": _to_alg(omega.grad, dims)}
    V = math.prod(dims)
    odd = _odd(dims, U.device)
    w1, w2 = torch.zeros(3, dtype=torch.float64), torch.zeros(5, dtype=torch.float64)
    h, plaq, loop = 0.0, 0.0, 0.0
    chi = sum(o.int() for o in odd)
    for mu, nu in _planes():
        one, two = _loop(U, mu, nu, 1, 1), _loop(U, mu, nu, 2, 2)
        cmn = sum(odd[r].int() for r in range(4) if r not in (mu, nu))
        for d in range(3):
            w1[d] += one[cmn == d].sum().cpu()
        for d in range(5):
            w2[d] += two[chi == d].sum().cpu()
        h = max(h, float(3 * (1 - one).max()))
        plaq += float(one.sum()) / (6 * V)
        loop += float(_loop(U, mu, nu, case["m"], case["n"]).sum()) / (6 * V)
    binom = [math.comb(4, d) for d in range(5)]
    partial = [float(w1[d]) / (2 * (4 - d) * (3 - d) * binom[d] * V / 16) for d in range(3)]
    partial += [float(w2[d]) / (6 * binom[d] * V / 16) for d in range(5)] + [h]
    Q = [float(_charge(U, m)) for m in (1, 2, 3)]
    imp = 1.5 * Q[0] - 0.6 * Q[1] / 16 + 0.1 * Q[2] / 81
    return {"plaquette": plaq, "loop": loop, "partial": np.array([partial]), "EQ": np.array([[float(_energy(U)), Q[0]]]),
            "Q": np.array([[imp] + Q]), "links": _to_links(U, dims, prec)}
