"""The adjoint of one flow step far beyond the step sizes in use, where the exponentials'
arguments are of O(1) and their differential's series is long: against torch's
differentiation of the step in 64 bits."""
import numpy as np
import pytest
import torch

from _helpers import gell_mann

pytestmark = pytest.mark.gpu

DIMS = [2, 2, 2, 4]
X = torch.from_numpy(0.5j * gell_mann())


def _neighbours():
    V = int(np.prod(DIMS))
    st = np.cumprod([1] + DIMS[:3])
    x = np.stack([(np.arange(V) // st[m]) % DIMS[m] for m in range(4)], axis=1)
    out = []
    for mu in range(4):
        f = x.copy()
        f[:, mu] = (f[:, mu] + 1) % DIMS[mu]
        b = x.copy()
        b[:, mu] = (b[:, mu] - 1) % DIMS[mu]
        out.append((torch.from_numpy(f @ st), torch.from_numpy(b @ st)))
    return out


def _alg(c):
    return torch.einsum("vma,aij->vmij", c.to(torch.complex128), X)


def _coeffs(M):
    """Coefficients of TA(M): Tr(X_a X_b) = -delta_ab / 2."""
    return -2 * torch.einsum("aij,vmji->vma", X, (M - M.mH) / 2).real


def _generator(W, nb):
    Z = []
    for mu in range(4):
        A = 0
        for nu in range(4):
            if nu != mu:
                fm, (fn, bn) = nb[mu][0], nb[nu]
                A = A + W[fm, nu] @ W[fn, mu].mH @ W[:, nu].mH + W[bn[fm], nu].mH @ W[bn, mu].mH @ W[bn, nu]
        Z.append(W[:, mu] @ A)
    return -_alg(_coeffs(torch.stack(Z, dim=1)))


def _step(W, eps, nb):
    Z0 = eps * _generator(W, nb)
    W = torch.linalg.matrix_exp(Z0 / 4) @ W
    Z1 = eps * _generator(W, nb)
    W = torch.linalg.matrix_exp(8 / 9 * Z1 - 17 / 36 * Z0) @ W
    Z2 = eps * _generator(W, nb)
    return torch.linalg.matrix_exp(0.75 * Z2 - 8 / 9 * Z1 + 17 / 36 * Z0) @ W


def reference(U, lam, eps):
    """d/domega of lam . (coefficients of W3(exp(omega) U) W3(U)^+) at omega = 0."""
    nb = _neighbours()
    W0, lam = torch.from_numpy(U), torch.from_numpy(lam)
    omega = torch.zeros(lam.shape, dtype=torch.float64, requires_grad=True)
    W3 = _step(torch.linalg.matrix_exp(_alg(omega)) @ W0, eps, nb)
    (lam * _coeffs(W3 @ W3.detach().mH)).sum().backward()
    return omega.grad.numpy()


# A cotangent passes some 60 products of 3-term sums, 180 roundings, in each of three stages: 540 x 2^-53 = 6e-14 and
# 540 x 2^-24 = 3.2e-5, times the 10 by which a relative change of the links changes the gradient of a step of 1 (largest
# entries, on the reference), times 5 for the alternating series of arguments up to 5
@pytest.mark.parametrize("prec,tol", [("f64", 3e-12), ("f32", 1.6e-3), ("f32c12", 1.6e-3)])
def test_step_adjoint_at_a_large_step(gpu, orc, prec, tol):
    U = orc.init_links(DIMS, 1, seed=8)
    if prec != "f64":
        U = U.astype(np.complex64).astype(np.complex128)
    lam = np.random.default_rng(4).standard_normal((U.shape[0], 4, 8)).astype(np.float32).astype(np.float64)
    lat = gpu.Lattice(DIMS, prec)
    lat.from_numpy(U)
    buf = gpu.alg_from_numpy(lat, lam)
    gpu.mgq_wilson_flow_step_adjoint(lat, 1.0, buf, gpu.flow_adjoint_scratch(lat))
    ref = reference(U, lam, 1.0)
    assert np.max(np.abs(gpu.alg_to_numpy(lat, buf) - ref)) < tol * np.max(np.abs(ref))
