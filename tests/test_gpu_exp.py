"""The SU(3) exponential over the range of |Q| its forms share out: the series
below rho = 1/2 and 1 (rho = sqrt(4 c1 / 3) bounds the eigenvalues), the closed
form above, both signs of det Q and degenerate eigenvalues, against scipy."""
import numpy as np
import pytest

from _helpers import expm, gell_mann

pytestmark = pytest.mark.gpu

DIMS = [4, 4, 4, 6]


def _fields(seed):
    """Algebra fields whose rho covers 1e-9 .. 4, dense around the limits 1/2 and 1."""
    rng = np.random.default_rng(seed)
    V = int(np.prod(DIMS))
    P = rng.standard_normal((V, 4, 8))
    P[::7] = 0.0
    P[::7, :, 7] = rng.choice([-1.0, 1.0], (len(P[::7]), 4))       # two equal eigenvalues
    P[1::7] = 0.0
    P[1::7, :, 2] = 1.0                                            # det Q = 0
    rho = np.concatenate([10.0 ** rng.uniform(-9, np.log10(4.0), 2 * V), 0.5 + 1e-7 * rng.standard_normal(V),
                          1.0 + 1e-7 * rng.standard_normal(V)]).reshape(V, 4)
    c1 = 0.25 * (P ** 2).sum(-1)                                   # Tr Q^2 / 2, Q = sum_a p_a lambda_a / 2
    P *= (rho / np.sqrt(4 * c1 / 3))[..., None]
    P[5, 2] = 0.0
    return P


# 20 roundings of O(1) intermediates (coefficients, Q^2, the two products): 20 x 2^-53 and 20 x 2^-24, times 3 entries a sum
@pytest.mark.parametrize("prec,tol", [("f64", 7e-15), ("f32", 3.6e-6), ("f32c12", 3.6e-6)])
def test_exponential_over_its_forms(gpu, prec, tol):
    P = _fields(11)
    lat = gpu.Lattice(DIMS, prec)
    gpu.mgq_init_links(lat, 0)
    buf = gpu.alg_from_numpy(lat, P)
    P = gpu.alg_to_numpy(lat, buf)          # as rounded to the precision
    gpu.mgq_link_exp_update(lat, buf, 1.0)
    got = lat.to_numpy()
    X = np.einsum("vma,aij->vmij", P, 0.5j * gell_mann())
    ref = np.stack([[expm(X[v, m]) for m in range(4)] for v in range(len(P))])
    assert np.max(np.abs(got - ref)) < tol
