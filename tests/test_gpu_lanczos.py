"""The small exponential and the vector kernels of a Lanczos run at the sizes where they change
path: one site with bond dimensions 1 and w = 1, so that H_eff is the d x d Hermitian matrix in W
and the local space has d entries (up to 62: two components per lane from 33 on, a full Krylov
space at every size), against the matrix exponential from the eigendecomposition.

Tolerance: the Chebyshev expansion and the projections carry rounding of a few ulp per order and
per vector, |delta| times the spectral radius (at most 40 here) orders: 40 * 62 * 2.2e-16 = 5e-13,
held to 2e-12.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 2e-12


@pytest.fixture(scope="module")
def g():
    assert torch.cuda.is_available()
    from paper_2005_06104_gb300 import gse_tdvp
    return gse_tdvp


def _hermitian(rng, d, radius):
    a = rng.standard_normal((d, d)) + 1j * rng.standard_normal((d, d))
    e, u = np.linalg.eigh(a + a.conj().T)
    return (u * np.linspace(-radius, radius, d)) @ u.conj().T if d > 1 else np.array([[radius + 0j]])


@pytest.mark.parametrize("d", [1, 2, 31, 32, 33, 62])
@pytest.mark.parametrize("radius,delta,kind", [(1e-9, 0.5, 0), (1.0, 0.5, 0), (40.0, -1.0, 0), (1.0, 0.5, 1),
                                               (20.0, -0.5, 1), (20.0, 0.5, 1)])
def test_exponential_of_a_dense_matrix(g, d, radius, delta, kind):
    rng = np.random.default_rng(d)
    h = _hermitian(rng, d, radius)
    x = rng.standard_normal(d) + 1j * rng.standard_normal(d)
    one = torch.ones(1, 1, 1, dtype=torch.complex128, device="cuda")
    xd = torch.from_numpy(x.reshape(1, d, 1)).cuda()
    y = torch.empty_like(xd)
    it = g.expm_contract(one, h.reshape(1, d, d, 1), one, xd, y, delta, kind=kind, tol=1e-13, nmax=62)
    e, u = np.linalg.eigh(h)
    ref = u @ (np.exp((-1j if kind == 0 else -1.0) * delta * e) * (u.conj().T @ x))
    assert 1 <= it <= d
    assert np.linalg.norm(y.cpu().numpy().ravel() - ref) <= TOL * np.linalg.norm(ref)


@pytest.mark.parametrize("ml,mr", [(1, 1), (3, 5), (63, 33), (130, 129), (300, 280)])
def test_one_site_exponential_keeps_the_norm_and_zero_sectors(g, ml, mr):
    """W = Z (x) identity environments: H x is known, runs of exact zeros in x stay exact zeros and
    the vectors span one warp up to more entries than threads."""
    rng = np.random.default_rng(ml)
    x = rng.standard_normal((ml, 2, mr)) + 1j * rng.standard_normal((ml, 2, mr))
    x[: ml // 2, 0, :] = 0.0
    W = np.zeros((1, 2, 2, 1), dtype=complex)
    W[0, 0, 0, 0], W[0, 1, 1, 0] = 1.5, -0.5
    L = torch.eye(ml, dtype=torch.complex128, device="cuda").reshape(ml, 1, ml).contiguous()
    R = torch.eye(mr, dtype=torch.complex128, device="cuda").reshape(mr, 1, mr).contiguous()
    xd = torch.from_numpy(x).cuda()
    y = torch.empty_like(xd)
    it = g.expm_contract(L, W, R, xd, y, 0.7)
    ref = x * np.exp(-0.7j * np.array([1.5, -0.5]))[None, :, None]
    got = y.cpu().numpy()
    assert it == (2 if np.any(x[:, 0, :]) else 1)
    assert np.linalg.norm(got - ref) <= TOL * np.linalg.norm(ref)
    assert not np.any(got[: ml // 2, 0, :])


def test_zero_and_non_finite_start_vectors(g):
    one = torch.ones(1, 1, 1, dtype=torch.complex128, device="cuda")
    h = np.array([[1.0, 0.5], [0.5, -1.0]], dtype=complex).reshape(1, 2, 2, 1)
    x = torch.zeros(1, 2, 1, dtype=torch.complex128, device="cuda")
    y = torch.ones_like(x)
    assert g.expm_contract(one, h, one, x, y, 0.5) == 0
    assert torch.all(y == 0)
    x[0, 1, 0] = float("nan")
    with pytest.raises(g.TDVPError) as e:
        g.expm_contract(one, h, one, x, y, 0.5)
    assert e.value.status == 5
