"""Singular vectors of blocks whose columns differ by many orders of magnitude, FP64 handles.

The middle site matrix of a chain holds one block with graded columns and, in rows and columns of
its own, a block of two equal columns, which makes the matrix rank deficient: the gauge move takes
the SVD and not the QR.  H = 0 (couplings of zero), so every evolution is the identity and what moves
the state is the factorisations.  Every singular value of the graded block is kept (above 1e-10 of
the largest), so the factors have to be isometries and the state has to stay.

A Jacobi sweep that leaves every pair orthogonal to rounding gives |U^H U - 1| of a few ulp times
sqrt(rows): 1e-15 to 4e-15 for these blocks (measured with the angles in FP64 throughout), held to
1e-13.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from exact import mps_to_dense
from paper_2005_06104_gb300 import workloads as wl

TOL = 1e-13


def _graded(rng, p, q, small, coupling, halves):
    """p x q: column norms from 1 down to `small`; overlaps of a column with those before it scaled
    by `coupling`.  halves: the first half of the columns orthonormal, the others of norm `small`."""
    m = rng.standard_normal((p, q)) + 1j * rng.standard_normal((p, q))
    for j in range(q):
        keep = 0.0 if halves and j < q // 2 else 1.0 if halves else coupling
        for _ in range(1 if keep else 2):
            if keep != 1.0 and j:
                b = np.linalg.qr(m[:, :j])[0]
                m[:, j] -= (1.0 - keep) * (b @ (b.conj().T @ m[:, j]))
        f = (1.0 if j < q // 2 else small) if halves else small ** (j / (q - 1))
        m[:, j] *= f / np.linalg.norm(m[:, j])
    return m


def _chain(rng, block):
    """Left sites: identity isometries up to ml = 2^k >= (p + 2) / 2 states; the block's site; random
    right sites down to 1."""
    p, q = block.shape
    k = int(np.ceil(np.log2((p + 2) / 2)))
    mps = [np.eye(2 ** (i + 1), dtype=complex).reshape(2 ** i, 2, 2 ** (i + 1)) for i in range(k)]
    m = np.zeros((2 ** (k + 1), q + 2), dtype=complex)
    m[:p, :q] = block
    v = rng.standard_normal(m.shape[0] - p) + 1j * rng.standard_normal(m.shape[0] - p)
    m[p:, q] = m[p:, q + 1] = v / np.linalg.norm(v)
    mps.append(m.reshape(2 ** k, 2, q + 2))
    left = q + 2
    while left > 1:                                # embeddings: state l goes to (s, r) = divmod(l, right)
        right = (left + 1) // 2
        a = np.zeros((left, 2, right), dtype=complex)
        for l in range(left):
            a[l, l // right, l % right] = 1.0
        mps.append(a)
        left = right
    return mps, k


def _isometry_error(mats):
    return max(np.max(np.abs(u.conj().T @ u - np.eye(u.shape[1]))) for u in mats)


def _left(mps):
    return [a.reshape(-1, a.shape[2]) for a in mps[:-1]]


def _right(mps):
    return [a.reshape(a.shape[0], -1).conj().T for a in mps[1:]]


def _direction_error(mps, ref):
    v, w = mps_to_dense(mps), mps_to_dense(ref)
    return np.linalg.norm(v / np.linalg.norm(v) - w / np.linalg.norm(w))


CASES = [(4, 2, 1e-4, 1.0, False), (4, 2, 1e-5, 1e-3, False), (4, 2, 1e-6, 1e-2, False), (4, 2, 1e-8, 1.0, False),
         (6, 3, 1e-7, 1.0, False), (8, 4, 1e-8, 1.0, True), (16, 8, 1e-6, 1.0, True), (60, 30, 1e-6, 1.0, True)]


@pytest.mark.parametrize("how", ["move", "imaginary", "two-site"])
@pytest.mark.parametrize("p,q,small,coupling,halves", CASES)
def test_graded_block_gives_an_isometry(p, q, small, coupling, halves, how):
    """The gauge move of a rank-deficient site (exact angles) and the truncating moves of imaginary time
    and of the two-site integrator (large angles in FP32)."""
    assert torch.cuda.is_available()
    from paper_2005_06104_gb300 import gse_tdvp as g
    iso = err = 0.0
    for seed in range(8):
        rng = np.random.default_rng(1000 * p + seed)
        mps, k = _chain(rng, _graded(rng, p, q, small, coupling, halves))
        h = g.GseTdvp(mps, wl.heisenberg_mpo(wl.chain(len(mps), 0.0)), chi_max=256)
        if how == "imaginary":
            h.sweep(0.1, g.IMAG)
        elif how == "two-site":
            h.sweep2(0.1, g.REAL)
        out = h.get_mps()
        h.close()
        assert out[k].shape[2] == q + 1            # the two equal columns are one direction
        iso = max(iso, _isometry_error(_left(out) if how == "move" else _right(out)))
        err = max(err, _direction_error(out, mps))
    assert iso < TOL and err < TOL


@pytest.mark.parametrize("tau", [0.1, -0.1j])
@pytest.mark.parametrize("p,q,small", [(4, 2, 1e-4), (4, 2, 1e-5), (8, 4, 1e-5), (60, 30, 1e-5)])
def test_graded_density_matrices_give_isometries(p, q, small, tau):
    """The same states through the density-matrix compression of the Krylov vectors (the operator is the
    identity): eigenvectors of graded positive semidefinite blocks, by Jacobi on Cholesky factors
    whose columns are graded by themselves; in imaginary time with the large angles in FP32."""
    from paper_2005_06104_gb300 import gse_tdvp as g
    worst = 0.0
    for seed in range(8):
        rng = np.random.default_rng(500 * p + seed)
        mps, k = _chain(rng, _graded(rng, p, q, small, 1.0, True))
        h = g.GseTdvp(mps, wl.heisenberg_mpo(wl.chain(len(mps), 0.0)), chi_max=256, tau=tau, eps_k=0.0)
        h.apply_krylov()
        worst = max(worst, _isometry_error(_left(h.get_mps())))
        h.close()
    assert worst < TOL
