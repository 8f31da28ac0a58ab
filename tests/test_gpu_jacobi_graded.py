"""Singular vectors of blocks whose columns differ by many orders of magnitude, FP64 handles.

The middle site matrix of a chain holds one block with graded columns and, in rows and columns of
its own, a block of two equal columns, which makes the matrix rank deficient: the gauge move takes
the SVD and not the QR.  Every singular value of the graded block is kept (above 1e-10 of the
largest), so the left factor has to be an isometry and the state has to stay.

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
    while left > 1:
        right = (left + 1) // 2
        a = rng.standard_normal((left, 2 * right)) + 1j * rng.standard_normal((left, 2 * right))
        mps.append(np.linalg.qr(a.conj().T)[0].conj().T.reshape(left, 2, right))
        left = right
    return mps, k


CASES = [(4, 2, 1e-4, 1.0, False), (4, 2, 1e-5, 1e-3, False), (4, 2, 1e-6, 1e-2, False), (4, 2, 1e-8, 1.0, False),
         (6, 3, 1e-7, 1.0, False), (8, 4, 1e-8, 1.0, True), (16, 8, 1e-6, 1.0, True), (60, 30, 1e-6, 1.0, True)]


@pytest.mark.parametrize("p,q,small,coupling,halves", CASES)
def test_graded_block_gives_an_isometry(p, q, small, coupling, halves):
    assert torch.cuda.is_available()
    from paper_2005_06104_gb300 import gse_tdvp as g
    worst = [0.0, 0.0]
    for seed in range(8):
        rng = np.random.default_rng(1000 * p + seed)
        mps, k = _chain(rng, _graded(rng, p, q, small, coupling, halves))
        h = g.GseTdvp(mps, wl.heisenberg_mpo(wl.chain(len(mps))), chi_max=256)
        out = h.get_mps()
        h.close()
        a = out[k]
        assert a.shape[2] == q + 1                 # the two equal columns are one direction
        u = a.reshape(-1, a.shape[2])
        worst[0] = max(worst[0], np.max(np.abs(u.conj().T @ u - np.eye(u.shape[1]))))
        v0, v1 = mps_to_dense(mps), mps_to_dense(out)
        worst[1] = max(worst[1], np.linalg.norm(v1 - v0) / np.linalg.norm(v0))
    assert worst[0] < TOL and worst[1] < TOL


@pytest.mark.parametrize("p,q,small", [(4, 2, 1e-4), (4, 2, 1e-5), (8, 4, 1e-5), (60, 30, 1e-5)])
def test_graded_density_matrices_give_isometries(p, q, small):
    """The same states through the density-matrix compression with tau = 0 (the operator is the
    identity): eigenvectors of graded positive semidefinite blocks, by Jacobi on Cholesky factors
    whose columns are graded by themselves."""
    from paper_2005_06104_gb300 import gse_tdvp as g
    worst = 0.0
    for seed in range(8):
        rng = np.random.default_rng(500 * p + seed)
        mps, k = _chain(rng, _graded(rng, p, q, small, 1.0, True))
        h = g.GseTdvp(mps, wl.heisenberg_mpo(wl.chain(len(mps))), chi_max=256, tau=0.0, eps_k=0.0)
        h.apply_krylov()
        for a in h.get_mps()[:-1]:
            u = a.reshape(-1, a.shape[2])
            worst = max(worst, np.max(np.abs(u.conj().T @ u - np.eye(u.shape[1]))))
        h.close()
    assert worst < TOL
