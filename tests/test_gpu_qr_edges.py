"""Gauge moves at the edges of the QR kernels' ranges: a cluster of CTAs takes blocks of up to 96
columns and 256 rows, a group of CTAs the wider ones; 32 columns and 64 / 128 rows are where the
cluster size and the reduction width change.  Dense random isometric states, so a block is the whole
site matrix (2 chi x chi).

Moving the centre to the far end and back leaves site tensors orthonormal to rounding: Householder
QR gives |Q^H Q - 1| of a few ulp times sqrt(columns), held to 1e-13; the state is unchanged,
overlap 1 to 1e-12.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O
from paper_2005_06104_gb300 import workloads as wl


@pytest.mark.parametrize("chi,n", [(2, 4), (31, 12), (32, 12), (33, 12), (64, 14), (96, 14), (97, 14), (128, 16),
                                   (130, 16)])
def test_canonical_forms(chi, n):
    assert torch.cuda.is_available()
    from paper_2005_06104_gb300 import gse_tdvp as g
    mps = wl.random_isometric_mps(n, chi, 5)
    h = g.GseTdvp(mps, wl.heisenberg_mpo(wl.chain(n)), chi_max=chi)
    left = h.get_mps()
    for a in left[:-1]:
        q = a.reshape(-1, a.shape[2])
        assert np.linalg.norm(q.conj().T @ q - np.eye(q.shape[1])) < 1e-13 * np.sqrt(q.shape[1])
    h.canonicalize(0)
    right = h.get_mps()
    for a in right[1:]:
        q = a.reshape(a.shape[0], -1)
        assert np.linalg.norm(q @ q.conj().T - np.eye(q.shape[0])) < 1e-13 * np.sqrt(q.shape[0])
    assert abs(abs(O.mps_overlap(right, mps)) - 1) < 1e-12 and abs(abs(O.mps_overlap(left, mps)) - 1) < 1e-12
    h.close()
