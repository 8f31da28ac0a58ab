"""Device memory of the FP64 tensor-core products: the digits and partial results of one product (or of
one H_eff apply, with the digits it keeps) stay within 8 GiB, larger products run in panels.

Operands whose digits alone are 15 and 30 GB.  Tolerance: the reference is an FP64 product, whose own
rounding grows with the square root of its K: 5e-15 at K = 5600 as in the tests of smaller sizes, so
2.5e-14 at the 131072 terms here."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2005_06104_gb300 import workloads as wl

GIB = 1 << 30
WORK = 8.6 * GIB           # 8 GiB in pool classes (at most 1/16 above)
TOL = 2.5e-14


@pytest.fixture(scope="module")
def g():
    assert torch.cuda.is_available()
    from paper_2005_06104_gb300 import gse_tdvp
    return gse_tdvp


def _rnd(gen, *shape):
    z = torch.empty(*shape, dtype=torch.complex128, device="cuda")
    torch.view_as_real(z).normal_(generator=gen)
    return z.mul_(1.0 / np.sqrt(shape[-1]))


def _grown(call):
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    call()
    torch.cuda.synchronize()
    return before - torch.cuda.mem_get_info()[0]


@pytest.mark.parametrize("ml,mr,w", [(4096, 64, 32), (64, 4096, 32), (4033, 65, 33)])
def test_products_in_panels(g, ml, mr, w):
    """Panels of A's rows (a large left environment) and of B's columns (a large right one)."""
    gen = torch.Generator(device="cuda").manual_seed(ml)
    L, R, x = _rnd(gen, ml, w, ml), _rnd(gen, mr, w, mr), _rnd(gen, ml, mr)
    y = torch.empty_like(x)
    torch.cuda.empty_cache()
    grown = _grown(lambda: g.keff_contract(L, R, x, y))
    t = (L.view(ml * w, ml) @ x).view(ml, w * mr)
    ref = t @ R.view(mr, w * mr).mT
    assert (torch.linalg.norm(y - ref) / torch.linalg.norm(ref)).item() < TOL
    assert grown <= WORK + 1.1 * 16 * ml * w * mr + 0.3 * GIB
    del L, R, x, y, t, ref
    torch.cuda.empty_cache()


def test_large_heff_keeps_no_digits(g):
    """H_eff at 2048 x 2048, w = 14: T1 and T2 are 1.9 GB each, the digits of everything 13 GB."""
    W = max(wl.heisenberg_mpo(wl.cylinder_snake(5)), key=lambda w: w.shape[0] * w.shape[3])
    wb, m = W.shape[0], 2048
    assert W.shape[3] == wb == 14
    gen = torch.Generator(device="cuda").manual_seed(1)
    L, R, x = _rnd(gen, m, wb, m), _rnd(gen, m, wb, m), _rnd(gen, m, 2, m)
    y = torch.empty_like(x)
    torch.cuda.empty_cache()
    grown = _grown(lambda: g.heff_contract(L, W, R, x, y))
    t = (L.view(m * wb, m) @ x.view(m, 2 * m)).view(m, wb, 2, m)
    t = torch.einsum("wstv,awtb->asvb", torch.from_numpy(W).cuda(), t).reshape(2 * m, wb * m)
    ref = (t @ R.view(m, wb * m).mT).view(m, 2, m)
    assert (torch.linalg.norm(y - ref) / torch.linalg.norm(ref)).item() < TOL
    assert grown <= WORK + 2 * 1.1 * 16 * m * wb * 2 * m + 0.3 * GIB
    del L, R, x, y, t, ref
    torch.cuda.empty_cache()
