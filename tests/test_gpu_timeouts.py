"""A bounded device wait that ran out is reported by the call it happened in, as status 6
(TDVP_ERR_TIMEOUT), and by no later one.  The mark a kernel would leave is set from the host."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2005_06104_gb300 import workloads as wl

TIMEOUT = 6


@pytest.fixture(scope="module")
def g():
    assert torch.cuda.is_available()
    from paper_2005_06104_gb300 import gse_tdvp
    return gse_tdvp


def _handle(g, **opts):
    return g.GseTdvp(wl.random_isometric_mps(10, 8, 3), wl.heisenberg_mpo(wl.chain(10)), chi_max=16, **opts)


def _keff(h):
    m = h.bond_dims()[4]
    x = torch.ones(m, m, dtype=torch.complex128, device="cuda")
    h.keff_apply(4, x, torch.empty_like(x))


def _heff(h):
    m = h.bond_dims()
    x = torch.ones(m[4], 2, m[5], dtype=torch.complex128, device="cuda")
    h.heff_apply(4, x, torch.empty_like(x))


CALLS = {"canonicalize": lambda h: h.canonicalize(2), "apply_krylov": lambda h: h.apply_krylov(),
         "expand_basis": lambda h: h.expand_basis(1), "sweep": lambda h: h.sweep(0.05),
         "sweep2": lambda h: h.sweep2(0.05), "energy": lambda h: h.energy(), "norm": lambda h: h.norm(),
         "get_mps": lambda h: h.get_mps(), "keff_apply": _keff, "heff_apply": _heff,
         "a call that fails by itself": lambda h: h.canonicalize(99)}


@pytest.mark.parametrize("call", CALLS)
@pytest.mark.parametrize("prec", ["fp64", "bf16x10"])
def test_handle_calls_report_the_time_out_once(g, call, prec):
    h = _handle(g, precision=g.PREC_FP64 if prec == "fp64" else g.PREC_BF16X10)
    g.inject_timeout(h)
    with pytest.raises(g.TDVPError) as e:
        CALLS[call](h)
    assert e.value.status == TIMEOUT
    h.norm()
    h.canonicalize(5)
    h.close()


def test_a_sweep_stops_at_its_first_lanczos_run(g):
    h = _handle(g)
    h.canonicalize(0)
    before = h.get_mps()
    g.inject_timeout(h)
    with pytest.raises(g.TDVPError) as e:
        h.sweep(0.05)
    assert e.value.status == TIMEOUT
    after = h.get_mps()
    assert all(np.array_equal(a, b) for a, b in zip(before, after))
    h.close()


def test_handle_free_calls_report_the_time_out_once(g):
    rng = np.random.default_rng(1)
    L, x = (torch.from_numpy(rng.standard_normal(s) + 0j).cuda() for s in ((4, 3, 4), (4, 4)))
    y = torch.empty_like(x)
    g.keff_contract(L, L, x, y)
    ref = y.clone()
    g.inject_timeout()
    with pytest.raises(g.TDVPError) as e:
        g.keff_contract(L, L, x, y)
    assert e.value.status == TIMEOUT
    g.keff_contract(L, L, x, y)
    assert torch.equal(y, ref)
    W = np.zeros((3, 2, 2, 3), dtype=complex)
    s, t = torch.ones(4, 2, 4, dtype=torch.complex128, device="cuda"), torch.empty(4, 2, 4, dtype=torch.complex128, device="cuda")
    g.inject_timeout()
    with pytest.raises(g.TDVPError) as e:
        g.expm_contract(L, W, L, s, t, 0.1, tol=-1.0)
    assert e.value.status == TIMEOUT
    g.expm_contract(L, W, L, s, t, 0.1)
