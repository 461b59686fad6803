"""M2L by spectral products (csrc/m2l_spec.cu) against the FP64 oracle, through
the C-ABI: every order it is built for, on trees whose levels take each of its
kernels (level 2 periodic and isolated, double-float, row chains, FP32), with
one cell per leaf and more.

Tolerance: the plain form's 1e-6 (FP32 spectra, sums over a plane's terms apart
from the total, double-float transforms: rounding of ~1e-7 per level times the
far field's cancellation of a few); the mixed form transforms in FP32 and keeps
its bf16x3 bound 2e-5."""
import numpy as np
import pytest

from oracle import fmm as ofmm
from oracle import nonperiodic as npo
from paper_2011_07099_gb300 import inputs
from parity_util import assert_close

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2011_07099_gb300 import binding, build
    build.build()
    binding.lib()
    return binding


def _solve(B, rho, L, p, iso=False, prec=0, timing=False):
    plan = B.Plan(rho.shape[0], L, p)
    if iso:
        B.fmm_plan_set_boundary(plan.handle, B.FMM_BOUNDARY_ISOLATED)
    if prec:
        plan.set_precision(prec)
    B.fmm_plan_set_timing(plan.handle, timing)
    phi, acc = plan.solve(torch.from_numpy(rho).cuda())
    torch.cuda.synchronize()
    assert B.lib().fmm_plan_check(plan.handle) == B.FMM_OK
    plan.close()
    return phi.cpu().numpy(), acc.cpu().numpy()


@pytest.mark.parametrize("p", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("N,L", [(12, 2), (16, 3), (16, 4)])
def test_spectral_m2l_matches_oracle(B, N, L, p):
    rho = inputs.lognormal(N, sigma=0.8, seed=N + L + p)
    phi, acc = _solve(B, rho, L, p)
    ophi, og = ofmm.solve(rho, L, p)
    assert_close(phi, ophi, 1e-6, f"phi {N}^3 L={L} p={p}")
    assert_close(acc, og, 1e-6, f"g {N}^3 L={L} p={p}")


@pytest.mark.parametrize("N,L,p", [(8, 2, 3), (16, 2, 6), (16, 3, 5), (16, 4, 6), (8, 3, 8)])
def test_spectral_m2l_isolated_matches_oracle(B, N, L, p):
    rho = inputs.lognormal(N, sigma=0.8, seed=N + p)
    phi, acc = _solve(B, rho, L, p, iso=True)
    ophi, og = npo.solve_isolated(rho, L, p)
    assert_close(phi, ophi, 1e-6, f"isolated phi {N}^3 L={L} p={p}")
    assert_close(acc, og, 1e-6, f"isolated g {N}^3 L={L} p={p}")


@pytest.mark.parametrize("N,L,p", [(32, 4, 5), (16, 4, 6), (32, 4, 7), (16, 4, 8)])
def test_mixed_form_spectral_levels_match_oracle(B, N, L, p):
    rho = inputs.lognormal(N, sigma=0.5, seed=N + L + p)
    phi, acc = _solve(B, rho, L, p, prec=B.FMM_PREC_BF16X3)
    ophi, og = ofmm.solve(rho, L, p)
    assert_close(phi, ophi, 2e-5, f"mixed phi {N}^3 L={L} p={p}")
    assert_close(acc, og, 2e-5, f"mixed g {N}^3 L={L} p={p}")


def test_levels_in_one_launch_equal_levels_one_by_one_bitwise(B):
    # timed solves launch each level on its own, untimed ones all levels of one
    # arithmetic together, on two streams
    rho = inputs.lognormal(32, sigma=0.5, seed=4)
    for p in (4, 7):
        a, b = _solve(B, rho, 5, p), _solve(B, rho, 5, p, timing=True)
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("N,L,p", [(8, 2, 4), (8, 3, 3), (8, 3, 5), (16, 4, 2)])
def test_spectral_table_gradient_matches_oracle_differences(B, N, L, p):
    # the loss is quadratic in the table values, so central differences of the
    # FP64 oracle are exact up to its rounding; entries at window edges
    # (components that are multiples of p, and the largest 4p - 1), inside
    # windows and on the axes.  FP32 residual, adjoint and sums: rounding of
    # ~1e-5 of the largest gradient; bound 1e-3 of it.
    from oracle import learn as olearn
    rho = inputs.lognormal(N, sigma=0.8, seed=N + p)
    n, G = olearn.grid_size(L, p), 4 * p
    theta = np.zeros(n)
    tphi, tg = (np.asarray(x) * 1.3 for x in olearn.pm_target(rho))
    w_phi, w_g = 1.0 / np.sum(tphi ** 2), 1.0 / np.sum(tg ** 2)
    plan = B.Plan(N, L, p)
    grad = torch.zeros(n, dtype=torch.float32, device="cuda")
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    f32 = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    B.fmm_table_grid_grad(plan.handle, f32(rho), f32(tphi), f32(tg), w_phi, w_g, grad, loss)
    got = grad.cpu().numpy().astype(np.float64)
    plan.close()
    for lev in range(2, L + 1):
        blk = got[(lev - 2) * 4 * G ** 3:(lev - 1) * 4 * G ** 3]
        for f, a in [(0, (0, 0, 2 * p)), (0, (p, 2 * p - 1, 3)), (1, (2 * p - 1, p, 0)), (2, (1, 2 * p - 1, 2 * p - 1)),
                     (3, (0, min(p + 1, 2 * p - 1), 2 * p - 1)), (0, (min(4 * p - 1, 2 ** lev * p // 2), 1, 0))]:
            i = (lev - 2) * 4 * G ** 3 + ((f * G + a[2]) * G + a[1]) * G + a[0]
            h = 1e-2 * 2.0 ** lev * p
            tp_, tm_ = theta.copy(), theta.copy()
            tp_[i] += h
            tm_[i] -= h
            fd = (olearn.grid_loss(tp_, rho, L, p, tphi, tg, w_phi, w_g)
                  - olearn.grid_loss(tm_, rho, L, p, tphi, tg, w_phi, w_g)) / (2 * h)
            assert abs(got[i] - fd) <= 1e-3 * np.abs(blk).max(), (lev, f, a, got[i], fd, np.abs(blk).max())
