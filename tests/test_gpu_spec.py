"""M2L by spectral products (csrc/m2l_spec.cu, on the tensor cores
csrc/m2l_spec_tc.cu) against the FP64 oracle, through the C-ABI, on trees whose
levels take each of its kernels (level 2 periodic and isolated, double-float,
row chains, FP32, tensor cores), with one cell per leaf and more.

Tolerance: the plain form's 1e-6 (FP32 spectra, sums over a plane's terms apart
from the total, double-float transforms: rounding of ~1e-7 per level times the
far field's cancellation of a few); the mixed form (FP16 pairs, 22 bits, FP32
accumulation and transforms) keeps its bf16x3 bound 2e-5."""
import numpy as np
import pytest

from oracle import fmm as ofmm
from oracle import nonperiodic as npo
from paper_2011_07099_gb300 import inputs
from parity_util import assert_close, leaf_values

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


LEAVES = {2: [[0, 0, 0], [3, 1, 2]], 3: [[7, 0, 5]], 4: [[15, 0, 6]]}   # on the faces: every wrap is taken


def _check(B, N, L, p, tol, iso=False, prec=0):
    rho = inputs.lognormal(N, sigma=0.8, seed=N + L + p)
    phi, acc = _solve(B, rho, L, p, iso, prec)
    leaves = np.array(LEAVES[L])
    ref = (npo.solve_isolated_at if iso else ofmm.solve_at)(rho, L, p, leaves)
    got = leaf_values(phi, acc, leaves, N >> L)
    what = f"{N}^3 L={L} p={p} iso={iso} prec={prec}"
    assert_close(got[:, 0], ref[:, 0], tol, "phi " + what)
    assert_close(got[:, 1:], ref[:, 1:], tol, "g " + what)


# odd and even orders; p = 8 is in the full-size tests of the plain and the mixed form
@pytest.mark.parametrize("N,L,p", [(12, 2, 5), (12, 2, 7), (16, 3, 4), (16, 4, 2), (16, 4, 3), (16, 4, 5), (16, 4, 6),
                                   (16, 3, 7)])
def test_spectral_m2l_matches_oracle(B, N, L, p):
    _check(B, N, L, p, 1e-6)


@pytest.mark.parametrize("N,L,p", [(8, 2, 3), (16, 2, 6), (16, 3, 5), (16, 4, 4)])
def test_spectral_m2l_isolated_matches_oracle(B, N, L, p):
    _check(B, N, L, p, 1e-6, iso=True)


# the tensor-core form: two parents per forward CTA (p <= 6) and one (p = 7),
# periodic halo copies and the isolated problem's zeros
@pytest.mark.parametrize("N,L,p,iso", [(16, 4, 4, False), (16, 4, 5, True), (16, 4, 6, False), (16, 4, 7, False),
                                       (32, 5, 4, False)])
def test_tensor_core_spectral_levels_match_oracle(B, N, L, p, iso):
    LEAVES.setdefault(5, [[31, 0, 17]])
    _check(B, N, L, p, 2e-5, iso=iso, prec=B.FMM_PREC_BF16X3)


def test_tensor_core_form_follows_the_boundary(B):
    # the periodic halo of an earlier solve must not leak into the isolated problem, nor zeros into the periodic one
    N, L, p = 32, 4, 4
    rho = torch.from_numpy(inputs.lognormal(N, sigma=0.8, seed=6)).cuda()
    plan = B.Plan(N, L, p, precision=B.FMM_PREC_BF16X3)
    out = []
    for b in (B.FMM_BOUNDARY_PERIODIC, B.FMM_BOUNDARY_ISOLATED, B.FMM_BOUNDARY_PERIODIC, B.FMM_BOUNDARY_ISOLATED):
        B.fmm_plan_set_boundary(plan.handle, b)
        phi, acc = plan.solve(rho)
        torch.cuda.synchronize()
        out.append((phi, acc))
    plan.close()
    assert torch.equal(out[0][0], out[2][0]) and torch.equal(out[0][1], out[2][1])
    fresh = B.Plan(N, L, p)
    B.fmm_plan_set_boundary(fresh.handle, B.FMM_BOUNDARY_ISOLATED)
    fresh.set_precision(B.FMM_PREC_BF16X3)
    phi, acc = fresh.solve(rho)
    torch.cuda.synchronize()
    for k in (1, 3):
        assert torch.equal(out[k][0], phi) and torch.equal(out[k][1], acc)
    fresh.close()


def test_tensor_core_scale_follows_the_field(B):
    # the FP16 split is scaled by the level's largest mass sum: densities 1e12
    # apart in size give the same solution up to rounding, and zeros give zeros
    N, L, p = 32, 4, 4
    rho = inputs.plummer(N, n_clumps=4, seed=3)
    plan = B.Plan(N, L, p, precision=B.FMM_PREC_BF16X3)
    ref = plan.solve(torch.from_numpy(rho).cuda())[0].double()
    for s in (2.0 ** 40, 2.0 ** -40):
        phi = plan.solve(torch.from_numpy((rho * np.float32(s)).astype(np.float32)).cuda())[0].double() / s
        assert float((phi - ref).norm() / ref.norm()) < 1e-6
    phi, acc = plan.solve(torch.full((N, N, N), 1.7, device="cuda"))
    assert torch.all(phi == 0) and torch.all(acc == 0)
    plan.close()


def test_tensor_core_bounded_wait_expires_and_context_survives(B):
    N, L, p = 32, 4, 4
    rho = torch.from_numpy(inputs.lognormal(N, sigma=0.5, seed=2)).cuda()
    plan = B.Plan(N, L, p, precision=B.FMM_PREC_BF16X3)
    ref = [x.clone() for x in plan.solve(rho)]
    B.fmm_plan_set_timeout_ms(plan.handle, 20)
    B.fmm_plan_inject_fault(plan.handle, B.FMM_FAULT_TC_STALL)
    plan.solve(rho)
    assert B.lib().fmm_plan_check(plan.handle) == B.FMM_ERR_TIMEOUT
    B.fmm_plan_inject_fault(plan.handle, B.FMM_FAULT_NONE)
    B.fmm_plan_set_timeout_ms(plan.handle, 2000)
    phi, acc = plan.solve(rho)
    assert B.lib().fmm_plan_check(plan.handle) == B.FMM_OK
    assert torch.equal(phi, ref[0]) and torch.equal(acc, ref[1])
    plan.close()


def test_levels_in_one_launch_equal_levels_one_by_one_bitwise(B):
    # timed solves launch each level on its own, untimed ones all levels of one
    # arithmetic together, on two streams
    rho = inputs.lognormal(32, sigma=0.5, seed=4)
    for p in (4, 7):
        a, b = _solve(B, rho, 5, p), _solve(B, rho, 5, p, timing=True)
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("N,L,p", [(8, 2, 5), (8, 3, 3), (8, 3, 2)])
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
