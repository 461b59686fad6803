"""Calls on a plan whose device allocations fail, through the C-ABI and the
host-side hook FMM_FAULT_ALLOC (the n-th allocation asks for more than any
device holds): the call falls back or reports FMM_ERR_ALLOC, and the plan then
solves as it did, with no half-made buffers."""
import numpy as np
import pytest

from oracle import nonperiodic as npo
from paper_2011_07099_gb300 import inputs
from parity_util import assert_close

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL_BF16X3 = 2e-5      # the dense form's bound, as in test_gpu_tensor.py


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2011_07099_gb300 import binding, build
    build.build()
    binding.lib()
    return binding


def _solve(B, plan, d):
    phi, acc = plan.solve(d)
    torch.cuda.synchronize()
    assert B.lib().fmm_plan_check(plan.handle) == B.FMM_OK
    return phi.cpu().numpy(), acc.cpu().numpy()


@pytest.mark.parametrize("n", [0, 1])
def test_a_level_without_room_for_its_tensor_core_spectra_runs_dense(B, n):
    # the sets of levels 4 and 5, one allocation each: the mixed form runs the
    # dense contraction at the level whose set fails, and a later re-tabulation
    # reaches no missing buffer.  Both forms are within 2e-5 of FP64.
    N, L, p = 32, 5, 4
    d = torch.from_numpy(inputs.lognormal(N, sigma=0.5, seed=9)).cuda()
    plan, whole = B.Plan(N, L, p), B.Plan(N, L, p, precision=B.FMM_PREC_BF16X3)
    B.fmm_plan_inject_fault(plan.handle, B.FMM_FAULT_ALLOC + n)
    plan.set_precision(B.FMM_PREC_BF16X3)
    T, C = B.FMM_FORM_DENSE_TC, B.FMM_FORM_SPECTRAL_TC
    assert B.fmm_plan_get_forms(plan.handle)[0][4:] == ([T, C] if n == 0 else [C, T])
    got, ref = _solve(B, plan, d), _solve(B, whole, d)
    assert_close(got[0], ref[0], 2 * TOL_BF16X3, f"set {n} phi")
    assert_close(got[1], ref[1], 2 * TOL_BF16X3, f"set {n} g")
    theta = torch.zeros(B.fmm_plan_table_grid_size(plan.handle))
    B.fmm_plan_set_table_grid(plan.handle, theta)          # a zero correction: the same tables again
    again = _solve(B, plan, d)
    assert np.array_equal(got[0], again[0]) and np.array_equal(got[1], again[1])
    plan.close()
    whole.close()


@pytest.mark.parametrize("n", range(4))
def test_each_set_of_spectra_is_one_allocation_and_is_left_out_alone(B, n):
    # the sets of levels 2 and 3 and of the near zone (an allocation takes tens
    # of microseconds of a plan's creation); there is no fourth
    N, L, p = 32, 3, 4
    d = torch.from_numpy(inputs.lognormal(N, sigma=0.5, seed=9)).cuda()
    plan, whole = B.Plan(N, L, p), B.Plan(N, L, p)
    B.fmm_plan_inject_fault(plan.handle, B.FMM_FAULT_ALLOC + n)
    B.fmm_plan_set_spectra_limit(plan.handle, None)
    forms = B.fmm_plan_get_forms(plan.handle)[0]
    assert [i for i in (2, 3, 0) if forms[i] == B.FMM_FORM_DENSE] == [[2], [3], [0], []][n]
    got, ref = _solve(B, plan, d), _solve(B, whole, d)
    assert_close(got[0], ref[0], 2e-6, f"set {n} phi")     # both within 1e-6 of FP64
    assert_close(got[1], ref[1], 2e-6, f"set {n} g")
    plan.close()
    whole.close()


@pytest.mark.parametrize("n", [0, 1, 2])
def test_a_first_level_that_cannot_be_prepared_is_not_taken(B, n):
    # order 2: the dense form's BF16 table, sources and tiles of level 4
    N, L, p = 32, 5, 2
    d = torch.from_numpy(inputs.lognormal(N, sigma=0.5, seed=3)).cuda()
    plan = B.Plan(N, L, p)
    B.fmm_plan_set_tc_min_level(plan.handle, 5)
    plan.set_precision(B.FMM_PREC_BF16X3)
    ref = _solve(B, plan, d)
    B.fmm_plan_inject_fault(plan.handle, B.FMM_FAULT_ALLOC + n)
    assert B.lib().fmm_plan_set_tc_min_level(plan.handle, 4) == B.FMM_ERR_ALLOC
    got = _solve(B, plan, d)                               # level 5 alone, as before
    assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])
    B.fmm_plan_set_tc_min_level(plan.handle, 4)            # and with room
    fresh = B.Plan(N, L, p)
    fresh.set_precision(B.FMM_PREC_BF16X3)
    a, b = _solve(B, plan, d), _solve(B, fresh, d)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    plan.close()
    fresh.close()


@pytest.mark.parametrize("n", range(6))
def test_training_buffers_are_made_all_or_none(B, n):
    # the call's allocations, in order: solve outputs, residual, table
    # gradients, network partials, one adjoint (level 2); then the set of the
    # spectral table gradient, without which the direct sums run
    N, L, p = 8, 2, 3
    rho = torch.from_numpy(inputs.lognormal(N, sigma=0.8, seed=2)).cuda()
    tphi, tg = torch.randn((N, N, N), device="cuda"), torch.randn((3, N, N, N), device="cuda")

    def gradient(plan, fault=None):
        grad = torch.zeros(B.fmm_plan_table_grid_size(plan.handle), device="cuda")
        loss = torch.zeros(1, device="cuda")
        if fault is not None:
            B.fmm_plan_inject_fault(plan.handle, B.FMM_FAULT_ALLOC + fault)
        ptr = lambda t: t.data_ptr()
        rc = B.lib().fmm_table_grid_grad(plan.handle, ptr(rho), ptr(tphi), ptr(tg), 1.0, 1.0, ptr(grad), ptr(loss), 0)
        torch.cuda.synchronize()
        return rc, grad.double(), float(loss)

    fresh, plan = B.Plan(N, L, p), B.Plan(N, L, p)
    rc, want, want_loss = gradient(fresh)
    assert rc == B.FMM_OK
    rc, got, _ = gradient(plan, n)
    assert rc == (B.FMM_ERR_ALLOC if n < 5 else B.FMM_OK)
    if n < 5:
        rc, got, loss = gradient(plan)
        assert rc == B.FMM_OK and loss == want_loss
    # FP32 sums of ~1e4 terms in another order: 1e-5 of the gradient
    assert float((got - want).norm() / want.norm()) < 1e-5
    plan.close()
    fresh.close()


@pytest.mark.parametrize("n", [0, 1])
def test_a_boundary_that_cannot_be_set_is_not_taken(B, n):
    # order 1 runs the dense sums: the new interaction list, then the scratch
    # of its offset ranges
    N, L, p = 8, 3, 1
    rho = inputs.lognormal(N, sigma=0.5, seed=4)
    d = torch.from_numpy(rho).cuda()
    plan = B.Plan(N, L, p)
    ref = _solve(B, plan, d)
    B.fmm_plan_inject_fault(plan.handle, B.FMM_FAULT_ALLOC + n)
    assert B.lib().fmm_plan_set_boundary(plan.handle, B.FMM_BOUNDARY_ISOLATED) == B.FMM_ERR_ALLOC
    got = _solve(B, plan, d)
    assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])
    B.fmm_plan_set_boundary(plan.handle, B.FMM_BOUNDARY_ISOLATED)
    got = _solve(B, plan, d)
    ophi, og = npo.solve_isolated(rho, L, p)
    assert_close(got[0], ophi, 1e-6, "isolated phi")
    assert_close(got[1], og, 1e-6, "isolated g")
    plan.close()


def test_spectra_limit_sets_the_forms_and_is_undone_bitwise(B):
    N, L, p = 64, 4, 4
    d = torch.from_numpy(inputs.lognormal(N, sigma=0.5, seed=7)).cuda()
    plan = B.Plan(N, L, p, precision=B.FMM_PREC_BF16X3)
    forms, held = B.fmm_plan_get_forms(plan.handle)
    S, D, T, C = B.FMM_FORM_SPECTRAL, B.FMM_FORM_DENSE, B.FMM_FORM_DENSE_TC, B.FMM_FORM_SPECTRAL_TC
    assert forms == [S, B.FMM_FORM_NONE, S, S, C] and held > 0
    ref = _solve(B, plan, d)
    B.fmm_plan_set_spectra_limit(plan.handle, 0)
    assert B.fmm_plan_get_forms(plan.handle) == ([D, B.FMM_FORM_NONE, D, D, T], 0)
    dense = _solve(B, plan, d)
    assert_close(dense[0], ref[0], 2e-5, "dense against spectral phi")
    B.fmm_plan_set_near_algorithm(plan.handle, B.FMM_NEAR_DIRECT)
    assert B.fmm_plan_get_forms(plan.handle)[1] == 0
    for limit in (6 << 20, 1 << 25):                # level 2 fits (5.4 MB); levels 2 and 3 (18 MB)
        B.fmm_plan_set_spectra_limit(plan.handle, limit)
        f, b = B.fmm_plan_get_forms(plan.handle)
        assert 0 < b <= limit and f[2] == S and f[0] == D, (f, b)
    B.fmm_plan_set_spectra_limit(plan.handle, None)
    assert B.fmm_plan_get_forms(plan.handle) == (forms, held)
    got = _solve(B, plan, d)
    assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])
    plan.close()


def test_a_limit_whose_buffers_cannot_be_made_stops_the_solves(B):
    # the scratch of the dense coarse levels is the only allocation of the limit 0 in the plain form
    N, L, p = 16, 3, 4
    d = torch.from_numpy(inputs.lognormal(N, sigma=0.5, seed=8)).cuda()
    plan, fresh = B.Plan(N, L, p), B.Plan(N, L, p)
    B.fmm_plan_inject_fault(plan.handle, B.FMM_FAULT_ALLOC + 0)
    assert B.lib().fmm_plan_set_spectra_limit(plan.handle, 0) == B.FMM_ERR_ALLOC
    with pytest.raises(B.FMMError) as e:
        plan.solve(d)
    assert e.value.code == B.FMM_ERR_ALLOC
    for pl in (plan, fresh):
        B.fmm_plan_set_spectra_limit(pl.handle, 0)
    a, b = _solve(B, plan, d), _solve(B, fresh, d)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    plan.close()
    fresh.close()


def test_a_statement_without_scratch_leaves_no_error_behind(B):
    # CUDA keeps a failed allocation's error until it is read: the next solve must not report it
    N, L, p = 16, 2, 3
    d = torch.from_numpy(inputs.lognormal(N, sigma=0.5, seed=5)).cuda()
    plan = B.Plan(N, L, p)
    phi, acc = plan.solve(d)
    B.fmm_plan_inject_fault(plan.handle, B.FMM_FAULT_ALLOC + 0)
    with pytest.raises(B.FMMError) as e:
        plan.error_stats(d, phi, acc, samples=32, seed=1)
    assert e.value.code == B.FMM_ERR_ALLOC
    again = plan.solve(d)
    torch.cuda.synchronize()
    assert torch.equal(again[0], phi) and torch.equal(again[1], acc)
    assert max(plan.error_stats(d, phi, acc, samples=32, seed=1)) < 1.0
    plan.close()


@pytest.mark.parametrize("n", [0, 1])
def test_host_staging_is_made_on_the_next_call(B, n):
    N, L, p = 16, 2, 3
    host = torch.from_numpy(inputs.lognormal(N, sigma=0.5, seed=5))
    phi, acc = torch.empty((N, N, N)), torch.empty((3, N, N, N))
    plan = B.Plan(N, L, p)
    ref = _solve(B, plan, host.cuda())
    B.fmm_plan_inject_fault(plan.handle, B.FMM_FAULT_ALLOC + n)
    with pytest.raises(B.FMMError) as e:
        B.fmm_solve_host(plan.handle, host, phi, acc)
    assert e.value.code == B.FMM_ERR_ALLOC
    B.fmm_solve_host(plan.handle, host, phi, acc)
    assert np.array_equal(phi.numpy(), ref[0]) and np.array_equal(acc.numpy(), ref[1])
    plan.close()
