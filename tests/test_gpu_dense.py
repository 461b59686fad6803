"""The dense kernels that run where spectra have no room, through the C-ABI
with the plan's spectra limit at 0 (fmm_plan_set_spectra_limit): M2L by dense
sums on the CUDA cores (csrc/m2l_fp32.cu: double-float, split tables, FP32) and
on the tensor cores (csrc/m2l_tc.cu), the near zone by pairs (csrc/p2p.cu) and
the direct table gradient (csrc/learn.cu), against the spectral kernels, which
the FP64 oracle checks (test_gpu_spec.py, test_gpu_near_spec.py).

Tolerances: each form is held to 1e-6 of FP64 (plain) and 2e-5 (bf16x3) over a
mesh, so the two are held to twice that between them."""
import numpy as np
import pytest

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


def _plan(B, N, L, p, iso=False, prec=0):
    plan = B.Plan(N, L, p)
    B.fmm_plan_set_spectra_limit(plan.handle, 0)
    if iso:
        B.fmm_plan_set_boundary(plan.handle, B.FMM_BOUNDARY_ISOLATED)
    if prec:
        plan.set_precision(prec)
    forms, held = B.fmm_plan_get_forms(plan.handle)
    assert held == 0 and not {B.FMM_FORM_SPECTRAL, B.FMM_FORM_SPECTRAL_TC} & set(forms)
    return plan


def _solve(B, plan, rho):
    phi, acc = plan.solve(torch.from_numpy(rho).cuda())
    torch.cuda.synchronize()
    assert B.lib().fmm_plan_check(plan.handle) == B.FMM_OK
    return phi.cpu().numpy(), acc.cpu().numpy()


def _check(B, N, L, p, tol, iso=False, prec=0):
    rho = inputs.lognormal(N, sigma=0.8, seed=N + L + p)
    plan, spectral = _plan(B, N, L, p, iso, prec), B.Plan(N, L, p)
    if iso:
        B.fmm_plan_set_boundary(spectral.handle, B.FMM_BOUNDARY_ISOLATED)
    if prec:
        spectral.set_precision(prec)
    got, ref = _solve(B, plan, rho), _solve(B, spectral, rho)
    plan.close()
    spectral.close()
    what = f"{N}^3 L={L} p={p} iso={iso} prec={prec}"
    assert_close(got[0], ref[0], tol, "phi " + what)
    assert_close(got[1], ref[1], tol, "g " + what)


# level 2 (double-float), 3 (split tables; orders >= 7 double-float) and 4 (FP32); leaves of 1 cell
@pytest.mark.parametrize("N,L,p", [(16, 4, 2), (16, 4, 3), (16, 4, 5), (16, 4, 6), (8, 3, 7), (8, 3, 8)])
def test_dense_m2l_matches_the_spectral_one(B, N, L, p):
    _check(B, N, L, p, 2e-6)


@pytest.mark.parametrize("N,L,p", [(8, 2, 3), (16, 3, 5), (16, 4, 4)])
def test_dense_m2l_isolated_matches_the_spectral_one(B, N, L, p):
    _check(B, N, L, p, 2e-6, iso=True)


# every leaf size that has a spectral near zone, orders below and above it
@pytest.mark.parametrize("S,L,p", [(4, 2, 1), (4, 3, 3), (6, 2, 4), (6, 3, 2), (8, 2, 6), (8, 3, 3), (16, 2, 3), (16, 2, 6)])
def test_near_zone_by_pairs_matches_the_spectral_one(B, S, L, p):
    _check(B, S << L, L, p, 2e-6)


@pytest.mark.parametrize("S", [4, 8])
def test_near_zone_by_pairs_isolated_matches_the_spectral_one(B, S):
    _check(B, S << 2, 2, 4, 2e-6, iso=True)


@pytest.mark.parametrize("N,L,p,iso", [(16, 4, 4, False), (16, 4, 5, True), (16, 4, 6, False), (16, 4, 7, False), (32, 5, 4, False)])
def test_dense_tensor_core_levels_match_the_spectral_ones(B, N, L, p, iso):
    _check(B, N, L, p, 4e-5, iso=iso, prec=B.FMM_PREC_BF16X3)


@pytest.mark.parametrize("group", [1, 3, 189])
def test_dense_tensor_core_promotion_groups(B, group):
    N, L, p = 32, 4, 4
    rho = inputs.plummer(N, n_clumps=16, seed=5)
    plan = _plan(B, N, L, p, prec=B.FMM_PREC_BF16X3)
    B.fmm_plan_set_m2l_group(plan.handle, group)
    spectral = B.Plan(N, L, p, precision=B.FMM_PREC_BF16X3)
    (phi, acc), ref = _solve(B, plan, rho), _solve(B, spectral, rho)
    plan.close()
    spectral.close()
    tol = 4e-5 if group <= 3 else 1e-3          # one partial for all 189 offsets drifts furthest
    assert_close(phi, ref[0], tol, f"group {group} phi")
    assert_close(acc, ref[1], tol, f"group {group} g")


def test_dense_tensor_core_tile_of_128_targets_equals_256_bitwise(B):
    N, L, p = 64, 5, 4                          # tensor-core levels 4 and 5
    rho = inputs.lognormal(N, sigma=0.5, seed=11)
    out = []
    for tile in (256, 128):
        plan = _plan(B, N, L, p, prec=B.FMM_PREC_BF16X3)
        for lev in (4, 5):
            B.fmm_plan_set_tc_tile(plan.handle, lev, tile)
        out.append(_solve(B, plan, rho))
        plan.close()
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("N,L,p", [(128, 6, 2), (96, 5, 3), (64, 3, 6)])
def test_direct_and_spectral_table_gradients_agree_at_every_depth(B, N, L, p):
    # FP32 spectra and chains of 128 terms leave ~1e-7 of a level's gradient
    # against FP64, as the direct sums do: 2e-7 between the two at the leaf level
    # (one FP32 chain over a level of 2^6 nodes per axis left 3.2e-7).  Above it
    # the two solves' own roundings (1e-7 of the residual each) come in: 2e-6.
    rho = torch.from_numpy(inputs.lognormal(N, sigma=0.8, seed=N)).cuda()
    zero = torch.zeros((4, N, N, N), device="cuda")
    G3, out = 4 * (4 * p) ** 3, []
    for plan in (B.Plan(N, L, p), _plan(B, N, L, p)):
        grad = torch.zeros(B.fmm_plan_table_grid_size(plan.handle), device="cuda")
        loss = torch.zeros(1, device="cuda")
        B.fmm_table_grid_grad(plan.handle, rho, zero[0].contiguous(), zero[1:].contiguous(), 1.0, 1e-3, grad, loss)
        torch.cuda.synchronize()
        out.append(grad.double().reshape(L - 1, G3))
        held = B.fmm_plan_get_forms(plan.handle)[1]
        plan.close()
    assert held == 0                                       # the direct sums ran on the last plan
    err = ((out[0] - out[1]).norm(dim=1) / out[1].norm(dim=1)).tolist()
    assert err[-1] < 2e-7 and max(err) < 2e-6, err


def test_tile_autotuner_times_only_levels_that_have_a_tile(B):
    N, L, p = 64, 5, 4
    rho = torch.from_numpy(inputs.lognormal(N, sigma=0.5, seed=12)).cuda()
    plan = B.Plan(N, L, p, precision=B.FMM_PREC_BF16X3)       # levels 4 and 5 on the spectral form
    B.fmm_plan_autotune_tiles(plan.handle, rho)
    with pytest.raises(B.FMMError):                          # no solve was timed
        B.fmm_plan_stage_times(plan.handle)
    plan.close()
    plan = _plan(B, N, L, p, prec=B.FMM_PREC_BF16X3)
    before = plan.solve(rho)
    tiles = B.fmm_plan_autotune_tiles(plan.handle, rho)
    assert tiles[3] == 0 and tiles[4] in (128, 256) and tiles[5] in (128, 256)
    assert B.fmm_plan_stage_times(plan.handle)[B.FMM_TIME_M2L] > 0
    after = plan.solve(rho)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(before, after))
    plan.close()


def test_m2l_ablation_times_the_dense_contractions(B, monkeypatch):
    from paper_2011_07099_gb300 import ablation
    seen, solve = [], B.Plan.solve

    def recorded(self, *a, **k):
        seen.append(tuple(B.fmm_plan_get_forms(self.handle)[0][2:]))
        return solve(self, *a, **k)
    monkeypatch.setattr(B.Plan, "solve", recorded)
    d = torch.from_numpy(inputs.lognormal(32, sigma=0.5, seed=1)).cuda()
    rows = ablation.m2l_forms(32, 4, 4, d, steps=1)
    D, T, F = B.FMM_FORM_DENSE, B.FMM_FORM_DENSE_TC, B.FMM_FORM_FFT
    assert list(dict.fromkeys(seen)) == [(D, D, D), (D, D, T), (D, D, F)] and len(rows) == 3
