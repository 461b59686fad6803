"""The dense kernels that run where spectra have no room, through the C-ABI
with the plan's spectra limit at 0 (fmm_plan_set_spectra_limit): M2L by dense
sums on the CUDA cores (csrc/m2l_fp32.cu: double-float, split tables, FP32) and
on the tensor cores (csrc/m2l_tc.cu), the near zone by pairs (csrc/p2p.cu) and
the direct table gradient (csrc/learn.cu), against the FP64 oracle.

Tolerances as for the same kernels elsewhere: 1e-6 for the plain form, 2e-5 for
bf16x3 (test_gpu_tensor.py), 1e-3 of the largest gradient (test_gpu_spec.py)."""
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
    plan = _plan(B, N, L, p, iso, prec)
    phi, acc = _solve(B, plan, rho)
    plan.close()
    n = 1 << L
    leaves, S = np.array([[n - 1, 0, n // 2 + 1]]), N >> L
    cells = np.arange(0, S ** 3, 1 if S < 16 else 37)
    if iso:
        ref = npo.solve_isolated_at(rho, L, p, leaves)[:, :, cells]
    else:
        ref = ofmm.solve_at(rho, L, p, leaves, cells=cells)
    got = leaf_values(phi, acc, leaves, S)[:, :, cells]
    # the tolerances are of the whole mesh's norm: errors in one leaf, whose own
    # values may be small, against the mesh's root mean square
    for what, f, mesh in (("phi", slice(0, 1), phi), ("g", slice(1, 4), acc)):
        rms = np.sqrt(np.mean(mesh.astype(np.float64) ** 2))
        err = np.sqrt(np.mean((got[:, f].astype(np.float64) - ref[:, f]) ** 2)) / rms
        print(f"{what} {N}^3 L={L} p={p} iso={iso} prec={prec}: {err:.3e} of the mesh's RMS (tol {tol:.1e})")
        assert err <= tol, (what, err, tol)


# level 2 (double-float), 3 (split tables; orders >= 7 double-float) and 4 (FP32); leaves of 1 cell
@pytest.mark.parametrize("N,L,p", [(16, 4, 2), (16, 4, 3), (16, 4, 5), (16, 4, 6), (8, 3, 7), (8, 3, 8)])
def test_dense_m2l_matches_oracle(B, N, L, p):
    _check(B, N, L, p, 1e-6)


@pytest.mark.parametrize("N,L,p", [(8, 2, 3), (16, 3, 5), (16, 4, 4)])
def test_dense_m2l_isolated_matches_oracle(B, N, L, p):
    _check(B, N, L, p, 1e-6, iso=True)


# every leaf size that has a spectral near zone, orders below and above it
@pytest.mark.parametrize("S,L,p", [(4, 2, 1), (4, 3, 3), (6, 2, 4), (6, 3, 2), (8, 2, 6), (8, 3, 3), (16, 2, 3), (16, 2, 6)])
def test_near_zone_by_pairs_matches_oracle(B, S, L, p):
    _check(B, S << L, L, p, 1e-6)


@pytest.mark.parametrize("S", [4, 8])
def test_near_zone_by_pairs_isolated_matches_oracle(B, S):
    _check(B, S << 2, 2, 4, 1e-6, iso=True)


@pytest.mark.parametrize("N,L,p,iso", [(16, 4, 4, False), (16, 4, 5, True), (16, 4, 6, False), (16, 4, 7, False), (32, 5, 4, False)])
def test_dense_tensor_core_levels_match_oracle(B, N, L, p, iso):
    _check(B, N, L, p, 2e-5, iso=iso, prec=B.FMM_PREC_BF16X3)


@pytest.mark.parametrize("group", [1, 3, 189])
def test_dense_tensor_core_promotion_groups(B, group):
    N, L, p = 32, 4, 4
    rho = inputs.plummer(N, n_clumps=16, seed=5)
    plan = _plan(B, N, L, p, prec=B.FMM_PREC_BF16X3)
    B.fmm_plan_set_m2l_group(plan.handle, group)
    phi, acc = _solve(B, plan, rho)
    plan.close()
    ophi, og = ofmm.solve(rho, L, p)
    tol = 2e-5 if group <= 3 else 1e-3          # one partial for all 189 offsets drifts furthest
    assert_close(phi, ophi, tol, f"group {group} phi")
    assert_close(acc, og, tol, f"group {group} g")


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


@pytest.mark.parametrize("N,L,p", [(8, 2, 5), (8, 3, 3)])
def test_direct_table_gradient_of_a_periodic_plan_matches_oracle_differences(B, N, L, p):
    # the loss is quadratic in the table values: central differences are exact
    from oracle import learn as olearn
    rho = inputs.lognormal(N, sigma=0.8, seed=N + p)
    n, G = olearn.grid_size(L, p), 4 * p
    theta = np.zeros(n)
    tphi, tg = (np.asarray(x) * 1.3 for x in olearn.pm_target(rho))
    w_phi, w_g = 1.0 / np.sum(tphi ** 2), 1.0 / np.sum(tg ** 2)
    plan = _plan(B, N, L, p)
    grad = torch.zeros(n, dtype=torch.float32, device="cuda")
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    f32 = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    B.fmm_table_grid_grad(plan.handle, f32(rho), f32(tphi), f32(tg), w_phi, w_g, grad, loss)
    got = grad.cpu().numpy().astype(np.float64)
    assert B.fmm_plan_get_forms(plan.handle)[1] == 0
    plan.close()
    for lev in range(2, L + 1):
        blk = got[(lev - 2) * 4 * G ** 3:(lev - 1) * 4 * G ** 3]
        for f, a in [(0, (0, 0, 2 * p)), (0, (p, 2 * p - 1, 3)), (1, (2 * p - 1, p, 0)), (3, (0, p + 1, 2 * p - 1))]:
            i = (lev - 2) * 4 * G ** 3 + ((f * G + a[2]) * G + a[1]) * G + a[0]
            h = 1e-2 * 2.0 ** lev * p
            tp_, tm_ = theta.copy(), theta.copy()
            tp_[i] += h
            tm_[i] -= h
            fd = (olearn.grid_loss(tp_, rho, L, p, tphi, tg, w_phi, w_g)
                  - olearn.grid_loss(tm_, rho, L, p, tphi, tg, w_phi, w_g)) / (2 * h)
            assert abs(got[i] - fd) <= 1e-3 * np.abs(blk).max(), (lev, f, a, got[i], fd, np.abs(blk).max())


@pytest.mark.parametrize("N,L,p", [(128, 6, 2), (96, 5, 3), (64, 3, 6)])
def test_spectral_table_gradient_rounds_like_the_direct_one_at_depth(B, N, L, p):
    # FP32 spectra and chains of 128 terms leave ~1e-7 of the leaf level's
    # gradient against FP64, as the direct sums do: 2e-7 between the two.  (One
    # FP32 chain over a level of 2^6 nodes per axis left 3.2e-7.)
    rho = torch.from_numpy(inputs.lognormal(N, sigma=0.8, seed=N)).cuda()
    zero = torch.zeros((4, N, N, N), device="cuda")
    G3, out = 4 * (4 * p) ** 3, []
    for plan in (B.Plan(N, L, p), _plan(B, N, L, p)):
        grad = torch.zeros(B.fmm_plan_table_grid_size(plan.handle), device="cuda")
        loss = torch.zeros(1, device="cuda")
        B.fmm_table_grid_grad(plan.handle, rho, zero[0].contiguous(), zero[1:].contiguous(), 1.0, 1e-3, grad, loss)
        torch.cuda.synchronize()
        out.append(grad[-G3:].double())
        plan.close()
    err = float((out[0] - out[1]).norm() / out[1].norm())
    assert err < 2e-7, err


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
