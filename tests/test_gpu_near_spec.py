"""Near zone by spectral products (csrc/near_spec.cu) in the plain form, against
the FP64 oracle: every leaf size it is built for, periodic (the tile's halo
wraps onto itself at L = 2) and isolated (out-of-box leaves), orders below and
above the leaf size.

Tolerance: the plain form's 1e-6 (FP32 spectra of double-float transforms, 27
products per sum; double-float throughout for 16-cell leaves)."""
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


def _solve(B, rho, L, p, iso=False):
    plan = B.Plan(rho.shape[0], L, p)
    if iso:
        B.fmm_plan_set_boundary(plan.handle, B.FMM_BOUNDARY_ISOLATED)
    phi, acc = plan.solve(torch.from_numpy(rho).cuda())
    torch.cuda.synchronize()
    assert B.lib().fmm_plan_check(plan.handle) == B.FMM_OK
    plan.close()
    return phi.cpu().numpy(), acc.cpu().numpy()


@pytest.mark.parametrize("S,L,p", [(4, 2, 1), (4, 2, 8), (4, 3, 3), (6, 2, 4), (6, 3, 5), (8, 2, 2), (8, 2, 7), (8, 3, 5),
                                   (16, 2, 3), (16, 2, 6)])
def test_near_zone_matches_oracle_at_a_face_leaf(B, S, L, p):
    N = S << L
    rho = inputs.plummer(N, n_clumps=6, seed=N + p, a_min=0.5, a_max=3.0)
    phi, acc = _solve(B, rho, L, p)
    leaves = np.array([[(1 << L) - 1, 0, 1]])
    cells = np.arange(0, S ** 3, 1 if S < 16 else 37)
    ref = ofmm.solve_at(rho, L, p, leaves, cells=cells)
    got = leaf_values(phi, acc, leaves, S)[:, :, cells]
    assert_close(got[:, 0], ref[:, 0], 1e-6, f"phi S={S} L={L} p={p}")
    assert_close(got[:, 1:], ref[:, 1:], 1e-6, f"g S={S} L={L} p={p}")


@pytest.mark.parametrize("S,L,p", [(4, 2, 4), (6, 2, 3), (8, 2, 6), (4, 3, 2)])
def test_near_zone_isolated_matches_oracle(B, S, L, p):
    N = S << L
    rho = inputs.plummer(N, n_clumps=4, seed=N, a_min=0.5, a_max=3.0)
    phi, acc = _solve(B, rho, L, p, iso=True)
    ophi, og = npo.solve_isolated(rho, L, p)
    assert_close(phi, ophi, 1e-6, f"isolated phi S={S} L={L} p={p}")
    assert_close(acc, og, 1e-6, f"isolated g S={S} L={L} p={p}")


@pytest.mark.parametrize("N,L,p,phi_bound,g_bound", [(64, 3, 6, 1.63e-7, 1.57e-7), (32, 2, 4, 2.33e-7, 1.68e-7)])
def test_fp32_transforms_round_no_more_than_radix_2_ones(B, N, L, p, phi_bound, g_bound):
    # FMM_NEAR_FFT against FMM_NEAR_DIRECT, clumped fields, mean of three: the
    # bounds are what radix-2 FP32 transforms of 16 points differ by from the
    # sums over pairs on the same fields
    err = []
    for seed in (1, 2, 3):
        d = torch.from_numpy(inputs.plummer(N, n_clumps=16, seed=seed)).cuda()
        plan = B.Plan(N, L, p)
        direct = plan.solve(d)
        B.fmm_plan_set_near_algorithm(plan.handle, B.FMM_NEAR_FFT)
        fft = plan.solve(d)
        torch.cuda.synchronize()
        err.append([float((a.double() - b.double()).norm() / a.double().norm()) for a, b in zip(direct, fft)])
        plan.close()
    phi, g = np.mean(err, axis=0)
    assert phi <= phi_bound and g <= g_bound, (phi, g)


@pytest.mark.parametrize("S", [4, 6, 8, 16])
def test_a_plan_holds_the_kernel_spectra_of_half_the_offsets(B, S):
    # order 1 has no M2L spectra: 14 of the 27 offsets' kernels (the others are
    # their conjugates), 4 fields of 16 complex values per chunk of 16
    # frequencies; the leaves' spectra and one of zeros; the targets' 4 fields
    L = 2
    plan = B.Plan(S << L, L, 1)
    _, held = B.fmm_plan_get_forms(plan.handle)
    plan.close()
    chunks, leaves = -(-(2 * S - 1) ** 2 * S // 16), 8 ** L
    assert held == chunks * (14 * 512 + (leaves + 1) * 128 + leaves * 4 * 128)
