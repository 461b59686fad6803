"""Host-side logic of bench.py (no GPU)."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)


def test_launch_count_claim_matches_the_profiled_launch_list():
    # the ncu launch list of the 256^3 p = 6 bench counts per solve of the
    # headline form: mean 2, P2M 1, M2M 3, M2L 8 (level 2 double-float +
    # range sum, level 3 split table + range sum, levels 4-5 BF16 split +
    # tensor core), L2L 3, near zone by FFT 4 (forward, sums, L2P, inverse):
    # 21; the direct near zone is 1 kernel, and the plain form replaces each
    # tensor-core pair by one FP32 kernel
    import bench
    assert bench.launches_per_solve(5, True, 6, near_fft=True) == 21
    assert bench.launches_per_solve(5, True, 6) == 18
    assert bench.launches_per_solve(5, False, 6) == 16


def test_launch_count_of_the_forms_that_run():
    import bench
    from paper_2011_07099_gb300 import binding as B
    S, D, T, C, N = (B.FMM_FORM_SPECTRAL, B.FMM_FORM_DENSE, B.FMM_FORM_DENSE_TC, B.FMM_FORM_SPECTRAL_TC,
                     B.FMM_FORM_NONE)
    # 256^3 p = 6: mean 2, P2M, M2M 3, levels 2-3 spectral 3, levels 4-5 on the tensor cores 8, L2L 3, near 3
    assert bench.launches_of_forms([S, N, S, S, C, C], 6, 8) == 23
    assert bench.launches_of_forms([S, N, S, S, S, S], 6, 8) == 18          # plain: FP32 and double-float spectra
    assert bench.launches_of_forms([D, N, D, D, T, T], 6, 8) == bench.launches_per_solve(5, True, 6)
    assert bench.launches_of_forms([D, N, D, D, D, D], 6, 8) == bench.launches_per_solve(5, False, 6)
