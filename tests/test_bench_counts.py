"""The flop and byte models of bench.py against what the current kernels do."""

import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_fp64_smoother_flops():
    """A colour pass: 3 x 5 additions of neighbours, then the Newton solve
    (pfc_device.cuh, point_solve): st1, st3, q4, 2a + b, 4 extra, the two of st2, Q,
    det, the two of the numerator, the four of the quotient, phi and omega are FMAs;
    a^2, b^2, s^2, b^3 and a r products; a + b a sum."""
    sys.path.insert(0, ROOT)
    import bench
    assert bench.FP64_SMOOTH_FLOPS == 15 + 2 * (1 + 1 + 1 + 1 + 1 + 2 + 1 + 1 + 2 + 4 + 1 + 1) + 5 + 1


def test_fp64_prolongation_is_one_launch():
    """u += P (v - w): u read and written, v and w read on the coarse level."""
    sys.path.insert(0, ROOT)
    import bench
    assert bench.KERNEL_BYTES["prolong"] == (48.0 + 2 * 24.0 / 8, 1)


def test_vcycle_bytes_of_a_large_jacobi_level_and_of_odd_sweeps():
    """A 128^3 Jacobi level prolongs in a launch of its own, and an odd count of
    sweeps ends without a copy (the level's buffers change places)."""
    sys.path.insert(0, ROOT)
    import bench
    from paper_1611_06288_gb300 import binding as B
    from paper_1611_06288_gb300 import opbench as OB
    p = B.pfc_default_params()
    for factor in (4, 3):
        p.nu1, p.nu2, p.jacobi_factor, p.jacobi_factor0 = 0, 1, factor, factor
        top = [(256, B.PFC_SWEEP_RB)]
        assert bench.vcycle_bytes(p, top + [(128, B.PFC_SWEEP_JACOBI)]) - \
            bench.vcycle_bytes(p, top) == OB.algorithmic_bytes("lin_restrict_zero", 128) + \
            OB.algorithmic_bytes("lin_prolong_assign", 128) + \
            factor * OB.algorithmic_bytes("lin_jacobi", 128)
        top = [(128, B.PFC_SWEEP_RB)]
        assert bench.vcycle_bytes(p, top + [(64, B.PFC_SWEEP_JACOBI)]) - \
            bench.vcycle_bytes(p, top) == OB.algorithmic_bytes("lin_restrict_zero", 64) + \
            OB.algorithmic_bytes("lin_prolong_jacobi_assign", 64) + \
            (factor - 1) * OB.algorithmic_bytes("lin_jacobi", 64)
