"""Strengths near the ends of FP64's range: a density times a power of two gives the
potential times that power, as long as nothing overflows.  The fixed-point passes
scale every box by its largest exponent, so they have to hold at both ends: List 2
of p_fmm >= 16, List 3 far and M2M."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,q", [(10, 5), (15, 8), (20, 8), (30, 7)])
@pytest.mark.parametrize("kern", ["S", "D"])
def test_powers_of_two(p, q, kern):
    """m2l = 1: the tensor-core kernels have their own range.  The largest strengths'
    sums stay below 2^1020.  2^-1010: strengths and multipoles are subnormal, rounded
    at 2^-1074, which the potentials (2^-1010) feel at 2^-60; elsewhere the scaling is
    exact, and only the direct sums change between fixed point and FP64 (1e-13, as
    between the other variants of the direct sums)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_04070_gb300 import Geometry, params_default
    g = workloads.small_grid(3, 2, 24, 2000, seed=3)
    geo = Geometry(g, params_default(p_qbx=q, p_fmm=p, n_max=32, m2l=1))
    geo.build()
    base = geo.eval(kern, g["density"])
    for e in (-1010, -990, -700, 700, 970, 990, 1005):
        v = geo.eval(kern, np.ldexp(g["density"], e))
        assert np.isfinite(v).all(), e
        assert np.abs(np.ldexp(v, -e) - base).max() <= (1e-12 if e < -1000 else 1e-13) * np.abs(base).max(), e
    geo.close()
