"""What the two streams of an evaluation share."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _need_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


@pytest.mark.parametrize("nx,off", [(1, 300), (3, 2000), (5, 20000)])
def test_orders_lowered_after_the_build(nx, off):
    """Built at an order above the tensor-core kernels' range, evaluated within it:
    their tiles and pairs are then made by the first evaluation.  The values are
    those of a geometry built at the lower order, bit for bit."""
    _need_cuda()
    from paper_1801_04070_gb300 import Geometry, params_default
    g = workloads.small_grid(nx, nx, 24, off, seed=nx)
    for p, q in ((12, 8), (15, 5)):
        ref = Geometry(g, params_default(p_qbx=q, p_fmm=p, n_max=32))
        ref.build()
        want = ref.eval("S", g["density"])
        ref.close()
        for _ in range(3):
            geo = Geometry(g, params_default(p_qbx=q, p_fmm=20, n_max=32))
            geo.build()
            geo.set_orders(q, p)
            first = geo.eval("S", g["density"])
            again = geo.eval("S", g["density"])
            geo.close()
            assert np.array_equal(first, want) and np.array_equal(again, want)
