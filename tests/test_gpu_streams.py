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


def test_two_threads_on_one_context():
    """Two host threads evaluate geometries of one context at the same time: an
    evaluation leaves the context's stream alone, so the other thread's work stays
    ordered on it.  Bits as from one thread."""
    _need_cuda()
    import ctypes as C
    import threading

    from paper_1801_04070_gb300 import lib, params_default
    from paper_1801_04070_gb300._lib import GeometryDesc, Stats
    L, ctx = lib(), C.c_void_p()
    assert L.gq_create(0, None, C.byref(ctx)) == 0
    keys = ("ref_b", "ref_u", "base_xy", "base_n", "up_xy", "up_n", "up_w", "panel_len")
    geoms, work = [], []
    for i, (p, off) in enumerate(((10, 3000), (18, 500))):
        g = workloads.small_grid(3, 2, 24, off, seed=i)
        a = {k: np.ascontiguousarray(g[k], np.float64) for k in keys + ("tgt_xy", "density")}
        node = np.ascontiguousarray(g["tgt_onsurf"], np.int32)
        desc = GeometryDesc(int(g["npanels"]), int(g["nb"]), int(g["nu"]), *[a[k].ctypes.data for k in keys])
        geom, prm = C.c_void_p(), params_default(p_qbx=5, p_fmm=p, n_max=32)
        assert L.gq_geometry_create(ctx, C.byref(desc), C.byref(prm), C.byref(geom)) == 0
        assert L.gq_targets_set(geom, len(node), a["tgt_xy"].ctypes.data, node.ctypes.data) == 0
        assert L.gq_build(geom) == 0
        geoms.append(geom)
        work.append((a["density"], len(node)))

    def evaluate(i, kernel):
        out, st = np.empty(work[i][1]), Stats()
        assert L.gq_eval(geoms[i], kernel, work[i][0].ctypes.data, out.ctypes.data, C.byref(st)) == 0
        return out
    want = [[evaluate(i, k) for k in (0, 1)] for i in (0, 1)]
    wrong = []

    def loop(i):
        for n in range(60):
            if not np.array_equal(evaluate(i, n & 1), want[i][n & 1]):
                wrong.append((i, n))
    threads = [threading.Thread(target=loop, args=(i,)) for i in (0, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for geom in geoms:
        assert L.gq_geometry_destroy(geom) == 0
    assert L.gq_destroy(ctx) == 0
    assert not wrong
