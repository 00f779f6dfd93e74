"""gq_eval_stages: the values of gq_eval and each stage's own time."""
import numpy as np
import pytest


def test_null_arguments():
    import ctypes as C

    import paper_1801_04070_gb300 as pkg
    from paper_1801_04070_gb300._lib import Stats
    assert pkg.lib().gq_eval_stages(None, 0, None, None, None) == -1
    assert pkg.lib().gq_eval_stages(None, 0, None, None, C.byref(Stats())) == -1


@pytest.mark.gpu
@pytest.mark.parametrize("kw", [{}, {"eps": 1e-8, "precision": 1, "p_qbx": 0, "p_fmm": 0}])
@pytest.mark.parametrize("kern", [0, 1])
def test_stages_in_order(kern, kw):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import ctypes as C

    import workloads
    from paper_1801_04070_gb300 import Geometry, params_default
    from paper_1801_04070_gb300._lib import Stats
    g = workloads.small_grid(4, 4, 32, 20000, seed=1, on_surface="up")
    geo = Geometry(g, params_default(**{"p_qbx": 8, "p_fmm": 15, "n_max": 32, **kw}))
    geo.build()
    want, st = geo.eval("SD"[kern], g["density"]), Stats()
    out = np.empty_like(want)
    for _ in range(3):
        assert geo.L.gq_eval_stages(geo._geom, kern, g["density"].ctypes.data, out.ctypes.data, C.byref(st)) == 0
    geo.close()
    assert np.array_equal(out, want)
    # in order, the stages neither overlap nor leave more than the joins between them
    assert 0.8 * st.ms_total <= sum(st.ms_stage[:11]) <= 1.001 * st.ms_total
