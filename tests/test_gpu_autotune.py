"""Tuning on nine-node elements, whose kernels have one launch shape each: it picks nothing, and leaves
nothing behind that a pixel context of the same size class would take for its own."""
import pytest

from test_gpu_eval import random_mag

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_elements_keep_their_configuration():
    import paper_1306_1122_gb300 as dbie
    from paper_1306_1122_gb300 import _native as N
    f = dbie.DBIEField.from_magnetogram(random_mag(9, 9, 91))
    f.set_quadrature(4)
    before = N.dbie_get_config(f.handle)
    start = [(c + 1) % 6 for c in before]   # a configuration that no pick of equal shapes is likely to be
    f.set_config(start)
    assert f.autotune() == start
    f.set_quadrature(0)
    f.set_config(before)
    assert all(0 <= c < 6 for c in f.autotune())
    f.close()
