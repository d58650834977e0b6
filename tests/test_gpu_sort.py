"""The one-launch cluster sort of up to 32,768 keys (csrc/k_tree.cu) against numpy's stable sort.

Sizes at the edges of its parts: one block of 1024 keys, the next cluster sizes (2, 4, 8 and 16
blocks of 1024 or 2048, the last of them ragged or empty), its largest size, and one key more (the
one-sweep sort).
Most keys occur several times, so the order also shows that the sort is stable.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ff():
    from paper_1212_2934_gb300 import _build, ff

    _build.build()
    ff.lib()
    return ff


@pytest.mark.parametrize("n", [2, 33, 1023, 1024, 1025, 2049, 4097, 16384, 16385, 32767, 32768, 32769])
def test_keys_and_stable_order(ff, n):
    rng = np.random.default_rng(n)
    pts = rng.uniform(0.0, 50.0, (max(n // 3, 1), 3))
    pos = pts[rng.integers(0, len(pts), size=n)].astype(np.float32)
    u = np.tile(np.array([[0.0, 0.0, 1.0]], dtype=np.float32), (n, 1))
    ctx = ff.ff_create(ff.ff_params_default(n=n, lj_eps=0.0, leaf_max=64))
    ff.ff_set_particles(ctx, pos, u)
    ff.ff_dipolar_field(ctx, ff.FF_ALGO_BH, 0.9, False)
    g = ff.ff_get_tree(ctx)
    import oracle

    keys, _ = oracle.morton(pos.astype(np.float64), "f32")
    order = np.argsort(keys, kind="stable")
    assert np.array_equal(g["keys"], keys[order])
    assert np.array_equal(g["order"].astype(np.int64), order)
