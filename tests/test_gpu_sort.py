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


def _repeats(n, seed):
    """Positions drawn with repeats from n / 3 points: most keys occur several times."""
    rng = np.random.default_rng(seed)
    pts = rng.uniform(0.0, 50.0, (max(n // 3, 1), 3))
    return pts[rng.integers(0, len(pts), size=n)].astype(np.float32)


# the one-sweep sort: tiles of 1024, 2048 and 4096 keys (4, 8 and 16 a thread), the sizes where it
# changes over, whole tiles and ragged ones
@pytest.mark.parametrize("n", [32769, 40960, 65535, 65536, 65537, 67584, 100003, 393216, 393217,
                               397312, 400003])
def test_tiled_sort_keys_and_stable_order(ff, n):
    import oracle

    pos = _repeats(n, n)
    u = np.tile(np.array([[0.0, 0.0, 1.0]], dtype=np.float32), (n, 1))
    ctx = ff.ff_create(ff.ff_params_default(n=n, lj_eps=0.0, leaf_max=64))
    ff.ff_set_particles(ctx, pos, u)
    ff.ff_dipolar_field(ctx, ff.FF_ALGO_BH, 0.9, False)
    g = ff.ff_get_tree(ctx)
    keys, _ = oracle.morton(pos.astype(np.float64), "f32")
    order = np.argsort(keys, kind="stable")
    assert np.array_equal(g["keys"], keys[order])
    assert np.array_equal(g["order"].astype(np.int64), order)


@pytest.mark.parametrize("sizes", [[20001, 3, 12000], [30000, 35537], [65536, 1, 300000, 27679],
                                   [200001, 200002]])
def test_sort_of_batches(ff, sizes):
    """Keys in order within each system, systems in order (the digit passes over the systems use
    the same tiles)."""
    import oracle

    n = sum(sizes)
    pos = np.concatenate([_repeats(k, 7 + k) for k in sizes])
    u = np.tile(np.array([[0.0, 0.0, 1.0]], dtype=np.float32), (n, 1))
    ctx = ff.ff_create(ff.ff_params_default(n=n, lj_eps=0.0, leaf_max=64))
    ff.ff_set_systems(ctx, sizes)
    ff.ff_set_particles(ctx, pos, u)
    ff.ff_dipolar_field(ctx, ff.FF_ALGO_BH, 0.9, False)
    g = ff.ff_get_tree(ctx)
    off = 0
    for k in sizes:
        keys, _ = oracle.morton(pos[off:off + k].astype(np.float64), "f32")
        order = np.argsort(keys, kind="stable")
        assert np.array_equal(g["keys"][off:off + k], keys[order])
        assert np.array_equal(g["order"][off:off + k].astype(np.int64), order + off)
        off += k
