"""The shared walk of small single-precision contexts (csrc/k_walk.cu) against the counting walk.

Contexts of up to 106,496 particles without interaction counts take a walk in which a warp
serves 8, 16 or 32 particles (n <= 8192, <= 26,624, above); with counts they take the one-lane
walk.  Both add every particle's sources in the same order with the same operations, so fields
and forces agree bit for bit, over the edges of the task sizes, leaves of several particles,
LJ on and off, opening angles from 0 (every cell opened) to 0.9, tasks that span several
systems, and coincident particles; the energies (sums of the same terms) agree too.
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


def _gas(n, seed):
    """Random sites of a jittered lattice (no two centres closer than 1)."""
    rng = np.random.default_rng(seed)
    m = max(2, int(np.ceil((3.1 * n) ** (1.0 / 3.0))))
    site = rng.permutation(m ** 3)[:n]
    q = np.stack([site // (m * m), (site // m) % m, site % m], axis=1)
    u = rng.standard_normal((n, 3))
    u /= np.linalg.norm(u, axis=1)[:, None]
    return ((q + rng.uniform(-0.16, 0.16, (n, 3))) * 1.5).astype(np.float32), u.astype(np.float32)


def _both(ff, pos, u, theta, sizes=None, **kw):
    out = []
    for count in (0, 1):
        ctx = ff.ff_create(ff.ff_params_default(n=len(pos), count_interactions=count, **kw))
        if sizes is not None:
            ff.ff_set_systems(ctx, sizes)
        ff.ff_set_particles(ctx, pos, u)
        out.append(ff.ff_dipolar_field(ctx, ff.FF_ALGO_BH, theta, True, dtype=np.float32))
    return out


@pytest.mark.parametrize("n", [1, 2, 7, 9, 33, 1000, 8191, 8193, 26623, 26625, 40009, 106496])
def test_equals_counting_walk_at_task_edges(ff, n):
    pos, u = _gas(n, n)
    (hp, fp), (hc, fc) = _both(ff, pos, u, 0.5)
    assert np.array_equal(hp, hc) and np.array_equal(fp, fc)


@pytest.mark.parametrize("theta", [0.0, 0.3, 0.9])
@pytest.mark.parametrize("leaf_max", [1, 5, 64])
@pytest.mark.parametrize("lj", [0.0, 1.0])
def test_equals_counting_walk_over_options(ff, theta, leaf_max, lj):
    pos, u = _gas(2011, 3)
    (hp, fp), (hc, fc) = _both(ff, pos, u, theta, leaf_max=leaf_max, lj_eps=lj)
    assert np.array_equal(hp, hc) and np.array_equal(fp, fc)


@pytest.mark.parametrize("n", [3000, 9001, 30011])
def test_tasks_spanning_systems(ff, n):
    rng = np.random.default_rng(n)
    sizes = []
    while sum(sizes) < n:
        sizes.append(min(int(rng.integers(1, 40)), n - sum(sizes)))
    parts = [_gas(k, i)[0] for i, k in enumerate(sizes)]
    _, u = _gas(n, 1)
    (hp, fp), (hc, fc) = _both(ff, np.concatenate(parts), u, 0.5, sizes=sizes)
    assert np.array_equal(hp, hc) and np.array_equal(fp, fc)


def test_coincident_particles_and_flat_systems(ff):
    pos, u = _gas(4000, 9)
    pos[100:190] = pos[100]           # one leaf of 90 particles at the deepest level
    pos[500:2500, 2] = 0.0            # a layer, some of its pairs near enough to overflow LJ
    (hp, fp), (hc, fc) = _both(ff, pos, u, 0.6)
    assert np.array_equal(hp, hc) and np.array_equal(fp, fc, equal_nan=True)
    line = np.zeros((3000, 3), dtype=np.float32)
    line[:, 0] = np.arange(3000) * 1.25
    (hp, fp), (hc, fc) = _both(ff, line, u[:3000], 0.5)
    assert np.array_equal(hp, hc) and np.array_equal(fp, fc)
