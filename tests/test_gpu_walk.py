"""The walks that serve several particles a warp: of small single-precision contexts
(csrc/k_walk.cu) against the counting walk, and of double precision (csrc/k_walk64.cu) against
the oracle.

Contexts of up to 106,496 particles without interaction counts take a walk in which a warp
serves 4, 8, 16 or 32 particles (n <= 4096, <= 8192, <= 26,624, above); with counts they take the one-lane
walk.  Both add every particle's sources in the same order with the same operations, so fields
and forces agree bit for bit, over the edges of the task sizes, leaves of several particles,
LJ on and off, opening angles from 0 (every cell opened) to 0.9, tasks that span several
systems, and coincident particles.  The double-precision walk is held to the repository's 1e-10
and to exact interaction counts over the same options.
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


def _both(ff, pos, u, theta, sizes=None, dtype=np.float32, **kw):
    out = []
    for count in (0, 1):
        ctx = ff.ff_create(ff.ff_params_default(n=len(pos), count_interactions=count, **kw))
        if sizes is not None:
            ff.ff_set_systems(ctx, sizes)
        ff.ff_set_particles(ctx, pos, u)
        out.append(ff.ff_dipolar_field(ctx, ff.FF_ALGO_BH, theta, True, dtype=dtype))
    return out


@pytest.mark.parametrize("n", [1, 2, 3, 5, 9, 33, 1000, 4095, 4097, 8191, 8193, 26623, 26625, 40009, 106496])
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


@pytest.mark.parametrize("theta", [0.0, 0.3, 0.9])
@pytest.mark.parametrize("leaf_max", [1, 5, 64])
@pytest.mark.parametrize("lj", [0.0, 1.0])
def test_fp64_matches_oracle(ff, theta, leaf_max, lj):
    import oracle
    from conftest import rel_err

    for n in (1, 7, 8, 9, 1501):
        pos, u = _gas(n, 40 + n)
        # off the single-precision grid, far from the origin
        pos = pos.astype(np.float64) * (1.0 + 1e-9) + np.array([1000.0, -300.0, 7.0]) / 3.0
        u = u.astype(np.float64)
        (hp, fp), (hc, fc) = [(a, b) for a, b in _both(ff, pos, u, theta, precision="f64",
                                                      leaf_max=leaf_max, lj_eps=lj,
                                                      dtype=np.float64)]
        assert np.array_equal(hp, hc) and np.array_equal(fp, fc)
        if n == 1:
            assert not hp.any() and not fp.any()
            continue
        ref = oracle.bh(pos, u, theta, leaf_max, "f64", 1.0, lj, 1.0, 2.5, True)
        assert rel_err(hp, ref["h"]).max() <= 1e-10
        assert rel_err(fp, ref["f"]).max() <= 1e-10
        ctx = ff.ff_create(ff.ff_params_default(n=n, precision="f64", leaf_max=leaf_max,
                                                lj_eps=lj, count_interactions=1))
        ff.ff_set_particles(ctx, pos, u)
        ff.ff_dipolar_field(ctx, ff.FF_ALGO_BH, theta, True)
        acc, pairs, opened = ff.ff_get_counts(ctx)
        assert np.array_equal(acc, ref["nacc"]) and np.array_equal(pairs, ref["npair"])
        assert np.array_equal(opened, ref["nopen"])


def test_fp64_tasks_spanning_systems(ff):
    rng = np.random.default_rng(5)
    sizes = [int(k) for k in rng.integers(1, 30, 200)]
    parts = [_gas(k, i) for i, k in enumerate(sizes)]
    pos = np.concatenate([p for p, _ in parts]).astype(np.float64)
    u = np.concatenate([q for _, q in parts]).astype(np.float64)
    (hp, fp), (hc, fc) = _both(ff, pos, u, 0.5, sizes=sizes, precision="f64", dtype=np.float64)
    assert np.array_equal(hp, hc) and np.array_equal(fp, fc)
    # each system alone gives the same bits: a particle's sums depend on its own sources
    off = 0
    for k, (p, q) in list(zip(sizes, parts))[:25]:
        ctx = ff.ff_create(ff.ff_params_default(n=k, precision="f64"))
        ff.ff_set_particles(ctx, p.astype(np.float64), q.astype(np.float64))
        h, f = ff.ff_dipolar_field(ctx, ff.FF_ALGO_BH, 0.5, True)
        assert np.array_equal(h, hp[off:off + k]) and np.array_equal(f, fp[off:off + k])
        off += k


@pytest.mark.parametrize("leaf_max", [1, 6])
def test_fp64_long_lists_do_not_depend_on_neighbours(ff, leaf_max):
    """A particle's sources are summed 480 to 512 at a time, all of a warp's particles when the
    longest list is full; which of its four partial sums a source goes to does not depend on that.
    Systems whose lists are cut several times, at offsets that put other particles in the warps,
    have the bits they have alone."""
    sizes = [3001, 1500, 2503, 7, 1999]
    parts = [_gas(k, 60 + k) for k in sizes]
    pos = np.concatenate([p for p, _ in parts]).astype(np.float64)
    u = np.concatenate([q for _, q in parts]).astype(np.float64)
    (hp, fp), (hc, fc) = _both(ff, pos, u, 0.3, sizes=sizes, precision="f64", leaf_max=leaf_max,
                               dtype=np.float64)
    assert np.array_equal(hp, hc) and np.array_equal(fp, fc)
    off = 0
    for k, (p, q) in zip(sizes, parts):
        ctx = ff.ff_create(ff.ff_params_default(n=k, precision="f64", leaf_max=leaf_max,
                                                count_interactions=1))
        ff.ff_set_particles(ctx, p.astype(np.float64), q.astype(np.float64))
        h, f = ff.ff_dipolar_field(ctx, ff.FF_ALGO_BH, 0.3, True)
        assert np.array_equal(h, hp[off:off + k]) and np.array_equal(f, fp[off:off + k])
        acc, pairs, _ = ff.ff_get_counts(ctx)
        assert k < 100 or (acc + pairs).max() > 512  # longer than a list
        off += k


@pytest.mark.parametrize("theta", [1e-19, 0.5, 9.0, 11.0, 1e6, 1e25])
def test_fp64_decides_exactly_at_any_angle(ff, theta):
    """Particles about the LJ cut away from the upper face of a cube a million wide, whose own
    particles lie at that face: at opening angles that accept it, the distance from its cube
    decides, and the far corner it is formed from is a million away."""
    import oracle
    from conftest import rel_err

    s = 2.0 ** 20
    k = np.arange(64)
    pos = np.zeros((68, 3))
    pos[0, 1:] = s
    pos[1, 0] = s
    pos[2:4] = [[s / 2 - 0.3, 5000.0, 4000.0], [s / 2 - 0.4, 5003.0, 4001.0]]
    pos[4:, 0] = s / 2 + 2.4 + 0.2 * k / 63
    pos[4:, 1] = 4900.0 + 3.1 * k
    pos[4:, 2] = 4000.0 + 0.7 * (k % 5)
    u = np.random.default_rng(8).standard_normal((68, 3))
    u /= np.linalg.norm(u, axis=1)[:, None]
    ref = oracle.bh(pos, u, theta, 1, "f64", 1.0, 1.0, 1.0, 2.5, True)
    ctx = ff.ff_create(ff.ff_params_default(n=68, precision="f64", count_interactions=1))
    ff.ff_set_particles(ctx, pos, u)
    h, f = ff.ff_dipolar_field(ctx, ff.FF_ALGO_BH, theta, True)
    acc, pairs, opened = ff.ff_get_counts(ctx)
    assert np.array_equal(acc, ref["nacc"]) and np.array_equal(pairs, ref["npair"])
    assert np.array_equal(opened, ref["nopen"])
    assert rel_err(h, ref["h"]).max() <= 1e-10 and rel_err(f, ref["f"]).max() <= 1e-10


@pytest.mark.parametrize("leaf_max", [1, 6])
@pytest.mark.parametrize("n", [1, 31, 33, 3001, 120011])
def test_gradient_records_match_lists(ff, n, leaf_max):
    """The gradient from the shared walk's records and from the lists of the counting walk (a
    context that counts): the same sources in the same order, so the same bits; and the counts
    of the gradient's evaluation can be asked for after either."""
    pos, u = _gas(n, n + leaf_max)
    if n > 3000:
        pos[11:60] = pos[11]  # a leaf of several particles at any leaf_max
    res = []
    for count in (0, 1):
        ctx = ff.ff_create(ff.ff_params_default(n=n, leaf_max=leaf_max, count_interactions=count))
        ff.ff_set_particles(ctx, pos, u)
        e, gp, gu = ff.ff_energy_grad(ctx, ff.FF_ALGO_BH, 0.5, dtype=np.float32)
        e2, gp2, gu2 = ff.ff_energy_grad(ctx, ff.FF_ALGO_BH, 0.5, dtype=np.float32)
        assert e == e2 and np.array_equal(gp, gp2) and np.array_equal(gu, gu2)
        res.append((e, gp, gu, *ff.ff_get_counts(ctx), ff.ff_tree_info(ctx)["interactions"]))
        ff.ff_step(ctx, 2)  # steps after a gradient
        res[-1] += tuple(ff.ff_get_particles(ctx))
    for a, b in zip(*res):
        assert np.array_equal(a, b)


def test_counts_taken_after_a_gradient(ff):
    """Without interaction counting the counts of a gradient's evaluation are taken when first
    asked for: by either call, once, as one of the context's launches."""
    pos, u = _gas(3001, 21)
    res = []
    for first in (0, 1):
        ctx = ff.ff_create(ff.ff_params_default(n=3001))
        ff.ff_set_particles(ctx, pos, u)
        grad = ff.ff_energy_grad(ctx, ff.FF_ALGO_BH, 0.5, dtype=np.float32)
        ff.ff_profile(ctx, True)
        if first:
            counts = ff.ff_get_counts(ctx)
            n0 = ff.ff_profile_read(ctx)["launches"]
            info = ff.ff_tree_info(ctx)
            assert ff.ff_profile_read(ctx)["launches"] == n0
        else:
            info = ff.ff_tree_info(ctx)
            assert ff.ff_profile_read(ctx)["launches"] == 1
            counts = ff.ff_get_counts(ctx)
        assert info["interactions"] == int(counts[0].sum()) + int(counts[1].sum()) > 0
        again = ff.ff_energy_grad(ctx, ff.FF_ALGO_BH, 0.5, dtype=np.float32)
        assert again[0] == grad[0] and np.array_equal(again[1], grad[1])
        res.append(counts)
    for a, b in zip(*res):
        assert np.array_equal(a, b)


def test_gradient_records_outgrow_their_pool(ff):
    """At a small opening angle a task's records need more chunks than the pool's first
    allocation (6000 particles, nearly all of them a source of each task: 17,600 chunks against
    10,024): the walk is redone with room for what it took, and the result is that of a second
    call and of the lists."""
    pos, u = _gas(6000, 17)
    res = []
    for count in (0, 1):
        ctx = ff.ff_create(ff.ff_params_default(n=6000, count_interactions=count))
        ff.ff_set_particles(ctx, pos, u)
        for _ in range(2):
            res.append(ff.ff_energy_grad(ctx, ff.FF_ALGO_BH, 0.05, dtype=np.float32))
    for r in res[1:]:
        assert r[0] == res[0][0]
        assert np.array_equal(r[1], res[0][1]) and np.array_equal(r[2], res[0][2])
