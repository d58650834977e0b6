"""The single-precision all-pairs kernel (k_ap2) against the FP64 oracle.

Sizes at the edges of its parts: one to a few targets, blocks of 16 (below 65,536 targets) and
of 32, batches of 32 sources (16 pairs), the 256-source rows that a block's warps share out, and
a ragged end of each.  Bar: the repository's 1e-5 for single-precision fields and forces.
Coincident particles add nothing to each other.
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


@pytest.fixture(scope="module")
def ora():
    import oracle

    return oracle


def _system(n, seed):
    rng = np.random.default_rng(seed)
    m = max(2, int(np.ceil((3.1 * n) ** (1.0 / 3.0))))
    site = rng.permutation(m ** 3)[:n]
    q = np.stack([site // (m * m), (site // m) % m, site % m], axis=1)
    u = rng.standard_normal((n, 3))
    u /= np.linalg.norm(u, axis=1)[:, None]
    return ((q + rng.uniform(-0.16, 0.16, (n, 3))) * 1.5).astype(np.float32), u.astype(np.float32)


def _err(a, b):
    rms = np.sqrt((b * b).sum(1).mean())
    return (np.linalg.norm(a - b, axis=1) / np.maximum(np.linalg.norm(b, axis=1), 0.1 * rms)).max()


@pytest.mark.parametrize("n", [2, 15, 16, 17, 33, 255, 256, 257, 2049, 65535, 65536, 65569])
def test_matches_oracle(ff, ora, n):
    pos, u = _system(n, n)
    ctx = ff.ff_create(ff.ff_params_default(n=n, algo="ap"))
    ff.ff_set_particles(ctx, pos, u)
    h, f = ff.ff_dipolar_field(ctx, ff.FF_ALGO_AP, 0.0, True)
    only = None if n < 4000 else np.concatenate([np.arange(40), np.arange(n - 60, n)])
    rh, rf, _ = ora.allpairs(pos.astype(np.float64), u.astype(np.float64), 1.0, 1.0, 1.0, 2.5, True,
                             only=only)
    sel = slice(None) if only is None else only
    assert _err(h[sel], rh[sel]) <= 1e-5
    assert _err(f[sel], rf[sel]) <= 1e-5


def test_coincident_and_single(ff):
    one = ff.ff_create(ff.ff_params_default(n=1, algo="ap"))
    ff.ff_set_particles(one, np.ones((1, 3), np.float32), np.ones((1, 3), np.float32))
    h, f = ff.ff_dipolar_field(one, ff.FF_ALGO_AP, 0.0, True)
    assert not h.any() and not f.any()
    pos, u = _system(300, 4)
    pos[7:40] = pos[7]
    ctx = ff.ff_create(ff.ff_params_default(n=300, algo="ap", lj_eps=0.0))
    ff.ff_set_particles(ctx, pos, u)
    h, f = ff.ff_dipolar_field(ctx, ff.FF_ALGO_AP, 0.0, True)
    keep = np.r_[0:7, 40:300]
    for k in (7, 21, 39):  # a coincident particle feels the others alone
        sub = np.r_[k, keep]
        c = ff.ff_create(ff.ff_params_default(n=len(sub), algo="ap", lj_eps=0.0))
        ff.ff_set_particles(c, pos[sub], u[sub])
        hs, fs = ff.ff_dipolar_field(c, ff.FF_ALGO_AP, 0.0, True)
        np.testing.assert_allclose(h[k], hs[0], rtol=1e-5, atol=1e-5 * np.abs(hs).max())
        np.testing.assert_allclose(f[k], fs[0], rtol=1e-5, atol=1e-5 * np.abs(fs).max())


@pytest.mark.parametrize("n", [1, 40, 600, 65569])
@pytest.mark.parametrize("case", ["nan position", "infinite moment", "nan moment", "huge moment"])
def test_undefined_and_huge_inputs(ff, n, case):
    """What adds nothing adds nothing whatever its numbers are, as in double precision: a source
    at an undefined distance (a position that is not a number, for the others and for itself),
    and the target itself (its own moment infinite, undefined, or so large that its square
    overflows).  The defined values agree with double precision within the bar."""
    pos, u = _system(n, 5)
    bad = [0] if n == 1 else [7, n // 2, n - 1]
    if case == "nan position":
        pos[bad[0], 1] = np.nan
        pos[bad[-1]] = np.nan
    elif case == "infinite moment":
        u[bad[0]] = [0.0, np.inf, 0.0]
    elif case == "nan moment":
        u[bad[0], 2] = np.nan
    else:
        u[bad[0]] *= np.float32(1e25)
    out = []
    for prec, dt in (("f32", np.float32), ("f64", np.float64)):
        ctx = ff.ff_create(ff.ff_params_default(n=n, algo="ap", precision=prec, lj_eps=0.0))
        ff.ff_set_particles(ctx, pos.astype(dt), u.astype(dt))
        out.append(ff.ff_dipolar_field(ctx, ff.FF_ALGO_AP, 0.0, True, dtype=dt))
    (h, f), (h64, f64) = out
    for a, b in ((h, h64), (f, f64)):
        ok = np.isfinite(b)
        assert np.array_equal(np.isfinite(a), ok)
        rows = ok.all(axis=1)
        none = rows & ~b.any(axis=1)
        assert not a[none].any()
        rows &= ~none
        if rows.any():
            assert _err(a[rows].astype(np.float64), b[rows]) <= 1e-5
