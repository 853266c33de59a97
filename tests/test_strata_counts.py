"""Strata counts of systematic resampling: the count found from one rounded estimate and one
probe (FP32, up to 2^20 strata) or three probes equals #{j : u_j <= c}.

The CPU tests evaluate the same FP32 expressions with numpy and compare with a search over
every point; the GPU test compares the ancestors of a step, at the sizes where the rule
changes (2^20) and beyond, with the oracle's resampling of the CDF the step computed.
"""
import numpy as np
import pytest

F = np.float32


def _points(n, u0):
    inv_n = F(1.0) / F(n)
    return (np.arange(n).astype(F) + F(u0)) * inv_n


def _values(rng, n, u):
    """CDF values: random ones, the points themselves and their neighbours, and the ends."""
    pick = u[rng.integers(0, n, 4000)]
    c = np.concatenate([rng.random(8000).astype(F), pick, np.nextafter(pick, F(0)), np.nextafter(pick, F(2)),
                        np.array([0.0, 1.0, u[0], u[-1], np.nextafter(u[0], F(0)), 1e-30], F)])
    return np.minimum(c, F(1.0))


def _estimate(c, n, u0, fused):
    if fused:
        return (c.astype(np.float64) * n - np.float64(F(u0))).astype(F)   # the product is exact in FP64
    return c * F(n) - F(u0)


@pytest.mark.parametrize("fused", [False, True])
@pytest.mark.parametrize("n", [1, 2, 3, 1000, 4097, 65535, 300007, (1 << 20) - 1, 1 << 20])
def test_one_probe_counts_every_stratum(n, fused):
    rng = np.random.default_rng(n)
    for u0 in (2.0 ** -24, 0.5, 0.37152, 1.0 - 2.0 ** -24):
        u = _points(n, u0)
        c = _values(rng, n, u)
        m = np.clip(_estimate(c, n, u0, fused), F(0), F(n) - F(1)) + F(12582912.0)
        jf = m - F(12582912.0)
        got = jf.astype(np.int64) + ((jf + F(u0)) * (F(1.0) / F(n)) <= c)
        assert np.array_equal(got, np.searchsorted(u, c, side="right")), (n, u0)


@pytest.mark.parametrize("n", [5, (1 << 20) + 1, 3 * (1 << 20) + 7, 1 << 22, (1 << 22) + 12345])
def test_three_probes_decide_or_ask_for_the_general_count(n):
    rng = np.random.default_rng(n)
    for u0 in (2.0 ** -24, 0.613, 1.0 - 2.0 ** -24):
        u = _points(n, u0)
        c = _values(rng, n, u)
        inv_n = F(1.0) / F(n)
        j = np.clip(np.rint(_estimate(c, n, u0, True)).astype(np.int64), 0, n - 1)
        jf = j.astype(F)
        lo = (j == 0) | ((jf - F(1) + F(u0)) * inv_n <= c)
        mid = (jf + F(u0)) * inv_n <= c
        hi = (j < n - 1) & ((jf + F(1) + F(u0)) * inv_n <= c)
        ok = lo & ~hi
        want = np.searchsorted(u, c, side="right")
        assert np.array_equal((j + mid)[ok], want[ok]), (n, u0)
        assert ok.mean() > 0.99


@pytest.mark.gpu
@pytest.mark.parametrize("prec,n", [("f32", 1 << 20), ("f32", (1 << 20) + 1), ("f16", 3 * (1 << 20) + 7),
                                    ("f32", (1 << 23) + 3), ("f32", 1 << 24), ("ref64", 70001), ("f16", 1)])
def test_ancestors_equal_the_oracle_where_the_rule_changes(prec, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import oracle
    import paper_2308_00763_gb300 as pf
    from paper_2308_00763_gb300 import synth
    pf.lib(build_if_missing=True)
    v = synth.make_video(128, 96, 3, 4, noise=8.0, seed=9, v=(1.0, -1.0))
    f = pf.Filter(v.W, v.H, n, 4, prec, init=tuple(v.centres[0]), seed=6, sigma=(2.0, 2.0),
                  flags=pf.PF_FLAG_DEBUG_ARRAYS)
    f.run(torch.from_numpy(v.frames).cuda())
    anc = f.debug(0).astype(np.int64)
    c = f.debug(1).astype(np.float64)
    f.close()
    assert np.array_equal(anc, oracle.resample(c, oracle.resample_u0(6, v.T - 2), "f64" if prec == "ref64" else "f32"))
