"""Routes of the step that ordinary videos seldom take, against the oracle: every particle outside
any likelihood table (the direct route), tables built from row sums in bands, the FP64 draws
of a whole frame, the multinomial search at the edges of its levels, and Gumbel-max draws over
flat weights (no particle can be ruled out).
"""
import numpy as np
import pytest

import oracle
from paper_2308_00763_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pf():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2308_00763_gb300 as m
    m.lib(build_if_missing=True)
    return m


def _cuda(frames):
    import torch
    return torch.from_numpy(frames).cuda()


def _check_likelihoods(pf, f, prec, frame, r, flags=0):
    st = f.get_state()
    half = prec in ("f16", "bf16")
    x = st["x"] + (st["anchor_x"] if half else 0.0)
    y = st["y"] + (st["anchor_y"] if half else 0.0)
    if half:   # the same operations, each rounded once: bit for bit
        kind = "f16acc32" if prec == "f16" and flags & pf.PF_FLAG_ACCUM32 else prec
        assert np.array_equal(st["L"], oracle.likelihood_half(x, y, frame, r, kind))
    elif prec == "ref64":
        assert np.array_equal(st["L"], oracle.likelihood_all(x, y, frame, r))
    else:
        np.testing.assert_allclose(st["L"], oracle.likelihood_all(x, y, frame, r), rtol=2 ** -23, atol=1e-4)


@pytest.mark.parametrize("prec,accum32", [("ref64", 0), ("f32", 0), ("f16", 0), ("f16", 1), ("bf16", 0)])
@pytest.mark.parametrize("r", [0, 5, 40])
def test_direct_route_of_every_particle(pf, prec, accum32, r):
    """Draws of 40 px: no window fits a table, so every lane's two particles go to the frame
    (whole warps, partial warps at the tile's end and the straddling pairs)."""
    v = synth.make_video(200, 150, 3, 6, noise=8.0, seed=21)
    flags = pf.PF_FLAG_DEBUG_ARRAYS | (pf.PF_FLAG_ACCUM32 if accum32 else 0)
    f = pf.Filter(v.W, v.H, 1027, r, prec, init=tuple(v.centres[0]), seed=8, sigma=(40.0, 40.0), flags=flags)
    f.run(_cuda(v.frames))
    assert np.all(f.debug(2)[:, 2] == 0)
    _check_likelihoods(pf, f, prec, v.frames[-1], r, flags)
    f.close()


@pytest.mark.parametrize("prec,accum32", [("f16", 0), ("f16", 1), ("bf16", 0)])
@pytest.mark.parametrize("r", [1, 7, 14, 20])
def test_tables_by_row_sums_and_bands(pf, prec, accum32, r):
    v = synth.make_video(160, 140, 3, r, noise=8.0, seed=22, c0=(60.0, 60.0))
    flags = pf.PF_FLAG_DEBUG_ARRAYS | (pf.PF_FLAG_ACCUM32 if accum32 else 0)
    for resampler in ("systematic", "multinomial"):
        f = pf.Filter(v.W, v.H, 3000, r, prec, init=tuple(v.centres[0]), seed=8, flags=flags, resampler=resampler)
        f.run(_cuda(v.frames))
        assert np.all(f.debug(2)[:, 2] > 0)
        _check_likelihoods(pf, f, prec, v.frames[-1], r, flags)
        f.close()


def test_fp64_draws_of_a_frame(pf):
    """2^20 normal pairs around the origin.  Radii are below 5.77, within 1 ulp (9e-16) on either
    side; the step's sine and cosine are within 1.7e-16, the oracle's within 1.2e-16 of those of
    its angle, whose product 2 pi u is off by up to 7e-16: 5.77 x 9.9e-16 + 2 x 9e-16 < 8e-15."""
    v = synth.make_video(64, 64, 1, 3, noise=5.0, seed=23)
    n = 1 << 20
    f = pf.Filter(v.W, v.H, n, 3, "ref64", init=(0.0, 0.0), seed=24)
    f.run(_cuda(v.frames))
    st = f.get_state()
    f.close()
    nx, ny = oracle.normals(24, 0, n)
    assert np.abs(st["x"] - nx).max() <= 8e-15 and np.abs(st["y"] - ny).max() <= 8e-15


@pytest.mark.parametrize("prec,n", [("f32", n) for n in (7, 8, 9, 63, 64, 65, 511, 4097, (1 << 20) + 9)] +
                         [("ref64", 65), ("ref64", 70001), ("f16", 130), ("f16", 700001)])
def test_multinomial_search_at_the_edges_of_its_levels(pf, prec, n):
    v = synth.make_video(128, 128, 3, 5, noise=5.0, seed=25)
    f = pf.Filter(v.W, v.H, n, 5, prec, init=tuple(v.centres[0]), seed=26, flags=pf.PF_FLAG_DEBUG_ARRAYS,
                  resampler="multinomial")
    f.run(_cuda(v.frames))
    anc, c = f.debug(0).astype(np.int64), f.debug(1).astype(np.float64)
    f.close()
    want = oracle.resample_multinomial(c, oracle.stratified_offsets(26, v.T - 2, n), "f64" if prec == "ref64" else "f32")
    assert np.array_equal(anc, want)


@pytest.mark.parametrize("prec", ["ref64", "f32", "f16"])
def test_gumbel_over_flat_weights(pf, prec):
    """A frame of one level: every likelihood is the same, no particle can be ruled out."""
    frames = np.full((2, 64, 64), 100, np.uint8)
    n = 1500
    f = pf.Filter(64, 64, n, 3, prec, init=(32.0, 32.0), seed=27, flags=pf.PF_FLAG_DEBUG_ARRAYS, resampler="gumbel")
    f.step(_cuda(frames)[0])
    like = f.get_state()["L"].astype(np.float64)
    assert np.all(like == like[0])
    f.step(_cuda(frames)[1])
    anc = f.debug(0).astype(np.int64)
    f.close()
    want = oracle.resample_gumbel(like, 27, 0, 0, "f64" if prec == "ref64" else "f32")
    bad = np.nonzero(anc != want)[0]   # (near ties of the two sides' logarithms)
    assert bad.size <= 2
    for j in bad:
        g = oracle.gumbel_variates(27, 0, int(j), n)
        assert abs(g[want[j]] - g[anc[j]]) <= (1e-12 if prec == "ref64" else 1e-5) * max(1.0, abs(like[0]))


@pytest.mark.parametrize("n", [1, 2, 5, 33, 2047, 2049, 4101])
def test_gumbel_list_chunks(pf, n):
    """Flat weights list every quad, so n sets the list: a part of one quad, quads fewer than a
    pass takes, and the edges of the 2048 particles whose weights are staged at a time."""
    frames = np.full((2, 64, 64), 100, np.uint8)
    f = pf.Filter(64, 64, n, 3, "f32", init=(32.0, 32.0), seed=29, flags=pf.PF_FLAG_DEBUG_ARRAYS, resampler="gumbel")
    f.step(_cuda(frames)[0])
    like = f.get_state()["L"].astype(np.float64)
    f.step(_cuda(frames)[1])
    anc = f.debug(0).astype(np.int64)
    f.close()
    want = oracle.resample_gumbel(like, 29, 0, 0, "f32")
    bad = np.nonzero(anc != want)[0]   # (near ties of the two sides' logarithms)
    assert bad.size <= 2
    for j in bad:
        g = oracle.gumbel_variates(29, 0, int(j), n)
        assert abs(g[want[j]] - g[anc[j]]) <= 1e-5 * max(1.0, abs(like[0]))


@pytest.mark.parametrize("prec", ["ref64", "f32"])
@pytest.mark.parametrize("x,y", [(10.5, 9.5), (10.499999, 9.500001), (-0.5, -1.5), (0.0, -0.25), (63.5, 31.75),
                                 (1e-30, -1e-30), (70000.0, -5e5)])
def test_pixels_at_half_integers(pf, prec, x, y):
    """Particles without noise exactly on, and next to, the positions where a pixel ends."""
    v = synth.make_video(64, 48, 2, 3, noise=8.0, seed=30)
    f = pf.Filter(v.W, v.H, 37, 3, prec, init=(x, y), seed=31, sigma=(0.0, 0.0))
    f.run(_cuda(v.frames))
    _check_likelihoods(pf, f, prec, v.frames[-1], 3)
    f.close()


@pytest.mark.parametrize("n,tries", [(31, 0), (33, 0), (19456, 0), (19457, 0), (155649, 0), (5000, 63), (5000, 64),
                                     (5000, 65), (5000, 129), (200003, 9)])
def test_rejection_pools_and_lists(pf, n, tries):
    """Pools of less than a thread's share, at the sizes where a pool grows, and beyond the threads
    of a CTA; try limits around the 64 tries that a warp takes at once."""
    v = synth.make_video(128, 128, 3, 5, noise=5.0, seed=32)
    f = pf.Filter(v.W, v.H, n, 5, "f32", init=tuple(v.centres[0]), seed=33, flags=pf.PF_FLAG_DEBUG_ARRAYS,
                  resampler="rejection", resampler_steps=tries)
    fr = _cuda(v.frames)
    f.run(fr[:2])
    st = f.get_state()
    f.step(fr[2])
    anc = f.debug(0).astype(np.int64)
    f.close()
    L, M, t = st["L"].astype(np.float64), float(st["max_l"]), int(st["t"]) - 1
    tries = tries or 4096
    bad = np.nonzero(anc != oracle.resample_rejection(L, M, 33, t, 0, "f32", tries))[0]
    assert bad.size <= max(1, n // 1000)   # (tests within rounding of their threshold)
    for j in bad:
        assert min(oracle.rejection_trace(L, M, 33, t, int(j), 0, tries)[1]) <= 1e-4


def test_fp64_draws_are_accurate_next_to_the_axes(pf):
    """Every draw of a frame around the origin relative to its own size, against extended
    precision from the generator's words.  In units of 2^-52: the radius is within 0.852, the sine
    or cosine within 1.093, and their product's rounding adds 0.5, so 2.45; second-order terms
    and the reference (64 bits or more) stay below 0.05.  (Drift 0 and sigma 1 are exact.)"""
    ld = np.longdouble
    v = synth.make_video(64, 64, 1, 3, noise=5.0, seed=41)
    n = 1 << 20
    f = pf.Filter(64, 64, n, 3, "ref64", init=(0.0, 0.0), seed=42)
    f.run(_cuda(v.frames))
    st = f.get_state()
    f.close()
    ctr = np.zeros((n // 2, 4), np.uint32)
    ctr[:, 0] = np.arange(n // 2)
    w = oracle.philox(ctr, 42).reshape(n, 2)
    m = 2 * (w >> 9).astype(np.int64) + 1                    # u = m / 2^24
    rad = np.sqrt(-2 * np.log(m[:, 0].astype(ld) / (1 << 24)))
    quad, rem = m[:, 1] >> 22, m[:, 1] & 0x3fffff
    far = rem > 1 << 21                                      # nearer to the quarter's end
    pi = ld("3.14159265358979323846264338327950288")
    a = pi * np.where(far, (1 << 22) - rem, rem).astype(ld) / (1 << 23)
    swap = far != (quad % 2 == 1)
    c, s = np.where(swap, np.sin(a), np.cos(a)), np.where(swap, np.cos(a), np.sin(a))
    want_x = np.where((quad == 1) | (quad == 2), -c, c) * rad
    want_y = np.where(quad >= 2, -s, s) * rad
    for got, want in ((st["x"], want_x), (st["y"], want_y)):
        assert np.abs((got - want) / want).max() <= 2.5 * 2.0 ** -52


@pytest.mark.parametrize("prec,accum32", [("ref64", 0), ("f32", 0), ("f16", 0), ("f16", 1), ("bf16", 0)])
@pytest.mark.parametrize("n,r,sigma", [(40001, 0, (5.0, 2.0)), (40001, 12, (5.0, 2.0)), (70, 5, (5.0, 2.0)),
                                       (5001, 3, (40.0, 30.0)), (7, 5, (40.0, 40.0))])
def test_direct_route_of_few_and_of_all(pf, prec, accum32, n, r, sigma):
    """Production trackers (no debug arrays): a few draws beyond a window of 3.5 sigma, which the lanes
    of a warp score together, and noise that no window fits, where each lane scores its own."""
    v = synth.make_video(200, 150, 3, 6, noise=8.0, seed=43)
    flags = pf.PF_FLAG_ACCUM32 if accum32 else 0
    f = pf.Filter(v.W, v.H, n, r, prec, init=tuple(v.centres[0]), seed=44, sigma=sigma, flags=flags)
    f.run(_cuda(v.frames))
    _check_likelihoods(pf, f, prec, v.frames[-1], r, flags)
    f.close()


@pytest.mark.parametrize("prec,accum32", [("f16", 0), ("f16", 1), ("bf16", 0)])
@pytest.mark.parametrize("r", [5, 12, 14])
@pytest.mark.parametrize("low", [0.0, -1.5, -6.0])
def test_ancestors_of_tiles_with_row_sum_tables(pf, prec, accum32, r, low):
    """The row sums of a tile's table lie in the memory of its strata counts and ancestor map: the
    ancestors behind them are those of the CDF, in the first tile and in later ones, with the map's
    first part in use, nearly all of it (low = -1.5: 7000 offspring of the first tile) and the counts
    in its place (low = -6: more offspring than it holds)."""
    v = synth.make_video(160, 140, 2, r, noise=8.0, seed=45, c0=(60.0, 60.0))
    n = 9001
    flags = pf.PF_FLAG_DEBUG_ARRAYS | (pf.PF_FLAG_ACCUM32 if accum32 else 0)
    f = pf.Filter(v.W, v.H, n, r, prec, init=tuple(v.centres[0]), seed=46, flags=flags)
    fr = _cuda(v.frames)
    f.step(fr[0])
    st = f.get_state()
    st["L"] = np.where(np.arange(n) < 4096, 0.0, low)
    st["max_l"], st["sum_e"] = 0.0, float(np.exp(st["L"]).sum())
    f.set_state(st)
    f.step(fr[1])
    anc, c = f.debug(0).astype(np.int64), f.debug(1).astype(np.float64)
    assert np.all(f.debug(2)[:, 2] > 0)
    _check_likelihoods(pf, f, prec, v.frames[1], r, flags)
    f.close()
    assert np.array_equal(anc, oracle.resample(c, oracle.resample_u0(46, 0), "f32"))


@pytest.mark.parametrize("prec,n", [("f32", 31), ("f16", 5003), ("bf16", 150001), ("ref64", 2047), ("f16", 200003)])
def test_rejection_over_flat_weights(pf, prec, n):
    """Equal weights accept the first try, which is the offspring's own index."""
    frames = _cuda(np.full((2, 64, 64), 100, np.uint8))
    f = pf.Filter(64, 64, n, 3, prec, init=(32.0, 32.0), seed=47, flags=pf.PF_FLAG_DEBUG_ARRAYS, resampler="rejection")
    f.step(frames[0])
    f.step(frames[1])
    anc = f.debug(0)
    f.close()
    assert np.array_equal(anc, np.arange(n))


@pytest.mark.parametrize("prec,accum32", [("f16", 0), ("f16", 1), ("bf16", 0)])
@pytest.mark.parametrize("r", [5, 10, 14, 16])
@pytest.mark.parametrize("resampler", ["systematic", "multinomial", "metropolis", "rejection"])
def test_production_tables_by_row_sums(pf, prec, accum32, r, resampler):
    """Trackers without debug arrays: the pull kernel's row sums lie over the ancestor map (debug arrays
    keep it in use, and the sums away), in one band up to radius 10 in F16 and in several beyond; the
    step kernel's pairs take their fast copy.  A second tracker with debug arrays has a table in
    every tile, and the same particles."""
    v = synth.make_video(160, 140, 3, r, noise=8.0, seed=48, c0=(60.0, 60.0))
    flags = pf.PF_FLAG_ACCUM32 if accum32 else 0
    states = []
    for debug in (0, pf.PF_FLAG_DEBUG_ARRAYS):
        f = pf.Filter(v.W, v.H, 3001, r, prec, init=tuple(v.centres[0]), seed=49, flags=flags | debug, resampler=resampler)
        f.run(_cuda(v.frames))
        _check_likelihoods(pf, f, prec, v.frames[-1], r, flags)
        states.append(f.get_state())
        if debug:
            assert np.all(f.debug(2)[:, 2] > 0)
        f.close()
    for k in ("x", "y", "L", "est_x", "est_y", "sum_e"):
        assert np.array_equal(states[0][k], states[1][k])


@pytest.mark.parametrize("prec", ["ref64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("resampler", ["multinomial", "metropolis"])
@pytest.mark.parametrize("n,sigma", [(40001, (5.0, 2.0)), (3001, (40.0, 40.0))])
def test_direct_route_of_the_pull_kernel(pf, prec, resampler, n, sigma):
    v = synth.make_video(200, 150, 3, 6, noise=8.0, seed=50)
    f = pf.Filter(v.W, v.H, n, 5, prec, init=tuple(v.centres[0]), seed=51, sigma=sigma, resampler=resampler)
    f.run(_cuda(v.frames))
    _check_likelihoods(pf, f, prec, v.frames[-1], 5)
    f.close()
