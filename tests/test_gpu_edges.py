"""Edges of the GPU kernels' runs, tiles and launches against the FP64 oracles: column
heights of every remainder in the sampler, prefilter rows at any byte and narrow images,
the seed search staged and not, propagation around obstacles (more waves than the
distance to the corners, fronts larger than their launch), strain tiles of 32 x 32 points
and displacements that are no FP32 numbers, and FFT windows of every length.

Tolerances: those of parity_util for correlations; FP32 coefficients within 2e-6 of the
largest (two recursions of about 16 significant terms at 6e-8 each); seeds and waves exact;
strain within 1e-6 (as in test_gpu_strain); window peaks within 2e-5 (test_gpu_fft)."""
import numpy as np
import pytest

import oracle
import synth
from oracle import dic_oracle as O
from oracle import fft_oracle as F
from oracle import strain_oracle as SO

from parity_util import GPU_PARAMS, ORACLE_PARAMS, compare

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def pkg():
    import paper_2601_12941_gb300 as P
    from paper_2601_12941_gb300 import build

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    build.build()
    P.load()
    return P


def _speckle(W, H, fld=synth.IDENTITY, dtype="u8", gray=250.0, tag=1):
    sp = synth.Speckle(seed=77, density=0.03, sigma=(1.5, 3.0), cell=16)
    return synth.render(synth.ImageSpec(sp, field=fld, gray_max=gray, noise=0.01 * gray, noise_tag=tag), W, H, dtype)


# band heights: 9 -> 2, 13 -> 4, 17 -> 6, 19 -> 7, 23 -> 12, 25 -> 13, 35 -> 12, 45 -> 23 rows; the
# strains move floor crossings through the runs
@pytest.mark.parametrize("shape,S", [("rigid", 9), ("rigid", 13), ("rigid", 45), ("affine", 17), ("affine", 19),
                                     ("affine", 23), ("affine", 25), ("affine", 35), ("affine", 45),
                                     ("quadratic", 23), ("quadratic", 25), ("quadratic", 35), ("quadratic", 45)])
def test_column_heights_of_every_remainder(pkg, shape, S):
    W, H = 140, 128
    e = 0.0 if shape == "rigid" else 1.0
    fld = synth.affine_field(W, H, u0=0.97, v0=-1.03, exx=e * 8e-3, exy=e * 3e-3, eyx=-e * 2e-3, eyy=-e * 6e-3)
    ref, dfm = _speckle(W, H), _speckle(W, H, fld, tag=2)
    seed = (W // 2, H // 2)
    ora = oracle.correlate(ref, dfm, None, S, 16, shape, [seed], dict(ORACLE_PARAMS, search_radius=4))
    c = pkg.Correlation(torch.from_numpy(ref).cuda(), torch.from_numpy(dfm).cuda(), None, S, 16, shape,
                        precision="mixed", search_radius=4, **GPU_PARAMS["mixed"])
    c.run([seed])
    stats = compare(c.results(), ora, W, H, S)
    assert stats["accepted"] > 10
    c.close()


@pytest.mark.parametrize("dtype", ["u8", "u16", "f32"])
@pytest.mark.parametrize("W,H,offset", [(33, 40, 0), (150, 31, 1), (191, 64, 3), (193, 70, 2), (331, 300, 1), (257, 33, 0)])
def test_prefilter_rows_at_any_byte_and_narrow_images(pkg, W, H, offset, dtype):
    from paper_2601_12941_gb300 import binding as B

    img = _speckle(W, H, dtype=dtype, gray=250.0 if dtype == "u8" else 4000.0)
    host = img.view(np.int16) if dtype == "u16" else img
    wide = np.zeros((H, W + offset + 2), host.dtype)       # a view that starts `offset` elements into its rows
    wide[:, offset:offset + W] = host
    dev = torch.from_numpy(wide).cuda()[:, offset:offset + W]
    c = pkg.Correlation(dev, dev, None, 9, 5, "rigid", precision="mixed")
    c.run([(W // 2, H // 2)])
    ptr, ld, _ = pkg.dic_get_coefficients(c.h, 0)
    got = torch.as_tensor(B._DeviceArray(ptr, (H, ld), "<f4"), device="cuda")[:, :W].double().cpu().numpy()
    want = O.bspline_coefficients(img.astype(np.float64))
    assert np.abs(got - want).max() < 2e-6 * np.abs(want).max()
    c.close()


# widths whose last whole run ends up to three bytes before the row does: its last word is the buffer's last
@pytest.mark.parametrize("dtype", ["u8", "u16", "f32"])
@pytest.mark.parametrize("W,H,offset", [(240, 200, 1), (241, 200, 3), (242, 193, 2), (208, 192, 3)])
def test_prefilter_of_the_last_row(pkg, W, H, offset, dtype):
    test_prefilter_rows_at_any_byte_and_narrow_images(pkg, W, H, offset, dtype)


# radius 20 at subset 61 fits the staged rows for integers, not for FP64; 40 at 61 for neither
@pytest.mark.parametrize("dtype", ["u8", "f32"])
@pytest.mark.parametrize("S,R", [(3, 2), (21, 8), (33, 16), (61, 20), (61, 40)])
def test_seed_search_finds_integer_shifts(pkg, S, R, dtype):
    W = H = 2 * (S + 2 * R) + 30
    du, dv = R - 1, -(R // 2)
    big = _speckle(W + 2 * R, H + 2 * R, dtype=dtype)
    ref = np.ascontiguousarray(big[R:R + H, R:R + W])
    dfm = np.ascontiguousarray(big[R - dv:R - dv + H, R - du:R - du + W])
    c = pkg.Correlation(ref, dfm, None, S, 7, "rigid", search_radius=R)
    c.run([(W // 2, H // 2)])
    r = c.results()
    q = int(np.flatnonzero(r["wave"] == 0)[0])
    assert r["status"][q] == 0 and abs(r["u"][q] - du) < 1e-3 and abs(r["v"][q] - dv) < 1e-3
    c.close()


# the lanes per offset: one (subsets up to 7), two (up to 15), eight (up to 49) where there are many
# offsets, eight or 32 where there are few; the last radius whose rows are staged at subset 61
@pytest.mark.parametrize("dtype", ["u8", "f32"])
@pytest.mark.parametrize("S,R", [(7, 22), (7, 23), (9, 40), (15, 40), (15, 22), (17, 23), (49, 24), (51, 23), (61, 39)])
def test_seed_search_by_lanes_per_offset(pkg, S, R, dtype):
    test_seed_search_finds_integer_shifts(pkg, S, R, dtype)


@pytest.mark.parametrize("S,R", [(7, 24), (15, 24), (21, 24), (61, 24)])
def test_seed_search_beside_the_border(pkg, S, R):
    """Two seeds beside opposite corners: most offsets of each leave the image."""
    W = H = 2 * S + 70
    du, dv = 5, -4
    big = _speckle(W + 40, H + 40)
    ref = np.ascontiguousarray(big[20:20 + H, 20:20 + W])
    dfm = np.ascontiguousarray(big[20 - dv:20 - dv + H, 20 - du:20 - du + W])
    c = pkg.Correlation(ref, dfm, None, S, 7, "rigid", search_radius=R)
    c.run([(0, H - 1), (S // 2, 2 * S)])
    r = c.results()
    at = np.flatnonzero(r["wave"] == 0)
    assert len(at) == 2 and (r["status"][at] == 0).all()
    assert np.abs(r["u"][at] - du).max() < 1e-3 and np.abs(r["v"][at] - dv).max() < 1e-3
    c.close()


def test_waves_around_obstacles_and_from_many_seeds(pkg):
    """A serpentine region: several times the waves that the grid's corners suggest. Then
    one seed per grid point of a line: the first front is a whole row."""
    W, H, S, step = 300, 200, 9, 6
    roi = np.ones((H, W), np.uint8)
    for k, y in enumerate(range(30, H, 30)):
        roi[y:y + 4, (0 if k % 2 else 30):(W - 30 if k % 2 else W)] = 0
    img = _speckle(W, H)
    c = pkg.Correlation(img, img, roi, S, step, "affine")
    for seeds in ([(10, 10)], [(x, 100) for x in range(4, 290, step)]):
        c.run(seeds)
        r = c.results()
        nx, ny = r["nx"], r["ny"]
        ok = r["status"].reshape(ny, nx) == 0
        dist = np.full((ny, nx), -1)
        front = [divmod(int(q), nx) for q in np.flatnonzero(r["wave"] == 0)]
        for j, i in front:
            dist[j, i] = 0
        k = 0
        while front:
            k += 1
            new = []
            for j, i in front:
                for a, b in ((j, i - 1), (j, i + 1), (j - 1, i), (j + 1, i)):
                    if 0 <= a < ny and 0 <= b < nx and ok[a, b] and dist[a, b] < 0:
                        dist[a, b] = k
                        new.append((a, b))
            front = new
        assert np.array_equal(dist[ok], r["wave"].reshape(ny, nx)[ok])
        assert ok.sum() > 0.5 * nx * ny and (r["n_waves"] > nx + ny if len(seeds) == 1 else True)
    c.close()


@pytest.mark.parametrize("n", [1, 2, 3])
def test_next_frame_on_the_smallest_grids(pkg, n):
    """One to three points: fewer waves allowed than a frame launches ahead."""
    W, H = 26 + 40 * (n - 1), 50
    big = _speckle(W + 20, H + 20)
    ref = np.ascontiguousarray(big[10:10 + H, 10:10 + W])
    dfm = np.ascontiguousarray(big[8:8 + H, 8:8 + W])      # content moved by (2, 2): inside the bounds
    c = pkg.Correlation(ref, dfm, None, 21, 40, "affine")
    c.run([(10, 10)])
    for _ in range(2):
        c.set_deformed(dfm)
        c.run_next()
    r = c.results()
    assert r["n_points"] == n and (r["status"] == 0).all() and (r["wave"] == 0).all()
    assert np.abs(r["u"] - 2.0).max() < 1e-3 and np.abs(r["v"] - 2.0).max() < 1e-3
    c.close()


# the fields and the tolerance of test_gpu_strain, on tiles of every remainder, with values
# that are FP32 numbers and values that are not; windows above 15 on full windows only
@pytest.mark.parametrize("fp32_values", [True, False])
@pytest.mark.parametrize("nx,ny,window", [(31, 33, 3), (32, 32, 5), (33, 64, 9), (65, 40, 15), (63, 97, 9), (70, 67, 21),
                                          (96, 80, 31)])
def test_strain_tiles_and_displacement_types(pkg, nx, ny, window, fp32_values):
    from test_gpu_strain import KEYS, TOL, _field, _gpu

    u, v, st = _field(nx, ny, 5, 1.0, seed=window, hole_frac=0.04 if window <= 15 else 0.0)
    if fp32_values:
        u, v = u.astype(np.float32).astype(np.float64), v.astype(np.float32).astype(np.float64)
    g = _gpu(pkg, u, v, st, nx, ny, 5, window, SO.BIQUADRATIC, SO.HENCKY)
    o = SO.strain_field(u, v, st, nx, ny, 5, window, SO.BIQUADRATIC, SO.HENCKY)
    ok = o["valid"]
    assert np.array_equal(g["valid"].astype(bool), ok)
    h = (window - 1) // 2
    bad = np.pad((st.reshape(ny, nx) != 0).astype(int), h, constant_values=1)
    full = np.array([[bad[j:j + window, i:i + window].sum() == 0 for i in range(nx)] for j in range(ny)]).ravel()
    at = ok & (full if window > 15 else True)
    assert at.any()
    for k in KEYS:
        assert np.isnan(g[k][~ok]).all()
        assert np.abs(g[k][at].astype(np.float64) - o[k][at]).max() <= TOL, k


# grids large enough for two and four points per thread (the ones above take one): crops at the first
# and the last tiles and across a tile's corner against the oracle. Above window 15 the bilinear
# basis, whose general fits keep the tolerance: with slopes up to 0.04 px a point, sum |i u| / sum i^2 is
# at most 0.041, so 961 FP32 additions leave a slope within 961 x 6e-8 x 0.041 / 5 = 5e-7
@pytest.mark.parametrize("nx,ny,window", [(560, 520, 3), (400, 300, 5), (400, 300, 9), (701, 603, 9), (401, 299, 15),
                                          (2201, 2003, 15), (1101, 1003, 31)])
def test_strain_grids_of_several_points_per_thread(pkg, nx, ny, window):
    from test_gpu_strain import KEYS, TOL, _field, _gpu

    basis, h = SO.BIQUADRATIC if window <= 15 else SO.BILINEAR, window // 2
    u, v, st = _field(nx, ny, 5, 500.0 / max(nx, ny) / 5, seed=window, hole_frac=0.01)
    g = _gpu(pkg, u, v, st, nx, ny, 5, window, basis, SO.GREEN_LAGRANGE)
    u, v, st = (a.reshape(ny, nx) for a in (u, v, st))
    for i0, j0 in ((0, 0), (nx - 24, ny - 18), (320 - 10, 256 - 9)):
        i1, j1 = i0 + 24, j0 + 18
        ya, yb, xa, xb = max(j0 - h, 0), min(j1 + h, ny), max(i0 - h, 0), min(i1 + h, nx)
        o = SO.strain_field(u[ya:yb, xa:xb].ravel(), v[ya:yb, xa:xb].ravel(), st[ya:yb, xa:xb].ravel(), xb - xa, yb - ya, 5,
                            window, basis, SO.GREEN_LAGRANGE)
        cut = lambda a: a.reshape(yb - ya, xb - xa)[j0 - ya:j1 - ya, i0 - xa:i1 - xa]
        ok = cut(o["valid"])
        assert ok.any() and np.array_equal(g["valid"].reshape(ny, nx)[j0:j1, i0:i1].astype(bool), ok)
        for k in KEYS:
            got = g[k].reshape(ny, nx)[j0:j1, i0:i1]
            assert np.isnan(got[~ok]).all()
            assert np.abs(got[ok].astype(np.float64) - cut(o[k])[ok]).max() <= TOL, k


@pytest.mark.parametrize("window", range(17, 32, 2))
def test_general_fits_of_the_large_windows(pkg, window):
    from test_gpu_strain import _compare, _field, _gpu

    nx, ny = 45, 41
    u, v, st = _field(nx, ny, 5, 1.0, seed=window, hole_frac=0.04)
    g = _gpu(pkg, u, v, st, nx, ny, 5, window, SO.BILINEAR, SO.HENCKY)
    assert _compare(g, SO.strain_field(u, v, st, nx, ny, 5, window, SO.BILINEAR, SO.HENCKY)) > 0.8 * nx * ny


# an accepted point whose displacement is not finite (or no FP32 number), inside a tile and as a
# tile's first point. u takes part in the test of a fit: the windows that hold the point have no strain,
# a NaN counts as a missing point. v does not: the slopes of u stand, those of v are not finite
@pytest.mark.parametrize("at", [(12, 14), (32, 32)])
@pytest.mark.parametrize("value", [np.inf, -np.inf, 1e300, np.nan])
@pytest.mark.parametrize("comp", ["u", "v"])
@pytest.mark.parametrize("window,basis", [(5, SO.BILINEAR), (9, SO.BIQUADRATIC)])
def test_strain_of_an_accepted_point_that_is_not_finite(pkg, window, basis, comp, value, at):
    from test_gpu_strain import KEYS, TOL, _field, _gpu

    nx, ny, (i, j), h = 100, 70, at, window // 2
    u, v, st = _field(nx, ny, 5, 1.0, seed=7, hole_frac=0.0)   # its hole lies outside the windows that hold the point
    q = j * nx + i
    so = st.copy()
    if comp == "u" and np.isnan(value):
        so[q] = 5
    o = SO.strain_field(u, v, so, nx, ny, 5, window, basis, SO.GREEN_LAGRANGE)
    (u if comp == "u" else v)[q] = value
    g = _gpu(pkg, u, v, st, nx, ny, 5, window, basis, SO.GREEN_LAGRANGE)
    jj, ii = np.divmod(np.arange(nx * ny), nx)
    holds = (np.abs(ii - i) <= h) & (np.abs(jj - j) <= h)
    if np.isnan(value) and comp == "u":
        holds[:] = False
    ok = o["valid"] & ~holds if comp == "u" else o["valid"]
    assert np.array_equal(g["valid"].astype(bool), ok)
    for k in KEYS:
        assert np.isnan(g[k][~ok]).all(), k
        at_k = ok if comp == "v" and k in ("dudx", "dudy") else ok & ~holds
        assert np.abs(g[k][at_k].astype(np.float64) - o[k][at_k]).max() <= TOL, k
    if comp == "v":
        assert not np.isfinite(g["dvdx"][holds]).any() and not np.isfinite(g["dvdy"][holds]).any()


@pytest.mark.parametrize("window", [3, 9, 15])
def test_strain_beside_an_accepted_outlier(pkg, window):
    """An accepted point 1e4 px off, the first point of the halo of the tile that starts at (32, 32):
    the windows of that tile that do not hold it keep the tolerance (offsets from it would be
    rounded to 1e-3 px)."""
    from test_gpu_strain import KEYS, TOL, _field, _gpu

    nx, ny, h = 100, 70, window // 2
    i = j = 32 - h
    u, v, st = _field(nx, ny, 5, 1.0, seed=7, hole_frac=0.0)
    o = SO.strain_field(u, v, st, nx, ny, 5, window, SO.BIQUADRATIC, SO.GREEN_LAGRANGE)
    u[j * nx + i] = v[j * nx + i] = 1e4
    g = _gpu(pkg, u, v, st, nx, ny, 5, window, SO.BIQUADRATIC, SO.GREEN_LAGRANGE)
    jj, ii = np.divmod(np.arange(nx * ny), nx)
    ok = o["valid"] & ((np.abs(ii - i) > h) | (np.abs(jj - j) > h))
    assert np.array_equal(g["valid"].astype(bool), o["valid"])
    for k in KEYS:
        assert np.abs(g[k][ok].astype(np.float64) - o[k][ok]).max() <= TOL, k


@pytest.mark.parametrize("L", [64, 128, 256, 512, 1024, 2048, 4096])
def test_windows_of_every_length(pkg, L):
    from paper_2601_12941_gb300 import binding as B

    N = L + 40
    ref = _speckle(N, N)
    dfm = _speckle(N, N, synth.affine_field(N, N, u0=5.0, v0=-3.0), tag=2)
    c = pkg.Correlation(ref, dfm, None, 21, 64, "affine")
    origins = [(0, 0, 0, 0), (17, 23, 12, 40 - 3), (40, 40, 39, 40)]
    org = torch.tensor(origins, dtype=torch.int32, device="cuda")
    u, v, pk = (torch.empty(3, dtype=torch.float32, device="cuda") for _ in range(3))
    B.dic_fftcc_windows(c.h, L, org, L <= 64, u, v, pk)
    torch.cuda.synchronize()
    for k, (x0, y0, gx, gy) in enumerate(origins):
        R = F.fftcc(ref[y0:y0 + L, x0:x0 + L], dfm[gy:gy + L, gx:gx + L])
        dx, dy, peak = F.peak(R, L <= 64)
        assert abs(float(u[k]) - (gx - x0 + dx)) < 1e-4 and abs(float(v[k]) - (gy - y0 + dy)) < 1e-4
        assert abs(float(pk[k]) - peak) < 2e-5
    c.close()
