"""Timed workloads of the correlation library, through its public entry points.

Image pairs are synthetic speckle: a seeded random lattice interpolated by cubic
B-splines at the exactly mapped position of every pixel, squashed to dark and bright
blobs, with 1 % camera noise, quantised to the gray type. Sizes, gray types, subset
settings and options are those of the repository's workloads (synth/workloads.py,
bench.py) and of the ranges its serving stream declares.

A case is a dict; `kind` selects the entry point:
  pair      both images replaced, then one correlation from seeds, results on the device
  sequence  the next frame against the resident reference, started from the last one
  update    two frames with a reference update between them, total warps
  job       one serving job: re-grid, host image in, correlation, results on the host
  static    the allocation-free correlation into caller-owned arrays
  fft       the multi-window FFT initialiser over the grid
  strain    strain of a displacement field

`exact` computes the same outputs with plain torch in FP64, sharing no code with the library.
"""
import math

import numpy as np
import torch

import paper_2601_12941_gb300 as pkg
from paper_2601_12941_gb300 import binding

GRAY_MAX = {"u8": 255.0, "u16": 65535.0, "bf16": 255.0, "f32": 4095.0, "f64": 4095.0}
DEV = "cuda"


# ---------------------------------------------------------------- the cases
def _pair(name, w, h, dtype, S, step, shape, **kw):
    c = dict(name=name, kind="pair", w=w, h=h, dtype=dtype, S=S, step=step, shape=shape, precision="mixed",
             optimizer="gn", cost="znssd", interp="bspline3", roi=False, seeds=1, radius=8, pitch=3.5)
    c.update(kw)
    return c


def listed():
    return [
        # a live camera crop in a loop that may not allocate: the smallest call, all latency
        _pair("static_384x288_u8", 384, 288, "u8", 21, 8, "affine", kind="static"),
        # the 256^2 quick-look pair (2,304 points), mixed precision: short waves, launches and latency
        _pair("pair_256_u8", 256, 256, "u8", 21, 5, "affine"),
        # the same pair in plain FP64, the form used for reference results
        _pair("pair_256_u8_fp64", 256, 256, "u8", 21, 5, "affine", precision="fp64"),
        # an optical 2048^2 pair, dense quadratic grid of 1.02 M points
        _pair("pair_2048_u16_quadratic", 2048, 2048, "u16", 31, 2, "quadratic", radius=4),
        # odd sizes with unaligned rows, a region of interest with a hole, Levenberg-Marquardt
        _pair("pair_1531x1103_u8_lm_roi", 1531, 1103, "u8", 25, 4, "affine", optimizer="lm", roi=True),
        # the 1.07 Gpx SEM-like pair (10.7 M points), several seeds: the headline workload
        _pair("pair_32768_u8", 32768, 32768, "u8", 41, 10, "affine", seeds=16, radius=32, pitch=2.0),
        # video: frames of a 4096 x 3000 camera against one reference, small and large subsets
        _pair("sequence_4096x3000_u16_s21", 4096, 3000, "u16", 21, 10, "affine", kind="sequence"),
        _pair("sequence_4096x3000_u16_s41_quadratic", 4096, 3000, "u16", 41, 10, "quadratic", kind="sequence"),
        # incremental reference updating on a medium camera
        _pair("update_1600x1200_bf16", 1600, 1200, "bf16", 31, 7, "affine", kind="update"),
        # one job of the serving stream: resident reference, host image in, host results out
        _pair("job_2896_u16_s45", 2896, 2896, "u16", 45, 4, "affine", kind="job"),
        # the multi-window FFT initialiser with the SEM study's window settings
        dict(name="fft_8192_u8", kind="fft", w=8192, h=8192, dtype="u8", S=31, step=15, displacement=1000,
             subpixel=True, pitch=2.0),
        # strain of a gigapixel pair's field (10.7 M points), a crack-like band and stray points rejected
        dict(name="strain_3273", kind="strain", nx=3273, ny=3273, step=10, window=9, basis="biquadratic",
             measure="green_lagrange"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pair", "pair", "pair", "sequence", "update", "job", "static", "fft", "strain"])
    if kind == "strain":
        return dict(kind="strain", nx=_log_int(rng, 40, 3273), ny=_log_int(rng, 40, 3273), step=rng.randint(1, 15),
                    window=2 * rng.randint(1, 10) + 1, basis=rng.choice(["bilinear", "biquadratic"]),
                    measure=rng.choice(["green_lagrange", "hencky", "euler_almansi", "biot_right", "biot_left"]))
    if kind == "fft":
        side = _log_int(rng, 512, 8192)
        return dict(kind="fft", w=side, h=max(256, int(side * rng.uniform(0.6, 1.0))),
                    dtype=rng.choice(["u8", "u16", "bf16", "f32"]), S=2 * rng.randint(7, 20) + 1,
                    step=rng.randint(8, 20), displacement=min(side // 8, _log_int(rng, 16, 1000)),
                    subpixel=rng.random() < 0.5, pitch=rng.choice([2.0, 3.5]))
    if kind == "static":
        c = _pair("", rng.randint(160, 640), rng.randint(160, 512), rng.choice(["u8", "u16", "bf16"]),
                  2 * rng.randint(5, 20) + 1, rng.randint(4, 12), rng.choice(["rigid", "affine", "quadratic"]),
                  kind="static")
    else:
        side = _log_int(rng, 256, 4096)
        S = 2 * rng.randint(7, 30) + 1
        step = rng.randint(1, 12)
        while (side / step) ** 2 > 1.1e6:
            step += 1
        c = _pair("", side, max(192, int(side * rng.uniform(0.6, 1.0))), rng.choice(["u8", "u8", "u16", "bf16", "f32"]),
                  S, step, rng.choice(["affine", "affine", "quadratic", "rigid"]), kind=kind)
    if kind in ("pair", "job"):
        c["roi"] = rng.random() < 0.3
        option = rng.choice(["", "", "", "lm", "nssd", "keys", "fp64", "solve64"])
        if option == "lm":
            c["optimizer"] = "lm"
        elif option == "nssd":
            c["cost"] = rng.choice(["nssd", "ssd"])
        elif option == "keys":
            c["interp"] = "bicubic"
        elif option == "fp64":
            c["precision"] = "fp64"
            c["step"] = max(c["step"], c["w"] // 200 + 1)    # FP64 runs at a small fraction of the FP32 rate
        elif option == "solve64":
            c["precision"] = "mixed_fp64_solve"
    if kind == "update" and c["shape"] == "quadratic":
        c["shape"] = "affine"                                 # reference updating is rigid or affine
    if kind == "job" and c["dtype"] == "bf16":
        c["dtype"] = "u16"                                    # host images are numpy arrays
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs
def _lattice(case, seed):
    pitch = case["pitch"]
    nx, ny = int(case["w"] / pitch) + 96, int(case["h"] / pitch) + 96
    g = torch.Generator(device=DEV).manual_seed(7919 * seed + 1)
    return torch.rand(ny, nx, device=DEV, generator=g)


def _field(case, seed, frame):
    """Backward map of a frame: reference position = x - d(x), d affine about the centre."""
    if frame == 0:
        return (0.0,) * 6
    r = np.random.default_rng(1000003 * seed + 17)
    if case["kind"] in ("sequence", "update"):
        e = 0.02 * frame / 16.0
        return (0.0, e, 0.0, 0.0, 0.0, -0.3 * e) if case["kind"] == "update" else \
            (0.3, 1e-3 * frame, 2e-4, 0.1, 1e-4, -3e-4 * frame)
    u0, v0 = r.uniform(-3.5, 3.5, 2)
    e = r.uniform(-1.0, 1.0, 4) * min(2e-3, 8.0 / max(case["w"], case["h"]))
    return (u0, e[0], e[1], v0, e[2], e[3])


def _render(case, lat, seed, frame):
    """The frame as a float32 gray plane in row chunks, quantised to the case's type."""
    w, h, pitch, dtype = case["w"], case["h"], case["pitch"], case["dtype"]
    G = GRAY_MAX[dtype]
    kinds = dict(u8=torch.uint8, u16=torch.int16, bf16=torch.bfloat16, f32=torch.float32, f64=torch.float64)
    out = torch.empty(h, w, device=DEV, dtype=kinds[dtype])
    u0, ux, uy, v0, vx, vy = _field(case, seed, frame)
    gen = torch.Generator(device=DEV).manual_seed(104729 * seed + 13 * frame + 5)
    x = torch.arange(w, device=DEV, dtype=torch.float64) - 0.5 * (w - 1)
    ld = lat.shape[1]
    flat = lat.reshape(-1)
    rows = max(1, (1 << 25) // w)
    for a in range(0, h, rows):
        y = (torch.arange(a, min(a + rows, h), device=DEV, dtype=torch.float64) - 0.5 * (h - 1))[:, None]
        X = (x - (u0 + ux * x + uy * y) + 0.5 * (w - 1)) / pitch + 48.0
        Y = (y - (v0 + vx * x + vy * y) + 0.5 * (h - 1)) / pitch + 48.0
        ix, iy = X.floor(), Y.floor()
        tx, ty = (X - ix).float(), (Y - iy).float()
        base = (iy.long() - 1) * ld + (ix.long() - 1)
        wx, wy = _bspline(tx), _bspline(ty)
        v = torch.zeros_like(tx)
        for j in range(4):
            row = sum(wx[i] * flat[base + (j * ld + i)] for i in range(4))
            v += wy[j] * row
        v = 0.1 + 0.8 * torch.sigmoid(14.0 * (v - 0.5))
        v += 0.01 * torch.randn(v.shape, device=DEV, generator=gen)
        v = (G * v).clamp_(0.0, G)
        if dtype not in ("f32", "f64"):
            v = v.round_()
        if dtype == "u16":
            v = v.to(torch.int32)                 # the 16 bits of the level in an int16 tensor
        out[a:a + rows] = v.to(out.dtype)
    return out


def _bspline(t):
    s = 1.0 - t
    return (s * s * s / 6.0, (3.0 * t - 6.0) * t * t / 6.0 + 2.0 / 3.0, (3.0 * s - 6.0) * s * s / 6.0 + 2.0 / 3.0,
            t * t * t / 6.0)


def _images(case, seed, frames):
    lat = _lattice(case, seed)
    return [_render(case, lat, seed, f) for f in frames]


def _seeds(case):
    w, h = case["w"], case["h"]
    if case["seeds"] == 1:
        return [(w // 2, h // 2)] if not case["roi"] else [(w // 4, h // 4)]
    m = int(round(math.sqrt(case["seeds"])))
    return [(w // (2 * m) + i * (w // m), h // (2 * m) + j * (h // m)) for j in range(m) for i in range(m)]


def _roi(case):
    """A frame of 6 px and a round hole in the middle are outside the region of interest."""
    if not case["roi"]:
        return None
    w, h = case["w"], case["h"]
    y, x = np.mgrid[0:h, 0:w]
    m = (x >= 6) & (x < w - 6) & (y >= 6) & (y < h - 6)
    m &= (x - w / 2) ** 2 + (y - h / 2) ** 2 > (min(w, h) / 8) ** 2
    return m.astype(np.uint8)


def _params(case):
    return dict(precision=case["precision"], optimizer=case["optimizer"], cost=case["cost"],
                search_radius=case["radius"])


def _host(t, dtype):
    a = t.cpu().numpy()
    return a.view(np.uint16) if dtype == "u16" else a


def _strain_inputs(case, seed):
    nx, ny = case["nx"], case["ny"]
    g = torch.Generator(device=DEV).manual_seed(7919 * seed + 3)
    i = torch.arange(nx, device=DEV, dtype=torch.float64) * case["step"]
    j = torch.arange(ny, device=DEV, dtype=torch.float64)[:, None] * case["step"]
    u = 3.3 + 5e-4 * i + 1e-4 * j + 0.3 * torch.sin(i / 97.0) * torch.cos(j / 61.0)
    v = -1.2 + 1e-4 * i - 2e-4 * j + 0.2 * torch.cos(i / 83.0 + j / 71.0)
    u = u + 1e-3 * torch.randn(ny, nx, device=DEV, dtype=torch.float64, generator=g)
    v = v + 1e-3 * torch.randn(ny, nx, device=DEV, dtype=torch.float64, generator=g)
    # displacements as the mixed path writes them: FP32 values in FP64 arrays
    u, v = u.float().double(), v.float().double()
    status = (torch.rand(ny, nx, device=DEV, generator=g) < 2e-5).to(torch.uint8) * binding.PT_LOW_ZNCC
    status[(i[None, :] / case["step"] - j * (0.9 / case["step"])).abs() < 1.5] = binding.PT_LOW_ZNCC
    return u.reshape(-1), v.reshape(-1), status.reshape(-1)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, kind=kind)
    if kind == "strain":
        u, v, status = _strain_inputs(case, seed)
        st.update(u=u, v=v, status=status, out=binding.strain_outputs(case["nx"] * case["ny"]))
        return st
    if kind == "fft":
        ref, dfm = _images(case, seed, (0, 1))
        st["c"] = pkg.Correlation(ref, dfm, None, case["S"], case["step"], "affine")
        return st
    st["seeds"] = _seeds(case)
    if kind == "static":
        ref, dfm = _images(case, seed, (0, 1))
        n = int(np.prod(binding.grid_size(case["w"], case["h"], case["S"], case["step"])))
        npar = binding.N_PARAMS[binding.SHAPES[case["shape"]]]
        new = lambda m, dt: torch.zeros(m, device=DEV, dtype=dt)
        st["out"] = dict(u=new(n, torch.float64), v=new(n, torch.float64), p=new(n * npar, torch.float64),
                         zncc=new(n, torch.float32), iters=new(n, torch.int32), converged=new(n, torch.uint8),
                         status=new(n, torch.uint8), wave=new(n, torch.int32))
        st.update(ref=ref, dfm=dfm, prm=binding.params(**_params(case)))
        return st
    frames = _images(case, seed, (0, 1, 2) if kind in ("sequence", "update") else (0, 1))
    if kind == "job":
        frames[1] = _host(frames[1], case["dtype"])
        ref = _host(frames[0], case["dtype"])
        st["roi"] = _roi(case)
        st["c"] = pkg.Correlation(ref, frames[1], st["roi"], case["S"], case["step"], case["shape"], case["interp"],
                                  **_params(case))
    else:
        st["c"] = pkg.Correlation(frames[0], frames[1], _roi(case), case["S"], case["step"], case["shape"],
                                  case["interp"], **_params(case))
    st["frames"] = frames
    if kind == "sequence":
        st["c"].run(st["seeds"])                  # the first frame, from the seed
        st["next"] = 2
    return st


FIELDS = ("u", "v", "p", "zncc", "iters", "converged", "status", "wave")


def _views(c, r, names):
    """Device results are views of the handle's arrays: each keeps its handle alive, so that
    reading one after the state is gone stays valid."""
    out = {k: r[k] for k in names}
    for t in out.values():
        t.handle = c
    return out


def run(state):
    kind, case = state["kind"], state["case"]
    if kind == "strain":
        binding.dic_strain_field(state["u"], state["v"], state["status"], case["nx"], case["ny"], case["step"],
                                 case["window"], case["basis"], case["measure"], state["out"])
        return state["out"]
    if kind == "static":
        binding.dic_correlate_static(state["ref"], state["dfm"], case["S"], case["step"],
                                     binding.SHAPES[case["shape"]], state["prm"], state["seeds"], state["out"])
        return state["out"]
    c = state["c"]
    if kind == "fft":
        r = c.fft_field(max_displacement=case["displacement"], subpixel=case["subpixel"])
        return _views(c, r, ("u", "v", "peak", "status", "replaced"))
    frames = state["frames"]
    if kind == "update":
        c.set_reference(frames[0])
        c.set_deformed(frames[1])
        c.run(state["seeds"])
        c.update_reference()
        c.set_deformed(frames[2])
        c.run_next()
        r = c.totals(on_device=True)
        return _views(c, r, ("u", "v", "p", "status"))
    if kind == "sequence":
        c.set_deformed(frames[state["next"]])     # frames 2, 1, 2, 1, ...
        state["next"] = 3 - state["next"]
        c.run_next()
    elif kind == "job":
        c.set_subsets(case["S"], case["step"], case["shape"], state["roi"])
        c.set_deformed(frames[1])
        c.run(state["seeds"])
        r = c.results()
        return {k: r[k] for k in FIELDS}
    else:
        c.set_reference(frames[0])
        c.set_deformed(frames[1])
        c.run(state["seeds"])
    return _views(c, c.results(on_device=True), FIELDS)


# ---------------------------------------------------------------- work
def work(case):
    """Bytes: images (and prefiltered planes where a later step reads them) once, results
    once. Flops: the method's own count per point, two sampling passes of c S^2 (c = 64,
    84, 108) and the reference terms n (n + 1) S^2; transforms 5 N log2 N."""
    if case["kind"] == "strain":
        n = case["nx"] * case["ny"]
        return dict(bytes=n * (17 + 29), flops=n * (12.0 * case["window"] + 60))
    es = dict(u8=1, u16=2, bf16=2, f32=4, f64=8)[case["dtype"]]
    px = case["w"] * case["h"]
    nx, ny = binding.grid_size(case["w"], case["h"], case["S"], case["step"])
    n = nx * ny
    if case["kind"] == "fft":
        flops = 0.0
        for L in _fft_sizes(case):
            m = n if L == case["S"] else (case["w"] // L) * (case["h"] // L)
            flops += m * L * L * (2 * 5 * 2 * math.log2(L) + 12)
        return dict(bytes=2 * es * px + 14 * n, flops=flops)
    npar = dict(rigid=2, affine=6, quadratic=12)[case["shape"]]
    c = dict(rigid=64, affine=84, quadratic=108)[case["shape"]]
    frames = 2 if case["kind"] == "update" else 1
    S2 = case["S"] ** 2
    planes = {"sequence": 1, "job": 1}.get(case["kind"], 1 + frames)
    return dict(bytes=planes * es * px + n * (16 + 8 * npar + 14),
                flops=frames * n * S2 * (2.0 * c + npar * (npar + 1)) + planes * px * 16.0)


# ---------------------------------------------------------------- the same outputs in FP64, plain torch
def _levels(img, dtype):
    if dtype == "u16":
        return (img.to(torch.int32) & 0xFFFF).double()
    return img.double()


def _reflect(a, k):
    return torch.nn.functional.pad(a[None, None], (k, k, k, k), mode="reflect")[0, 0]


def _spline_coefficients(img):
    """Interpolating cubic B-spline coefficients, whole-sample mirror: the two-sided
    exponential -6 z / (1 - z^2) z^|k| along both axes."""
    z = math.sqrt(3.0) - 2.0
    K = 28
    a = _reflect(img, K)
    for dim in (1, 0):
        n = a.shape[dim] - 2 * K
        out = a.narrow(dim, K, n).clone()
        for k in range(1, K + 1):
            out += z ** k * (a.narrow(dim, K - k, n) + a.narrow(dim, K + k, n))
        a = out * (-6.0 * z / (1.0 - z * z))
    return a


def _keys(t):
    s = 1.0 - t
    return (-0.5 * t * s * s, 1.0 + t * t * (1.5 * t - 2.5), 1.0 + s * s * (1.5 * s - 2.5), -0.5 * s * t * t)


class _Exact:
    """Frontier-wave correlation in FP64 over one resident reference."""

    def __init__(self, case, ref):
        self.case = case
        self.keys = case["interp"] == "bicubic"
        self.h, self.w = ref.shape
        self.S, self.step = case["S"], case["step"]
        self.r = (self.S - 1) // 2
        self.nx = (self.w - 1 - 2 * self.r) // self.step + 1
        self.ny = (self.h - 1 - 2 * self.r) // self.step + 1
        self.n = self.nx * self.ny
        self.NP = dict(rigid=2, affine=6, quadratic=12)[case["shape"]]
        d = torch.arange(-self.r, self.r + 1, device=DEV)
        self.dy, self.dx = (t.reshape(-1) for t in torch.meshgrid(d, d, indexing="ij"))
        q = torch.arange(self.n, device=DEV)
        self.xc, self.yc = self.r + (q % self.nx) * self.step, self.r + (q // self.nx) * self.step
        self.in_roi = torch.ones(self.n, dtype=torch.bool, device=DEV)
        roi = _roi(case)
        if roi is not None:
            m = torch.from_numpy(roi).to(DEV).double()
            full = torch.nn.functional.avg_pool2d(m[None, None], self.S, 1)[0, 0]
            self.in_roi = full[self.yc - self.r, self.xc - self.r] > 1.0 - 0.5 / self.S ** 2
        self.set_reference(ref)

    def set_reference(self, ref):
        self.f = ref
        c = ref if self.keys else _spline_coefficients(ref)
        p = _reflect(c, 1)
        gx, gy = 0.5 * (p[:, 2:] - p[:, :-2]), 0.5 * (p[2:] - p[:-2])
        if self.keys:
            self.fx, self.fy = gx[1:-1], gy[:, 1:-1]
        else:
            self.fx = (gx[:-2] + 4.0 * gx[1:-1] + gx[2:]) / 6.0
            self.fy = (gy[:, :-2] + 4.0 * gy[:, 1:-1] + gy[:, 2:]) / 6.0

    def set_deformed(self, dfm):
        self.g = dfm
        self.c = dfm if self.keys else _spline_coefficients(dfm)

    def monomials(self):
        x, y = self.dx.double(), self.dy.double()
        return [torch.ones_like(x), x, y] + ([x * x, x * y, y * y] if self.NP == 12 else [])

    def sample(self, q, p):
        """g at the warped pixels and whether all lie inside the sampling bounds."""
        x, y = self.dx.double(), self.dy.double()
        P = lambda k: p[:, k, None]
        X = self.xc[q, None] + x + P(0)
        Y = self.yc[q, None] + y + P(1)
        if self.NP >= 6:
            X, Y = X + P(2) * x + P(3) * y, Y + P(4) * x + P(5) * y
        if self.NP == 12:
            X = X + P(6) * (x * x) + P(7) * (x * y) + P(8) * (y * y)
            Y = Y + P(9) * (x * x) + P(10) * (x * y) + P(11) * (y * y)
        ok = ((X >= 1) & (X < self.w - 2) & (Y >= 1) & (Y < self.h - 2)).all(1)
        X, Y = X.nan_to_num(1.0).clamp(1, self.w - 2.001), Y.nan_to_num(1.0).clamp(1, self.h - 2.001)
        ix, iy = X.floor(), Y.floor()
        wt = _keys if self.keys else _bspline
        wx, wy = wt(X - ix), wt(Y - iy)
        base = (iy.long() - 1) * self.w + (ix.long() - 1)
        flat = self.c.reshape(-1)
        g = 0.0
        for j in range(4):
            g = g + wy[j] * sum(wx[i] * flat[base + (j * self.w + i)] for i in range(4))
        return g, ok

    def compose(self, p, dp):
        """p o dp^-1 through the second-order monomial maps of [x^2, xy, y^2, x, y, 1]."""
        def full(v):
            z = torch.zeros(v.shape[0], 12, dtype=torch.float64, device=DEV)
            z[:, :self.NP] = v
            return z
        p, d = full(p), full(dp)
        R = torch.stack([torch.stack([p[:, 6], p[:, 7], p[:, 8], 1 + p[:, 2], p[:, 3], p[:, 0]], 1),
                         torch.stack([p[:, 9], p[:, 10], p[:, 11], p[:, 4], 1 + p[:, 5], p[:, 1]], 1)], 1)
        u, v, a, b, c, e = d[:, 0], d[:, 1], 1 + d[:, 2], d[:, 3], d[:, 4], 1 + d[:, 5]
        q = [d[:, k] for k in range(6, 12)]
        one, zero = torch.ones_like(u), torch.zeros_like(u)
        rows = [[a * a + 2 * u * q[0], 2 * a * b + 2 * u * q[1], b * b + 2 * u * q[2], 2 * u * a, 2 * u * b, u * u],
                [a * c + u * q[3] + v * q[0], a * e + b * c + u * q[4] + v * q[1], b * e + u * q[5] + v * q[2],
                 u * c + v * a, u * e + v * b, u * v],
                [c * c + 2 * v * q[3], 2 * c * e + 2 * v * q[4], e * e + 2 * v * q[5], 2 * v * c, 2 * v * e, v * v],
                [q[0], q[1], q[2], a, b, u], [q[3], q[4], q[5], c, e, v], [zero, zero, zero, zero, zero, one]]
        M = torch.stack([torch.stack(r, 1) for r in rows], 1)
        Z = torch.linalg.solve(M.transpose(1, 2), R.transpose(1, 2)).transpose(1, 2)
        X, Y = Z[:, 0], Z[:, 1]
        out = torch.stack([X[:, 5], Y[:, 5], X[:, 3] - 1, X[:, 4], Y[:, 3], Y[:, 4] - 1, X[:, 0], X[:, 1], X[:, 2],
                           Y[:, 0], Y[:, 1], Y[:, 2]], 1)
        return out[:, :self.NP]

    def points(self, q, p):
        """Correlates the points q from the warps p: final p, zncc, accepted."""
        chunk = max(1, (1 << 24) // self.S ** 2)
        parts = [self.some(q[a:a + chunk], p[a:a + chunk]) for a in range(0, len(q), chunk)]
        return [torch.cat(t) for t in zip(*parts)]

    def some(self, q, p):
        case, NP, r, N = self.case, self.NP, float(self.r), float(self.S ** 2)
        pix = (self.yc[q, None] + self.dy) * self.w + self.xc[q, None] + self.dx
        f, fx, fy = (t.reshape(-1)[pix] for t in (self.f, self.fx, self.fy))
        m = self.monomials()
        order = [(0, 0), (1, 0), (0, 1), (0, 2), (1, 1), (1, 2), (0, 3), (0, 4), (0, 5), (1, 3), (1, 4), (1, 5)]
        SD = torch.stack([(fy if t else fx) * m[k] for t, k in order[:NP]], 2)
        H = SD.transpose(1, 2) @ SD
        wgt = torch.tensor([1.0] * 2 + [r * r] * 4 + [r ** 4] * 6, dtype=torch.float64, device=DEV)[:NP]
        fb = f - f.mean(1, keepdim=True)
        df = fb.norm(dim=1)
        nf = f.norm(dim=1)
        lm = case["optimizer"] == "lm"
        n = len(q)
        p = p.clone()
        zncc = torch.full((n,), math.nan, dtype=torch.float64, device=DEV)
        accepted = torch.zeros(n, dtype=torch.bool, device=DEV)
        act = torch.arange(n, device=DEV)
        best = dict(p=p.clone(), b=torch.zeros_like(p), c=torch.full((n,), math.inf, dtype=torch.float64, device=DEV),
                    s=torch.full((n,), math.inf, dtype=torch.float64, device=DEV),
                    lam=torch.full((n,), 1e-3, dtype=torch.float64, device=DEV))
        for _ in range(40):
            if not len(act):
                break
            g, ok = self.sample(q[act], p[act])
            act, g = act[ok], g[ok]                           # a sample out of bounds ends the point
            gb = g - g.mean(1, keepdim=True)
            dg, ng = gb.norm(dim=1), g.norm(dim=1)
            if case["cost"] == "ssd":
                e = f[act] - g
                cval = (e * e).sum(1)
            elif case["cost"] == "nssd":
                e = f[act] - (nf[act] / ng)[:, None] * g
                cval = 2 - 2 * (f[act] * g).sum(1) / (nf[act] * ng)
            else:
                e = fb[act] - (df[act] / dg)[:, None] * gb
                cval = 2 - 2 * (fb[act] * gb).sum(1) / (df[act] * dg)
            b = (SD[act] * e[:, :, None]).sum(1)
            dp = -torch.linalg.solve(H[act], b)
            n2 = (wgt * dp * dp).sum(1)
            z = (fb[act] * gb).sum(1) / (df[act] * dg)
            if lm:
                keep = (cval < best["c"][act]) | (n2 < best["s"][act])
                k = act[keep]
                best["p"][k], best["b"][k], best["c"][k], best["s"][k] = p[k], b[keep], cval[keep], n2[keep]
                best["lam"][act] *= torch.where(keep, 0.1, 10.0).double()
                conv = best["s"][act] < 1e-4
                Hd = H[act] + torch.diag_embed(torch.diagonal(H[act], dim1=1, dim2=2) *
                                               torch.where(conv, 0.0, best["lam"][act])[:, None])
                p[act] = self.compose(best["p"][act], -torch.linalg.solve(Hd, best["b"][act]))
            else:
                conv = n2 < 1e-4
                p[act] = self.compose(p[act], dp)
            done, z = act[conv], z[conv]
            if lm and len(done):                              # the coefficient at the final warp
                g, ok = self.sample(q[done], p[done])
                gb = g - g.mean(1, keepdim=True)
                z = (fb[done] * gb).sum(1) / (df[done] * gb.norm(dim=1))
                done, z = done[ok], z[ok]
            zncc[done] = z
            accepted[done] = z >= 0.70
            act = act[~conv]
        return p, zncc, accepted

    def start(self):
        """Seeds: the best integer shift by ZNCC within the search radius."""
        self.p = torch.zeros(self.n, self.NP, dtype=torch.float64, device=DEV)
        R, r, S = self.case["radius"], self.r, self.S
        qs = []
        for x, y in _seeds(self.case):
            gi = min(max(-((-(2 * (x - r) - self.step)) // (2 * self.step)), 0), self.nx - 1)
            gj = min(max(-((-(2 * (y - r) - self.step)) // (2 * self.step)), 0), self.ny - 1)
            q = gj * self.nx + gi
            xc, yc = r + gi * self.step, r + gj * self.step
            f = self.f[yc - r:yc + r + 1, xc - r:xc + r + 1].reshape(-1)
            f = f - f.mean()
            best = (-2.0, 0, 0)
            for dv in range(-R, R + 1):
                y0 = yc + dv - r
                x0, x1 = max(xc - R - r, 0), min(xc + R + r, self.w - 1)
                if y0 < 0 or y0 + S > self.h:
                    continue
                g = self.g[y0:y0 + S, x0:x1 + 1].unfold(1, S, 1).permute(1, 0, 2).reshape(-1, S * S)
                g = g - g.mean(1, keepdim=True)
                z = (g @ f) / (g.norm(dim=1) * f.norm())
                k = int(z.argmax())
                if float(z[k]) > best[0]:
                    best = (float(z[k]), k + x0 - (xc - r), dv)
            self.p[q, 0], self.p[q, 1] = best[1], best[2]
            qs.append(q)
        return torch.tensor(sorted(set(qs)), device=DEV)

    def correlate(self, front):
        """Waves from the front (its starts in self.p): fills p, zncc and status."""
        n, nx = self.n, self.nx
        wave = torch.full((n,), -1, dtype=torch.long, device=DEV)
        self.acc = torch.zeros(n, dtype=torch.bool, device=DEV)
        self.zncc = torch.full((n,), math.nan, dtype=torch.float64, device=DEV)
        front = front[self.in_roi[front]]
        wave[front] = 0
        k = 0
        while len(front):
            p = self.p[front]
            if k:
                gi = front % nx
                nb = torch.stack([front - 1, front + 1, front - nx, front + nx], 1)
                ok = torch.stack([gi > 0, gi < nx - 1, front >= nx, front < n - nx], 1)
                nb = torch.where(ok, nb, 0)
                ok &= self.acc[nb] & (wave[nb] < k)
                z = torch.where(ok, self.zncc[nb], torch.full_like(self.zncc[nb], -3.0))
                best = nb.gather(1, z.argmax(1, keepdim=True))[:, 0]
                d = (self.xc[front] - self.xc[best]).double(), (self.yc[front] - self.yc[best]).double()
                p = self.shift(self.p[best], *d)
            self.p[front], self.zncc[front], a = self.points(front, p)
            self.acc[front] = a
            src = front[a]
            gi = src % nx
            nxt = torch.cat([src[gi > 0] - 1, src[gi < nx - 1] + 1, src[src >= nx] - nx, src[src < n - nx] + nx])
            nxt = torch.unique(nxt)
            nxt = nxt[(wave[nxt] < 0) & self.in_roi[nxt]]
            k += 1
            wave[nxt] = k
            front = nxt
        self.p[wave < 0] = 0.0

    def shift(self, p, dx, dy):
        """The warp p re-expanded about a centre (dx, dy) away."""
        o = p.clone()
        if self.NP >= 6:
            o[:, 0] += p[:, 2] * dx + p[:, 3] * dy
            o[:, 1] += p[:, 4] * dx + p[:, 5] * dy
        if self.NP == 12:
            o[:, 0] += p[:, 6] * dx * dx + p[:, 7] * dx * dy + p[:, 8] * dy * dy
            o[:, 1] += p[:, 9] * dx * dx + p[:, 10] * dx * dy + p[:, 11] * dy * dy
            o[:, 2] += 2 * p[:, 6] * dx + p[:, 7] * dy
            o[:, 3] += p[:, 7] * dx + 2 * p[:, 8] * dy
            o[:, 4] += 2 * p[:, 9] * dx + p[:, 10] * dy
            o[:, 5] += p[:, 10] * dx + 2 * p[:, 11] * dy
        return o

    def next_frame(self):
        keep = self.acc.clone()
        self.p[~keep] = 0.0
        self.correlate(torch.nonzero(keep)[:, 0])

    def outputs(self):
        # the outputs hold the last warp of every attempted point, accepted or not
        return dict(u=self.p[:, 0].contiguous(), v=self.p[:, 1].contiguous(), p=self.p, zncc=self.zncc,
                    iters=None, converged=None, status=None, wave=None)


def _exact_update(case, ref, d1, d2):
    e = _Exact(case, ref)
    e.set_deformed(d1)
    e.correlate(e.start())
    acc_p, acc_ok = e.p.clone(), e.acc.clone()
    e.set_reference(d1)
    e.set_deformed(d2)
    e.p.zero_()
    e.acc = e.in_roi.clone()
    e.next_frame()
    # a point's total: the increment of the grid point nearest to where it has moved,
    # re-expanded there, after its accumulated warp
    x, y = e.xc + acc_p[:, 0], e.yc + acc_p[:, 1]
    i, j = (((t - e.r) / e.step - 0.5).ceil().long() for t in (x, y))
    inside = (i >= 0) & (i < e.nx) & (j >= 0) & (j < e.ny)
    best_q = torch.where(inside, j * e.nx + i, 0)
    inc = e.shift(e.p[best_q], x - e.xc[best_q], y - e.yc[best_q])
    good = acc_ok & inside & e.acc[best_q]
    tot = torch.zeros_like(acc_p)
    tot[:, :2] = acc_p[:, :2] + inc[:, :2]
    if e.NP == 6:
        A = lambda p: torch.stack([1 + p[:, 2], p[:, 3], p[:, 4], 1 + p[:, 5]], 1).reshape(-1, 2, 2)
        M = A(inc) @ A(acc_p)
        tot[:, 2], tot[:, 3], tot[:, 4], tot[:, 5] = M[:, 0, 0] - 1, M[:, 0, 1], M[:, 1, 0], M[:, 1, 1] - 1
    tot[~good] = 0.0
    return tot


def _fft_sizes(case):
    L = 1
    while L <= case["displacement"]:
        L *= 2
    out = []
    while L > case["S"]:
        if L <= min(case["w"], case["h"]):
            out.append(L)
        L //= 2
    return out + [case["S"]]


def _exact_fft(case, ref, dfm):
    H, W = ref.shape
    S, r = case["S"], (case["S"] - 1) // 2
    ar = lambda n: torch.arange(n, device=DEV)
    prev = None
    for L in _fft_sizes(case):
        last = L == S
        if last:
            nx, ny = (W - 1 - 2 * r) // case["step"] + 1, (H - 1 - 2 * r) // case["step"] + 1
            cx, cy, half = r + ar(nx) * case["step"], r + ar(ny) * case["step"], r
        else:
            nx, ny = W // L, H // L
            cx, cy, half = ar(nx) * L + L // 2, ar(ny) * L + L // 2, L // 2
        X, Y = cx.repeat(ny), cy.repeat_interleave(nx)
        x0, y0 = X - half, Y - half
        gu = gv = torch.zeros(nx * ny, dtype=torch.long, device=DEV)
        if prev is not None:
            pu, pv, c0, st = prev
            gu, gv = ((_bilinear(t, c0, st, X, Y) + 0.5).floor().long() for t in (pu, pv))
        gx, gy = (x0 + gu).clamp(0, W - L), (y0 + gv).clamp(0, H - L)
        u, v, pk = (torch.empty(nx * ny, dtype=torch.float64, device=DEV) for _ in range(3))
        chunk = max(1, (1 << 24) // (L * L))
        o = (ar(L)[:, None] * W + ar(L)).reshape(-1)
        for a in range(0, nx * ny, chunk):
            s = slice(a, a + chunk)
            win = lambda img, xx, yy: img.reshape(-1)[(yy[s] * W + xx[s])[:, None] + o].reshape(-1, L, L)
            f, g = win(ref, x0, y0), win(dfm, gx, gy)
            f, g = f - f.mean((1, 2), keepdim=True), g - g.mean((1, 2), keepdim=True)
            R = torch.fft.irfft2(torch.fft.rfft2(f) * torch.fft.rfft2(g).conj(), s=(L, L)).reshape(-1, L * L)
            R = R / (f.flatten(1).norm(dim=1) * g.flatten(1).norm(dim=1))[:, None]
            m, k = R.max(1)
            ky, kx = k // L, k % L
            wrap = lambda t: ((-t + L // 2) % L - L // 2).double()
            du, dv = wrap(kx), wrap(ky)
            if last and case["subpixel"]:
                at = lambda yy, xx: R.gather(1, ((yy % L) * L + xx % L)[:, None])[:, 0]
                du = du - _gauss3(at(ky, kx - 1), m, at(ky, kx + 1))
                dv = dv - _gauss3(at(ky - 1, kx), m, at(ky + 1, kx))
            u[s], v[s], pk[s] = (gx - x0)[s] + du, (gy - y0)[s] + dv, m
        u, v = _median_rule(u.reshape(ny, nx), v.reshape(ny, nx))
        prev = (u, v, float(L // 2), float(L))
    return dict(u=u.reshape(-1), v=v.reshape(-1), peak=pk, status=None, replaced=None)


def _gauss3(a, b, c):
    ok = (a > 0) & (b > 0) & (c > 0)
    la, lb, lc = (torch.where(ok, t, torch.ones_like(t)).log() for t in (a, b, c))
    den = 2 * (la - 2 * lb + lc)
    return torch.where(ok & (den < 0), (la - lc) / den, torch.zeros_like(a))


def _bilinear(field, c0, st, X, Y):
    ny, nx = field.shape
    tx, ty = ((X - c0) / st).clamp(0, nx - 1), ((Y - c0) / st).clamp(0, ny - 1)
    i0, j0 = tx.floor().long().clamp(max=max(nx - 2, 0)), ty.floor().long().clamp(max=max(ny - 2, 0))
    i1, j1 = (i0 + 1).clamp(max=nx - 1), (j0 + 1).clamp(max=ny - 1)
    fx, fy = tx - i0, ty - j0
    top = (1 - fx) * field[j0, i0] + fx * field[j0, i1]
    return (1 - fy) * top + fy * ((1 - fx) * field[j1, i0] + fx * field[j1, i1])


def _median_rule(u, v):
    """A value far from the median of its 3 x 3 neighbourhood (3 (1.4826 MAD + 0.5 px)) in
    either component is replaced by the medians."""
    def nine(t):
        p = torch.nn.functional.pad(t[None, None], (1, 1, 1, 1), value=math.nan)[0, 0]
        return torch.stack([p[j:j + t.shape[0], i:i + t.shape[1]] for j in range(3) for i in range(3)], 2)

    def median(t):
        s = torch.sort(t, 2).values                           # NaN last
        n = (~t.isnan()).sum(2)
        return 0.5 * (s.gather(2, ((n - 1) // 2)[..., None]) + s.gather(2, (n // 2)[..., None]))[..., 0]

    bad, med = False, []
    for t in (u, v):
        k = nine(t)
        m = median(k)
        d = median((k - m[..., None]).abs())
        bad = bad | ((t - m).abs() > 3.0 * (1.4826 * d + 0.5))
        med.append(m)
    return torch.where(bad, med[0], u), torch.where(bad, med[1], v)


def _exact_strain(case, u, v, status):
    nx, ny, N = case["nx"], case["ny"], case["window"]
    h = (N - 1) // 2
    quad = case["basis"] == "biquadratic"
    ok = (status == 0).reshape(ny, nx)
    pad = lambda t: torch.nn.functional.pad(t[None, None], (h, h, h, h), value=0.0)[0, 0]
    val = pad(ok.double())
    flds = [pad(torch.where(ok, t.reshape(ny, nx), torch.zeros_like(t.reshape(ny, nx)))) for t in (u, v)]
    k = torch.arange(-h, h + 1, device=DEV, dtype=torch.float64)
    s2, s4 = float((k ** 2).sum()), float((k ** 4).sum())
    wa, wb = (s4 / (s2 * (N * s4 - s2 * s2)), -1.0 / (N * s4 - s2 * s2)) if quad else (1.0 / (N * s2), 0.0)

    def axis(t, w, dim):
        n = t.shape[dim] - 2 * h
        return sum(float(w[a]) * t.narrow(dim, a, n) for a in range(N))

    one = torch.ones_like(k)
    full = axis(axis(val, one, 1), one, 0) > N * N - 0.5
    G = []
    for t in flds:
        G.append(axis(axis(t, k, 1), wa + wb * k * k, 0))
        G.append(wa * axis(axis(t, one, 1), k, 0) + wb * axis(axis(t, k * k, 1), k, 0))
    # points with missing neighbours: normal equations with a unit diagonal, elimination in order
    jj, ii = torch.nonzero(ok & ~full, as_tuple=True)
    dy, dx = (t.reshape(-1) for t in torch.meshgrid(k, k, indexing="ij"))
    P = [torch.ones_like(dx), dx, dy] + ([dx * dx, dy * dy, dx * dx * dy, dx * dy * dy, dx * dx * dy * dy] if quad else [])
    P = torch.stack(P, 1)
    K = P.shape[1]
    valid = ok.clone()
    offs = (dy + h).long() * val.shape[1] + (dx + h).long()
    for a in range(0, len(ii), 1 << 18):
        i, j = ii[a:a + (1 << 18)], jj[a:a + (1 << 18)]
        e = (j * val.shape[1] + i)[:, None] + offs
        m = val.reshape(-1)[e]
        M = torch.einsum("nw,wr,wc->nrc", m, P, P)
        rhs = []
        for t in flds:
            c = t[j + h, i + h][:, None]
            rhs.append(torch.einsum("nw,wr->nr", m * (t.reshape(-1)[e] - c), P))
        rhs = torch.stack(rhs, 2)
        diag = torch.diagonal(M, dim1=1, dim2=2)
        good = (m.sum(1) > K - 0.5) & (diag > 0).all(1)
        d = diag.clamp(min=1e-300).rsqrt()
        A = M * d[:, :, None] * d[:, None, :]
        L = A.clone()
        for s in range(K):
            piv = L[:, s, s]
            good &= piv > 1e-5
            f = L[:, s + 1:, s] / torch.where(piv > 1e-5, piv, torch.ones_like(piv))[:, None]
            L[:, s + 1:] = L[:, s + 1:] - f[:, :, None] * L[:, s:s + 1]
        A[~good] = torch.eye(K, dtype=torch.float64, device=DEV)
        z = torch.linalg.solve(A, rhs * d[:, :, None]) * d[:, :, None]
        for n, t in enumerate((z[:, 1, 0], z[:, 2, 0], z[:, 1, 1], z[:, 2, 1])):
            G[n][j, i] = t
        valid[j[~good], i[~good]] = False
    a, b, c, d = (t / case["step"] for t in G)                # dudx, dudy, dvdx, dvdy
    left = case["measure"] in ("euler_almansi", "biot_left")
    # D = F^T F - I (right) or F F^T - I (left)
    D11 = 2 * a + a * a + (b * b if left else c * c)
    D22 = 2 * d + d * d + (c * c if left else b * b)
    D12 = b + c + (a * c + b * d if left else a * b + c * d)
    if case["measure"] == "green_lagrange":
        E = [0.5 * D11, 0.5 * D22, 0.5 * D12]
    elif case["measure"] == "euler_almansi":
        det = D11 * D22 - D12 * D12
        s = 0.5 / (1 + D11 + D22 + det)
        E = [(D11 + det) * s, (D22 + det) * s, D12 * s]
    else:
        m, t = 0.5 * (D11 + D22), (0.25 * (D11 - D22) ** 2 + D12 * D12).sqrt()
        fn = (lambda x: 0.5 * torch.log1p(x)) if case["measure"] == "hencky" else (lambda x: x / (1 + (1 + x).sqrt()))
        der = (lambda x: 0.5 / (1 + x)) if case["measure"] == "hencky" else (lambda x: 0.5 / (1 + x).sqrt())
        f1, f2 = fn(m + t), fn(m - t)
        g = torch.where(t > 1e-7, (f1 - f2) / (2 * t).clamp(min=1e-300), der(m))
        E = [0.5 * (f1 + f2) + g * (D11 - m), 0.5 * (f1 + f2) + g * (D22 - m), g * D12]
    nan = torch.full_like(a, math.nan)
    out = dict(zip(("dudx", "dudy", "dvdx", "dvdy", "exx", "eyy", "exy"),
                   (torch.where(valid, t, nan).reshape(-1) for t in (a, b, c, d, *E))))
    out["valid"] = None
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "strain":
        return _exact_strain(case, *_strain_inputs(case, seed))
    if case["w"] * case["h"] > 7e7:
        return None                                           # the gigapixel pair takes minutes in FP64
    img = [_levels(t, case["dtype"]) for t in _images(case, seed, (0, 1, 2))]
    if kind == "fft":
        return _exact_fft(case, img[0], img[1])
    if kind == "update":
        p = _exact_update(case, *img)
        return dict(u=p[:, 0].contiguous(), v=p[:, 1].contiguous(), p=p, status=None)
    if kind != "sequence" and work(case)["flops"] > 4e11:
        return None
    e = _Exact(case, img[0])
    e.set_deformed(img[1])
    e.correlate(e.start())
    if kind == "sequence":
        e.set_deformed(img[2])
        e.next_frame()
    out = e.outputs()
    if kind == "static":
        out["p"] = out["p"].reshape(-1)
    return out
