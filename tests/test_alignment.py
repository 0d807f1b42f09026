"""Device images whose rows do not start on element boundaries (a raw 16- or 32-bit frame behind an
odd header, an odd row stride). Calls that read gray levels through typed loads refuse them before
any device work; the frames of a sequence, whose FP32 spline prefilter reads any byte, give
the aligned frames' results bit for bit."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def B():
    from paper_2601_12941_gb300 import binding, build

    build.build()
    binding.load()
    return binding


@pytest.mark.parametrize("data,stride,dtype", [(0x1001, 0, "DIC_U16"), (0x1000, 129, "DIC_BF16"), (0x1002, 0, "DIC_F32"),
                                               (0x1004, 0, "DIC_F64"), (0x1000, 516, "DIC_F64")])
def test_the_allocation_free_call_refuses_them(B, data, stride, dtype):
    good = B.DicImage(0x1000, 64, 48, 0, getattr(B, dtype), 1)
    bad = B.DicImage(data, 64, 48, stride, getattr(B, dtype), 1)
    if stride == 516:
        good = B.DicImage(0x1000, 64, 48, 520, B.DIC_F64, 1)
    prm, acc = B.dic_default_params(), ctypes.c_int64(0)
    out = B.DicStaticOutputs(*([16] * 8), ctypes.cast(ctypes.byref(acc), ctypes.c_void_p))
    seeds = (ctypes.c_int32 * 2)(32, 24)
    err = ctypes.create_string_buffer(256)
    for ref, dfm in ((bad, good), (good, bad)):
        rc = B.load().dic_correlate_static(ctypes.byref(ref), ctypes.byref(dfm), 21, 5, B.DIC_AFFINE, ctypes.byref(prm), seeds,
                                           1, ctypes.byref(out), None, err, 256)
        assert rc == B.DIC_EINVAL and b"element boundaries" in err.value


def _frames(dtype):
    import synth

    W, H = 250, 210
    sp = synth.Speckle(seed=77, density=0.03, sigma=(1.5, 3.0), cell=16)
    out = []
    for k in range(3):
        fld = synth.affine_field(W, H, u0=0.3 * k, v0=-0.2 * k, exx=1e-3 * k, exy=0.0, eyx=0.0, eyy=-1e-3 * k)
        out.append(synth.render(synth.ImageSpec(sp, field=fld, gray_max=4000.0, noise=20.0, noise_tag=k), W, H, dtype))
    return W, H, out


def _raw(B, img, header, dtype):
    """The image in a device buffer behind `header` bytes with an odd row stride."""
    H, row = img.shape[0], img.shape[1] * img.itemsize
    stride = row + 1
    host = np.zeros(header + H * stride, np.uint8)
    for y in range(H):
        host[header + y * stride:header + y * stride + row] = np.ascontiguousarray(img[y]).view(np.uint8)
    dev = torch.from_numpy(host).cuda()
    return B.DicImage(dev.data_ptr() + header, img.shape[1], H, stride, dtype, 1), dev


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["u16", "f32"])
def test_frames_behind_an_odd_header(B, dtype):
    import paper_2601_12941_gb300 as pkg

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    W, H, frames = _frames(dtype)
    code = B.DIC_U16 if dtype == "u16" else B.DIC_F32
    got = []
    for odd in (False, True):
        c = pkg.Correlation(frames[0], frames[1], None, 21, 10, "affine")
        c.run([(W // 2, H // 2)])
        if odd:
            im, keep = _raw(B, frames[2], 3, code)
            assert B.load().dic_set_deformed(c.h, ctypes.byref(im)) == B.DIC_OK
        else:
            c.set_deformed(frames[2])
        c.run_next()
        got.append(c.results())
        if odd:
            # the calls with typed loads refuse the frame and leave the handle usable
            with pytest.raises(B.DicError, match="element boundaries"):
                c.run([(W // 2, H // 2)])
            with pytest.raises(B.DicError, match="element boundaries"):
                c.fft_field(max_displacement=16)
            org = torch.zeros((1, 4), dtype=torch.int32, device="cuda")
            u, v, pk = (torch.empty(1, dtype=torch.float32, device="cuda") for _ in range(3))
            with pytest.raises(B.DicError, match="element boundaries"):
                B.dic_fftcc_windows(c.h, 32, org, False, u, v, pk)
            c.run_next()
            # and so does a bicubic or an FP64 sequence
            for kw, interp in ((dict(precision="fp64"), "bspline3"), (dict(), "bicubic")):
                d = pkg.Correlation(frames[0], frames[1], None, 21, 40, "rigid", interp, **kw)
                d.run([(W // 2, H // 2)])
                assert B.load().dic_set_deformed(d.h, ctypes.byref(im)) == B.DIC_OK
                with pytest.raises(B.DicError, match="element boundaries"):
                    d.run_next()
                d.close()
        c.close()
    for k in ("u", "v", "p", "zncc", "iters", "status"):
        assert np.array_equal(got[0][k], got[1][k], equal_nan=True), k
