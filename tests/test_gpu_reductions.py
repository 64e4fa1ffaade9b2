"""GPU tests of the filtered FP64 extrema: the largest |v| (the reported CFL)
against the same maximum formed in FP64 on the host, at the sizes and
magnitudes where the FP32 filter could lose it."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _ctx(n, **opts):
    from paper_2209_08189_gb300 import claire
    return claire.Context(n, 1e-2, 4, stream=torch.cuda.current_stream().cuda_stream, **opts)


@pytest.mark.parametrize("n", [(8, 8, 8), (10, 14, 22), (40, 36, 30), (64, 32, 96)])
@pytest.mark.parametrize("scale", [0.0, 1e-30, 1e-16, 1.0, 1e12, 1e25])
def test_cfl_is_the_fp64_maximum(n, scale):
    rng = np.random.default_rng(7)
    v = rng.standard_normal((3,) + n)
    # many near ties: a quarter of the points within FP32 rounding of the largest norm
    v /= np.sqrt((v * v).sum(0))
    v *= np.where(rng.random(n) < 0.25, 1.0, rng.random(n))
    v = (v * scale).astype(np.float32)
    ctx = _ctx(n, max_gn=0, spectral_iterate=0)
    z = torch.zeros(n, device="cuda")
    ctx.set_images(z, z)
    h = float(min(np.float32(2.0 * math.pi / s) for s in n))  # the grid spacing is held in FP32
    v64 = v.astype(np.float64)
    # three squares and two sums in FP64, in any order and with or without FMA: a few ulps
    want = math.sqrt(np.max((v64 * v64).sum(0))) * 0.25 / h
    for off in (0, 1):  # 16-byte aligned, and offset by one float
        buf = torch.empty(v.size + 4, device="cuda")
        t = buf[off:off + v.size].view(v.shape)
        t.copy_(torch.from_numpy(v))
        if scale <= 1.0:  # beyond, the transport itself overflows
            _, rep = ctx.register(t, check=False)
            assert abs(rep["cfl"] - want) <= 1e-14 * want
        d = torch.empty(v.shape, device="cuda")
        ctx.backtrace(t, d)  # screened: finite magnitudes pass
    ctx.close()


@pytest.mark.parametrize("n", [(8, 8, 8), (40, 36, 30)])
@pytest.mark.parametrize("bad", [float("nan"), -float("nan"), float("inf"), -float("inf")])
def test_screen_finds_one_bad_value_anywhere(n, bad):
    from paper_2209_08189_gb300 import claire
    ctx = _ctx(n, kernels_only=1)
    N = n[0] * n[1] * n[2]
    d = torch.empty((3,) + n, device="cuda")
    for where in (0, 31, N - 1, N, 2 * N + N // 2, 3 * N - 1):
        v = torch.full((3 * N,), 0.25, device="cuda")
        v[where] = bad
        with pytest.raises(claire.ClaireError) as e:
            ctx.backtrace(v.view((3,) + n), d)
        assert e.value.status == -5
    ctx.close()
