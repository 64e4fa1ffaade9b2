"""GPU tests of single kernels on inputs that the entry points cannot give them
directly (direct_calls.cu, linked against libclaire.so)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import __graft_entry__ as entry

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def direct(tmp_path_factory):
    entry.build()
    from paper_2209_08189_gb300 import build
    so = str(tmp_path_factory.mktemp("direct") / "direct_calls.so")
    cmd = [os.path.join(build._cuda_home(), "bin", "nvcc"), *build.ARCH, "-O1", "-std=c++17", "-Xcompiler", "-fPIC",
           "-shared", "-cudart", "shared", "--expt-relaxed-constexpr", "-I" + build.INCLUDE, "-I" + build.CSRC,
           os.path.join(ROOT, "tests", "direct_calls.cu"), build.LIB, "-Xlinker", "-rpath=" + build.PKG, "-o", so]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stdout + res.stderr
    return ctypes.CDLL(so)


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def _differences(n, u):
    """The nine FP32 differences of u, as the FD8 gradient forms them."""
    from paper_2209_08189_gb300 import claire
    ctx = claire.Context(n, 1e-2, 4, stream=torch.cuda.current_stream().cuda_stream, kernels_only=1)
    out = np.empty((3, 3) + n)
    for c in range(3):
        g = torch.empty((3,) + n, device="cuda")
        ctx.fd8_grad(u[c], g)
        out[c] = g.cpu().numpy()
    ctx.close()
    return out


def _det(e):
    F = e + np.eye(3).reshape(3, 3, 1, 1, 1)
    return (F[0, 0] * (F[1, 1] * F[2, 2] - F[1, 2] * F[2, 1]) - F[0, 1] * (F[1, 0] * F[2, 2] - F[1, 2] * F[2, 0]) +
            F[0, 2] * (F[1, 0] * F[2, 1] - F[1, 1] * F[2, 0]))


def _plateau(n, slope):
    """Periodic function with the slope `slope` on a third of the period."""
    x = np.arange(n) * 2 * np.pi / n
    ramp = np.clip((np.abs(x - np.pi) - np.pi / 3) / (2 * np.pi / 3), 0, 1)
    bump = ramp ** 3 * (10 - 15 * ramp + 6 * ramp ** 2)     # 0 on the plateau
    d = slope * (1 - bump / bump.mean())
    u = np.cumsum(d + np.roll(d, 1)) * np.pi / n
    return u - u[n // 2]


@pytest.mark.parametrize("size", [10.0, 1.0, 1e-1, 1e-2, 1e-3, 3e-6, 1e-12])
def test_det_bounds_hold(direct, size):
    """det(I + e) in FP64 lies between its FP32 bounds for entries of I + e up to
    `size`, down to maps that compress a thousandfold and to products that
    underflow, and the bounds are no wider than stated (8e-6 m^3 and its rounding)."""
    n, rng = 1 << 18, np.random.default_rng(7)
    ih = np.array([64, 90, 52], dtype=np.float32) / np.float32(2 * np.pi)
    F = rng.uniform(-size, size, (3, 3, n)) * 10.0 ** rng.uniform(-1, 0, (3, 3, n))
    diff = ((F - np.eye(3)[:, :, None]) / ih[None, :, None]).astype(np.float32)
    d, i = torch.from_numpy(diff).cuda(), torch.from_numpy(ih).cuda()
    lo, hi = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")
    det = torch.empty(n, device="cuda", dtype=torch.float64)
    assert direct.direct_det_bounds(_ptr(d), _ptr(i), n, _ptr(lo), _ptr(det), _ptr(hi)) == 0
    assert bool((lo.double() <= det).all()) and bool((det <= hi.double()).all())
    assert float((hi - lo).max()) <= 1.1e-5 * max(size, 2e-7) ** 3 + 3e-36
    e = (diff * ih[None, :, None]).astype(np.float64)
    assert np.abs(det.cpu().numpy() - _det(e.reshape(3, 3, 1, 1, n)).ravel()).max() <= 1e-14 * max(size, 2e-7) ** 3 + 1e-300


@pytest.mark.parametrize("compression", [1e-1, 1e-2])
def test_detj_extrema_of_a_compressing_map(direct, compression):
    """The FP32 filter of the determinant never loses an extremum: where the map
    compresses by 1 / compression on every axis the entries of I + grad u are
    small and thousands of points nearly tie.  The extrema are those of the
    determinants in FP64 of the same FP32 differences, up to the rounding of the
    FP64 formula (1e-14 of six products of the largest entries)."""
    n = (48, 40, 64)
    for seed in range(4):
        rng = np.random.default_rng(seed)
        ax = [_plateau(s, compression - 1.0) for s in n]
        u = np.stack([np.broadcast_to(ax[c].reshape([-1 if a == c else 1 for a in range(3)]), n) for c in range(3)])
        u = u + rng.uniform(-1, 1, u.shape) * 2e-8
        d = torch.from_numpy(u.astype(np.float32)).cuda()
        det = _det(_differences(n, d))
        assert (det < 2 * det.min()).sum() > 1000  # near ties
        out = (ctypes.c_double * 2)()
        assert direct.direct_detj(*n, _ptr(d), 608, out) == 0
        assert abs(out[0] - det.min()) <= 1e-14 * 6 * (2 * compression) ** 3
        assert abs(out[1] - det.max()) <= 1e-14 * 6 * 3.0 ** 3


@pytest.mark.parametrize("where", [(0, 0, 0), (47, 39, 63), (20, 17, 31)])
def test_detj_keeps_a_nan(direct, where):
    n = (48, 40, 64)
    u = torch.zeros((3,) + n, device="cuda")
    u[1][where] = float("nan")
    out = (ctypes.c_double * 2)()
    assert direct.direct_detj(*n, _ptr(u), 608, out) == 0
    assert np.isnan(out[0]) and np.isnan(out[1])


def _fixed_to_float(direct, acc, maxabs, out, mult=1.0, accumulate=True):
    a = torch.from_numpy(np.asarray(acc, dtype=np.int64)).cuda()
    m = torch.tensor([maxabs], dtype=torch.float64, device="cuda")
    o = torch.from_numpy(np.asarray(out, dtype=np.float32)).cuda()
    assert direct.direct_fixed_to_float(_ptr(a), _ptr(m), int(accumulate), ctypes.c_float(mult), _ptr(o),
                                        ctypes.c_longlong(o.numel())) == 0
    assert int(a.abs().max()) == 0  # cleared for the next scatter
    return o.cpu().numpy()


def test_fixed_point_sum_onto_infinities(direct):
    """Added to an infinity the sum is that infinity, as it is in FP64; a NaN stays a
    NaN, and a finite sum beyond the FP32 range becomes an infinity.  Seven values:
    the vector path and the tail."""
    big = np.float32(3e38)
    old = [np.inf, -np.inf, np.nan, big, 1.0, np.inf, -big]
    acc = [1 << 40, 1 << 40, 5, 1 << 47, 1 << 20, 0, -(1 << 47)]
    got = _fixed_to_float(direct, acc, 2.5e38, old, mult=2.0)  # 2^47 stands for 2^127
    assert got[0] == np.inf and got[1] == -np.inf and np.isnan(got[2]) and got[3] == np.inf
    assert got[5] == np.inf and got[6] == -np.inf


@pytest.mark.parametrize("n", [1, 6, 4096])
def test_fixed_point_sum_uses_all_bits(direct, n):
    """acc / scale enters the sum with all 64 bits.  Added to minus its FP32 rounding
    the rest remains, held to 2^-22 of it (three FP32 roundings), however many
    bits of the sum cancel; plain, it is the FP32 rounding (2^-23, for ties that
    an intermediate rounding makes)."""
    rng = np.random.default_rng(3)
    acc = [int(rng.integers(1, 1 << 62)) >> int(rng.integers(0, 62)) for _ in range(n)]
    acc = [((a >> 40) << 40 | (a & ((1 << int(rng.integers(1, 33))) - 1))) or 1 for a in acc]  # low words after zeros
    acc = [a if rng.random() < 0.5 else -a for a in acc]
    maxabs = 1.0  # 2^47 stands for 1
    val = [a / 2 ** 47 for a in acc]  # a Python division is correctly rounded
    plain = _fixed_to_float(direct, acc, maxabs, np.zeros(n), accumulate=False)
    assert np.all(np.abs(plain - np.array(val)) <= 2.0 ** -23 * np.abs(val))
    got = _fixed_to_float(direct, acc, maxabs, -plain)
    for a, p, g in zip(acc, plain, got):
        rest = a - int(float(p) * 2 ** 47)  # exact: p is an FP32 value of at least 2^-47
        assert abs(float(g) * 2 ** 47 - rest) <= 2.0 ** -22 * abs(rest), (a, p, g)
