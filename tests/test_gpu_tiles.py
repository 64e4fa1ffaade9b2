"""GPU tests of the tiled kernels at the sizes where a tile can go wrong: grids
that their tiles do not cover, tiles wider than the grid, and boxes that do
not fit in shared memory."""
import numpy as np
import pytest

import oracle
from paper_2209_08189_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _ctx(n, **opts):
    from paper_2209_08189_gb300 import claire
    return claire.Context(n, 1e-2, 4, stream=torch.cuda.current_stream().cuda_stream, **opts)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def _rel(a, b):
    a = a.cpu().numpy().astype(np.float64)
    return float(np.abs(a - b).max() / np.abs(b).max())


@pytest.mark.parametrize("n", [(8, 8, 8), (10, 14, 22), (12, 10, 66), (34, 18, 40), (70, 44, 104)])
def test_fd8_on_partial_columns(n):
    """Columns of 8 x 32 nodes past the end of the grid, and halos that wrap
    onto the column itself; random fields, so every wrong neighbour shows.
    Tolerance: the oracle parity of the FD8 kernels (FP32 sums of 8 terms)."""
    rng = np.random.default_rng(3)
    f, v = rng.standard_normal(n).astype(np.float32), rng.standard_normal((3,) + n).astype(np.float32)
    ctx = _ctx(n, kernels_only=1)
    g, d = torch.empty((3,) + n, device="cuda"), torch.empty(n, device="cuda")
    ctx.fd8_grad(_dev(f), g)
    ctx.fd8_div(_dev(v), d)
    ref = oracle.fd8_grad(f.astype(np.float64))
    for c in range(3):
        assert _rel(g[c], ref[c]) <= 1e-5
    assert _rel(d, oracle.fd8_div(v.astype(np.float64))) <= 1e-5
    ctx.close()


@pytest.mark.parametrize("n", [(16, 24, 8), (12, 10, 66), (70, 44, 104)])
@pytest.mark.parametrize("order", [3, 1, 4])
def test_detj_on_partial_tiles(n, order):
    """Map steps and determinant extrema; tolerance of the existing parity test."""
    v = synth.mode_velocity(n, seed=12, vmax=0.8, kmax=2).astype(np.float32)
    ctx = _ctx(n, interp=order)
    lo, hi = ctx.detj(_dev(v))
    ref = oracle.detj(v.astype(np.float64), oracle.Params(nt=4, order=order))
    assert abs(lo - ref.min()) <= 1e-5 * abs(ref.min()) and abs(hi - ref.max()) <= 1e-5 * ref.max()
    ctx.close()


@pytest.mark.parametrize("n", [(12, 10, 66), (32, 16, 64), (70, 44, 104)])
@pytest.mark.parametrize("rough", [False, True])
def test_vjp_tiles_and_fallback(n, rough):
    """The reverse pass with boxes in shared memory (smooth velocity) and with
    boxes that do not fit (rough: every point moves on its own, so tiles take the
    global-memory paths), against the oracle.  The image cotangent is a sum of
    64 FP32 products per node (1e-5); the velocity cotangent of a rough map
    has kinks at every cell face, so only the smooth one is compared (1e-4).
    A cotangent scaled by a power of two scales the result exactly: the
    fixed-point scale follows max |gbar|.  (Scaled down, the velocity
    cotangent's FP32 products with small image gradients become subnormal and
    lose bits, so only the image cotangent scales exactly there.)"""
    rng = np.random.default_rng(5)
    v = rng.uniform(-3, 3, (3,) + n) if rough else synth.mode_velocity(n, seed=4, vmax=1.0, kmax=2)
    v = v.astype(np.float32)
    m0 = synth.blob_template(n, seed=5, sigma=0.9).astype(np.float32)
    gbar = rng.standard_normal(n).astype(np.float32)
    gbar[rng.random(n) < 0.1] = 0.0
    ctx = _ctx(n)
    out = {}
    for k in (0, 90, -90):
        gm, gv = torch.empty(n, device="cuda"), torch.empty((3,) + n, device="cuda")
        ctx.transport_vjp(_dev(v), _dev(m0), _dev(gbar * np.float32(2.0 ** k)), gm, gv)
        out[k] = (gm, gv)
    rm, rv = oracle.transport_vjp(m0.astype(np.float64), v.astype(np.float64), gbar.astype(np.float64),
                                  oracle.Params(nt=4))
    l2 = lambda a, b: float(np.linalg.norm(a.cpu().numpy().astype(np.float64) - b) / np.linalg.norm(b))
    assert l2(out[0][0], rm) < 1e-5
    if not rough:
        assert l2(out[0][1], rv) < 1e-4
    for k in (90, -90):
        assert torch.equal(out[k][0], out[0][0] * 2.0 ** k)
        if k > 0:
            assert torch.equal(out[k][1], out[0][1] * 2.0 ** k)
    ctx.close()


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_vjp_non_finite_cotangent_gives_nan(bad):
    n = (16, 24, 8)
    v = synth.mode_velocity(n, seed=4, vmax=0.5, kmax=2)
    g = np.ones(n, dtype=np.float32)
    g[3, 4, 5] = bad
    ctx = _ctx(n)
    gm = torch.empty(n, device="cuda")
    ctx.transport_vjp(_dev(v), _dev(np.ones(n)), _dev(g), gm)
    assert bool(torch.isnan(gm).all())
    ctx.close()


@pytest.mark.parametrize("n", [(8, 8, 8), (32, 32, 32), (12, 14, 30), (34, 18, 70), (20, 28, 44), (64, 24, 96)])
@pytest.mark.parametrize("order", [3, 1])
def test_table_and_chunk_widths_agree(n, order):
    """The solver's gathers take their boxes from the backtrace's tile-bounds
    table and stage them with the widest copies the row length and the address
    allow; the kernel-level gather reduces the bounds itself.  A transport and
    the same steps through the kernel-level calls, from fields at every 4-byte
    alignment, give the same bits, and a smooth displacement of under two cells
    fits the box on every grid, however short its axes."""
    from paper_2209_08189_gb300 import claire
    rng = np.random.default_rng(9)
    v = synth.mode_velocity(n, seed=3, vmax=1.0, kmax=1)
    v = (v * (1.5 * 4 * 2 * np.pi / max(n)) / np.abs(v).max()).astype(np.float32)  # at most 1.5 cells per step
    m = rng.standard_normal(n).astype(np.float32)
    ctx, out = _ctx(n, interp=order), torch.empty(n, device="cuda")
    claire.claire_gather_fallback_tiles(reset=True)
    ctx.transport(_dev(v), _dev(m), out)
    d = torch.empty((3,) + n, device="cuda")
    ctx.backtrace(_dev(v), d)
    for off in range(4):
        buf = torch.empty(m.size + 4, device="cuda")
        cur = buf[off:off + m.size].view(n)
        cur.copy_(_dev(m))
        for _ in range(4):
            nxt = torch.empty(n, device="cuda")
            ctx.interp(cur, d, nxt, order)
            cur.copy_(nxt)
        assert torch.equal(cur, out)
    assert claire.claire_gather_fallback_tiles() == 0
    ctx.close()


@pytest.mark.parametrize("n", [(32, 32, 32), (12, 14, 30), (34, 18, 70), (20, 28, 44)])
@pytest.mark.parametrize("storage", [0, 1, 2])
def test_boxes_on_every_row_length_carry_a_shift(n, storage):
    """Rows staged in 16-, 8- and 4-byte copies, for each storage type.  A
    constant velocity of whole cells per step carries an image of values that
    the type holds exactly; each step interpolates at a point within FP32
    rounding of a node, so it returns the node's value up to 1e-6 of it, which
    16-bit rounding removes (values in [1/2, 1], spacing at least 2^-12): the
    mismatch against the shifted image is 0, or in FP32 of that order squared."""
    rng = np.random.default_rng(4)
    m0 = (0.5 + rng.integers(0, 64, n) / 128.0).astype(np.float32)  # seven bits: exact in every type
    step = (1, -2, 3)
    v = np.empty((3,) + n, dtype=np.float32)
    for c in range(3):
        v[c] = step[c] * 4 * 2 * np.pi / n[c]
    # m(1)(x) = m0(x - v): four steps of `step` cells
    m1 = np.roll(m0, [4 * s for s in step], (0, 1, 2))
    ctx = _ctx(n, storage=storage)
    ctx.set_images(_dev(m0), _dev(m1))
    _, mis = ctx.objective(_dev(v))
    vol = float(np.prod([2 * np.pi / s for s in n]))
    assert mis <= (0.0 if storage else 0.5 * vol * m0.size * (4 * 4e-6) ** 2)
    ctx.close()


@pytest.mark.parametrize("nt", [1, 4])
def test_results_formed_in_the_callers_array(nt):
    """Results are formed in the caller's array when it is aligned and shares no
    byte with the input, else in scratch and copied: outputs into separate,
    unaligned and partly or fully shared arrays hold the same bits, and an input
    that is not shared is left alone."""
    from paper_2209_08189_gb300 import claire
    n = (16, 24, 40)
    N = n[0] * n[1] * n[2]
    ctx = claire.Context(n, 1e-2, nt, stream=torch.cuda.current_stream().cuda_stream)
    v = _dev(synth.mode_velocity(n, seed=3, vmax=0.4, kmax=2))
    vt = _dev(synth.mode_velocity(n, seed=4, vmax=0.4, kmax=2))
    m0, m1 = _dev(synth.blob_template(n, seed=1, sigma=0.9)), _dev(synth.blob_template(n, seed=2, sigma=0.9))
    ctx.set_images(m0, m1)
    new = lambda k: torch.empty(k * N, device="cuda")

    def layouts(x, k):
        """(input, output) views of k N floats; the input holds x."""
        size = x.numel()
        for out_off, shared in ((0, None), (1, None), (0, 0), (0, 4), (0, 3)):
            if shared is None:  # separate arrays, output at out_off
                inp, out = x.clone().reshape(-1), new(k + 1)[out_off:out_off + k * N]
            else:               # one array, output `shared` floats behind the input
                buf = new(max(k, size // N) + 1)
                inp, out = buf[:size], buf[shared:shared + k * N]
                inp.copy_(x.reshape(-1))
            yield inp, out, shared is None

    calls = {
        "gradient": (v, 3, lambda i, o: ctx.gradient(i, o)),
        "matvec": (vt, 3, lambda i, o: (ctx.gradient(v, new(3)), ctx.hessian_matvec(i, o))),
        "precond": (vt, 3, lambda i, o: ctx.precond(i, o)),
        "forward": (m0, 1, lambda i, o: ctx.transport(v, i, o)),
        "adjoint": (m0, 1, lambda i, o: ctx.transport(v, i, o, claire.TRANSPORT_ADJ)),
        "vjp": (v, 3, lambda i, o: ctx.transport_vjp(i, m0, m1, new(1), o)),
        "vjp_image": (m1, 1, lambda i, o: ctx.transport_vjp(v, m0, i, o)),
    }
    for name, (x, k, call) in calls.items():
        want = None
        for inp, out, separate in layouts(x, k):
            call(inp, out)
            got = out.clone()
            want = got if want is None else want
            assert torch.equal(got, want), name
            if separate:
                assert torch.equal(inp, x.reshape(-1)), name
    ctx.close()



@pytest.mark.parametrize("n", [(64, 64, 64), (70, 44, 104)])
def test_trilinear_values_do_not_depend_on_the_box(n):
    """Trilinear tiles take a wider box where the displacement is large, and go to
    global memory where no box holds them.  The value at a point is the same bits on
    every path: a displacement below the line, one above it whose tiles fit, and
    tiles made to overflow by one far point each, whose other points are compared."""
    from paper_2209_08189_gb300 import claire
    rng = np.random.default_rng(2)
    f = _dev(rng.standard_normal(n))
    far = np.zeros((3,) + n, dtype=np.float32)
    far[:, ::4, ::8, ::32] = 40.0  # the first point of every tile
    near = rng.uniform(-1.5, 1.5, (3,) + n).astype(np.float32)
    out = {}
    for vmax in (0.5, 20.0):  # below and above 12 cells per step on these grids
        v = synth.mode_velocity(n, seed=3, vmax=vmax, kmax=1).astype(np.float32)
        ctx = _ctx(n, interp=claire.INTERP_LINEAR)
        d = torch.empty((3,) + n, device="cuda")
        ctx.backtrace(_dev(v), d)
        for name, disp in (("near", near), ("far", near + far)):
            claire.claire_gather_fallback_tiles(reset=True)
            o = torch.empty(n, device="cuda")
            ctx.interp(f, _dev(disp), o, claire.INTERP_LINEAR)
            tiles = -(-n[0] // 4) * -(-n[1] // 8) * -(-n[2] // 32)
            assert claire.claire_gather_fallback_tiles() == (tiles if name == "far" else 0)
            out[name, vmax] = o.cpu().numpy()
        ctx.close()
    same = far[0] == 0
    for key in out:
        assert np.array_equal(out[key][same], out["near", 0.5][same]), key
