"""The folded form of uniform axes (csrc/fold_kernel.cuh): n = R*m with R = 4, 8 or 16 and m <= 64 (TF32 pieces: 32).

Bound: both operands carry 22 bits (2^-23 relative rounding each), sums and phases are fp32 (2^-24 per operation), the
chains truncate at most 24 times: below 4e-7 per axis in the 2-norm; 1e-6 is asserted for up to three axes.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

BOUND = 1e-6


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2002_03260_b200 as d
    return d


MARGIN = 1 << 12


def _with_margins(x):
    """A buffer that holds a copy of x between two margins of sevens: (buffer, the copy)."""
    buf = torch.full((x.numel() + 2 * MARGIN,), 7.0 + 7.0j, dtype=torch.complex64, device="cuda")
    inner = buf[MARGIN:MARGIN + x.numel()].view(x.shape)
    inner.copy_(x)
    return buf, inner


def _run(lib, x, **kw):
    plan = lib.Plan(*x.shape, **kw)
    y = plan(x)
    torch.cuda.synchronize()
    plan.status()
    plan.destroy()
    return y


def _run_guarded(lib, x, **kw):
    """As _run, with margins round the input (which must not change) and round an output full of NaN (every word of which
    must be written)."""
    plan = lib.Plan(*x.shape, **kw)
    xin, xi = _with_margins(x)
    yout, yi = _with_margins(torch.full_like(x, complex(float("nan"), float("nan"))))
    plan(xi, yi)
    torch.cuda.synchronize()
    plan.status()
    plan.destroy()
    for buf in (xin, yout):
        assert bool((buf[:MARGIN] == 7.0 + 7.0j).all()) and bool((buf[-MARGIN:] == 7.0 + 7.0j).all())
    assert torch.equal(xi, x) and bool(torch.isfinite(yi).all())
    return yi.clone()


def _rel(a, b):
    a, b = a.to(torch.complex128), b.to(torch.complex128)
    return (torch.linalg.vector_norm((a - b).flatten()) / torch.linalg.vector_norm(b.flatten())).item()


# every R, m from 1 to 64 with and without a remainder of the groups (of 4 and 2 points) and of the K = 16 steps, tiles that
# are not full, batches that end inside a tile, n2 a multiple of 16 (blocked hand-over between axes 0 and 1) or not
@pytest.mark.parametrize("shape", [(4, 4, 4), (8, 20, 12), (100, 68, 36), (256, 12, 252), (264, 8, 16), (296, 4, 24),
                                   (512, 4, 20), (20, 504, 4), (528, 4, 32), (4, 544, 12), (36, 1008, 16), (1024, 8, 4),
                                   (4, 12, 1008), (4, 4, 1024), (64, 64, 48)])
@pytest.mark.parametrize("sign", [-1, +1])
def test_folded_axes_against_the_oracle(lib, oracle, shape, sign):
    from paper_2002_03260_b200 import inputs
    x = inputs.cube(shape, "normal", 301, device="cuda")
    y = _run_guarded(lib, x, sign=sign)
    assert oracle.rel_l2(y.cpu().numpy(), oracle.dft3d(x.cpu().numpy(), sign=sign, scaled_inverse=sign > 0)) < BOUND


# TF32 pieces: R and m as they fall there, groups and K = 8 steps with remainders, beside axes that are not folded (odd, and
# more than 512 points), and the FFT formulation's 256 and 512 points with and without the blocked order and in place
@pytest.mark.parametrize("mode,shape,axes", [("kdft", (100, 8, 4), None), ("kdft", (4, 128, 36), None), ("kdft", (252, 5, 12), None),
                                             ("kdft", (20, 256, 16), None), ("kdft", (500, 4, 6), None), ("kdft", (4, 512, 8), None),
                                             ("kdft", (3, 2, 496), None), ("kdft", (520, 12, 512), None), ("kdft", (64, 100, 32), None),
                                             # not multiples of four: R = 1, 2, 3, 5, 6 and 10, m up to 32, odd and even, alone or together
                                             ("kdft", (31, 1, 2), None), ("kdft", (29, 25, 30), None), ("kdft", (62, 58, 54), None),
                                             ("kdft", (93, 87, 6), None), ("kdft", (155, 5, 10), None), ("kdft", (66, 186, 6), None),
                                             ("kdft", (250, 310, 4), None), ("kdft", (7, 3, 310), None), ("kdft", (9, 66, 250), None),
                                             ("kdft", (3, 70, 190), (1, 2)), ("kdft", (5, 14, 186), (2,)), ("kdft", (66, 33, 18), (0,)),
                                             ("fft", (256, 512, 256), None), ("fft", (64, 512, 64), (1,)),
                                             ("fft", (512, 64, 64), (0,)), ("fft", (3, 256, 512), (1, 2))])
@pytest.mark.parametrize("sign", [-1, +1])
def test_folded_axes_with_tf32_pieces(lib, oracle, mode, shape, axes, sign):
    from paper_2002_03260_b200 import inputs
    x = inputs.cube(shape, "normal", 305, device="cuda")
    kw = dict(mode=lib.DFT3D_FFT if mode == "fft" else lib.DFT3D_KDFT, sign=sign, flags=lib.DFT3D_SPLIT_TF32, axes=axes)
    y = _run_guarded(lib, x, **kw)
    want = x.cpu().numpy().astype(np.complex128)
    for a in axes or (0, 1, 2):
        want = oracle.dft_axis(want, a, sign=sign, scale=1.0 / shape[a] if sign > 0 else 1.0)
    radices = lambda n: (4, 8, 16) if n % 4 == 0 else (1, 2, 3, 5, 6, 10)
    folded = all(any(shape[a] % r == 0 and shape[a] // r <= 32 for r in radices(shape[a])) for a in axes or (0, 1, 2))
    assert oracle.rel_l2(y.cpu().numpy(), want) < (BOUND if folded else 5e-6)   # 2e-6 per axis with the full matrix
    if mode == "fft" and axes is None:
        in_place = _run(lib, x, workspace_limit=1, **kw)
        assert _rel(in_place, y) < BOUND


# 512-point axes of FFT plans that leave the pieces open, in every schedule they appear in: beside axes that keep fp16 pieces
# (whose blocked orders they share), in slices of the last axis, in place, alone, and after a KDFT axis; against the plan
# that insists on fp16 pieces
@pytest.mark.parametrize("shape,mode,axes,limit", [((512, 256, 64), "fft", None, 0), ((256, 512, 128), "fft", None, 0),
                                                   ((512, 512, 256), "fft", None, 1 << 28), ((512, 256, 256), "fft", None, 1 << 26),
                                                   ((1024, 512, 256), "fft", None, 1 << 28), ((512, 512, 512), "fft", None, 1),
                                                   ((512, 2048, 64), "fft", None, 0), ((2048, 512, 64), "fft", None, 0),
                                                   ((5, 512, 512), "fft", (1, 2), 0), ((12, 512, 256), "auto", None, 0)])
def test_512_point_fft_axes(lib, shape, mode, axes, limit):
    from paper_2002_03260_b200 import inputs
    if mode == "fft" and axes is None and shape[2] % 256:
        axes = (0, 1)
    x = inputs.cube(shape, "normal", 306, device="cuda")
    kw = dict(mode=lib.DFT3D_FFT if mode == "fft" else lib.DFT3D_AUTO, axes=axes, workspace_limit=limit)
    y = _run(lib, x, **kw)
    assert _rel(y, _run(lib, x, flags=lib.DFT3D_SPLIT_FP16, **kw)) < BOUND
    if axes is None and mode == "fft":             # the transform itself, in 64 bits
        assert _rel(y, torch.fft.fftn(x.to(torch.complex128))) < BOUND


# the full matrix, which an axis with (uniform) nodes given keeps, in every form a plan takes
@pytest.mark.parametrize("axes", [(0,), (1,), (2,), (0, 1), (0, 2), (1, 2), (0, 1, 2)])
@pytest.mark.parametrize("sign,flag,limit", [(-1, "", 0), (+1, "UNSCALED_INVERSE", 0), (+1, "", 1 << 17)])
def test_folded_axes_against_the_full_matrix(lib, axes, sign, flag, limit):
    from paper_2002_03260_b200 import inputs
    shape = (24, 272, 40)
    x = inputs.cube(shape, "uniform", 302, device="cuda")
    flags = lib.DFT3D_UNSCALED_INVERSE if flag else 0
    if limit and 0 in axes and len(axes) == 2:
        limit = 0                                  # such plans need a whole cube of workspace
    uniform = [np.arange(n) / n for n in shape]
    got = _run(lib, x, sign=sign, flags=flags, axes=axes, workspace_limit=limit)
    want = _run(lib, x, sign=sign, flags=flags, axes=axes, nodes=uniform)
    assert _rel(got, want) < 5e-6                  # the full matrix: 2e-6 per axis


@pytest.mark.parametrize("scale", [2.0 ** 100, 2.0 ** 118, 2.0 ** -110])
def test_folded_scales_at_the_ends_of_the_float_range(lib, oracle, scale):
    """Inputs whose R-point sums would leave the float range, or that are nearly subnormal, scale like any other."""
    from paper_2002_03260_b200 import inputs
    shape = (4, 12, 528)
    x = inputs.cube(shape, "normal", 303, device="cuda")
    y = _run(lib, x, axes=(2,))
    ys = _run(lib, x * scale, axes=(2,))
    assert torch.equal(torch.view_as_real(ys), torch.view_as_real(y) * scale)
    assert oracle.rel_l2(y.cpu().numpy(), oracle.dft_axis(x.cpu().numpy().astype(np.complex128), 2)) < BOUND


def test_lines_beside_an_infinity_keep_their_values(lib):
    """One infinite and one NaN sample: their lines are lost, the others are what they are without them."""
    from paper_2002_03260_b200 import inputs
    x = inputs.cube((4, 8, 528), "normal", 304, device="cuda") * 1e5
    y = _run(lib, x, axes=(2,))
    bad = x.clone()
    bad[1, 3, 7] = complex(float("inf"), 0.0)
    bad[2, 5, 9] = complex(0.0, float("nan"))
    z = _run(lib, bad, axes=(2,))
    lost = torch.zeros(4, 8, dtype=torch.bool, device="cuda")
    lost[1, 3] = lost[2, 5] = True
    assert not bool(torch.isfinite(torch.view_as_real(z[lost])).all())
    assert _rel(z[~lost], y[~lost]) < 1e-6         # the scale may differ by a power of two, the pieces with it


@pytest.mark.parametrize("n", [64, 260, 2048])     # the folded, the real-matrix and the paired-CTA kernel
def test_scaled_inverse_of_the_largest_floats(lib, n):
    """The largest sample lies between 3.0e38 and the largest float: it is scaled like any other."""
    x = torch.zeros((4, 4, n), dtype=torch.complex64, device="cuda")
    x[1, 2, 5] = 3.2e38 - 1e37j
    y = _run(lib, x, axes=(2,), sign=+1)
    assert _rel(torch.view_as_complex(torch.view_as_real(y) * 2.0 ** -40),
                torch.fft.ifft(x.to(torch.complex128), dim=2) * 2.0 ** -40) < BOUND


def test_slices_do_the_work_of_their_lines_only(lib):
    """An eighth of a cube of workspace: the strided passes run once per slice, and each takes the time of its own lines.
    (The same schedule with fp16 pieces has always done that; four times its time means whole-cube work per slice.)"""
    shape = (256, 512, 512)
    x = torch.zeros(shape, dtype=torch.complex64, device="cuda")
    out = torch.empty_like(x)
    took = []
    for flags in (0, lib.DFT3D_SPLIT_FP16):
        plan = lib.Plan(*shape, mode=lib.DFT3D_FFT, workspace_limit=1 << 26, flags=flags)
        assert plan.launches == 17
        for _ in range(3):
            plan(x, out)
        best = float("inf")
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            plan(x, out)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        plan.status()
        plan.destroy()
        took.append(best)
    assert took[0] < 2.0 * took[1]


@pytest.mark.parametrize("shape,axes", [((2, 2048, 8), (1, 2)), ((4, 4, 2048), (0, 2))])
def test_an_overflow_in_a_paired_pass_spares_the_lines_beside_it(lib, shape, axes):
    """A 2048-point pass (paired CTAs) before a shorter one: a line of 3e35 sums to an infinity at frequency zero, which
    has no say in the second pass's scale; the lines that it does not reach keep their values."""
    from paper_2002_03260_b200 import inputs
    x = inputs.cube(shape, "normal", 307, device="cuda") * 1e30
    y = _run(lib, x, axes=axes)
    bad = x.clone()
    keep = torch.ones(shape, dtype=torch.bool, device="cuda")
    if 0 in axes:
        bad[1, 3] = 3e35
        keep[:, 3] = False                         # axis 0 spreads it over the planes
    else:
        bad[1, :, 5] = 3e35
        keep[1] = False
    z = _run(lib, bad, axes=axes)
    assert not bool(torch.isfinite(torch.view_as_real(z[~keep])).all())
    assert _rel(torch.view_as_complex(torch.view_as_real(z[keep]) * 2.0 ** -100),
                torch.view_as_complex(torch.view_as_real(y[keep]) * 2.0 ** -100)) < 1e-6   # the scale may differ


# ------------------------------------------------------------------ TF32 pieces: the ends of the float range, and the pieces

# every R, contiguous and strided, in the formulation and with the pieces that choose it; "" leaves the pieces open
RANGE_AXES = [("fft", "", 0, 256), ("fft", "", 0, 512), ("fft", "", 1, 512), ("fft", "", 2, 512), ("fft", "tf32", 1, 256),
              ("fft", "tf32", 2, 256), ("fft", "tf32", 2, 512), ("kdft", "tf32", 1, 100), ("kdft", "tf32", 2, 100)]
RANGE_AXES += [("kdft", "", a, n) for a in (1, 2) for n in (30, 62, 66, 150, 186, 250)]


@pytest.mark.parametrize("mode,pieces,axis,n", RANGE_AXES)
@pytest.mark.parametrize("sign", [-1, +1])
@pytest.mark.parametrize("low,high", [(-120, 60), (-146, 124), (0, 0)])
def test_every_line_keeps_its_precision_at_any_magnitude(lib, mode, pieces, axis, n, sign, low, high):
    """Lines whose magnitudes differ by any power of two, side by side: each comes out with an error of 1e-6 of its own norm,
    or half a step of the subnormal numbers per component."""
    from paper_2002_03260_b200 import inputs
    shape = [64, 64, 64] if mode == "fft" else [10, 34, 18]
    shape[axis] = n
    x = inputs.cube(tuple(shape), "uniform", 308, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(309)
    lines = [1 if d == axis else shape[d] for d in range(3)]
    power = torch.randint(low, high + 1, lines, generator=g, device="cuda").double()
    if sign < 0:
        power[power > 60] -= n.bit_length()        # the sums of n samples are floats
    xs = torch.view_as_complex((torch.view_as_real(x).double() * torch.exp2(power)[..., None]).float())
    y = _run(lib, xs, mode=lib.DFT3D_FFT if mode == "fft" else lib.DFT3D_KDFT, axes=(axis,), sign=sign,
             flags=lib.DFT3D_SPLIT_TF32 if pieces else 0).to(torch.complex128)
    want = (torch.fft.fft if sign < 0 else torch.fft.ifft)(xs.to(torch.complex128), dim=axis)
    error = torch.linalg.vector_norm(y - want, dim=axis)
    assert bool((error <= BOUND * torch.linalg.vector_norm(want, dim=axis) + 2.0 ** -149 * np.sqrt(n)).all())


@pytest.mark.parametrize("pieces", ["", "tf32"])
@pytest.mark.parametrize("limit", [0, 1 << 28, 1])
@pytest.mark.parametrize("power", [-104, 100])
def test_whole_cubes_near_the_ends_of_the_range(lib, pieces, limit, power):
    """Lines of every pass that are taken twice, out of place, in slices and in place: bit for bit the scaled result."""
    from paper_2002_03260_b200 import inputs
    x = inputs.cube((512, 256, 512), "uniform", 310, device="cuda")
    kw = dict(mode=lib.DFT3D_FFT, sign=+1, flags=(lib.DFT3D_SPLIT_TF32 if pieces else 0) | lib.DFT3D_UNSCALED_INVERSE,
              workspace_limit=limit)
    x[:, :, ::3] = 0                               # samples and lines of zeros among them
    y = torch.view_as_real(_run(lib, x, **kw))
    z = torch.view_as_real(_run(lib, torch.view_as_complex(torch.view_as_real(x) * 2.0 ** power), **kw))
    want = y * 2.0 ** power
    normal = want.abs() >= 2.0 ** -126
    assert torch.equal(z[normal], want[normal]) and bool(((z - want)[~normal].abs() <= 2.0 ** -148).all())


def test_more_units_than_a_block_can_mark(lib):
    """3.2e8 lines of four points: with more than 65536 units a block scales every line by its own largest component."""
    n0, n1 = 40000, 8000
    x = torch.zeros((n0, n1, 4), dtype=torch.complex64, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(312)
    rows = [0, 1, 19999, n0 - 1]
    for i, r in enumerate(rows):
        x[r] = torch.view_as_complex(torch.randn((n1, 4, 2), generator=g, device="cuda") * 2.0 ** (0, -110, 120, 3)[i])
    y = _run(lib, x, axes=(2,), flags=lib.DFT3D_SPLIT_TF32)
    for r in rows:
        want = torch.fft.fft(x[r].to(torch.complex128), dim=1)
        assert _rel(y[r].to(torch.complex128), want) < BOUND
        y[r] = 0
    assert not bool(torch.view_as_real(y).any())


@pytest.mark.parametrize("axis", [0, 1, 2])
def test_lines_beside_infinities_with_tf32_pieces(lib, axis):
    from paper_2002_03260_b200 import inputs
    shape = [64, 64, 64]
    shape[axis] = 512
    x = inputs.cube(tuple(shape), "normal", 313, device="cuda")
    y = _run(lib, x, mode=lib.DFT3D_FFT, axes=(axis,))
    bad = x.clone()
    bad[1, 3, 7] = complex(float("inf"), 0.0)
    bad[2, 5, 9] = complex(0.0, float("nan"))
    z = _run(lib, bad, mode=lib.DFT3D_FFT, axes=(axis,))
    lost = torch.zeros(shape, dtype=torch.bool, device="cuda")
    for at in ([1, 3, 7], [2, 5, 9]):
        at[axis] = slice(None)
        lost[tuple(at)] = True
    assert not bool(torch.isfinite(z[lost]).any()) and torch.equal(z[~lost], y[~lost])


@pytest.mark.parametrize("pieces", ["", "fp16", "tf32"])
def test_named_pairs_are_used_and_the_query_reports_what_runs(lib, pieces):
    """The folded form computes 256 = 8*32 and 512 = 16*32; a plan that names 16*16 or 32*16 runs those two products."""
    from paper_2002_03260_b200 import inputs
    shape = (256, 512, 512)
    flags = {"": 0, "fp16": lib.DFT3D_SPLIT_FP16, "tf32": lib.DFT3D_SPLIT_TF32}[pieces]
    x = inputs.cube(shape, "normal", 314, device="cuda")
    want = torch.fft.fftn(x.to(torch.complex128))
    named = [(16, 16), (32, 16), (32, 16)]
    own = named if pieces == "fp16" else [(8, 32), (16, 32), (16, 32)]
    for pairs in (None, named, [named[0], None, None], [None, named[1], None], [None, None, named[2]]):
        for limit in (0, 1):
            plan = lib.Plan(*shape, mode=lib.DFT3D_FFT, flags=flags, fft_split=pairs, workspace_limit=limit)
            assert [plan.fft_split(a) for a in range(3)] == [(pairs or own)[a] or own[a] for a in range(3)]
            y = plan(x)
            torch.cuda.synchronize()
            plan.status()
            plan.destroy()
            assert _rel(y, want) < BOUND
