"""KDFT axes with nodes as products with a real matrix about the centre of the frequencies (csrc/kdft_real_kernel.cuh).

Bound: the chain of the tensor core's accumulator is 48 products long, which truncates to about 1e-6 per axis (as with the
complex matrix it replaces); 5e-6 is asserted for up to three axes, 2e-5 for a solve of jittered nodes (growth below 10).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2002_03260_b200 as d
    return d


# a single quadruple, ragged stages (64 points), tiles (64 lines, 256 outputs) and batches, more than one table panel; the
# uniform 260 points have no folded form and run here too
@pytest.mark.parametrize("shape,axes", [((4, 8, 12), (0, 1, 2)), ((68, 60, 36), (0, 1, 2)), ((252, 20, 4), (0,)),
                                        ((12, 260, 20), (1,)), ((5, 4, 516), (2,)), ((8, 516, 36), (1,)), ((260, 4, 100), (0,)),
                                        ((2, 36, 256), (1, 2)), ((3, 128, 68), (1,))])
@pytest.mark.parametrize("on_output", [False, True])
@pytest.mark.parametrize("sign", [-1, +1])
def test_nodes_on_single_axes(lib, oracle, shape, axes, on_output, sign):
    from paper_2002_03260_b200 import inputs
    x = inputs.cube(shape, "normal", 401, device="cuda")
    full = inputs.sorted_nodes(shape, 402)
    nodes = [full[a] * 3.0 - 1.0 if a in axes else None for a in range(3)]     # any finite value, used modulo 1
    flags = lib.DFT3D_NODES_ON_OUTPUT if on_output else 0
    plan = lib.Plan(*shape, nodes=nodes, axes=axes, sign=sign, flags=flags)
    # input and output (all NaN before) between margins that must not change
    margin = 1 << 12
    bufs = [torch.full((x.numel() + 2 * margin,), 7.0 + 7.0j, dtype=torch.complex64, device="cuda") for _ in range(2)]
    xi, y = [b[margin:margin + x.numel()].view(shape) for b in bufs]
    xi.copy_(x)
    y.fill_(complex(float("nan"), float("nan")))
    plan(xi, y)
    torch.cuda.synchronize()
    plan.status()
    plan.destroy()
    assert all(bool((b[:margin] == 7.0 + 7.0j).all()) and bool((b[-margin:] == 7.0 + 7.0j).all()) for b in bufs)
    assert torch.equal(xi, x)
    want = x.cpu().numpy().astype(np.complex128)
    for a in axes:
        want = oracle.dft_axis(want, a, sign=sign, scale=1.0 / shape[a] if sign > 0 else 1.0, nodes=nodes[a],
                               nodes_on_output=on_output)
    assert oracle.rel_l2(y.cpu().numpy(), want) < 5e-6


@pytest.mark.parametrize("on_output", [False, True])
@pytest.mark.parametrize("shape,axis", [((20, 12, 8), 0), ((4, 260, 12), 1), ((3, 5, 68), 2)])
def test_solve_on_single_axes(lib, oracle, shape, axis, on_output):
    from paper_2002_03260_b200 import inputs
    x = inputs.cube(shape, "normal", 403, device="cuda")
    n = shape[axis]
    jitter = np.random.default_rng(404).uniform(-0.3, 0.3, n)
    nodes = [None] * 3
    nodes[axis] = (np.arange(n) + jitter) / n
    flags = lib.DFT3D_INVERSE_SOLVE | (lib.DFT3D_NODES_ON_OUTPUT if on_output else 0)
    plan = lib.Plan(*shape, nodes=nodes, axes=(axis,), sign=+1, flags=flags)
    y = plan(x)
    torch.cuda.synchronize()
    plan.status()
    plan.destroy()
    want = oracle.solve_axis(x.cpu().numpy().astype(np.complex128), axis, nodes[axis], nodes_on_output=on_output)
    assert oracle.rel_l2(y.cpu().numpy(), want) < 2e-5


def _one_axis(lib, x, axis, nodes, **kw):
    plan = lib.Plan(*x.shape, nodes=nodes, axes=(axis,), **kw)
    y = plan(x)
    torch.cuda.synchronize()
    plan.status()
    plan.destroy()
    return y


# (axis, points, nodes): every form of the kernel; the uniform 260 points have no folded form
RANGE_CASES = [(0, 64, "in"), (0, 64, "out"), (1, 64, "in"), (1, 64, "out"), (2, 64, "in"), (2, 64, "out"), (2, 260, "")]


def _range_case(lib, axis, n, where):
    shape = [4, 4, 4]
    shape[axis] = n
    nodes = [None] * 3
    if where:
        nodes[axis] = (np.arange(n) + np.random.default_rng(405).uniform(-0.3, 0.3, n)) / n
    return shape, nodes, lib.DFT3D_NODES_ON_OUTPUT if where == "out" else 0


@pytest.mark.parametrize("axis,n,where", RANGE_CASES)
@pytest.mark.parametrize("sign,unscaled", [(-1, False), (+1, False), (+1, True)])
@pytest.mark.parametrize("power", [100, 118, 123, 126, -100, -110])
def test_single_samples_scale_like_any_other(lib, axis, n, where, sign, unscaled, power):
    """A single sample spreads over its line with its own magnitude, so the result at 2^power is a normal number and
    equals the scaled result bit for bit: every scale is a power of two, and no step may leave the float range."""
    shape, nodes, flags = _range_case(lib, axis, n, where)
    flags |= lib.DFT3D_UNSCALED_INVERSE if unscaled else 0
    x = torch.zeros(shape, dtype=torch.complex64, device="cuda")
    at = [1, 2, 3]
    at[axis] = n // 3
    x[tuple(at)] = 0.75 - 0.5j
    y = _one_axis(lib, x, axis, nodes, sign=sign, flags=flags)
    z = _one_axis(lib, x * 2.0 ** power, axis, nodes, sign=sign, flags=flags)
    want = torch.view_as_real(y) * 2.0 ** power
    normal = want.abs() >= 2.0 ** -126         # small components of the phases may be subnormal: they round once more
    assert torch.equal(torch.view_as_real(z)[normal], want[normal])
    assert (torch.view_as_real(z) - want).abs().max().item() <= (2.0 ** -149 if power < 0 else 0.0)


@pytest.mark.parametrize("axis,n,where", RANGE_CASES)
@pytest.mark.parametrize("kind", ["inverse", "solve"])
def test_samples_at_the_top_of_the_range(lib, axis, n, where, kind):
    """Two samples that a pair sum adds, both components at 2.9e38: their sums and their products with the phases are no
    floats, the results (scaled by 1/n, or a solve's) are, and equal those of the samples 2^-40 as large."""
    if kind == "solve" and not where:
        pytest.skip("a solve needs nodes")
    shape, nodes, flags = _range_case(lib, axis, n, where)
    flags |= lib.DFT3D_INVERSE_SOLVE if kind == "solve" else 0
    x = torch.zeros(shape, dtype=torch.complex64, device="cuda")
    for j in (n // 2 - 3, n // 2 + 2):
        at = [1, 2, 3]
        at[axis] = j
        x[tuple(at)] = 2.9e38 + 2.9e38j
    y = torch.view_as_real(_one_axis(lib, torch.view_as_complex(torch.view_as_real(x) * 2.0 ** -40), axis, nodes, sign=+1, flags=flags))
    z = torch.view_as_real(_one_axis(lib, x, axis, nodes, sign=+1, flags=flags))
    assert torch.equal(z, y * 2.0 ** 40) and bool(torch.isfinite(z).all())


@pytest.mark.parametrize("axis,n,where", RANGE_CASES)
@pytest.mark.parametrize("sign", [-1, +1])
def test_subnormal_samples_lose_nothing_before_the_store(lib, axis, n, where, sign):
    """Dense data of 2^-140, multiples of 2^-149 all: the results are what the same samples 2^120 as large give, rounded
    to the grid of the subnormal numbers (half a step; one is asserted)."""
    shape, nodes, flags = _range_case(lib, axis, n, where)
    flags |= lib.DFT3D_UNSCALED_INVERSE if sign > 0 else 0
    g = torch.Generator(device="cuda").manual_seed(406)
    steps = torch.randint(-512, 513, shape + [2], generator=g, device="cuda").double()
    big = torch.view_as_complex((steps * 2.0 ** -29).float())
    small = torch.view_as_complex((steps * 2.0 ** -149).float())
    y = torch.view_as_real(_one_axis(lib, big, axis, nodes, sign=sign, flags=flags)).double() * 2.0 ** -120
    z = torch.view_as_real(_one_axis(lib, small, axis, nodes, sign=sign, flags=flags)).double()
    assert (z - y).abs().max().item() <= 2.0 ** -149
