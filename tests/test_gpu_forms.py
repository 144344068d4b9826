"""GPU tests of kernel forms beside one another: where the packages of a dust
source start, and the descent to the leaf within a pass against one level per
pass."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1206_3710_gb300 import synth  # noqa: E402


@pytest.fixture(scope="module")
def rt():
    from paper_1206_3710_gb300 import build
    build.build()
    from paper_1206_3710_gb300 import rt as _rt
    return _rt


DEV = "cuda:0"


def _zeros(*shape):
    return torch.zeros(shape, dtype=torch.float64, device=DEV)


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("n", [1, 255, 1023, 1024, 1025, 2049])
def test_dust_packages_start_in_their_cells(rt, orc, n, precision):
    """Cell c sends floor(E / w + u) packages of bin b, u from its own Philox
    block: at the edges of the chunks that the counts are taken in, the
    deposits per cell, and the energy per bin and cell, are those packages'.
    The medium is opaque (1e12 optical depths a cell) and does not scatter: a
    package deposits all of its energy in the cell it starts in."""
    ctx = rt.Context(0)
    desc = synth.uniform_tree((n, 1, 1), (n * 1e15, 1e15, 1e15), 1e-19)
    g = rt.Grid(ctx, desc)
    lam = np.array([3.0, 30.0, 300.0])
    kabs, dnu = np.array([100.0, 10.0, 0.1]), synth.bin_dnu(lam)
    T = np.random.default_rng(n).uniform(0.0, 60.0, n)
    Td = torch.from_numpy(T).to(DEV)
    em = _zeros(3, n)
    tot = rt.rt_dust_emission(ctx, g, Td, lam, kabs, dnu, em)
    em = em.cpu().numpy()
    budget, seed = 5 * n + 7, 17
    u = np.array([[orc.philox4x32(np.array([c, 0x80000000, 0, b], np.uint32), np.array([seed, 0], np.uint32))[0]
                   for c in range(n)] for b in range(3)], dtype=np.float64)
    w = tot / budget
    k = np.floor(em / w[:, None] + (u + 0.5) * 2.0 ** -32).astype(np.int64)
    # the neighbour's packages are another number: a shifted sum would show
    assert n == 1 or not np.array_equal(k, np.roll(k, 1, axis=1))
    optics = synth.Optics(lambda_um=lam, kappa_ext=np.full(3, 1e16), albedo=np.zeros(3), g_hg=np.zeros(3), dnu=dnu)
    absorbed, hits = _zeros(3, n), torch.zeros(n, dtype=torch.int32, device=DEV)
    led = rt.rt_trace(ctx, g, [rt.DustSource(Td, lam, kabs, dnu)], optics, absorbed, seed=seed, precision=precision,
                      packets_per_bin=budget, hits=hits)
    assert led["n_packets"] == k.sum()
    np.testing.assert_array_equal(hits.cpu().numpy(), k.sum(axis=0))
    # (a weight is rounded to f32 in the FP32 tracer)
    np.testing.assert_allclose(absorbed.cpu().numpy() / w[:, None], k, rtol=1e-6 if precision == 32 else 1e-12, atol=0)


def _refined(depth):
    """A 2^3 root, all of it refined to level 2, then around one corner: from
    depth 2 on more than half of the cells lie below level 1, so that launches
    keep the path above the leaf."""
    rng = np.random.default_rng(depth)
    desc = synth.grow_tree((2, 2, 2), (8e16,) * 3, depth,
                           lambda l, x, y, z: 1e-20 * 10.0 ** rng.uniform(-1, 1, x.size),
                           lambda l, x, y, z, r: (l < 2) | ((x < 2) & (y < 2) & (z < 2)))
    below = desc.n_cells - 8 - 64
    assert 2 * below >= desc.n_cells
    optics = synth.Optics(lambda_um=np.array([0.5, 2.0]), kappa_ext=np.array([3e3, 5e2]), albedo=np.array([0.6, 0.4]),
                          g_hg=np.array([0.4, 0.0]), dnu=np.array([1e13, 1e13]))
    return desc, optics, [synth.Source("external", bin_energy=np.array([1.0, 2.0]))]


_NPK = 3000
_OBS = synth.Observers(dirs=np.array([[0.36, 0.48, 0.8], [0.0, 0.0, -1.0]]), ups=np.array([[0.0, 1.0, 0.0]] * 2),
                       nx=24, ny=20, fov=(1e17, 1e17))


def _job(rt, ctx, depth, job, precision):
    desc, optics, src = _refined(depth)
    g = rt.Grid(ctx, desc)
    return rt.Job(g, src, optics, absorbed=_zeros(2, g.n_cells), observers=_OBS, images=_zeros(2, 2, _OBS.ny, _OBS.nx),
                  seed=5, job=job, packets_per_bin=_NPK, packet_log=_zeros(2 * _NPK, 10), precision=precision)


def _same(a, b):
    (ja, la), (jb, lb) = a, b
    assert la["n_scatter"] > 500 and la["n_peel_cross"] > 1000
    for k in ("n_cross", "n_scatter", "n_peel_cross", "n_peel_out"):
        assert la[k] == lb[k], k
    np.testing.assert_array_equal(ja.params["packet_log"].cpu().numpy(), jb.params["packet_log"].cpu().numpy())
    # the order of the FP64 additions differs
    for x, y in ((ja.absorbed, jb.absorbed), (ja.images, jb.images)):
        x, y = x.cpu().numpy(), y.cpu().numpy()
        np.testing.assert_allclose(y, x, rtol=1e-12, atol=1e-14 * x.max())


@pytest.mark.parametrize("depth", [2, 8])
def test_fp32_descent_forms(rt, depth):
    """FP32: a grid of at most 8 levels descends to the leaf within a pass
    alone, and a level per pass beside a 9-level one."""
    ctx = rt.Context(0)
    alone, beside = [_job(rt, ctx, depth, 0, 32)], [_job(rt, ctx, depth, 0, 32), _job(rt, ctx, 9, 1, 32)]
    _same((alone[0], rt.rt_trace_batch(ctx, alone)[0]), (beside[0], rt.rt_trace_batch(ctx, beside)[0]))


@pytest.mark.parametrize("depth", [2, 3, 8, 10])
def test_fp64_descent_forms(rt, depth):
    """FP64: untiled launches descend to the leaf within a pass whatever the
    depth, the rounds of a tiled one a level per pass."""
    ctx = rt.Context(0)
    res = []
    for edge in (0, 1):
        ctx.set_tiles(edge)
        j = _job(rt, ctx, depth, 0, 64)
        led = rt.rt_trace_batch(ctx, [j])[0]
        assert led["n_tiles"] == (8 if edge else 0)
        res.append((j, led))
    _same(*res)
