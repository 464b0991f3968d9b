"""The kernels that a lattice may step on (strips, tiles, a run of steps in one cluster)
do the same arithmetic on a site and round it to storage the same way: the same bits, in
every storage mode.  Slabs of a lattice, which may step on another kernel than the whole,
and runs that are cut into calls rely on it."""
import numpy as np
import pytest

from paper_1405_2232_gb300 import inputs as I

pytestmark = pytest.mark.gpu
PRECISIONS = ["fp64", "fp32", "fp16", "bf16"]
IDEAL = dict(a=0.0, b=0.0, R=0.5, G=1.0)


@pytest.fixture(scope="module")
def lb():
    from paper_1405_2232_gb300 import lb as _lb
    _lb.load()
    return _lb


def cases(lb, nx, ny):
    """Both treatments and the three force forms (beta = 0: an ideal gas, whose psi^2
    keeps its sign)."""
    slab = I.slab_fields(nx, ny, width=max(2, nx // 2), noise=1e-3)
    wave = I.sinusoid_fields(nx, ny, 1.0, 1.0, 0.05, mode=2 if nx > 4 else 1, axis=0)
    psi = dict(psi_uses_local_T=0, T_psi=0.85 * I.CS_TC)
    return [(*slab, dict(thermal=lb.LB_THERMAL_EQ24, beta=1.3, **psi)),
            (*slab, dict(thermal=lb.LB_THERMAL_EQ7, beta=1.0)),
            (*wave, dict(thermal=lb.LB_THERMAL_EQ24, beta=0.0, eos=lb.LB_EOS_IDEAL, **IDEAL))]


def state(L):
    L.synchronize()
    return L.populations()


def moved(a, b):
    """Every plane took part, at the interfaces at least."""
    return all(np.mean(a[k][i] != b[k][i]) > 0.02 for k in range(2) for i in range(9))


@pytest.mark.parametrize("prec", PRECISIONS)
@pytest.mark.parametrize("nx,ny", [(33, 5), (64, 64), (90, 91), (257, 36), (333, 200)])
def test_kernels_give_the_same_bits(lb, prec, nx, ny):
    strip = dict(tile_x=128, tile_y=0)
    for rho, T, kw in cases(lb, nx, ny):
        kw = dict(kw, nx=nx, ny=ny, precision=prec)
        with lb.Lattice(rho, T, **kw, **strip) as L:
            start = state(L)
            L.step(20)
            ref = state(L)
        assert moved(start, ref)
        for shape, calls in (({}, [20]), ({}, [1] * 20), ({}, [17, 3]), (dict(tile_x=32, tile_y=8), [20]),
                             (dict(tile_x=64, tile_y=4), [20])):
            with lb.Lattice(rho, T, **kw, **shape) as L:
                for n in calls:
                    L.step(n)
                got = state(L)
            assert all(np.array_equal(a, b) for a, b in zip(got, ref)), (shape, calls, kw["beta"])


@pytest.mark.parametrize("prec", PRECISIONS)
@pytest.mark.parametrize("nx,ny,world,steps", [(1100, 2000, 4, 5), (64, 96, 2, 35)])
def test_slabs_of_default_shape_match_the_whole(lb, prec, nx, ny, world, steps):
    """The whole on strips (1100 x 2000) or in a cluster (64 x 96, FP32 and 16-bit), its
    slabs on tiles."""
    import torch
    from paper_1405_2232_gb300 import decomp as D
    rho, T = I.slab_fields(nx, ny, noise=1e-3)
    kw = dict(precision=prec, psi_uses_local_T=0, T_psi=0.85 * I.CS_TC, beta=1.3)
    stream = torch.cuda.Stream()
    slabs = [D.SlabLattice(rho, T, rank=r, world=world, stream=stream, **kw) for r in range(world)]
    try:
        with lb.Lattice(rho, T, nx=nx, ny=ny, **kw) as W:
            W.step(steps)
            D.step_local(slabs, steps)
            whole = state(W)
        parts = [s.populations() for s in slabs]
        for k in range(2):
            assert np.array_equal(np.concatenate([p[k] for p in parts], axis=1), whole[k])
    finally:
        for s in slabs:
            s.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_batch_kernels_give_the_same_bits(lb, prec):
    """Batches on tiles (the default) and on strips; in FP64 lone lattices too."""
    sizes = [(3, 3), (33, 15), (64, 5), (31, 130), (97, 64), (260, 70)]
    for k in range(3):
        specs = [cases(lb, nx, ny)[k] for nx, ny in sizes]
        params = [lb.lb_params_default(nx=nx, ny=ny, precision=prec, **kw) for (nx, ny), (_, _, kw) in zip(sizes, specs)]
        rhos, Ts = [s[0] for s in specs], [s[1] for s in specs]
        with lb.Batch(params, rhos, Ts) as A, lb.Batch(params, rhos, Ts) as B:
            B.chunk_rows = 16
            A.step(25)
            B.step(25)
            for d, p in enumerate(params):
                a, b = A.fields(d), B.fields(d)
                assert not np.array_equal(a[0], rhos[d])
                assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]), (k, sizes[d])
                if prec == "fp64":
                    with lb.Lattice(rhos[d], Ts[d], tile_x=128, tile_y=0, nx=p.nx, ny=p.ny, precision=prec,
                                    **specs[d][2]) as L:
                        L.step(25)
                        m = L.moments()
                    assert np.array_equal(a[0], m[0]) and np.array_equal(a[1], m[3]), (k, sizes[d])


@pytest.mark.parametrize("prec,thermal,nx,ny,shape", [
    ("fp32", None, 64, 64, (0, 0)), ("fp64", None, 90, 70, (0, 0)), ("bf16", None, 300, 200, (0, 0)),
    ("fp32", "fd", 128, 96, (0, 0)), ("fp32", None, 2048, 1100, (256, 0)), ("fp64", None, 1100, 1000, (128, 0))])
def test_a_context_from_the_reported_parameters_runs_the_same_kernels(lb, prec, thermal, nx, ny, shape):
    """lb_get_params of a context without a shape: the strip kernel's width where it runs, else
    no shape; a context created from the parameters reports them again.  An explicit
    shape is reported as it is."""
    rho, T = np.full((ny, nx), 0.1), np.full((ny, nx), 0.075)
    kw = dict(nx=nx, ny=ny, precision=prec, thermal=lb.LB_THERMAL_FD26 if thermal else lb.LB_THERMAL_EQ24)
    with lb.Lattice(rho, T, **kw) as L:
        p = lb.lb_get_params(L.ctx)
    assert (p.tile_x, p.tile_y) == shape
    with lb.Lattice(rho, T, **{n: getattr(p, n) for n, _ in p._fields_}) as L:
        q = lb.lb_get_params(L.ctx)
    assert (q.tile_x, q.tile_y) == shape
    width = 128 if prec == "fp64" else 256
    with lb.Lattice(rho, T, tile_x=width, tile_y=0, **kw) as L:
        q = lb.lb_get_params(L.ctx)
    assert (q.tile_x, q.tile_y) == (width, 0)


@pytest.mark.parametrize("prec", ["fp16", "bf16"])
@pytest.mark.parametrize("nx,ny,tiles", [(1016, 765, True), (1024, 896, True), (1032, 896, False), (1024, 1024, False)])
def test_16bit_lattices_leave_the_tiles_where_strips_are_faster(lb, prec, nx, ny, tiles):
    """1024^2: 24.8 - 26.1 us per step on strips, 26.2 - 26.6 on tiles; 1016 x 765: 20.5 and
    18.6 at least."""
    with lb.Lattice(np.full((ny, nx), 0.1), np.full((ny, nx), 0.075), nx=nx, ny=ny, precision=prec) as L:
        assert lb.lb_get_params(L.ctx).tile_x == (0 if tiles else 256)


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_cluster_runs_under_stream_capture(lb, prec):
    """A captured run of an even number of steps replays in place."""
    import torch
    s = torch.cuda.Stream()
    rho, T = I.slab_fields(64, 48, noise=1e-3)
    kw = dict(nx=64, ny=48, precision=prec, psi_uses_local_T=0, T_psi=0.85 * I.CS_TC)
    with lb.Lattice(rho, T, stream=s, **kw) as A, lb.Lattice(rho, T, stream=s, **kw) as B:
        g = torch.cuda.CUDAGraph()
        s.synchronize()
        with torch.cuda.graph(g, stream=s):
            A.step(32)
        with torch.cuda.stream(s):
            for _ in range(3):
                g.replay()
        for _ in range(96):
            B.step(1)
        a, b = state(A), state(B)
        assert all(np.array_equal(x, y) for x, y in zip(a, b))
