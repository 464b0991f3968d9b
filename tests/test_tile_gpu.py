"""The tile kernel that small lattices run by default: the same state as the strip
kernel it replaces there (sizes at the edges of its tiles, single columns and rows
left over, lattices narrower than a tile), ghost columns that the strip kernel can
go on from, and its programmatic launches under stream capture."""
import numpy as np
import pytest

from paper_1405_2232_gb300 import inputs as I

pytestmark = pytest.mark.gpu

SIZES = [(32, 4), (33, 5), (31, 3), (3, 3), (5, 64), (64, 65), (97, 41), (160, 150), (257, 36)]


@pytest.fixture(scope="module")
def lb():
    import torch  # noqa: F401  (initialises CUDA in this process)
    from paper_1405_2232_gb300 import lb as _lb
    _lb.load()
    return _lb


def lattice(lb, nx, ny, precision, beta=1.3, strip=False, **kw):
    rho, T = I.slab_fields(nx, ny, width=max(2, nx // 2), noise=1e-3)
    shape = dict(tile_x=128, tile_y=0) if strip else {}
    return lb.Lattice(rho, T, nx=nx, ny=ny, precision=precision, beta=beta, psi_uses_local_T=0,
                      T_psi=0.85 * I.CS_TC, **shape, **kw)


@pytest.mark.parametrize("precision,eps", [("fp64", 0.0), ("fp32", 2.0 ** -24), ("fp16", 2.0 ** -11),
                                           ("bf16", 2.0 ** -8)])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_default_shape_equals_strip(lb, precision, eps, nx, ny):
    """Six steps: FP64 bit for bit; FP32 and 16-bit storage within one rounding
    (eps, of values below 0.2) per population, direction and step."""
    for thermal, beta in ((lb.LB_THERMAL_EQ24, 1.3), (lb.LB_THERMAL_EQ7, 1.0)):
        with lattice(lb, nx, ny, precision, beta, thermal=thermal) as A, \
                lattice(lb, nx, ny, precision, beta, strip=True, thermal=thermal) as B:
            A.step(6)
            B.step(6)
            A.synchronize()
            B.synchronize()
            for a, b in zip(A.populations(), B.populations()):
                assert np.abs(a - b).max() <= 6 * 9 * eps * 0.2


@pytest.mark.parametrize("precision", ["fp64", "fp32", "fp16"])
def test_kernels_alternate_on_one_state(lb, precision):
    """A caller-set wait limit runs the strip kernel: both kernels in turn on one
    context give the state of one of them (the ghost columns stay current)."""
    nx, ny = 70, 45
    with lattice(lb, nx, ny, precision) as A, lattice(lb, nx, ny, precision) as B:
        for k in range(6):
            lb.lb_set_wait_limit(A.ctx, 0 if k % 2 else 1 << 30)
            A.step(1)
        B.step(6)
        A.synchronize()
        tol = {"fp64": 0.0, "fp32": 2.0 ** -24, "fp16": 2.0 ** -11}[precision] * 6 * 9 * 0.2
        for a, b in zip(A.populations(), B.populations()):
            assert np.abs(a - b).max() <= tol


def test_steps_under_stream_capture(lb):
    """Captured steps replay as the same steps (an even number: the buffers end where
    they began)."""
    import torch
    s = torch.cuda.Stream()
    with lattice(lb, 64, 48, "fp32", stream=s) as A, lattice(lb, 64, 48, "fp32", stream=s) as B:
        A.step(2)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            A.step(4)
        with torch.cuda.stream(s):
            for _ in range(3):
                g.replay()
        B.step(2 + 4 * 3)
        s.synchronize()
        for a, b in zip(A.populations(), B.populations()):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("precision,eps", [("fp32", 2.0 ** -24), ("fp16", 2.0 ** -11), ("bf16", 2.0 ** -8)])
@pytest.mark.parametrize("nx,ny", [(3, 3), (33, 5), (5, 300), (64, 64), (90, 91), (256, 32), (257, 31), (128, 65)])
def test_runs_of_steps_equal_single_steps(lb, precision, eps, nx, ny):
    """Tiny lattices take a run of steps in one cluster of blocks, single steps as tiles
    (the last three sizes: both as tiles): the same state, odd and even runs, ghost columns
    included (the strip kernel goes on from them)."""
    ideal = dict(eos=lb.LB_EOS_IDEAL, a=0.0, b=0.0, R=0.5, G=1.0)
    for thermal, beta, kw in ((lb.LB_THERMAL_EQ24, 1.3, {}), (lb.LB_THERMAL_EQ7, 1.0, {}),
                              (lb.LB_THERMAL_EQ24, 0.0, ideal)):
        if kw:
            rho, T = I.sinusoid_fields(nx, ny, 1.0, 1.0, 0.05, mode=2, axis=0)
        else:
            rho, T = I.slab_fields(nx, ny, width=max(2, nx // 2), noise=1e-3)
            kw = dict(psi_uses_local_T=0, T_psi=0.85 * I.CS_TC)
        with lb.Lattice(rho, T, nx=nx, ny=ny, precision=precision, beta=beta, thermal=thermal, **kw) as A, \
                lb.Lattice(rho, T, nx=nx, ny=ny, precision=precision, beta=beta, thermal=thermal, **kw) as B:
            A.step(17)
            lb.lb_set_wait_limit(A.ctx, 1 << 30)
            A.step(1)
            lb.lb_set_wait_limit(A.ctx, 0)
            A.step(18)
            for _ in range(36):
                B.step(1)
            A.synchronize()
            B.synchronize()
            for a, b in zip(A.populations(), B.populations()):
                assert np.abs(a - b).max() <= 36 * 9 * eps * 0.2
