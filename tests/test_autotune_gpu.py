"""Autotuner on the GPU: the chosen shape is the fastest measured one, shapes
that do not apply are skipped, a tuned lattice gives the same results, and
tuning a batch leaves its state untouched."""
import math

import numpy as np
import pytest

import oracle as O
from paper_1405_2232_gb300 import autotune as A
from paper_1405_2232_gb300 import inputs as I


@pytest.fixture(scope="module")
def lb():
    from paper_1405_2232_gb300 import lb as _lb
    _lb.load()
    return _lb


@pytest.mark.gpu
@pytest.mark.parametrize("prec,nx,ny,invalid", [
    ("fp32", 512, 256, []),
    ("fp64", 256, 128, [0]),          # the FP64 strip kernel is 128 wide only
    ("fp32", 130, 64, []),            # any nx: the strip kernel's row copies are rounded up
    ("bf16", 1024, 512, []),
])
def test_autotune_picks_the_fastest_valid_shape(lb, prec, nx, ny, invalid):
    p = lb.lb_params_default(nx=nx, ny=ny, precision=prec, beta=1.3, psi_uses_local_T=0,
                             T_psi=0.075)
    best, ms = lb.lb_autotune(p, 6)
    for k in range(lb.LB_TUNE_N):
        assert math.isnan(ms[k]) == (k in invalid), (k, ms)
    k_best = int(np.nanargmin(ms))
    assert (best.tile_x, best.tile_y) == lb.lb_tune_candidate(k_best)
    assert best.nx == nx and best.precision == p.precision and best.beta == 1.3


@pytest.mark.gpu
def test_tuned_lattice_matches_default_bit_for_bit(lb, tmp_path):
    rho, T = I.slab_fields(96, 64)
    p = lb.lb_params_default(nx=96, ny=64, precision="fp64")
    q = A.tuned_params(p, A.TuneCache(str(tmp_path / "t.json")), steps=4)
    out = []
    for par in (p, q):
        with lb.Lattice(rho, T, **{n: getattr(par, n) for n, _ in par._fields_}) as L:
            L.step(50)
            out.append(L.populations())
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


@pytest.mark.gpu
def test_batch_autotune_restores_state(lb):
    specs = [(64, 48), (132, 36), (256, 200), (36, 260)]
    params, rhos, Ts = [], [], []
    for k, (nx, ny) in enumerate(specs):
        rho, T = I.droplet_fields(nx, ny, min(nx, ny) // 4, rho_l=0.3, rho_g=0.04)
        params.append(lb.lb_params_default(nx=nx, ny=ny, precision="fp64", tau_f=0.8 + 0.1 * k,
                                           psi_uses_local_T=0, T_psi=0.085))
        rhos.append(rho)
        Ts.append(np.full((ny, nx), 0.085))
    with lb.Batch(params, rhos, Ts) as A_, lb.Batch(params, rhos, Ts) as B_:
        A_.step(10)
        B_.step(10)
        before = [A_.fields(d) for d in range(len(specs))]
        rows, ms = A_.autotune(4)
        assert rows in (16, 32, 64, 128) and A_.chunk_rows == rows
        assert np.all(np.isfinite(ms)) and ms[[16, 32, 64, 128].index(rows)] == ms.min()
        assert A_.time == 10
        after = [A_.fields(d) for d in range(len(specs))]
        for (r0, t0), (r1, t1) in zip(before, after):
            assert np.array_equal(r0, r1) and np.array_equal(t0, t1)
        A_.step(30)
        B_.step(30)
        for d in range(len(specs)):
            (ra, ta), (rb, tb) = A_.fields(d), B_.fields(d)
            assert np.array_equal(ra, rb) and np.array_equal(ta, tb), d
        A_.chunk_rows = 16
        A_.step(2)
        B_.step(2)
        for d in range(len(specs)):
            assert np.array_equal(A_.fields(d)[0], B_.fields(d)[0]), d


def uniform_batch(lb, sizes):
    params = [lb.lb_params_default(nx=nx, ny=ny, precision="fp32", psi_uses_local_T=0, T_psi=0.075) for nx, ny in sizes]
    return params, [np.full((ny, nx), 0.1) for nx, ny in sizes], [np.full((ny, nx), 0.075) for nx, ny in sizes]


@pytest.mark.gpu
def test_batch_steps_on_the_same_kernel_with_a_cold_and_a_warm_cache(lb, tmp_path):
    cache = str(tmp_path / "t.json")
    args = uniform_batch(lb, [(64, 64), (90, 70)])
    kernels = []
    for _ in range(2):
        with lb.Batch(*args) as B:
            untuned = B.tile_rows
            rows = A.tuned_batch(B, A.TuneCache(cache), steps=4)
            assert B.chunk_rows == rows
            kernels.append(B.tile_rows)
    assert untuned > 0 and kernels[0] == kernels[1]


@pytest.mark.gpu
def test_tuned_strips_hold_for_half_of_the_sites(lb):
    """A tuning that chose strips applies while half of its sites are active; then the
    library's rule: tiles for the domains that are left, narrow ones among them (the
    longest tile list).  A height set by the caller stays."""
    # 2.6 million sites, too many for tiles; all but two domains are at rest and converge
    sizes = [(1024, 1024), (1024, 1024), (3, 100000), (5, 50000)]
    params, rhos, Ts = uniform_batch(lb, sizes)
    for d in (2, 3):
        nx, ny = sizes[d]
        rhos[d] = 0.1 + 1e-3 * np.sin(2 * np.pi * np.arange(ny) / 100)[:, None] * np.ones((1, nx))
    with lb.Batch(params, rhos, Ts) as B, lb.Batch(params, rhos, Ts) as C:
        B.apply_tuning(32, False)
        C.chunk_rows = 32
        assert (B.tile_rows, C.tile_rows) == (0, 0) and B.chunk_rows == 32
        rb, rc = B.run(1e-7, K=20, max_steps=40), C.run(1e-7, K=20, max_steps=40)
        assert rb[2][:2].tolist() == [0, 0] and rb[2][2] == lb.LB_ERR_NOT_CONVERGED
        assert B.tile_rows > 0 and C.tile_rows == 0 and B.chunk_rows == 32
        assert np.array_equal(rb[0], rc[0])
        for d in range(len(sizes)):
            assert np.array_equal(B.fields(d)[0], C.fields(d)[0]), d
        with pytest.raises(lb.LbError):
            B.apply_tuning(8, False)


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_batch_state_around_a_tuning_read_anew(lb, prec):
    """Mass, energy and fields after a tuning, each from the state (a check), equal those
    before; a step in between changes them."""
    rho, T = I.slab_fields(70, 45, noise=1e-3)
    p = [lb.lb_params_default(nx=70, ny=45, precision=prec, psi_uses_local_T=0, T_psi=0.08)] * 2
    with lb.Batch(p, [rho, rho], [T, T]) as B:
        B.step(7)
        before = B.check()[1:3], B.fields(1)
        B.autotune(3)
        after = B.fields(1), B.check()[1:3]
        B.step(1)
        moved = B.fields(1)
    assert np.array_equal(before[0], after[1])
    for k in range(2):
        assert np.array_equal(before[1][k], after[0][k]) and not np.array_equal(before[1][k], moved[k])


@pytest.mark.gpu
@pytest.mark.parametrize("prec,nx,ny", [("fp32", 64, 64), ("fp64", 90, 70)])
def test_tuned_lattice_is_not_slower_than_the_default(lb, tmp_path, prec, nx, ny):
    """Tuning keeps the library's choice where no shape beats it (64^2 FP32: 1.2 us per
    step in one cluster against 2.2 and more), so the tuned time is within the noise
    of two timings (20%) of it."""
    p = lb.lb_params_default(nx=nx, ny=ny, precision=prec, psi_uses_local_T=0, T_psi=0.075)
    q = A.tuned_params(p, A.TuneCache(str(tmp_path / "t.json")), steps=200)
    if prec == "fp32":
        assert (q.tile_x, q.tile_y) == (0, 0)
    assert lb.lb_time_step(q, 400) <= 1.2 * lb.lb_time_step(p, 400)
    with pytest.raises(lb.LbError):
        lb.lb_time_step(lb.lb_params_default(nx=nx, ny=ny, tile_x=7, tile_y=7), 4)
