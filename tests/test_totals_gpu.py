"""Mass and energy totals of FP32 states whose populations spread over many binades and
signs: the FP64 sums of the stored floats, as nine FP64 additions per site give them.

One block of equal sites, so that the reduction over the lattice adds equal doubles:
exact within a warp, one rounding for each of the eight warps.  With the eight
additions of a site that is at most 16 roundings of 2^-53: 2^-49 of the sum (its
greatest term carries it).  A site's rounding errors kept in one float miss it by
2^-46.3 (seed 37) and 2^-47.0 (seed 17)."""
import math

import numpy as np
import pytest


def populations(seed):
    r = np.random.default_rng(seed)
    return np.concatenate([[0.15], 0.05 * 10.0 ** -r.uniform(0, 9, 8) * r.choice([-1, 1], 8)]).astype(np.float32)


@pytest.mark.gpu
@pytest.mark.parametrize("seeds", [(37, 17), (17, 37), (14, 28)])
def test_fp32_totals_are_the_fp64_sums(seeds):
    from paper_1405_2232_gb300 import lb
    nx, ny = 32, 8
    f, g = (populations(s).astype(np.float64) for s in seeds)
    field = lambda v: np.ascontiguousarray(np.broadcast_to(v[:, None, None], (9, ny, nx)))
    with lb.Lattice(np.full((ny, nx), 0.1), np.full((ny, nx), 0.08), nx=nx, ny=ny, precision="fp32",
                    psi_uses_local_T=0, T_psi=0.08) as L:
        L.set_populations(field(f), field(g))
        back = L.populations()
        assert np.array_equal(back[0], field(f)) and np.array_equal(back[1], field(g))
        mass, energy = L.totals()[:2]
    for total, v in ((mass, f), (energy, g)):
        exact = nx * ny * math.fsum(v)
        assert abs(total - exact) <= 2.0 ** -49 * exact
