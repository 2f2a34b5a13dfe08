"""The adjoint's forward, replay and backward kernels with the grid and physics options fixed (cell
records) against the general ones (pair records): end states, J per particle and gradients per
particle equal to the bit, on uniform and block-AMR grids with linear and logarithmic r, in FP32 and
in 16 bits, reordered and not, on both sides of one wave, where the block size changes."""
import dataclasses
import math

import numpy as np
import pytest

from fte_inputs import amr, configs
from fte_inputs.configs import InjectSpec, Params, SmoothObserver

pytestmark = pytest.mark.gpu
DEG = math.pi / 180
STEPS, EVERY = 40, 16
OBS = SmoothObserver(r_o=1.3, sigma_r=0.2, e_c=0.05, sigma_lnE=0.7, t_c=200.0, sigma_t=300.0)
INJ = InjectSpec(region="box", r1=1.0, r2=1.6, th1=86 * DEG, th2=94 * DEG, ph1=math.pi, ph2=2 * math.pi,
                 divv_max=None, energy="powerlaw", e1=0.05, e2=0.5, gamma=3.0, weight="r-2", seed=6)


@pytest.fixture(scope="module")
def grids():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_12164_gb300 import api, build
    build.build()
    out = {}
    w = configs.scaled(configs.cir_uniform_1e6(), nr=64, nth=16, nph=32, n_snap=3)
    for radial in ("linear", "log"):
        g = dataclasses.replace(w.grid, radial=radial, periodic=False)
        bg = api.Background(g)
        w.grid = g
        api.fte_load_background(bg, configs.build_background(w))
        out[radial] = bg
        spec = amr.AmrSpec(nbr=4, nbt=2, nbp=4, bsize=8, levels=2, radial=radial, n_snap=2, periodic=False,
                           dt_snap=3600.0)
        leaves = amr.build_leaves(spec, amr.divv_refiner(spec, threshold=8e-6, r_from=0.9))
        bg = api.AmrBackground(spec, leaves)
        api.fte_load_background(bg, amr.fields(spec, leaves))
        api.fte_amr_prepare(bg)
        bg.leaves = leaves
        out["amr_" + radial] = bg
    return out


def _stored(bg, dtype, layout):
    from paper_2404_12164_gb300 import api
    if dtype == "f32" and layout == "cell":
        return bg
    if isinstance(bg, api.AmrBackground):
        out = api.AmrBackground(bg.grid, bg.leaves, dtype=dtype, layout=layout, share=bg)
    else:
        out = api.Background(bg.grid, dtype=dtype, layout=layout)
    api.fte_quantize_background(out, bg)
    return out


def _run(bg, prm, n):
    import torch
    from paper_2404_12164_gb300 import api
    pool, tally = api.Particles(n), api.Tally([])
    api.fte_inject(pool, bg, INJ, n, tally)
    adj = api.Adjoint(bg, prm, OBS, 0, STEPS, EVERY)
    _, Ji = adj.forward(pool, per_particle=True)
    _, pp = adj.reverse(pool, INJ, per_particle=True)
    torch.cuda.synchronize()
    return {**pool.state(), "J_i": Ji.cpu().numpy(), "per_particle": pp.cpu().numpy()}


@pytest.mark.parametrize("grid", ["linear", "log", "amr_linear", "amr_log"])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("sort,per_sm,more", [(0, 0, 3001), (16, 0, 3001), (0, 512, 0), (0, 512, 1), (0, 700, 9),
                                              (16, 700, 9)])
def test_fixed_options_equal_the_general_build(grids, grid, dtype, sort, per_sm, more):
    import torch
    n = torch.cuda.get_device_properties(0).multi_processor_count * per_sm + more
    prm = Params(dmumu="qlt", lambda_par=0.1, dt=10.0, seed=5, sort_every=sort)
    a, b = (_run(_stored(grids[grid], dtype, layout), prm, n) for layout in ("cell", "pair"))
    assert np.count_nonzero(a["J_i"]) > n // 2
    assert np.count_nonzero(a["per_particle"][:, 1:5]) > n // 2
    for k in a:
        assert np.array_equal(a[k], b[k]), k
