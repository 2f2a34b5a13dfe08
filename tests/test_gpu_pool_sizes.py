"""Step-kernel builds that are chosen by the size of a pool that is not reordered, against the
general kernel (fte_advance_noalloc; for ensembles the shared-memory layout): states, counts and
ledger equal to the bit on both sides of every line, which lie at so many particles per SM (8 warps,
one wave of 16 warps, 20 warps)."""
import dataclasses

import numpy as np
import pytest

from fte_inputs import amr, configs
from fte_inputs.configs import Observer

pytestmark = pytest.mark.gpu
STEPS = 12


@pytest.fixture(scope="module")
def grids():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_12164_gb300 import api, build
    build.build()
    out = {}
    for radial in ("linear", "log"):
        spec = amr.AmrSpec(nbr=4, nbt=2, nbp=4, bsize=8, levels=2, radial=radial, n_snap=2, periodic=False,
                           dt_snap=3600.0)
        leaves = amr.build_leaves(spec, amr.divv_refiner(spec, threshold=8e-6, r_from=0.9))
        bg = api.AmrBackground(spec, leaves)
        api.fte_load_background(bg, amr.fields(spec, leaves))
        api.fte_amr_prepare(bg)
        for dtype, layout in (("f32", "cell"), ("f32", "pair"), ("bf16", "cell")):
            img = bg
            if (dtype, layout) != ("f32", "cell"):
                img = api.AmrBackground(spec, leaves, dtype=dtype, layout=layout, share=bg)
                api.fte_quantize_background(img, bg)
            out[radial, dtype, layout] = img
    return out


def _run(bg, n, noalloc):
    from paper_2404_12164_gb300 import api
    w = configs.cir_uniform_1e6()
    t = dict(ne=8, t_lo=0.0, t_hi=STEPS * 10.0, nt=4, e_lo=0.01, e_hi=10.0)
    obs = [Observer(kind="shell", r=1.2, dr=0.05, **t), Observer(kind="shell", r=1.6, dr=0.1, **t)]
    pool, tally = api.Particles(n), api.Tally(obs)
    api.fte_inject(pool, bg, dataclasses.replace(w.inject, divv_max=None, energy="powerlaw", seed=5), n, tally)
    prm = dataclasses.replace(w.params, lambda_par=0.1, dt=10.0, seed=5, sort_every=0)
    (api.fte_advance_noalloc if noalloc else api.fte_advance)(pool, bg, prm, tally, 0, STEPS)
    return {**pool.state(), "C": tally.C.cpu().numpy(), "ledger": tally.ledger_n.cpu().numpy()}


@pytest.mark.parametrize("per_sm,more", [(256, 0), (256, 1), (640, -1), (640, 1), (1100, 7)])
@pytest.mark.parametrize("layout", ["cell", "pair"])
def test_amr_linear_r(grids, layout, per_sm, more):
    import torch
    n = torch.cuda.get_device_properties(0).multi_processor_count * per_sm + more
    bg = grids["linear", "f32", layout]
    got, ref = _run(bg, n, False), _run(bg, n, True)
    assert ref["C"].sum() > n // 10
    for k in ref:
        assert np.array_equal(got[k], ref[k]), k


@pytest.mark.parametrize("per_sm,more", [(512, 0), (512, 1), (1100, 7)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_amr_log_r(grids, dtype, per_sm, more):
    """One wave: up to it with the observers' reach test, above it without."""
    import torch
    n = torch.cuda.get_device_properties(0).multi_processor_count * per_sm + more
    bg = grids["log", dtype, "cell"]
    got, ref = _run(bg, n, False), _run(bg, n, True)
    assert ref["C"].sum() > n // 10
    for k in ref:
        assert np.array_equal(got[k], ref[k]), k


@pytest.mark.parametrize("per_sm,more", [(512, 0), (512, 1), (1100, 7)])
@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("threads", [128, 256])
@pytest.mark.parametrize("sort", [0, 8])
def test_ensemble(dtype, threads, per_sm, more, sort):
    """The ensemble kernels with the options fixed (global tally) against the general ones (shared)."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_12164_gb300 import api, build
    build.build()
    n = torch.cuda.get_device_properties(0).multi_processor_count * per_sm + more
    w = configs.scaled(configs.cir_uniform_1e6(), nr=64, nth=16, nph=32, n_snap=3)
    w.grid = dataclasses.replace(w.grid, periodic=False)
    cell = api.Background(w.grid)
    api.fte_load_background(cell, configs.build_background(w))
    bg = cell
    if dtype != "f32":
        bg = api.Background(w.grid, dtype=dtype)
        api.fte_quantize_background(bg, cell)
    t = dict(ne=4, t_lo=0.0, t_hi=STEPS * 10.0, nt=3, e_lo=0.01, e_hi=10.0)
    obs = [Observer(kind="shell", r=1.2, dr=0.05, **t), Observer(kind="slab", r=-1.0, dr=0.1, **t)]
    sets = [configs.EnsembleSet(0.1 + 0.3 * s, w.params.q, 0.05, 0.048, s, s, c,
                                dataclasses.replace(w.inject, divv_max=None, seed=s, set_id=s, e0=0.02 * (s + 1)))
            for s, c in enumerate((n // 3, 1, n - n // 3 - 1))]
    prm = dataclasses.replace(w.params, dt=10.0, sort_every=sort)
    runs = []
    for layout in ("global", "shared"):
        pool, tally = api.Particles(n), api.Tally(obs, n_sets=3)
        api.fte_inject_batched(pool, bg, sets, tally)
        api.fte_advance_batched(pool, bg, prm, sets, tally, 0, STEPS,
                                config={"threads": threads, "steps_per_launch": 8, "tally_layout": layout})
        runs.append({**pool.state(), "C": tally.C.cpu().numpy(), "ledger": tally.ledger_n.cpu().numpy()})
    assert runs[0]["C"].sum() > n // 10
    for k in runs[0]:
        assert np.array_equal(runs[0][k], runs[1][k]), k
