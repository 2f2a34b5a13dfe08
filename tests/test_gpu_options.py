"""Step kernels with the common options fixed at compile time against the general one.

fte_advance picks such a kernel by grid kind and physics options; fte_advance_noalloc always runs
the general kernel (options read from the parameters, shared-memory tally).  The arithmetic is the
same, so the particle states and the tally counts must be equal to the bit over every combination
that the choice looks at: each grid kind and storage form, each option switched off the common
value, reordered or not, and observer sets on both sides of the four that the reach test unrolls."""
import dataclasses
import math

import numpy as np
import pytest

from fte_inputs import amr, configs
from fte_inputs.configs import Observer

pytestmark = pytest.mark.gpu
DEG = math.pi / 180
N, STEPS = 3001, 70

COMMON = dict(dmumu="qlt", p_update="exp", dvdt_term=1, lambda_par=0.1, dt=10.0, seed=5)
OPTIONS = {"common": {}, "paper": dict(dmumu="paper"), "iso": dict(dmumu="iso"), "euler": dict(p_update="euler"),
           "no_dvdt": dict(dvdt_term=0), "rigidity": dict(p_ref=0.01, alpha=0.3), "cross_field": dict(lambda_perp=3e-4)}


def _observers(k):
    t = dict(ne=8, t_lo=0.0, t_hi=STEPS * 10.0, nt=7, e_lo=0.01, e_hi=10.0)
    obs = [Observer(kind="shell", r=1.2, dr=0.05, **t), Observer(kind="box", r=1.5, dr=0.1, ph=200 * DEG,
                                                               dph=40 * DEG, dth=3 * DEG, **t),
           Observer(kind="ring", r=1.7, dr=0.1, **t), Observer(kind="shell", r=1.05, dr=0.02, **t),
           Observer(kind="shell", r=1.9, dr=0.05, **t), Observer(kind="slab", r=-1.0, dr=0.05, **t)]
    return obs[:k]


@pytest.fixture(scope="module")
def backgrounds():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_12164_gb300 import api, build
    build.build()
    w = configs.scaled(configs.cir_uniform_1e6(), nr=64, nth=16, nph=32, n_snap=3)
    out = {}
    for radial in ("linear", "log"):
        w.grid = dataclasses.replace(w.grid, radial=radial, periodic=False)
        bg = api.Background(w.grid)
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
    return w, out


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


def _run(w, bg, prm, obs, noalloc):
    from paper_2404_12164_gb300 import api
    pool, tally = api.Particles(N), api.Tally(obs)
    spec = dataclasses.replace(w.inject, divv_max=None, energy="powerlaw", seed=5)
    api.fte_inject(pool, bg, spec, N, tally)
    if noalloc:
        api.fte_advance_noalloc(pool, bg, prm, tally, 0, STEPS)
    else:
        api.fte_advance(pool, bg, prm, tally, 0, STEPS)
    return pool.state(), tally.C.cpu().numpy(), tally.ledger_n.cpu().numpy()


def _same(a, b):
    for k in a[0]:
        assert np.array_equal(a[0][k], b[0][k]), k
    assert np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])


@pytest.mark.parametrize("grid", ["linear", "log", "amr_linear", "amr_log"])
@pytest.mark.parametrize("dtype,layout", [("f32", "cell"), ("bf16", "cell"), ("f16", "cell"), ("f32", "pair")])
def test_grid_kinds_and_storage(backgrounds, grid, dtype, layout):
    w, bgs = backgrounds
    bg = _stored(bgs[grid], dtype, layout)
    ref = None
    for sort in (0, 32):
        prm = dataclasses.replace(w.params, **COMMON, sort_every=sort)
        ref = ref or _run(w, bg, prm, _observers(2), True)
        assert ref[1].sum() > 1000
        _same(_run(w, bg, prm, _observers(2), False), ref)


@pytest.mark.parametrize("grid", ["linear", "amr_log"])
@pytest.mark.parametrize("option", list(OPTIONS))
def test_each_option(backgrounds, grid, option):
    w, bgs = backgrounds
    prm = dataclasses.replace(w.params, **{**COMMON, **OPTIONS[option]}, sort_every=32)
    _same(_run(w, bgs[grid], prm, _observers(1), False), _run(w, bgs[grid], prm, _observers(1), True))


@pytest.mark.parametrize("k", [0, 1, 2, 4, 5, 6])
@pytest.mark.parametrize("sort", [0, 32])
def test_observer_sets(backgrounds, k, sort):
    w, bgs = backgrounds
    prm = dataclasses.replace(w.params, **COMMON, sort_every=sort)
    _same(_run(w, bgs["linear"], prm, _observers(k), False), _run(w, bgs["linear"], prm, _observers(k), True))
