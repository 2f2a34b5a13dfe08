"""S and S2 of the shared-memory layouts are FP64 sums.

With one injection point every particle has the same weight, so the tallied terms of a step are
the same d = w dt (an FP32 product) everywhere and S = d C, S2 = d^2 C to the rounding of the FP64
additions: a bin gets at most one term per particle, launch and change of bin, each exact in FP64
but for one rounding, so the relative error stays below the number of terms times 2^-53.  FP32
partial sums per block are off by about 1e-9 and differ from run to run."""
import dataclasses

import numpy as np
import pytest

from fte_inputs import configs
from fte_inputs.configs import EnsembleSet, Observer

pytestmark = pytest.mark.gpu
STEPS, DT = 40, 10.0


@pytest.fixture(scope="module")
def parker():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_12164_gb300 import api, build
    build.build()
    w = configs.scaled(configs.parker_1e4(), nr=32, nth=8, nph=16)
    w.inject = dataclasses.replace(w.inject, region="point", r=1.1, weight="r-2")
    bg = api.Background(w.grid)
    api.fte_load_background(bg, configs.build_background(w))
    return w, bg


@pytest.mark.parametrize("entry", ["shared", "noalloc", "ensemble"])
@pytest.mark.parametrize("n", [33, 9001, 100_001])
def test_sums_are_fp64(parker, entry, n):
    from paper_2404_12164_gb300 import api
    w, bg = parker
    nt = 5
    obs = [Observer(kind="shell", r=1.1, dr=0.03, e_lo=0.01, e_hi=10.0, ne=16, t_lo=0.0, t_hi=STEPS * DT, nt=nt)]
    prm = dataclasses.replace(w.params, dt=DT, sort_every=0, tally_layout="shared")
    pool = api.Particles(n)
    sets = []
    if entry == "ensemble":
        cut = n // 3
        for s, c in enumerate((cut, n - cut)):
            sets.append(EnsembleSet(0.2 + 0.1 * s, 5 / 3, 0.05, 0.048, s, s, c, w.inject))
    tally = api.Tally(obs, n_sets=max(len(sets), 1))
    api.fte_tally_reset(tally)
    if sets:
        api.fte_inject_batched(pool, bg, sets, tally)
        api.fte_advance_batched(pool, bg, prm, sets, tally, 0, STEPS,
                                config={"threads": 256, "steps_per_launch": 32, "tally_layout": "shared"})
    else:
        api.fte_inject(pool, bg, w.inject, n, tally)
        (api.fte_advance_noalloc if entry == "noalloc" else api.fte_advance)(pool, bg, prm, tally, 0, STEPS)
    wgt = np.unique(pool.state()["w"])
    assert wgt.size == 1
    d = float(np.float32(wgt[0]) * np.float32(DT))
    assert d != round(d)
    S, S2, C = (t.cpu().numpy().astype(np.float64) for t in (tally.S, tally.S2, tally.C))
    assert C.sum() > 2 * n                  # most particles spend several steps in the shell
    # changes of bin: at most one per step; in earnest one per time bin and energy bin crossed
    tol = n * STEPS * 2.0 ** -53
    assert np.all(np.abs(S - d * C) <= tol * d * C)
    assert np.all(np.abs(S2 - d * d * C) <= tol * d * d * C)
