"""The step kernel's work list: every particle is advanced exactly once whatever the pool's size.

fte_advance hands out FP32 pools in per-SM ranges of whole 32-entry batches, or in blocks of one
warp for pools below one wave; fte_advance_noalloc hands the same particles out from one counter.
Each particle's trajectory depends on nothing but its own state and id, so the states must be
bitwise the same and the alive step count exact, at the sizes where ranges are empty, end inside
a batch or are one batch long, and on both sides of one wave."""
import dataclasses

import numpy as np
import pytest

from fte_inputs import configs

pytestmark = pytest.mark.gpu

STEPS = 20


@pytest.fixture(scope="module")
def parker():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_12164_gb300 import api, build
    build.build()
    w = configs.scaled(configs.parker_1e4(), nr=32, nth=8, nph=16)
    w.inject = dataclasses.replace(w.inject, r=1.0)
    bg = api.Background(w.grid)
    api.fte_load_background(bg, configs.build_background(w))
    return w, bg


def _run(w, bg, n, sort, noalloc):
    from paper_2404_12164_gb300 import api
    pool = api.Particles(n)
    tally = api.Tally(w.observers)
    api.fte_tally_reset(tally)
    api.fte_inject(pool, bg, w.inject, n, tally)
    prm = dataclasses.replace(w.params, sort_every=sort)
    if noalloc:
        api.fte_advance_noalloc(pool, bg, prm, tally, 0, STEPS)
    else:
        api.fte_advance(pool, bg, prm, tally, 0, STEPS)
    return pool.state(), tally.ledger_n.cpu().numpy(), tally.C.cpu().numpy()


@pytest.mark.parametrize("sort", [0, 8])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 2000, 152 * 32 - 1, 152 * 32 + 1, 10_000, 152 * 512 - 1, 152 * 512 + 1,
                               200_003])
def test_every_particle_once(parker, n, sort):
    w, bg = parker
    st, ledger, counts = _run(w, bg, n, sort, False)
    ref, rledger, rcounts = _run(w, bg, n, 0, True)
    for k in ref:
        assert np.array_equal(st[k], ref[k]), k
    assert np.array_equal(ledger, rledger)
    assert ledger[6] == n * STEPS            # nothing leaves the domain from 1 au in 200 s
    assert np.array_equal(counts, rcounts)


@pytest.mark.parametrize("per_sm,more", [(32, -1), (32, 0), (32, 1), (64, 1), (512, -1), (512, 0), (512, 1)])
@pytest.mark.parametrize("sort", [0, 8])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_every_particle_once_at_this_device_s_edges(parker, per_sm, more, sort, dtype):
    """Ranges of exactly one and two batches and one wave, by this device's number of SMs; 16-bit
    pools, which take their work from one counter, too."""
    import torch
    from paper_2404_12164_gb300 import api
    w, bg = parker
    if dtype != "f32":
        img = api.Background(w.grid, dtype=dtype)
        api.fte_quantize_background(img, bg)
        bg = img
    n = torch.cuda.get_device_properties(0).multi_processor_count * per_sm + more
    st, ledger, counts = _run(w, bg, n, sort, False)
    ref, rledger, rcounts = _run(w, bg, n, 0, True)
    for k in ref:
        assert np.array_equal(st[k], ref[k]), k
    assert np.array_equal(ledger, rledger) and ledger[6] == n * STEPS
    assert np.array_equal(counts, rcounts)
