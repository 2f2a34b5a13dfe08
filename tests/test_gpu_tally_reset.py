"""fte_tally_reset clears a tally wherever its arrays lie and however they are aligned, and nothing
beside them, eagerly and in a graph: one kernel for aligned memory of the current device, memsets by
address for everything else."""
import ctypes as C

import pytest

from fte_inputs.configs import Observer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("place", ["device", "pinned", "odd"])
@pytest.mark.parametrize("sets", [1, 3])
@pytest.mark.parametrize("how", ["stream", "null stream", "captured"])
def test_reset_clears_every_array(place, sets, how):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_12164_gb300 import api, build, _abi as A
    build.build()
    obs = [Observer(ne=3, nt=7), Observer(ne=1, nt=1)]
    nb = 22 * sets
    words = {"S": nb, "S2": nb, "C": nb, "S_class": nb * A.FTE_NCLASS, "ledger_w": A.FTE_LEDGER,
             "ledger_n": A.FTE_LEDGER}
    pad = 12 if place == "odd" else 16           # bytes before and after each array
    bufs = {}
    t = api.Tally(obs, n_sets=sets).c
    for k, n in words.items():
        b = torch.full((8 * n + 2 * pad,), 255, dtype=torch.uint8)
        bufs[k] = b.pin_memory() if place == "pinned" else b.cuda()
        setattr(t, k, bufs[k].data_ptr() + pad)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    if how == "captured":
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            assert A.lib().fte_tally_reset(C.byref(t), C.c_void_p(stream.cuda_stream)) == 0
        g.replay()
    else:
        s = None if how == "null stream" else C.c_void_p(stream.cuda_stream)
        assert A.lib().fte_tally_reset(C.byref(t), s) == 0
    torch.cuda.synchronize()
    for k, n in words.items():
        b = bufs[k].cpu()
        assert (b[pad:-pad] == 0).all(), k
        assert (b[:pad] == 255).all() and (b[-pad:] == 255).all(), k
