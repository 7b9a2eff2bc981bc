"""The few-row wavefront kernel on thread-block clusters against the CPU oracle, bit for bit, at the edges of its pieces (needs a B200)."""
import numpy as np
import pytest

from oracle import qlstm_ref as R
from tests.gpu_util import run_gpu
from tests.test_gpu_wave import VARIANTS
from workloads import random_layer_stack

pytestmark = pytest.mark.gpu

WAVE = 8
SHAPES = {"blocks without cells": (2, 16, 40, 24), "eights": (5, 32, 280, 48), "blocks without outputs": (2, 48, 272, 20), "several tiles": (2, 80, 640, 176), "odd": (3, 19, 333, 27)}


# h and m cross in pieces of 8 and 16 bytes, rows in groups of 8 up to 32; h alternates between two buffers; calls end at either
@pytest.mark.parametrize("T,B", [(1, 3), (2, 1), (7, 9), (12, 32)])
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("kw", VARIANTS, ids=lambda k: "+".join(sorted(k)) or "basic")
def test_wave_cluster(kw, shape, T, B):
    import paper_2101_05453_b200 as qlstm
    w = random_layer_stack(970 + B, *SHAPES[shape], T=T, B=B, **kw)
    want = R.run(w.layers, w.x, *w.initial_state())
    with qlstm.QLSTM(w.layers, T, B) as q:
        # (wide layers with a single exchange are left to more blocks)
        assert q.debug_wave_cluster(T, B) >= 8 or (shape == "several tiles" and not kw.get("layernorm"))
        for _ in range(2):                                     # (a second call: what the first one left behind)
            got = run_gpu(w, handle=q, impl=(0, WAVE))
            for name, g, r in zip(("y", "h", "c"), got[:3], want[:3]):
                assert np.array_equal(g, r), f"{name} differs at {np.argwhere(g != r)[:3].tolist()}"


# long calls of several layers: what a layer reads from the one below is announced by each of its blocks, and nothing holds those
# blocks together but the exchanges of their own recurrence (one per step without layer norm and projection)
@pytest.mark.parametrize("kw", [dict(), dict(cifg=True), dict(projection=True), dict(projection=True, layernorm=True)], ids=lambda k: "+".join(sorted(k)) or "basic")
def test_wave_cluster_long_calls_of_several_layers(kw):
    import paper_2101_05453_b200 as qlstm
    w = random_layer_stack(985, 4, 64, 320, 224, T=350, B=3, **kw)
    want = R.run(w.layers, w.x, *w.initial_state())
    with qlstm.QLSTM(w.layers, w.T, w.B) as q:
        assert q.debug_wave_cluster(w.T, w.B) >= 8
        for _ in range(20):
            got = run_gpu(w, handle=q, impl=(0, WAVE))
            for name, g, r in zip(("y", "h", "c"), got[:3], want[:3]):
                assert np.array_equal(g, r), f"{name} differs at {np.argwhere(g != r)[:3].tolist()}"


# stacks measured slower in clusters, whose few blocks stream more and finish more cells than the exchanges save
@pytest.mark.parametrize("layers,dims,B,kw", [(1, (512, 2048, 640), 32, dict(projection=True, peephole=True, layernorm=True)), (4, (128, 1120, 416), 20, dict(projection=True)),
                                              (2, (576, 1872, 352), 24, dict(projection=True, layernorm=True, cifg=True)), (6, (80, 704, 704), 1, dict())], ids=str)
def test_wave_cluster_is_left_alone_where_it_is_slower(layers, dims, B, kw):
    import paper_2101_05453_b200 as qlstm
    w = random_layer_stack(990 + B, layers, *dims, T=2, B=B, **kw)
    with qlstm.QLSTM(w.layers, 2, B) as q:
        assert q.debug_wave_cluster(2, B) == 0 and q.debug_wave_plan(2, B)[0] == 1


# a wait that runs out: reported, the caller's state untouched, nothing in flight for the calls that follow
@pytest.mark.parametrize("T", [3, 12])
@pytest.mark.parametrize("kw", VARIANTS, ids=lambda k: "+".join(sorted(k)) or "basic")
def test_wave_cluster_abort_leaves_state_and_handle_as_they_were(kw, T):
    import torch
    import paper_2101_05453_b200 as qlstm
    w = random_layer_stack(995, 3, 48, 272, 112, T=T, B=11, **kw)
    want = R.run(w.layers, w.x, *w.initial_state())
    dev = torch.device("cuda:0")
    with qlstm.QLSTM(w.layers, T, 11) as q:
        assert q.debug_wave_cluster(T, 11) >= 8
        x = torch.from_numpy(w.x).to(dev)
        y = torch.zeros((T, 11, w.layers[-1].n_output), dtype=torch.int8, device=dev)
        rng = np.random.default_rng(T)
        h0, c0 = (rng.integers(-100, 100, a.shape).astype(a.dtype) for a in w.initial_state())
        for limit in (300_000, 3_000_000):
            h, c = torch.from_numpy(h0).to(dev), torch.from_numpy(c0).to(dev)
            q.debug_barrier_timeout(1, limit)
            q.set_impl(0, WAVE)
            q.run(x, T, 11, h, c, y, stream=torch.cuda.current_stream().cuda_stream)
            with pytest.raises(qlstm.QlstmError) as e:
                q.last_status()
            assert e.value.code == qlstm.binding.ERR_TIMEOUT
            assert np.array_equal(h.cpu().numpy(), h0) and np.array_equal(c.cpu().numpy(), c0)
            q.debug_barrier_timeout(0)
            for _ in range(2):
                for name, g, r in zip(("y", "h", "c"), run_gpu(w, handle=q, impl=(0, WAVE))[:3], want[:3]):
                    assert np.array_equal(g, r), name
