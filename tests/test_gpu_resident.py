"""The wavefront kernel with resident weights against the CPU oracle, bit for bit, at the edges of its tiles and clusters (needs a B200)."""
import numpy as np
import pytest

from oracle import qlstm_ref as R
from tests.gpu_util import run_gpu
from tests.test_gpu_wave import VARIANTS
from workloads import random_layer_stack

pytestmark = pytest.mark.gpu

IDS = lambda k: "+".join(sorted(k)) or "basic"


def check(w, **plan):
    """One call through the kernel; `plan` pins what its plan must be (cluster: 1 or "many", tiles, groups)."""
    import paper_2101_05453_b200 as qlstm
    want = R.run(w.layers, w.x, *w.initial_state())
    with qlstm.QLSTM(w.layers, w.T, w.B) as q:
        cluster, groups, tiles, units = q.debug_resident_plan(w.T, w.B)
        assert cluster >= 1, "not taken"
        if "cluster" in plan:
            assert (cluster == 1) == (plan["cluster"] == 1), cluster
        if "tiles" in plan:
            assert tiles == plan["tiles"], tiles
        if "units" in plan:
            assert units >= plan["units"], units
        for _ in range(2):                                     # (a second call: what the first one left behind)
            got = run_gpu(w, handle=q)
            for name, g, r in zip(("y", "h", "c"), got[:3], want[:3]):
                assert np.array_equal(g, r), f"{name} differs at {np.argwhere(g != r)[:3].tolist()}, plan {(cluster, groups, tiles, units)}"


# one block per layer and row group (a single group of eight cells; with layer norm three), and clusters of several; one row to several
# tiles of eight; partial groups of eight cells
@pytest.mark.parametrize("B", [1, 7, 8, 40])
@pytest.mark.parametrize("kw", VARIANTS, ids=IDS)
def test_resident_one_block(kw, B):
    check(random_layer_stack(905 + B, 2, 32, 7, 5, T=7, B=B, **kw), cluster=1)
    if kw.get("layernorm"):
        check(random_layer_stack(907 + B, 2, 32, 21, 14, T=7, B=B, **kw), cluster=1)


@pytest.mark.parametrize("B", [1, 7, 8, 40])
@pytest.mark.parametrize("kw", VARIANTS, ids=IDS)
def test_resident_few_cells(kw, B):
    check(random_layer_stack(910 + B, 2, 32, 40, 24, T=7, B=B, **kw))


# shapes measured two to four times slower than others: several groups of cells per warp, one after the other, where more blocks fit
@pytest.mark.parametrize("layers,dims,B,kw", [(2, (16, 208, 24), 4, dict(projection=True, layernorm=True)), (3, (64, 104, 104), 11, dict(cifg=True)),
                                              (1, (64, 136, 136), 40, dict(layernorm=True)), (6, (32, 232, 24), 1, dict(projection=True, layernorm=True, peephole=True, cifg=True))],
                         ids=str)
def test_resident_shape(layers, dims, B, kw):
    import paper_2101_05453_b200 as qlstm
    w = random_layer_stack(915, layers, *dims, T=1, B=B, **kw)
    with qlstm.QLSTM(w.layers, 1, B) as q:
        cluster, _, _, units = q.debug_resident_plan(1, B)
        assert cluster >= 2 and units == 1


@pytest.mark.parametrize("B", [1, 9, 30, 60])
@pytest.mark.parametrize("kw", VARIANTS, ids=IDS)
def test_resident_clusters(kw, B):
    check(random_layer_stack(920 + B, 3, 80, 304, 208, T=7, B=B, **kw), cluster="many")


# dimensions that nothing divides (x and y in bytes), more blocks than outputs, calls of one and two steps
@pytest.mark.parametrize("T", [1, 2, 9])
@pytest.mark.parametrize("kw", VARIANTS, ids=IDS)
def test_resident_odd_dimensions(kw, T):
    check(random_layer_stack(930 + T, 2, 19, 37, 23, T=T, B=5, **kw))
    check(random_layer_stack(940 + T, 3, 83, 501, 9, T=T, B=13, **dict(kw, projection=True)))


# two and four tiles of eight rows, some groups with one tile fewer than others
@pytest.mark.parametrize("B,tiles", [(100, 2), (200, 4)])
@pytest.mark.parametrize("kw", VARIANTS, ids=IDS)
def test_resident_tiles_of_rows(kw, B, tiles):
    check(random_layer_stack(950 + B, 16, 32, 48, 32, T=3, B=B, **kw), tiles=tiles)


# two to four groups of eight cells per warp, with one, two and four tiles of rows: deep stacks, whose layers get few blocks each
@pytest.mark.parametrize("layers,dims,B", [(16, (32, 160, 80), 20), (8, (32, 256, 128), 60), (10, (32, 250, 125), 60), (8, (32, 64, 32), 200), (16, (32, 206, 101), 60)], ids=str)
@pytest.mark.parametrize("kw", [dict(projection=True, cifg=True), dict(projection=True, layernorm=True), dict(projection=True, peephole=True, layernorm=True, cifg=True)], ids=IDS)
def test_resident_groups_per_warp(kw, layers, dims, B):
    check(random_layer_stack(955, layers, *dims, T=4, B=B, **kw), units=2)


@pytest.mark.parametrize("layers,C,B", [(16, 160, 20), (8, 206, 60), (8, 160, 140), (10, 45, 140), (14, 112, 100)], ids=str)
def test_resident_groups_per_warp_basic(layers, C, B):
    check(random_layer_stack(956, layers, 32, C, C, T=4, B=B), units=2)


# a handle's smaller calls share the weight images of a few cluster sizes
def test_resident_calls_of_one_handle_share_shapes():
    import paper_2101_05453_b200 as qlstm
    w = random_layer_stack(957, 2, 32, 256, 256, T=1, B=64)
    with qlstm.QLSTM(w.layers, 4, 64) as q:
        assert len({q.debug_resident_plan(4, B)[0] for B in range(1, 65)} - {0}) <= 4


# gate sums so small that layer-norm quotients leave the fast range, or that whole rows are zero
@pytest.mark.parametrize("shift", [4, 9, 15])
@pytest.mark.parametrize("peephole", [False, True])
def test_resident_layernorm_of_small_deviations(shift, peephole):
    for dims in ((48, 112, 64), (64, 400, 160)):
        w = random_layer_stack(960, 3, *dims, projection=True, layernorm=True, peephole=peephole, T=5, B=5)
        for q in w.layers:
            q.eff_x = [(m, s - shift) for m, s in q.eff_x]
            q.eff_h = [(m, s - shift) for m, s in q.eff_h]
        check(w)


# long calls of several layers: what a layer reads from the one below is announced by each of its blocks, and nothing holds those
# blocks together but the exchanges of their own recurrence (one per step without layer norm and projection)
@pytest.mark.parametrize("kw", [dict(), dict(cifg=True), dict(projection=True), dict(projection=True, layernorm=True)], ids=IDS)
def test_resident_long_calls_of_several_layers(kw):
    import paper_2101_05453_b200 as qlstm
    w = random_layer_stack(965, 4, 64, 320, 224, T=350, B=3, **kw)
    want = R.run(w.layers, w.x, *w.initial_state())
    with qlstm.QLSTM(w.layers, w.T, w.B) as q:
        assert q.debug_resident_plan(w.T, w.B)[0] > 1, "not taken by clusters"
        for _ in range(20):
            got = run_gpu(w, handle=q)
            for name, g, r in zip(("y", "h", "c"), got[:3], want[:3]):
                assert np.array_equal(g, r), f"{name} differs at {np.argwhere(g != r)[:3].tolist()}"


# a wait that runs out: reported, the caller's state untouched, nothing in flight and no counter left behind for the calls that follow.
# One block and clusters per layer, x by bulk copies and by bytes, calls that end before the first exchange and after
@pytest.mark.parametrize("T", [1, 2, 7])
@pytest.mark.parametrize("dims", [(32, 40, 24), (19, 37, 23), (80, 304, 208), (83, 501, 9)], ids=str)
@pytest.mark.parametrize("kw", [dict(), dict(projection=True, peephole=True, layernorm=True)], ids=IDS)
def test_resident_abort_leaves_state_and_handle_as_they_were(kw, dims, T):
    import torch
    import paper_2101_05453_b200 as qlstm
    w = random_layer_stack(970 + T, 3, *dims, T=T, B=11, **kw)
    want = R.run(w.layers, w.x, *w.initial_state())
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(T)
    with qlstm.QLSTM(w.layers, T, 11) as q:
        assert q.debug_resident_plan(T, 11)[0] >= 1
        x = torch.from_numpy(w.x).to(dev)
        y = torch.zeros((T, 11, w.layers[-1].n_output), dtype=torch.int8, device=dev)
        h0, c0 = (rng.integers(-100, 100, a.shape).astype(a.dtype) for a in w.initial_state())
        for limit in (300_000, 3_000_000):
            h, c = torch.from_numpy(h0).to(dev), torch.from_numpy(c0).to(dev)
            q.debug_barrier_timeout(1, limit)
            q.run(x, T, 11, h, c, y, stream=torch.cuda.current_stream().cuda_stream)
            with pytest.raises(qlstm.QlstmError) as e:
                q.last_status()
            assert e.value.code == qlstm.binding.ERR_TIMEOUT
            assert np.array_equal(h.cpu().numpy(), h0) and np.array_equal(c.cpu().numpy(), c0)
            q.debug_barrier_timeout(0)
            for _ in range(2):
                for name, g, r in zip(("y", "h", "c"), run_gpu(w, handle=q)[:3], want[:3]):
                    assert np.array_equal(g, r), name


# clusters that the device has no room for (here: launches that the runtime refuses): the other kernels take the call
@pytest.mark.parametrize("dims,layers,B", [((80, 304, 208), 3, 9), ((83, 301, 131), 2, 5), ((48, 2048, 640), 1, 30), ((32, 40, 24), 2, 1)], ids=str)
def test_refused_cluster_launch(dims, layers, B):
    import paper_2101_05453_b200 as qlstm
    w = random_layer_stack(980 + B, layers, *dims, T=5, B=B, projection=True, peephole=True, layernorm=True)
    want = R.run(w.layers, w.x, *w.initial_state())
    with qlstm.QLSTM(w.layers, w.T, w.B) as q:
        for mode in (2, 0):
            q.debug_resident(mode)
            for name, g, r in zip(("y", "h", "c"), run_gpu(w, handle=q)[:3], want[:3]):
                assert np.array_equal(g, r), (mode, name)
        q.debug_resident(2)
        if q.debug_wave_cluster(w.T, w.B):                     # (forced: no other kernel may stand in)
            with pytest.raises(qlstm.QlstmError) as e:
                run_gpu(w, handle=q, impl=(0, 8))
            assert e.value.code == qlstm.binding.ERR_LAUNCH


@pytest.mark.parametrize("dims,layers", [((32, 96, 48), 2), ((64, 512, 512), 2)], ids=str)
def test_refused_cluster_launch_bidirectional(dims, layers):
    import torch
    import paper_2101_05453_b200 as qlstm
    from tests.test_gpu_bidirectional import two_directions
    T, B = 6, 7
    f, b = two_directions(985, layers, *dims, T, B)
    yf, hf, cf, _ = R.run(f.layers, f.x, *f.initial_state())
    yb, hb, cb, _ = R.run(b.layers, f.x[::-1], *b.initial_state())
    dev = torch.device("cuda:0")
    with qlstm.BiQLSTM(f.layers, b.layers, T, B) as q:
        for mode in (2, 0):
            q.debug_resident(mode)
            st = [torch.from_numpy(a.copy()).to(dev) for w in (f, b) for a in w.initial_state()]
            y = torch.zeros((T, B, q.n_output), dtype=torch.int8, device=dev)
            q.run(torch.from_numpy(np.ascontiguousarray(f.x)).to(dev), T, B, *st, y, stream=torch.cuda.current_stream().cuda_stream)
            q.last_status()
            assert np.array_equal(y.cpu().numpy(), np.concatenate([yf, yb[::-1]], axis=2)), mode
            for got, ref in zip(st, (hf, cf, hb, cb)):
                assert np.array_equal(got.cpu().numpy(), ref), mode
