"""The wavefront kernels against the CPU oracle, bit for bit, at the edges of their tiles (needs a B200)."""
import numpy as np
import pytest

from oracle import qlstm_ref as R
from tests.gpu_util import run_gpu
from workloads import make_workload, random_layer_stack

pytestmark = pytest.mark.gpu

WAVE = 8             # recurrent_impl: the wavefront kernel, forced

VARIANTS = [dict(), dict(projection=True), dict(cifg=True), dict(peephole=True, cifg=True), dict(projection=True, layernorm=True),
            dict(layernorm=True, cifg=True, projection=True), dict(projection=True, peephole=True, layernorm=True),
            dict(peephole=True, layernorm=True, cifg=True)]


FEW, MANY = 1, 0     # the kernels' forms, as qlstm_debug_wave_plan names them


def check(w, form=None, units=None):
    import paper_2101_05453_b200 as qlstm
    h0, c0 = w.initial_state()
    want = R.run(w.layers, w.x, h0, c0)
    with qlstm.QLSTM(w.layers, w.T, w.B) as q:
        plan = q.debug_wave_plan(w.T, w.B)
        assert form is None or plan[0] == form, plan
        assert units is None or plan[2] == units, plan
        got = run_gpu(w, handle=q, impl=(0, WAVE))
    for name, g, r in zip(("y", "h", "c"), got[:3], want[:3]):
        assert np.array_equal(g, r), f"{name} differs at {np.argwhere(g != r)[:3].tolist()}"


# few rows: one row; MMA columns of eight and 32 rows; two and four row groups of up to 32 rows.  Many rows: two units, odd and full
@pytest.mark.parametrize("B", [1, 8, 9, 32, 33, 64, 65, 128, 129, 256])
@pytest.mark.parametrize("kw", VARIANTS, ids=lambda k: "+".join(sorted(k)) or "basic")
def test_wave_variants(kw, B):
    check(random_layer_stack(810 + B, 3, 48, 112, 64, T=6, B=B, **kw))


# many rows in one unit (nine layers leave no room for row groups of the few-row form): rows twice in the lanes up to 64, once up to
# 128; then two units.  Fewer than four steps per layer and more order X differently
@pytest.mark.parametrize("B,T", [(33, 5), (64, 5), (65, 5), (128, 5), (129, 5), (33, 37), (100, 37)])
@pytest.mark.parametrize("kw", VARIANTS, ids=lambda k: "+".join(sorted(k)) or "basic")
def test_wave_many_rows(kw, B, T):
    check(random_layer_stack(815 + B, 9, 48, 112, 64, T=T, B=B, **kw), MANY, 1 if B <= 128 else 2)


# many rows with each row four times in the lanes: layers too wide for the few-row form's shared memory at 32 rows
@pytest.mark.parametrize("kw", [dict(projection=True, layernorm=True), dict(projection=True, peephole=True, cifg=True)], ids=lambda k: "+".join(sorted(k)))
def test_wave_many_rows_repeated_four_times(kw):
    check(random_layer_stack(817, 9, 64, 1600, 512, T=3, B=29, **kw), MANY, 1)


# dimensions that no tile, vector or pair of cells divides
@pytest.mark.parametrize("B", [3, 40, 131])
@pytest.mark.parametrize("kw", VARIANTS, ids=lambda k: "+".join(sorted(k)) or "basic")
def test_wave_odd_dimensions(kw, B):
    check(random_layer_stack(820 + B, 2, 19, 37, 23, T=7, B=B, **kw))
    check(random_layer_stack(830 + B, 4, 83, 301, 131, T=9, B=B, **kw))


# several gate tiles per block, long K; calls shorter than four steps per layer and longer ones order X differently
@pytest.mark.parametrize("index,kw", [(2, {}), (3, dict(batch=32, T=4)), (4, dict(batch=64, T=21)), (5, dict(batch=8, T=33)),
                                      (5, dict(batch=256, T=3))])
def test_wave_configs(index, kw):
    check(make_workload(index, **kw))


# gate sums so small that layer-norm quotients leave the fast range (2^4, 2^9 below the calibrated scale) or that whole rows
# are zero (sigma = 0): the division out of line
@pytest.mark.parametrize("B", [5, 70])
@pytest.mark.parametrize("shift", [4, 9, 15])
@pytest.mark.parametrize("peephole", [False, True])
def test_wave_layernorm_of_small_deviations(shift, B, peephole):
    w = random_layer_stack(840 + B, 3, 48, 112, 64, projection=True, layernorm=True, peephole=peephole, T=5, B=B)
    for q in w.layers:
        q.eff_x = [(m, s - shift) for m, s in q.eff_x]
        q.eff_h = [(m, s - shift) for m, s in q.eff_h]
    check(w)


# the same out-of-line division in the many-row form
@pytest.mark.parametrize("shift", [4, 9, 15])
@pytest.mark.parametrize("kw", [dict(projection=True), dict(peephole=True), dict(peephole=True, cifg=True)], ids=lambda k: "+".join(sorted(k)))
def test_wave_many_rows_layernorm_of_small_deviations(shift, kw):
    w = random_layer_stack(845, 9, 48, 112, 64, layernorm=True, T=5, B=70, **kw)
    for q in w.layers:
        q.eff_x = [(m, s - shift) for m, s in q.eff_x]
        q.eff_h = [(m, s - shift) for m, s in q.eff_h]
    check(w, MANY, 1)


# both directions in one launch: few and many rows, one and two units (and, where it fits, the kernel with resident weights)
@pytest.mark.parametrize("B", [3, 70, 140])
@pytest.mark.parametrize("kw", [dict(), dict(projection=True, layernorm=True)], ids=lambda k: "+".join(sorted(k)) or "basic")
def test_wave_bidirectional(kw, B):
    from tests.test_gpu_bidirectional import test_bidirectional_matches_two_oracle_runs
    test_bidirectional_matches_two_oracle_runs(kw, B, 9)


# memoised nonlinearities off (0: the definition, which only the many-row form evaluates) or the per-layer kernels' general form
# (2): whatever form the handle has, an ordinary call still runs, by the older kernels where it has to
@pytest.mark.parametrize("enable", [0, 2])
@pytest.mark.parametrize("dims,layers,B", [((48, 112, 64), 3, 5), ((19, 37, 23), 2, 5), ((48, 112, 64), 9, 40)])
def test_wave_without_tables(dims, layers, B, enable):
    import paper_2101_05453_b200 as qlstm
    w = random_layer_stack(850 + B, layers, *dims, projection=True, layernorm=True, T=6, B=B)
    h0, c0 = w.initial_state()
    want = R.run(w.layers, w.x, h0, c0)
    with qlstm.QLSTM(w.layers, w.T, w.B) as q:
        q.activation_tables(enable)
        got = run_gpu(w, handle=q)
        for name, g, r in zip(("y", "h", "c"), got[:3], want[:3]):
            assert np.array_equal(g, r), name
        if layers > 3:                                          # the many-row form without tables
            got = run_gpu(w, handle=q, impl=(0, WAVE))
            for name, g, r in zip(("y", "h", "c"), got[:3], want[:3]):
                assert np.array_equal(g, r), name


# a handle made for many rows, called with fewer: each call has the plan of a handle of its own size, whole row groups working
@pytest.mark.parametrize("dims,layers,kw,max_B", [((48, 112, 64), 2, dict(), 256), ((48, 112, 64), 3, dict(projection=True, layernorm=True), 200),
                                                  ((48, 112, 64), 9, dict(projection=True, layernorm=True, peephole=True), 140),
                                                  ((19, 37, 23), 1, dict(projection=True, layernorm=True, cifg=True), 600)])
def test_wave_calls_of_fewer_rows_than_the_handle(dims, layers, kw, max_B):
    import paper_2101_05453_b200 as qlstm
    w = random_layer_stack(870 + max_B, layers, *dims, T=6, B=300, **kw)
    with qlstm.QLSTM(w.layers, 6, max_B) as q:
        for T, B in ((6, 1), (5, 3), (6, 33), (2, 64), (6, 130), (6, 7), (6, 300)):
            if B > max_B:
                continue
            with qlstm.QLSTM(w.layers, 6, B) as own:
                assert q.debug_wave_plan(T, B) == own.debug_wave_plan(T, B)
            form, groups, _, _ = q.debug_wave_plan(T, B)
            assert form == (-1 if B > 256 else form) and groups <= B
            x = np.ascontiguousarray(w.x[:T, :B])
            h0, c0 = (np.concatenate([v.reshape(300, -1)[:B].ravel() for v in np.split(s, np.cumsum([300 * n for n in per])[:-1])])
                      for s, per in zip(w.initial_state(), ([p.n_output for p in w.layers], [p.n_cell for p in w.layers])))
            want = R.run(w.layers, x, h0, c0)
            got = run_gpu(w, handle=q, x=x, h0=h0, c0=c0, impl=(0, WAVE if form >= 0 else 0))
            for name, g, r in zip(("y", "h", "c"), got[:3], want[:3]):
                assert np.array_equal(g, r), (name, T, B)


# device memory for the handle but not for the wavefront plan (its weight images alone are 21 MB a stack): the handle goes without
@pytest.mark.parametrize("directions", [1, 2])
def test_wave_plan_that_does_not_fit_in_memory_is_left_out(directions):
    import torch
    import paper_2101_05453_b200 as qlstm
    from tests.test_gpu_bidirectional import two_directions
    f, b = two_directions(77, 1, 512, 2048, 2048, 2, 2)
    make = lambda: qlstm.QLSTM(f.layers, 2, 2) if directions == 1 else qlstm.BiQLSTM(f.layers, b.layers, 2, 2)
    h0, c0 = f.initial_state()
    want = R.run(f.layers, f.x, h0, c0)
    with qlstm.QLSTM(f.layers, 2, 2) as q:                      # (loads the kernels)
        run_gpu(f, handle=q)
        run_gpu(f, handle=q, impl=(0, WAVE))
        run_gpu(f, handle=q, impl=(0, 2))
    make().close()
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    q = make()
    size = before - torch.cuda.mem_get_info()[0]
    q.close()
    filler = torch.empty(torch.cuda.mem_get_info()[0] - size + (14 << 20), dtype=torch.uint8, device="cuda")
    try:
        q = make()
    finally:
        del filler
        torch.cuda.empty_cache()
    if directions == 1:
        got = run_gpu(f, handle=q)
        for g, r in zip(got[:3], want[:3]):
            assert np.array_equal(g, r)
        with pytest.raises(qlstm.QlstmError):
            run_gpu(f, handle=q, impl=(0, WAVE))
    q.close()


# the wavefront kernels' images of a long call lie in the per-layer path's workspace, and the two paths take turns on one handle
def test_wave_images_add_no_memory_and_paths_take_turns():
    import torch
    import paper_2101_05453_b200 as qlstm
    T, B = 1200, 64
    w = random_layer_stack(880, 3, 48, 256, 256, T=20, B=B)
    torch.cuda.empty_cache()
    qlstm.QLSTM(w.layers, 1, 1).close()
    before = torch.cuda.mem_get_info()[0]
    q = qlstm.QLSTM(w.layers, T, B)
    used = before - torch.cuda.mem_get_info()[0]
    rows = T * B
    per_layer_path = rows * (1024 * 2 + 2 * 256 + 48 + 256)     # X, the two sequences between layers, staged x and y
    assert used < per_layer_path + (48 << 20), used
    h0, c0 = w.initial_state()
    want = R.run(w.layers, w.x, h0, c0)
    for impl in ((0, WAVE), (0, 2), (0, WAVE), (1, 1), (0, 0)):
        got = run_gpu(w, handle=q, impl=impl)
        for g, r in zip(got[:3], want[:3]):
            assert np.array_equal(g, r), impl
    q.close()


# both directions in one launch of the many-row form, one and two units
@pytest.mark.parametrize("B,units", [(40, 1), (140, 2)])
def test_wave_bidirectional_many_rows(B, units):
    import torch
    import paper_2101_05453_b200 as qlstm
    from tests.test_gpu_bidirectional import two_directions
    T = 9
    f, b = two_directions(72, 8, 32, 96, 48, T, B, projection=True, layernorm=True)
    states = [a for w in (f, b) for a in w.initial_state()]
    yf, hf, cf, _ = R.run(f.layers, f.x, *f.initial_state())
    yb, hb, cb, _ = R.run(b.layers, f.x[::-1], *b.initial_state())
    with qlstm.BiQLSTM(f.layers, b.layers, T, B) as q:
        q.debug_resident(1)
        plan = q.debug_wave_plan(T, B)
        assert plan[0] == MANY and plan[2:] == (units, 1), plan
        dev = torch.device("cuda:0")
        st = [torch.from_numpy(a.copy()).to(dev) for a in states]
        y = torch.zeros((T, B, q.n_output), dtype=torch.int8, device=dev)
        q.run(torch.from_numpy(np.ascontiguousarray(f.x)).to(dev), T, B, *st, y, stream=torch.cuda.current_stream().cuda_stream)
        q.last_status()
        assert np.array_equal(y.cpu().numpy(), np.concatenate([yf, yb[::-1]], axis=2))
        for got, ref in zip(st, (hf, cf, hb, cb)):
            assert np.array_equal(got.cpu().numpy(), ref)


# which path a call takes, without the kernel with resident weights, where the wavefront kernels were measured slower (lines in
# wave_preferred and wave_row_groups): few steps of one row, wide single layers of many rows; and where the few-row form's groups would stream too much, the many-row form
@pytest.mark.parametrize("dims,layers,kw,T,B,taken,form", [
    ((64, 256, 256), 1, dict(), 2, 1, 0, 1), ((64, 256, 256), 1, dict(), 5, 1, 1, 1), ((64, 256, 128), 4, dict(projection=True), 8, 1, 0, 1),
    ((64, 256, 128), 4, dict(projection=True), 3, 1, 1, 1), ((64, 128, 128), 1, dict(), 1, 3, 0, 1), ((64, 256, 256), 2, dict(), 2, 2, 1, 1),
    ((512, 1536, 1536), 1, dict(), 4, 192, 0, 1), ((512, 1536, 1536), 1, dict(), 4, 128, 1, 1), ((512, 2048, 2048), 1, dict(cifg=True), 2, 200, 0, 0),
    ((512, 2048, 2048), 2, dict(), 2, 33, 1, 0), ((512, 2048, 2048), 2, dict(), 2, 200, 1, 0)])
def test_wave_selection(dims, layers, kw, T, B, taken, form):
    import paper_2101_05453_b200 as qlstm
    w = random_layer_stack(890 + T, layers, *dims, T=T, B=B, **kw)
    h0, c0 = w.initial_state()
    want = R.run(w.layers, w.x, h0, c0)
    with qlstm.QLSTM(w.layers, T, B) as q:
        q.debug_resident(1)
        plan = q.debug_wave_plan(T, B)
        assert (plan[3], plan[0]) == (taken, form), plan
        for resident, impl in ((1, (0, 0)), (1, (0, WAVE)), (0, (0, 0))):
            q.debug_resident(resident)
            got = run_gpu(w, handle=q, impl=impl)
            for name, g, r in zip(("y", "h", "c"), got[:3], want[:3]):
                assert np.array_equal(g, r), (name, resident, impl)
        # (with automatic selection the kernel with resident weights comes first)
        assert q.debug_wave_plan(T, B)[3] == (0 if q.debug_resident_plan(T, B)[0] else taken)


def test_wave_timeout_is_reported_and_the_handle_recovers():
    import paper_2101_05453_b200 as qlstm
    w = random_layer_stack(9, 3, 48, 112, 64, projection=True, layernorm=True, T=5, B=40)
    h0, c0 = w.initial_state()
    want = R.run(w.layers, w.x, h0, c0)
    with qlstm.QLSTM(w.layers, w.T, w.B) as q:
        q.debug_barrier_timeout(1, 3_000_000)
        with pytest.raises(qlstm.QlstmError) as e:
            run_gpu(w, handle=q, impl=(0, WAVE))
        assert e.value.code == qlstm.binding.ERR_TIMEOUT
        q.debug_barrier_timeout(0)
        got = run_gpu(w, handle=q, impl=(0, WAVE))
    for g, r in zip(got[:3], want[:3]):
        assert np.array_equal(g, r)


# both forms, copies and MMAs in flight when the wait runs out: later calls on the same handle are not disturbed
@pytest.mark.parametrize("layers,B,form", [(9, 40, MANY), (9, 128, MANY), (9, 20, FEW), (9, 150, MANY), (2, 150, FEW)])
def test_wave_abort_leaves_nothing_in_flight(layers, B, form):
    import paper_2101_05453_b200 as qlstm
    w = random_layer_stack(860 + B, layers, 48, 112, 64, projection=True, layernorm=True, T=12, B=B)
    h0, c0 = w.initial_state()
    want = R.run(w.layers, w.x, h0, c0)
    with qlstm.QLSTM(w.layers, w.T, w.B) as q:
        assert q.debug_wave_plan(w.T, w.B)[0] == form
        for limit in (300_000, 3_000_000):
            q.debug_barrier_timeout(1, limit)
            with pytest.raises(qlstm.QlstmError) as e:
                run_gpu(w, handle=q, impl=(0, WAVE))
            assert e.value.code == qlstm.binding.ERR_TIMEOUT
            q.debug_barrier_timeout(0)
            for _ in range(2):
                got = run_gpu(w, handle=q, impl=(0, WAVE))
                for g, r in zip(got[:3], want[:3]):
                    assert np.array_equal(g, r)
