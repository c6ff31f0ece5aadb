"""The two device-side waits of the library are bounded: when what they wait for never comes they
give up, record VIDKV_ERR_TIMEOUT in the cache's status word and leave in order, and the device
stays usable.  The test hook withholds the awaited event with nothing outstanding (no products
issued, no copy in flight), so nothing here faults, traps or waits without a limit."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _fresh_run_is_fine():
    from tests.helpers import Pair, TOL_ABS
    from workloads import CONFIGS
    pair = Pair(CONFIGS["tiny"], 352, B=1, L=1, p=0.0, max_new=2).prefill()
    out, ref = pair.decode()
    assert np.abs(out - ref).max() <= TOL_ABS
    assert pair.cache.status() == 0


def test_key_encoder_wait_runs_out_and_reports_timeout():
    import paper_2503_16257_b200 as P
    from workloads import CONFIGS, make_layer_kv
    wl = CONFIGS["tiny"]
    cfg = P.VidKVConfig(B=1, L=1, max_prefill_tokens=640, max_new_tokens=1)
    cache = P.VidKVCache(cfg)
    K, _ = make_layer_kv(wl, 0, "cuda", T=640, B=1)
    P.vidkv_debug_withhold_once(1)
    cache.quantize_keys(0, K)
    assert cache.status() == -7                    # VIDKV_ERR_TIMEOUT, read after a stream synchronisation
    # the hook cleared itself: a fresh cache quantizes and decodes as usual
    _fresh_run_is_fine()


DECODE_SHAPES = pytest.mark.parametrize("L,B,T,run_units", [
    (1, 1, 640, 1),      # stream kernel, nothing else in flight
    (1, 1, 640, 3),      # stream kernel, runs that cross slabs: the next unit's keys are in flight when the wait runs out
    (1, 1, 640, 0),      # small-call kernel, a unit per block: the wait behind the last unit
    (12, 4, 2029, -1),   # small-call kernel, four or five units per block, slabs of 13: the exit inside the walk
])


@DECODE_SHAPES
def test_cache_is_whole_after_a_decode_call_that_timed_out(L, B, T, run_units):
    """Only the affected call's results are lost: its key and value rows are in the residual, and the next call over
    the same cache is the oracle's (its status word keeps the first error)."""
    import paper_2503_16257_b200 as P
    from tests.test_gpu_launch_shapes import SampledRun
    from workloads import make_step_inputs
    run = SampledRun("tiny", L, B, T, 0.0, 4, sorted({(0, 0, 0), (L - 1, B - 1, 3), (L // 2, B // 2, 1)}))
    run.cache.debug_set_decode_plan(run_units=run_units)
    run.decode()
    P.vidkv_debug_withhold_once(2)
    run.decode(check=False)
    assert run.cache.status() == -7
    lay, row = run.cache.layout, run.cache.layer_state(0)["n_residual"] - 1
    slabs = run.cache.cache[lay["slab_offset"]:].view(L * B * 4, lay["slab_stride"])
    _, k, v = (torch.stack(t) for t in zip(*[make_step_inputs(run.wl, layer, 1, "cuda", T=T, B=B) for layer in range(L)]))
    for rows, at in ((k, lay["kres_offset"]), (v, lay["vres_offset"])):
        assert torch.equal(slabs[:, at + row * 256:at + (row + 1) * 256], rows.contiguous().view(torch.uint8).view(L * B * 4, 256))
    run.decode()
    run.decode()


@DECODE_SHAPES
def test_decode_wait_runs_out_and_reports_timeout(L, B, T, run_units):
    import paper_2503_16257_b200 as P
    from workloads import CONFIGS, make_layer_kv, make_step_inputs
    wl = CONFIGS["tiny"]
    cfg = P.VidKVConfig(B=B, L=L, max_prefill_tokens=T, max_new_tokens=2)
    cache = P.VidKVCache(cfg)
    for layer in range(L):
        K, V = make_layer_kv(wl, layer, "cuda", T=T, B=B)
        cache.quantize_keys(layer, K)
        cache.quantize_values(layer, V)
    assert cache.status() == 0
    cache.debug_set_decode_plan(run_units=run_units)
    q, k, v = (torch.stack(t) for t in zip(*[make_step_inputs(wl, layer, 0, "cuda", T=T, B=B) for layer in range(L)]))
    out = torch.empty((L, B, 28, 128), dtype=torch.float32, device="cuda")
    before = P.vidkv_launch_count()
    P.vidkv_debug_withhold_once(2)
    cache.decode_attention(0, L, q, k, v, out)
    assert P.vidkv_launch_count() - before == (3 if run_units > 0 else 1)      # the kernel that the case is about
    assert cache.status() == -7
    _fresh_run_is_fine()
