"""GPU parity at the launch shapes the benchmark times and at every way a decode call can be cut
into work: the named workloads at their full sizes (the oracle recomputes sampled slabs), and
small inputs on which every slab is checked while the test hook forces several run lengths of the
stream kernels (without and with protected tokens), including runs that end inside slabs, on slab
boundaries and span several slabs, and steps after a residual flush."""
import numpy as np
import pytest
import torch

from oracle import vidkv_oracle as O
from tests.helpers import Pair, TOL_ABS, to_np
from workloads import CONFIGS, make_layer_kv, make_saliency, make_step_inputs

pytestmark = pytest.mark.gpu


def _rel_tol(ref):
    """2e-3 absolute; where the outputs are large (heavy-tailed values) the bound scales with
    their magnitude."""
    return TOL_ABS * max(1.0, float(np.abs(ref).max()))


class SampledRun:
    """A workload at full size on the GPU; the oracle holds only the sampled (layer, b, h) slabs."""

    def __init__(self, name, L, B, T, p, max_new, samples):
        import paper_2503_16257_b200 as P
        self.P, self.wl, self.L, self.B, self.T, self.p = P, CONFIGS[name], L, B, T, p
        wl = self.wl
        in_dt = P.VIDKV_F16 if wl.dtype == "fp16" else P.VIDKV_BF16
        self.cfg = P.VidKVConfig(B=B, L=L, max_prefill_tokens=T, max_new_tokens=max_new, p_ratio=p,
                                 in_dtype=in_dt, out_dtype=P.VIDKV_F32)
        self.cache = P.VidKVCache(self.cfg, device="cuda")
        self.samples = samples
        self.slabs = {}
        self.step = 0
        Tq = T - T % 32
        E = {}
        if p > 0:
            l_v = min(wl.l_v, Tq)
            sal = make_saliency(wl, "cpu", l_v=l_v, B=B)
            self.cache.select_tokens(sal.cuda(), 0, l_v, T)
            for (_, b, _) in samples:
                if b not in E:
                    e = np.zeros(T, dtype=bool)
                    e[:Tq] = O.select_tokens(sal[b].numpy(), p, 0, Tq)
                    E[b] = e
        for layer in range(L):
            K, V = make_layer_kv(wl, layer, "cuda", T=T, B=B)
            self.cache.quantize_keys(layer, K)
            self.cache.quantize_values(layer, V)
            for (sl, b, h) in samples:
                if sl == layer:
                    sc = O.SlabCache()
                    sc.prefill(to_np(K[b, h]), to_np(V[b, h]), E.get(b))
                    self.slabs[(sl, b, h)] = sc
            del K, V

    def decode(self, check=True, triples=False):
        """triples: through the call that leaves (maximum, sum, output) triples, and their merge."""
        wl, L, B = self.wl, self.L, self.B
        q, k, v = (torch.stack(t) for t in zip(*[make_step_inputs(wl, layer, self.step, "cuda", T=self.T, B=B)
                                                  for layer in range(L)]))
        out = torch.empty((L, B, self.cfg.H_q, 128), dtype=torch.float32, device="cuda")
        if triples:
            part = torch.empty((1, L, B, self.cfg.H_q, 130), dtype=torch.float32, device="cuda")
            self.cache.decode_attention_partial(0, L, q, k, v, part[0])
            self.P.vidkv_merge_partials(part, out)
        else:
            self.cache.decode_attention(0, L, q, k, v, out)
        out = out.cpu().numpy().astype(np.float64)
        rep = self.cfg.H_q // self.cfg.H_kv
        worst = 0.0
        for (sl, b, h), sc in self.slabs.items():
            ref = sc.decode_step(to_np(q[sl, b, rep * h:rep * (h + 1)]), to_np(k[sl, b, h]), to_np(v[sl, b, h]))
            if check:
                err = np.abs(out[sl, b, rep * h:rep * (h + 1)] - ref).max()
                assert err <= _rel_tol(ref), f"step {self.step} slab {(sl, b, h)}: max abs error {err}"
                worst = max(worst, err)
        self.step += 1
        return worst


def _plan(run: SampledRun, n_residual):
    st = run.cache.layer_state(0)
    n_prefill_q = run.T - run.T % 32
    n_flush = (st["n_quantized"] - n_prefill_q) // 128
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    return run.P.vidkv_debug_decode_plan(run.cfg, n_prefill_q, n_flush, n_residual, st["n_protected"], run.L, sm_count=sm)


# ------------------------------------------------------------------ the benchmark's own shape
@pytest.mark.parametrize("L,p,steps", [
    (8, 0.0, 2),       # runs of about 23 units: three to four runs per slab
    (28, 0.0, 2),      # the launch bench.py times: runs of 80 units, every run crosses a slab boundary
    (28, 0.2, 2),      # the launch bench.py --p 0.2 times: runs of 120 units (two thirds of the warps)
])
def test_batched_workload_at_the_timed_launch_shape(L, p, steps):
    wl = CONFIGS["batched"]
    samples = [(0, 0, 0), (L // 2, 7, 2), (L - 1, 15, 3), (L - 1, 3, 1)]
    run = SampledRun("batched", L, wl.batch, wl.T, p, steps, samples)
    plan = _plan(run, 1)
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    assert plan["run_units"] == -(-(L * 64 * 79) // (sm * (12 if p == 0 else 8)))      # 80 / 120 at L = 28 on 148 SMs
    for _ in range(steps):
        run.decode()
    assert run.cache.status() == 0


@pytest.mark.parametrize("p", [0.0, 0.2])
def test_batched_shape_through_the_flush(p):
    """Two layers at batch 16 (128 slabs): 129 steps, so the 128-token residual is flushed and the step
    after it attends to the flushed chunk.  With p = 0.2 (2508 protected tokens per sequence) unit and
    run boundaries fall inside ternary supergroups and protected groups."""
    wl = CONFIGS["batched"]
    run = SampledRun("batched", 2, wl.batch, wl.T, p, 130, [(0, 0, 0), (1, 9, 2)])
    assert _plan(run, 1)["run_units"] > 2
    for s in range(129):
        run.decode(check=(s < 2 or s >= 126))
    assert run.cache.layer_state(1) == dict(n_quantized=wl.T + 128, n_residual=1, n_chunks=2,
                                            n_protected=int(np.float32(p) * wl.T) if p else 0)
    assert run.cache.status() == 0


# ------------------------------------------------------------------ the other named workloads
@pytest.mark.parametrize("name,p", [("llava", 0.0), ("llava", 0.2), ("qwen", 0.0), ("qwen", 0.2)])
def test_named_workload_one_layer_through_the_flush(name, p):
    """LLaVA-shaped (T = 6400, Student-t) and Qwen-shaped (T = 12 800, bfloat16, rotary keys) caches,
    one layer, every KV head against the oracle, through step 129 (the flush happens at step 128)."""
    wl = CONFIGS[name]
    run = SampledRun(name, 1, 1, wl.T, p, 130, [(0, 0, h) for h in range(4)])
    for s in range(129):
        run.decode(check=(s < 3 or s >= 126 or s % 16 == 0))
    assert run.cache.layer_state(0)["n_chunks"] == 2 and run.cache.status() == 0


@pytest.mark.parametrize("p", [0.0, 0.2])
def test_stress_length_slab(p):
    """196 000 tokens (1000 frames) on one sequence; the oracle recomputes one KV head."""
    wl = CONFIGS["stress"]
    run = SampledRun("stress", 1, 1, wl.T, p, 2, [(0, 0, 2)])
    for _ in range(2):
        run.decode()
    st = run.cache.layer_state(0)
    assert st["n_quantized"] == wl.T - wl.T % 32 and st["n_protected"] == (int(np.float32(0.2) * wl.l_v) if p else 0)
    assert run.cache.status() == 0


# ------------------------------------------------------------------ every plan on small inputs, all slabs checked
@pytest.mark.parametrize("run_units", [1, 2, 3, 5, 13, 40])
@pytest.mark.parametrize("name,T,B,L,p", [
    ("tiny", 2000, 2, 2, 0.2),       # 1984 quantized tokens = 12.4 units per slab, 16 residual tokens
    ("qwen", 1311, 1, 1, 0.5),       # bfloat16, half the visual tokens protected
    ("tiny", 1632, 1, 1, 0.9),       # long protected stream, short ternary one
])
def test_stream_kernel_with_protected_tokens_at_every_run_length(run_units, name, T, B, L, p):
    """Runs of 1 .. 40 units over caches with protected tokens: runs end inside ternary supergroups and
    protected groups, which both neighbours then multiply with their own probabilities."""
    pair = Pair(CONFIGS[name], T, B=B, L=L, p=p, max_new=4).prefill()
    pair.cache.debug_set_decode_plan(run_units=run_units)
    for _ in range(3):
        out, ref = pair.decode()
        assert np.abs(out - ref).max() <= _rel_tol(ref)
    assert pair.cache.status() == 0


@pytest.mark.parametrize("run_units", [1, 3])
def test_stream_kernel_with_protected_tokens_across_a_flush(run_units):
    pair = Pair(CONFIGS["tiny"], 1000, B=1, L=1, p=0.2, max_new=125).prefill()    # 992 + 8; flush at step 120
    pair.cache.debug_set_decode_plan(run_units=run_units)
    for s in range(123):
        out, ref = pair.decode()
        assert np.abs(out - ref).max() <= _rel_tol(ref), s
    assert pair.cache.layer_state(0)["n_chunks"] == 2 and pair.cache.status() == 0


@pytest.mark.parametrize("run_units", [1, 2, 3, 5, 13, 40])
def test_stream_kernel_at_every_run_length(run_units):
    """2000 tokens = 12.4 units per slab, 16 slabs: runs of 1 .. 40 units, so runs end inside slabs, on
    slab boundaries and span several slabs; every slab is checked."""
    pair = Pair(CONFIGS["tiny"], 2000, B=2, L=2, p=0.0, max_new=4).prefill()
    pair.cache.debug_set_decode_plan(run_units=run_units)
    for _ in range(3):
        out, ref = pair.decode()
        assert np.abs(out - ref).max() <= TOL_ABS
    assert pair.cache.status() == 0


@pytest.mark.parametrize("run_units", [1, 4])
def test_stream_kernel_across_two_flushes(run_units):
    """Chunks with their own channel splits inside one unit: 96 prefill tokens, then two flushed
    128-token chunks (a unit of 160 tokens then holds groups of two or three chunks)."""
    pair = Pair(CONFIGS["qwen"], 101, B=2, L=1, p=0.0, max_new=260).prefill()
    pair.cache.debug_set_decode_plan(run_units=run_units)
    for s in range(255):
        out, ref = pair.decode()
        assert np.abs(out - ref).max() <= _rel_tol(ref), s
    assert pair.cache.layer_state(0)["n_chunks"] == 3 and pair.cache.status() == 0


def _random_plans(n, seed):
    r = np.random.default_rng(seed)
    cases = []
    for _ in range(n):
        name = ["tiny", "llava", "qwen"][int(r.integers(0, 3))]
        T = int(r.integers(33, 2600))
        steps = int(r.integers(1, 4)) if r.random() < 0.75 else 128 - T % 32 + int(r.integers(1, 4))
        cases.append((name, T, int(r.integers(1, 3)), int(r.integers(1, 3)), [0.0, 0.05, 0.2, 0.5, 0.97][int(r.integers(0, 5))],
                      [1, 2, 3, 7, 19][int(r.integers(0, 5))], steps))
    return cases


@pytest.mark.parametrize("name,T,B,L,p,run_units,steps", _random_plans(14, 20250317))
def test_seeded_random_shapes_and_run_lengths(name, T, B, L, p, run_units, steps):
    """Shapes, protection ratios and run lengths nobody picked by hand (a quarter of the cases decode
    across a residual flush), every slab against the oracle."""
    pair = Pair(CONFIGS[name], T, B=B, L=L, p=p, max_new=steps + 1).prefill()
    pair.cache.debug_set_decode_plan(run_units=run_units)
    for s in range(steps):
        out, ref = pair.decode()
        assert np.abs(out - ref).max() <= _rel_tol(ref), s
    assert pair.cache.status() == 0


# ------------------------------------------------------------------ the one-launch kernel of small calls
@pytest.mark.parametrize("name,L,B,T,p,steps,check_from", [
    ("tiny", 1, 1, 160, 0.0, 2, 0),          # one unit and a residual block per slab
    ("qwen", 1, 1, 36000, 0.0, 2, 0),        # 225 units per slab, one or two to a block: about 148 parts, three levels of joins
    ("tiny", 12, 4, 2029, 0.0, 118, 113),    # 13 units per slab, five to a block, slabs shared by blocks; across a flush
    ("tiny", 28, 4, 362, 0.0, 3, 0),         # slabs of three units, the last one a single group; three to a block
    ("tiny", 4, 4, 2285, 0.0, 2, 0),         # 64 slabs of 14 units and a group: blocks end with their slabs
    ("qwen", 1, 1, 163, 0.5, 2, 0),          # protected tokens: one unit per slab
    ("tiny", 8, 4, 2029, 0.2, 118, 113),     # three or four units to a block, blocks end with their slabs; across a flush
    ("qwen", 4, 4, 2285, 0.3, 2, 0),         # bfloat16
    ("llava", 1, 2, 26000, 0.93, 2, 0),      # long protected stream, 1304 units
])
def test_small_calls_in_one_launch(name, L, B, T, p, steps, check_from):
    """Block and slab boundaries inside and on unit boundaries, the residual with a block of its own and with the slab's last
    block, every depth of the merge tree; the step behind the last one leaves triples."""
    samples = sorted({(0, 0, 0), (L - 1, B - 1, 3), (L // 2, B // 2, 1)})
    run = SampledRun(name, L, B, T, p, steps + 1, samples)
    run.cache.debug_set_decode_plan(run_units=-1)            # whichever kernel would be faster here
    for s in range(steps):
        before = run.P.vidkv_launch_count()
        run.decode(check=s >= check_from)
        assert run.P.vidkv_launch_count() - before == 1 or run.cache.layer_state(0)["n_residual"] == 0   # (a flush has its own)
    run.decode(triples=True)
    assert run.cache.status() == 0


@pytest.mark.parametrize("T", [2029, 20])
def test_a_new_prompt_starts_from_cleared_arrival_counters(T):
    """Two calls that overlap on one handle, against the rules, may leave arrival counters of the small-call kernel off
    zero, and every later call would then join too early or never.  vidkv_cache_reset and the next prompt recover."""
    import paper_2503_16257_b200 as P
    wl = CONFIGS["tiny"]
    cfg = P.VidKVConfig(B=1, L=2, max_prefill_tokens=2048, max_new_tokens=4, out_dtype=P.VIDKV_F32)
    kv = [[x[:, :, :T].contiguous() for x in make_layer_kv(wl, layer, "cuda", T=2048, B=1)] for layer in range(2)]

    def answer(c):
        for layer, (K, V) in enumerate(kv):
            c.quantize_keys(layer, K)
            c.quantize_values(layer, V)
        out = torch.empty((2, 1, 28, 128), dtype=torch.float32, device="cuda")
        q, k, v = (torch.stack(t) for t in zip(*[make_step_inputs(wl, layer, 0, "cuda", T=2048, B=1) for layer in range(2)]))
        c.decode_attention(0, 2, q, k, v, out)
        return out

    want = answer(P.VidKVCache(cfg))
    c = P.VidKVCache(cfg)
    answer(c)
    # the counters lie behind the channel ranges, the partial records and the query images (each from a 256-byte boundary)
    up = lambda n: -(-n // 256) * 256  # noqa: E731
    records = P.vidkv_debug_decode_plan(cfg, 2048, 0, 1, 0, 2)["records_capacity"]
    at = up(2 * 8 * 256 * 4) + up(records * 130 * 4) + up(8 * c.layout["max_chunks"] * 25 * 32 * 4)
    words = c.workspace[at:at + 4 * (records // 8 // 7 + 12 * 8 + 64)].view(torch.int32)
    assert not words.any()
    words.fill_(1)
    c.reset()
    assert torch.equal(answer(c), want) and not words.any()


# ------------------------------------------------------------------ one call, cut in different ways
@pytest.mark.parametrize("name,T,B,L,p,k_ratio,one_bit", [
    ("tiny", 2029, 2, 2, 0.0, 0.5, "fft"), ("qwen", 2003, 2, 1, 0.0, 0.5, "fft"), ("tiny", 2029, 2, 2, 0.2, 0.5, "fft"),
    ("tiny", 2029, 2, 1, 0.0, 0.75, "minmax")])
def test_outputs_do_not_depend_on_the_cut(name, T, B, L, p, k_ratio, one_bit):
    """Runs of 1, 3 and 40 units and the small-call kernel over the same cache: the rounding of a probability to
    binary16 must not depend on where a run began.  What is left is the order of the float32 sums, chains of at most
    about 100 additions (13 units of 5 groups, 13 records, the residual): 100 x 2^-24 = 6e-6 of the norm."""
    import paper_2503_16257_b200 as P
    wl = CONFIGS[name]
    cfg = P.VidKVConfig(B=B, L=L, max_prefill_tokens=T, max_new_tokens=4, p_ratio=p, k_ratio=k_ratio,
                        key_1bit_mode=P.VIDKV_KEY1BIT_PLAIN_MINMAX if one_bit == "minmax" else P.VIDKV_KEY1BIT_FFT_SIGN,
                        in_dtype=P.VIDKV_F16 if wl.dtype == "fp16" else P.VIDKV_BF16, out_dtype=P.VIDKV_F32)
    kv = [make_layer_kv(wl, layer, "cuda", T=T, B=B) for layer in range(L)]
    outs = {}
    for run_units in (0, 1, 3, 40):
        c = P.VidKVCache(cfg)
        if p > 0:
            l_v = min(wl.l_v, T - T % 32)
            c.select_tokens(make_saliency(wl, "cpu", l_v=l_v, B=B).cuda(), 0, l_v, T)
        for layer, (K, V) in enumerate(kv):
            c.quantize_keys(layer, K)
            c.quantize_values(layer, V)
        c.debug_set_decode_plan(run_units=run_units)
        out = torch.empty((3, L, B, 28, 128), dtype=torch.float32, device="cuda")
        for s in range(3):
            q, k, v = (torch.stack(t) for t in zip(*[make_step_inputs(wl, layer, s, "cuda", T=T, B=B) for layer in range(L)]))
            c.decode_attention(0, L, q, k, v, out[s])
        assert c.status() == 0
        outs[run_units] = out.double()
    for run_units in (1, 3, 40):
        assert float((outs[run_units] - outs[0]).norm() / outs[0].norm()) <= 6e-6, run_units


# ------------------------------------------------------------------ prompts shorter than one group
@pytest.mark.parametrize("T", [31, 0])
def test_flushes_after_a_prompt_with_nothing_to_quantize(T):
    """Fewer than 32 prompt tokens: chunk 0 of the chunk table stays empty and the flushed chunks
    follow it.  Decoded across two flushes through vidkv_decode_attention, and after each flush
    through vidkv_attend_noalloc as well."""
    import paper_2503_16257_b200 as P
    wl = CONFIGS["tiny"]
    steps = 2 * 128 - T + 3
    cfg = P.VidKVConfig(B=1, L=1, max_prefill_tokens=32, max_new_tokens=steps + 1, p_ratio=0.0, out_dtype=P.VIDKV_F32)
    cache = P.VidKVCache(cfg)
    K, V = make_layer_kv(wl, 0, "cpu", T=32, B=1)
    K, V = K[:, :, :T].contiguous(), V[:, :, :T].contiguous()
    cache.quantize_keys(0, K.cuda())
    cache.quantize_values(0, V.cuda())
    slabs = []
    for h in range(4):
        sc = O.SlabCache()
        sc.prefill(to_np(K[0, h]), to_np(V[0, h]), None)
        slabs.append(sc)
    flushes = 0
    for s in range(steps):
        q, k, v = make_step_inputs(wl, 0, s, "cpu", T=32, B=1)
        out = torch.empty((1, 1, 28, 128), dtype=torch.float32, device="cuda")
        cache.decode_attention(0, 1, q[None].cuda(), k[None].cuda(), v[None].cuda(), out)
        ref = np.concatenate([slabs[h].decode_step(to_np(q[0, 7 * h:7 * h + 7]), to_np(k[0, h]), to_np(v[0, h]))
                              for h in range(4)])
        assert np.abs(out[0, 0].cpu().numpy().astype(np.float64) - ref).max() <= TOL_ABS, s
        st = cache.layer_state(0)
        if st["n_quantized"] // 128 > flushes or s == steps - 1:
            flushes = st["n_quantized"] // 128
            # the same attention once more, without the append, through the workspace-free entry point
            again = torch.full((1, 1, 28, 128), float("nan"), dtype=torch.float32, device="cuda")
            P.vidkv_attend_noalloc(cfg, cache.cache, 0, flushes, st["n_residual"], 0, 0, 1, q[None].cuda(), again)
            if st["n_residual"] > 0:          # right after a flush the residual is empty and the attended set differs
                assert float((again - out).abs().max()) <= TOL_ABS
            else:
                # the flushed tokens are now read from their packed form: compare with the oracle's dequantized view
                Kd = [sl.dequant_k() for sl in slabs]
                Vd = [sl.dequant_v() for sl in slabs]
                r2 = np.concatenate([O.attention(to_np(q[0, 7 * h:7 * h + 7]), Kd[h], Vd[h], 1.0 / np.sqrt(128.0))
                                     for h in range(4)])
                assert np.abs(again[0, 0].cpu().numpy().astype(np.float64) - r2).max() <= TOL_ABS
    assert cache.layer_state(0) == dict(n_quantized=256, n_residual=T + steps - 256, n_chunks=2, n_protected=0)
    assert cache.status() == 0


@pytest.mark.parametrize("run_units", [0, 1, 3])
@pytest.mark.parametrize("T,p,steps", [(352, 0.0, 2), (416, 0.2, 2), (1664, 0.3, 130)])
def test_cache_memory_that_nobody_has_written_does_not_count(run_units, T, p, steps):
    """Cache memory full of NaN patterns before the prompt: the last unit of a slab, the last supergroup of a ternary
    stream and (a flush later) its gap have groups that do not exist, whose codes and scales nobody has written."""
    pair = Pair(CONFIGS["tiny"], T, B=1, L=1, p=p, max_new=steps)
    pair.cache.cache[256:] = 255                             # all but the header
    pair.prefill()
    pair.cache.debug_set_decode_plan(run_units=run_units)
    for s in range(steps):
        out, ref = pair.decode()
        if s < 2 or s >= 126:
            assert np.abs(out - ref).max() <= TOL_ABS, s
    assert pair.cache.status() == 0


@pytest.mark.parametrize("name,L,B,T,p,k_ratio,one_bit", [
    ("tiny", 27, 1, 362, 0.0, 0.5, "fft"),         # 108 slabs of three units and their residuals: 432 blocks, three to a multiprocessor
    ("tiny", 28, 1, 362, 0.0, 0.5, "fft"),         # 448 blocks: four
    ("qwen", 28, 4, 362, 0.0, 0.75, "minmax"),     # more slabs than blocks at three to a multiprocessor
    ("qwen", 28, 4, 330, 0.0, 0.75, "minmax"),     # the same of two units: four blocks on a multiprocessor for the general formats
    ("llava", 28, 5, 362, 0.2, 0.5, "fft"),        # the same with protected tokens
    ("tiny", 1, 4, 11300, 0.0, 0.75, "minmax"),    # 16 slabs of 71 units, two or three to a block
    ("tiny", 1, 1, 196000, 0.0, 0.5, "fft"),       # the longest slab: 1225 units, 111 parts
    ("llava", 1, 4, 22400, 0.2, 0.5, "fft"),       # protected tokens, 140 units, five or six to a block
])
def test_block_kernel_at_the_edges_of_its_variants(name, L, B, T, p, k_ratio, one_bit):
    """The small-call kernel against the stream kernel with runs of 40 units, over the same cache.  They differ by the order of
    float32 sums: chains of at most 40 units of 5 groups, 31 records and the residual, 250 x 2^-24 = 1.5e-5 of the norm."""
    import paper_2503_16257_b200 as P
    wl = CONFIGS[name]
    cfg = P.VidKVConfig(B=B, L=L, max_prefill_tokens=T, max_new_tokens=4, p_ratio=p, k_ratio=k_ratio,
                        key_1bit_mode=P.VIDKV_KEY1BIT_PLAIN_MINMAX if one_bit == "minmax" else P.VIDKV_KEY1BIT_FFT_SIGN,
                        in_dtype=P.VIDKV_F16 if wl.dtype == "fp16" else P.VIDKV_BF16, out_dtype=P.VIDKV_F32)
    q, k, v = (torch.stack(t) for t in zip(*[make_step_inputs(wl, layer, 0, "cuda", T=T, B=B) for layer in range(L)]))
    outs = []
    for run_units, launches in ((0, 1), (40, 3)):
        c = P.VidKVCache(cfg)
        if p > 0:
            l_v = min(wl.l_v, T - T % 32)
            c.select_tokens(make_saliency(wl, "cpu", l_v=l_v, B=B).cuda(), 0, l_v, T)
        for layer in range(L):
            K, V = make_layer_kv(wl, layer, "cuda", T=T, B=B)
            c.quantize_keys(layer, K)
            c.quantize_values(layer, V)
        c.debug_set_decode_plan(run_units=run_units)
        out = torch.empty((L, B, 28, 128), dtype=torch.float32, device="cuda")
        before = P.vidkv_launch_count()
        c.decode_attention(0, L, q, k, v, out)
        assert P.vidkv_launch_count() - before == launches
        assert c.status() == 0
        outs.append(out.double())
    assert float((outs[0] - outs[1]).norm() / outs[1].norm()) <= 1.5e-5


def test_attention_without_a_workspace_takes_longer_runs_where_its_scratch_is_short():
    """448 slabs of six units over eight chunks: the query images leave room for 1276 records, runs of one or two units would
    leave 1792 and more.  The same attention as the call with a workspace, but for the order of float32 sums (1.5e-5, above)."""
    import paper_2503_16257_b200 as P
    L, B, steps = 28, 4, 7 * 128 + 1
    cfg = P.VidKVConfig(B=B, L=L, max_prefill_tokens=64, max_new_tokens=steps, p_ratio=0.0, out_dtype=P.VIDKV_F32)
    c = P.VidKVCache(cfg)
    g = torch.Generator(device="cuda").manual_seed(11)
    K, V = (torch.randn((B, 4, 64, 128), device="cuda", generator=g).half() for _ in range(2))
    for layer in range(L):
        c.quantize_keys(layer, K)
        c.quantize_values(layer, V)
    q = torch.randn((L, B, 28, 128), device="cuda", generator=g).half()
    rows = torch.randn((2, 16, L, B, 4, 128), device="cuda", generator=g).half()
    out, again = (torch.empty((L, B, 28, 128), dtype=torch.float32, device="cuda") for _ in range(2))
    for s in range(steps):
        c.decode_attention(0, L, q, rows[0, s % 16], rows[1, s % 16], out)
    st = c.layer_state(0)
    assert (st["n_quantized"], st["n_residual"]) == (64 + 7 * 128, 1)
    P.vidkv_attend_noalloc(cfg, c.cache, 64, 7, 1, 0, 0, L, q, again)
    assert c.status() == 0
    assert float((again.double() - out.double()).norm() / out.double().norm()) <= 1.5e-5
