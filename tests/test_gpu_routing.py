"""Verification passes at the larger workloads' own context lengths, through the attention kernels with the rows on the lanes
(Section 3.4: attention over the KV cache plus the tree mask).

The library picks among five bf16 attention kernels by the number of heads, row count, context length and the number of (head,
sequence, row tile) CTAs.  Models of fewer than 24 heads, as here, take the four of this file; for the 7B, 13B and 33B shapes
they are the ones beyond the lines of the fifth (test_gpu_attention_kl.py).  The depth-reduced shape cases use prompts of about a
hundred tokens and so never reach the kernels of long contexts.  Each case here keeps what decides the routing -- head dimension, rows per
sequence, context length, enough CTAs -- on a model small enough for the oracle (2 layers, d_model 512-2048), runs one
planted-beam verification pass on top of a GPU-prefilled cache, checks it against the oracle element by element, and
asserts through redrafter_route_counts that the intended kernel did the work.
"""
import numpy as np
import pytest
import torch

from helpers import Rig, check_against_storage_noise, dev, top2_gap
from oracle import redrafter_oracle as ora
from paper_2403_09919_b200 import synth
from paper_2403_09919_b200.binding import ReDrafter

pytestmark = pytest.mark.gpu

REL = 3e-2
BASE = dict(synth.CONFIGS["tiny"], dtype="bf16", n_layers=2, d_ffn=1376, vocab=1000, beam_length=5)


def decided(ref_logits):
    bound = REL * np.abs(ref_logits).max(axis=-1)
    return top2_gap(ref_logits) > np.maximum(0.05, 2 * bound)


def verify_on_long_contexts(cfg, prompt_lens, follow, rho, seed, p_replace=0.3):
    """Prefill on the GPU, then one verification pass on planted beams; the oracle follows the sequences in `follow`
    (its own prefill, both storage modes) and every one of their packed rows is compared.  Returns the route counters
    of the verification pass alone."""
    rig = Rig(cfg=cfg, oracle_dtype=np.float32)
    B, BW, L, V = len(prompt_lens), cfg["beam_width"], cfg["beam_length"], cfg["vocab"]
    rng = np.random.default_rng(seed)
    prompts = [rng.integers(0, V, size=n) for n in prompt_lens]
    rig.eng.prefill(prompts)
    c_ctx, c_root, c_h = rig.eng.get_state()
    rig.eng.poll()
    roots, hs = c_root.cpu().numpy().copy(), c_h.cpu().numpy().copy()
    beams = np.stack([synth.plant_beams(rng.integers(0, V, size=L), BW, L, V, rng, p=p_replace, rho=rho) for _ in range(B)])
    refs = {}
    for b in follow:
        kv, kv_plain = rig.new_kv(), rig.new_kv()
        ctx, g, h = ora.prefill(rig.W, cfg, prompts[b], kv, np.float32, store="bf16")
        _, _, h_plain = ora.prefill(rig.W, cfg, prompts[b], kv_plain, np.float32)
        assert int(c_ctx[b]) == ctx == prompt_lens[b]
        check_against_storage_noise(hs[b][None], np.asarray(h)[None], np.asarray(h_plain)[None],
                                    f"sequence {b} ({ctx} tokens), h after the prompt", REL, l2_factor=1.25)
        roots[b], hs[b] = g, h
        refs[b] = (kv, kv_plain, ctx, g)
    rig.eng.set_state(None, dev(roots), dev(hs.astype(np.float32), torch.float32))
    before = rig.eng.route_counts()
    beams_d = dev(beams)
    pk = rig.eng.pack(beams_d)
    argmax, hidden, logits = rig.eng.verify(pk, want_logits=True)
    rig.eng.poll()
    after = rig.eng.route_counts()
    for b, (kv, kv_plain, ctx, g) in refs.items():
        aug = np.concatenate([np.full((BW, 1), g), beams[b]], axis=1)
        p = ora.pack_beam(aug, ctx)
        n = p["n"]
        assert int(pk.n[b]) == n and pk.tokens[b, :n].tolist() == p["tokens"].tolist()
        assert (pk.mask_bool(b) == p["mask"]).all()
        rh, rl = ora.llm_forward(rig.W, cfg, p["tokens"], p["pos"], p["mask"], kv, ctx, np.float32, store="bf16")
        _, rl_plain = ora.llm_forward(rig.W, cfg, p["tokens"], p["pos"], p["mask"], kv_plain, ctx, np.float32)
        got = logits[b, :n].cpu().numpy()
        check_against_storage_noise(got, rl, rl_plain, f"sequence {b} ({ctx} tokens, {n} rows), verification logits", REL)
        sure = decided(rl)
        assert sure.sum() >= n // 4
        assert (argmax[b, :n].cpu().numpy()[sure] == rl.argmax(1)[sure]).all()
        # the provisional K rows of this pass are in the cache at slots ctx + n
        kvg = rig.eng.kv_view()[:, 0, b, :, ctx:ctx + n].float().cpu().numpy().transpose(0, 2, 1, 3)
        assert np.abs(kvg - kv.k[:, ctx:ctx + n]).max() < REL * np.abs(kv.k[:, ctx:ctx + n]).max()
    rig.eng.close()
    return {k: after[k] - before[k] for k in after}, int(pk.n.max()), int(pk.n.sum())


def test_wide_beam_long_context_takes_the_tcgen05_kernel():
    """The 13B and 33B workloads' regime: head dimension 128, beam width 32 (up to 161 rows per sequence), more than a
    thousand tokens of context, more (head, sequence, tile) CTAs than four waves of 16-row tiles: tree-masked rows
    through 128-row tcgen05 tiles, the second tile of every sequence partly filled."""
    cfg = dict(BASE, d_model=2048, n_heads=16, d_rnn=2048, max_batch=4, beam_width=32, max_ctx=1200 + 161 + 16)
    route, n_max, n_sum = verify_on_long_contexts(cfg, [1200, 1100, 1150, 1030], follow=[0, 3], rho=0.2, seed=21, p_replace=0.6)
    assert n_max > 128
    assert route["att_rows128_tc5"] == cfg["n_layers"] and route["att_rows64"] == 0 and route["att_rows16"] == 0


def test_ragged_batch_takes_the_64_row_kernel_at_head_dimension_64():
    """Batch 16, beam width 16 (up to 81 rows per sequence), contexts from 256 to 900 tokens (4 to 15 chunks of keys), heads
    too small for the tcgen05 kernel: tree-masked 64-row tiles, every sequence with its own context length and row count."""
    cfg = dict(BASE, d_model=512, n_heads=8, d_rnn=512, max_batch=16, beam_width=16, max_ctx=900 + 81 + 16)
    lens = [int(x) for x in np.random.default_rng(22).integers(256, 901, size=16)]
    lens[0], lens[5], lens[15] = 900, 256, 640
    route, n_max, n_sum = verify_on_long_contexts(cfg, lens, follow=[0, 5, 15], rho=0.3, seed=22)
    assert n_sum > 512
    assert route["att_rows64"] == cfg["n_layers"] and route["att_rows128_tc5"] == 0 and route["att_rows16"] == 0


def test_ragged_batch_long_contexts_take_the_tcgen05_kernel():
    """The batched 7B workload's regime: batch 16, beam width 16 (up to 81 rows per sequence), contexts from 256 to 2048
    tokens (2 to 17 chunks of 128 keys): sequences that can fill half a 128-row tile go through the tcgen05 kernel (head
    dimension 128) from a thousand keys up, and these, whose tiles take one wave, from 320; every sequence with its own context length and row count, most of
    every tile unused."""
    cfg = dict(BASE, d_model=1024, n_heads=8, d_rnn=1024, max_batch=16, beam_width=16, max_ctx=2048 + 81 + 16)
    lens = [int(x) for x in np.random.default_rng(22).integers(256, 2049, size=16)]
    lens[0], lens[5], lens[15] = 2048, 256, 1400
    route, n_max, n_sum = verify_on_long_contexts(cfg, lens, follow=[0, 5, 15], rho=0.3, seed=22)
    assert n_sum > 512
    assert route["att_rows128_tc5"] == cfg["n_layers"] and route["att_rows64"] == 0 and route["att_rows16"] == 0


@pytest.mark.parametrize("heads,batch,bw,longest,tc5", [(8, 16, 16, 238, False), (8, 16, 16, 239, True),      # 128 tiles: one wave
                                                       (16, 12, 20, 218, False), (16, 12, 20, 219, True),    # up to 101 rows
                                                       (16, 16, 16, 942, False), (16, 16, 16, 943, True)])   # 81 rows, 256 tiles
def test_verification_lines_of_the_tcgen05_kernel(heads, batch, bw, longest, tc5):
    """Head dimension 128, either side of 320 keys (one wave of 128-row tiles, or 96 rows and more) and of 1024 keys (fewer
    rows on several waves): contexts from 40 tokens, less than a chunk of keys of either kernel's tiles, to the longest."""
    d = 128 * heads
    cfg = dict(BASE, d_model=d, n_heads=heads, d_rnn=d, max_batch=batch, beam_width=bw, max_ctx=longest + 1 + 5 * bw + 16)
    lens = [40 + (longest - 40) * b // (batch - 1) for b in range(batch)]
    route, n_max, n_sum = verify_on_long_contexts(cfg, lens, follow=[0, batch - 1], rho=0.3, seed=27)
    took, other = ("att_rows128_tc5", "att_rows64") if tc5 else ("att_rows64", "att_rows128_tc5")
    assert route[took] == cfg["n_layers"] and route[other] == 0 and route["att_rows16"] == 0


def test_long_context_few_heads_splits_the_keys():
    """The 33B workload's context length on few CTAs: 4096-token prompts, batch 2, 4 heads, beam width 8 (41 rows):
    16-row tiles whose keys are split over several CTAs and merged by the last one to arrive."""
    cfg = dict(BASE, d_model=512, n_heads=4, d_rnn=512, max_batch=2, beam_width=8, max_ctx=4096 + 41 + 16)
    route, n_max, n_sum = verify_on_long_contexts(cfg, [4096, 3000], follow=[0], rho=0.3, seed=23)
    assert route["att_rows16"] == cfg["n_layers"] and route["att_key_split"] == cfg["n_layers"]


def test_many_tiles_split_the_keys_too():
    """More 16-row tiles than half the SMs: the keys are split over up to three CTAs per SM (two-chunk ring), also for a
    sequence of one chunk of keys, which leaves one of its splits empty."""
    cfg = dict(BASE, d_model=1024, n_heads=8, d_rnn=1024, max_batch=4, beam_width=8, max_ctx=760 + 41 + 16)
    route, n_max, n_sum = verify_on_long_contexts(cfg, [760, 12, 400, 90], follow=[0, 1, 3], rho=0.3, seed=24)
    assert route["att_rows16_shallow"] == cfg["n_layers"] and route["att_key_split"] == cfg["n_layers"]


@pytest.mark.parametrize("heads,head_dim,batch", [(4, 128, 2), (8, 128, 4), (12, 64, 3)])
def test_key_splits_do_not_depend_on_the_hosts_bound(heads, head_dim, batch):
    """The host's bound of the contexts is lowered whenever a copy of the real lengths has arrived, so what a step computes
    must not follow it: the same verification pass and autoregressive step under a tight and a loose bound, bit for bit, with
    the keys split over several CTAs (few tiles, and more than half the SMs)."""
    d = heads * head_dim
    cfg = dict(BASE, d_model=d, n_heads=heads, d_rnn=d, max_batch=batch, beam_width=8, max_ctx=2000)
    eng = ReDrafter(cfg, synth.make_weights(cfg, "cuda:0"))
    gen = torch.Generator(device="cuda").manual_seed(4)
    eng.kv_view().normal_(generator=gen)
    kv0 = eng.kv_view().clone()
    rng = np.random.default_rng(25)
    lens = [900] + [int(x) for x in rng.integers(1, 900, size=batch - 1)]
    roots, h = dev(rng.integers(0, cfg["vocab"], size=batch)), torch.randn(batch, d, device="cuda", generator=gen)
    beams = dev(rng.integers(0, 3, size=(batch, 8, cfg["beam_length"])))
    seen = []
    for bound in (900, 1100, 1900):
        eng.kv_view().copy_(kv0)
        eng.set_state(dev(lens), roots, h, ctx_bound=bound)
        before = eng.route_counts()["att_key_split"]
        pk = eng.pack(beams)
        am, hid, lg = eng.verify(pk, want_logits=True)
        assert eng.route_counts()["att_key_split"] == before + cfg["n_layers"]
        eng.ar_step()
        eng.poll()
        assert eng.route_counts()["att_key_split"] == before + 2 * cfg["n_layers"]
        seen.append([am, hid, lg, eng.last_logits(batch), *eng.get_state()])
    for other in seen[1:]:
        for a, b in zip(seen[0], other):
            assert torch.equal(a, b)
    eng.close()


@pytest.mark.parametrize("tokens,split", [(1007, False), (1008, True), (1100, True)])
def test_tiles_of_one_wave_are_split_in_three_or_not_at_all(tokens, split):
    """16 heads, one sequence of up to 81 rows: 96 tiles on 148 SMs.  Up to seventeen chunks of keys would make two splits and
    stay whole.  From eighteen with all 81 rows (1008 tokens) the launch has three splits; the rows that are there leave
    seventeen chunks at 1008 tokens, so the kernel keeps them whole, and eighteen at 1100.  Against the oracle each time."""
    cfg = dict(BASE, d_model=2048, n_heads=16, d_rnn=2048, beam_width=16, max_ctx=1100 + 81 + 16)
    route, n_max, n_sum = verify_on_long_contexts(cfg, [tokens], follow=[0], rho=0.3, seed=29)
    assert 1008 + n_max <= 17 * 64
    assert route["att_key_split"] == (cfg["n_layers"] if split else 0) and route["att_rows16"] + route["att_rows16_shallow"] == cfg["n_layers"]


def test_the_feedback_of_context_lengths_changes_no_route():
    """The first step's copy of the real lengths (a hundred tokens) has arrived when the second is enqueued and lowers the
    host's bound: the second step takes the kernels that the calls alone decide on (here by the bound of 250)."""
    cfg = dict(BASE, d_model=1024, n_heads=8, d_rnn=1024, max_batch=16, beam_width=20, max_ctx=420)
    eng = ReDrafter(cfg, synth.make_weights(cfg, "cuda:0"))
    rng = np.random.default_rng(26)
    eng.set_state(dev(np.full(16, 100)), dev(rng.integers(0, cfg["vocab"], size=16)), torch.randn(16, 1024, device="cuda"), ctx_bound=250)
    seen = []
    for _ in range(2):
        before = eng.route_counts()
        eng.step(dev(rng.integers(0, cfg["vocab"], size=(16, 20, cfg["beam_length"]))))
        eng.poll()
        after = eng.route_counts()
        seen.append({k: after[k] - before[k] for k in after})
    assert seen[0]["att_rows128_tc5"] == cfg["n_layers"] and seen[0] == seen[1]
    eng.close()


@pytest.mark.parametrize("d_ffn,beam,verify_fused", [(9472, (102, 5), False), (9472, (73, 7), True),      # bounds of 511 and 512 rows
                                                     (1376, (58, 11), False), (1376, (71, 9), True)])     # ... of 639 and 640
def test_lines_of_the_projections_with_their_functions(d_ffn, beam, verify_fused):
    """gate|up with SwiGLU and QKV with rotary embedding: prompt passes from 352 rows; verification passes from a bound of 512
    rows where gate|up's tiles fill their waves (74 pairs of weight tiles at d_ffn = 9472), else from 640."""
    cfg = dict(BASE, d_model=128, n_heads=1, d_rnn=128, d_ffn=d_ffn, beam_width=beam[0], beam_length=beam[1], max_ctx=1100)
    eng = ReDrafter(cfg, synth.make_weights(cfg, "cuda:0"))
    rng = np.random.default_rng(28)

    def fused(call):
        before = eng.route_counts()
        call()
        eng.poll()
        after = eng.route_counts()
        n = {after[k] - before[k] for k in ("gemm_swiglu", "gemm_qkv")}
        assert n in ({0}, {cfg["n_layers"]})
        return n != {0}

    for rows in (351, 352):
        assert fused(lambda: eng.prefill([rng.integers(0, cfg["vocab"], size=rows)])) == (rows == 352)
    pk = eng.pack(dev(rng.integers(0, cfg["vocab"], size=(1, *beam))))
    assert fused(lambda: eng.verify(pk)) == verify_fused
    eng.close()
