"""Attention with the keys on the tensor-memory lanes (verification and autoregressive steps, head dimension 128): against the
oracle, and against the kernels that other passes take at the sizes where its tiles, chunks and references can go wrong."""
import numpy as np
import pytest
import torch

from helpers import dev
from paper_2403_09919_b200 import synth
from paper_2403_09919_b200.binding import ReDrafter
from test_gpu_routing import verify_on_long_contexts

pytestmark = pytest.mark.gpu

BASE = dict(synth.CONFIGS["tiny"], dtype="bf16", n_layers=2, d_ffn=1376, vocab=1000, beam_length=5)


def config(heads, **over):
    return dict(BASE, d_model=128 * heads, n_heads=heads, d_rnn=128 * heads, **over)


def outputs(monkeypatch, cfg, lens, beams, kv_scale=1.0, **env):
    """Logits of a verification pass and of an autoregressive step over a random cache; the attention routes they took."""
    for k, v in env.items():
        monkeypatch.setenv(k, str(v))
    eng = ReDrafter(cfg, synth.make_weights(cfg, "cuda:0"))
    for k in env:
        monkeypatch.delenv(k)
    gen = torch.Generator(device="cuda").manual_seed(4)
    eng.kv_view().normal_(0.0, 1.0, generator=gen)
    eng.kv_view()[:, 0].mul_(kv_scale)
    B, rng = len(lens), np.random.default_rng(5)
    roots, h = dev(rng.integers(0, cfg["vocab"], size=B)), torch.randn(B, cfg["d_model"], device="cuda", generator=gen)
    eng.set_state(dev(np.asarray(lens)), roots, h, batch=B, ctx_bound=max(lens))
    pk = eng.pack(dev(beams))
    _, hidden, logits = eng.verify(pk, want_logits=True)
    n = pk.n.cpu().numpy()
    rows = torch.cat([logits[b, :n[b]] for b in range(B)])
    eng.set_state(dev(np.asarray(lens)), roots, h, batch=B, ctx_bound=max(lens))
    eng.ar_step()
    eng.poll()
    ar = eng.last_logits(B)
    route = {k: v for k, v in eng.route_counts().items() if k.startswith("att_") and v}
    eng.close()
    return rows, ar, route, n


def distance(a, b):
    return float((a - b).norm() / b.norm())


@pytest.mark.parametrize("heads,lens,beam,distinct", [
    (1, [1], (1, 1), 9),                                   # two rows, one chunk
    (2, [63, 64, 65], (3, 5), 9),                          # around half a chunk: the second half of V is or is not fetched
    (3, [127, 128, 129, 250], (5, 3), 9),                  # around a whole one
    (4, [300, 5], (16, 3), 900),                           # 48 and 49 rows
    (2, [200, 700], (19, 5), 900),                         # 96 rows: the widest tile
    (16, [200, 90, 400, 77, 130, 256, 31, 500, 120, 384], (32, 3), 900),   # 97 rows, 160 tiles of two sizes and their rest: several per CTA
    (1, [1000], (64, 5), 900),                             # 321 rows on few tiles: narrow ones
    (4, [20 + 13 * b for b in range(40)], (4, 2), 9),      # more sequences than a warp lays out by lanes, 160 tiles
])
def test_matches_the_other_kernels(monkeypatch, heads, lens, beam, distinct):
    """One layer's attention differs by the rounding of the weights and the sums' order (bf16: 1e-2 of the logits, as between the
    other attention kernels); the hand-off by grid dependencies gives the same bits."""
    cfg = config(heads, max_batch=len(lens), beam_width=beam[0], beam_length=beam[1], max_ctx=max(lens) + 2 * (1 + beam[0] * beam[1]) + 8)
    beams = np.random.default_rng(6).integers(0, distinct, size=(len(lens), *beam))
    ours = outputs(monkeypatch, cfg, lens, beams, RD_ATT_KL=2)
    assert ours[2] == {"att_keys_on_lanes": 2 * cfg["n_layers"]}
    other = outputs(monkeypatch, cfg, lens, beams, RD_ATT_KL=0)
    assert "att_keys_on_lanes" not in other[2] and (ours[3] == other[3]).all()
    assert torch.isfinite(ours[0]).all() and distance(ours[0], other[0]) < 1e-2 and distance(ours[1], other[1]) < 1e-2
    plain = outputs(monkeypatch, cfg, lens, beams, RD_ATT_KL=2, RD_CHAIN=0)
    assert torch.equal(ours[0], plain[0]) and torch.equal(ours[1], plain[1])


@pytest.mark.parametrize("kv_scale", [12.0, 60.0, 400.0])
def test_scores_far_from_the_reference(monkeypatch, kv_scale):
    """Scores of some tens, hundreds and thousands (base 2): rows whose largest lies above what a reference of zero serves, in the
    first chunk and in later ones (below: test_gpu_attention_exact.py).  The softmax is then nearly a choice of one key, so that
    a lost or doubled rescale shows in the first digit."""
    cfg = config(4, max_batch=3, beam_width=9, max_ctx=700)
    beams = np.random.default_rng(7).integers(0, 900, size=(3, 9, 5))
    ours = outputs(monkeypatch, cfg, [600, 130, 260], beams, kv_scale, RD_ATT_KL=2)
    other = outputs(monkeypatch, cfg, [600, 130, 260], beams, kv_scale, RD_ATT_KL=0)
    assert torch.isfinite(ours[0]).all() and distance(ours[0], other[0]) < 2e-2 and distance(ours[1], other[1]) < 2e-2


def test_ragged_batch_against_the_oracle(monkeypatch):
    """Contexts of 40 to 900 tokens, up to 81 rows a sequence, two tiles per CTA, element by element; the layers' own rule."""
    monkeypatch.setenv("RD_ATT_KL", "2")
    cfg = config(16, max_batch=12, beam_width=16, max_ctx=900 + 81 + 16)
    route, n_max, n_sum = verify_on_long_contexts(cfg, [40 + 78 * b for b in range(12)], follow=[0, 7, 11], rho=0.3, seed=31)
    assert route["att_keys_on_lanes"] == cfg["n_layers"] and route["att_rows64"] == route["att_rows128_tc5"] == 0


@pytest.mark.parametrize("heads,batch,bw,tokens,taken", [
    (24, 1, 8, 40, True), (24, 6, 8, 40, True),        # up to one tile per SM: any context
    (24, 8, 8, 127, False), (24, 8, 8, 128, True),     # more: from 128 tokens
    (24, 4, 26, 200, False), (24, 4, 12, 200, True),   # 96 wide tiles, where the 64- or 128-row kernel would run
    (24, 3, 26, 200, True),                            # 72: can be halved
    (24, 2, 3, 1024, False), (24, 2, 3, 1023, True), (24, 2, 4, 1024, True), (24, 3, 3, 1024, True),   # 16 and 21 rows, 48 tiles and 72
    (23, 4, 8, 200, False)])
def test_lines_of_verification(heads, batch, bw, tokens, taken):
    cfg = config(heads, n_layers=1, max_batch=batch, beam_width=bw, max_ctx=tokens + 200)
    eng = ReDrafter(cfg, synth.make_weights(cfg, "cuda:0"))
    rng = np.random.default_rng(8)
    eng.set_state(dev(np.full(batch, tokens)), dev(rng.integers(0, 1000, size=batch)), torch.randn(batch, cfg["d_model"], device="cuda"),
                  batch=batch, ctx_bound=tokens)
    eng.verify(eng.pack(dev(rng.integers(0, 1000, size=(batch, bw, 5)))))
    eng.poll()
    assert eng.route_counts()["att_keys_on_lanes"] == (1 if taken else 0)
    eng.close()


@pytest.mark.parametrize("heads,bw,taken", [
    (49, 40, True), (50, 40, False), (50, 38, True), (40, 64, True),   # bounds of 201, 191 and 321 rows that the 64- or 128-row kernel would
                                                                       # take: more than two tiles' need room for three on the SMs
    (24, 16, False), (25, 16, True), (24, 12, True)])                  # 81 rows: 144 and 150 tiles of 16 rows; 61 rows
def test_lines_of_single_sequences(heads, bw, taken):
    cfg = config(heads, n_layers=1, beam_width=bw, max_ctx=700)
    eng = ReDrafter(cfg, synth.make_weights(cfg, "cuda:0"))
    rng = np.random.default_rng(8)
    eng.set_state(dev(np.full(1, 300)), dev(rng.integers(0, 1000, size=1)), torch.randn(1, cfg["d_model"], device="cuda"), batch=1, ctx_bound=300)
    eng.verify(eng.pack(dev(rng.integers(0, 1000, size=(1, bw, 5)))))
    eng.poll()
    assert eng.route_counts()["att_keys_on_lanes"] == (1 if taken else 0)
    eng.close()


@pytest.mark.parametrize("batch,tokens,taken", [(2, 300, False), (3, 255, False), (3, 256, True), (19, 40, True)])
def test_lines_of_autoregressive_steps(batch, tokens, taken):
    cfg = config(24, n_layers=1, max_batch=batch, beam_width=2, max_ctx=400)
    eng = ReDrafter(cfg, synth.make_weights(cfg, "cuda:0"))
    rng = np.random.default_rng(9)
    eng.set_state(dev(np.full(batch, tokens)), dev(rng.integers(0, 1000, size=batch)), torch.randn(batch, cfg["d_model"], device="cuda"),
                  batch=batch, ctx_bound=tokens)
    eng.ar_step()
    eng.poll()
    assert eng.route_counts()["att_keys_on_lanes"] == (1 if taken else 0)
    eng.close()
