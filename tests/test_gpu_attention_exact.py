"""Attention of verification passes and autoregressive steps against 64 bits, row by row and head by head (head dimension 128).

One layer whose output is its attention: embeddings of +-1/16 that the norm turns into +-1, queries and new keys that depend on
the first feature only (which is the same for every token), an output projection of 64 times the identity and no feed-forward
part.  The hidden row is then the normalised sum of a small known vector and 64 times the attention output, and scores are
whatever the cache is filled for."""
import math

import numpy as np
import pytest
import torch

from helpers import dev
from paper_2403_09919_b200 import synth
from paper_2403_09919_b200.binding import ReDrafter

pytestmark = pytest.mark.gpu

HD = 128
# A bf16 result is off by up to 2^-9 of each element; weights rounded to bf16 add as much at most.
CLOSE = 2.0 ** -8
LOG2E = 1 / math.log(2)


class Attention:
    """Verification passes and autoregressive steps of the model above.  `q`: the query of every row before its rotation,
    [heads, 128]; `k_new`: likewise the keys of the new rows."""

    def __init__(self, monkeypatch, heads, lens, beam, q, k_new, kl, max_ctx=None, seed=1):
        d = heads * HD
        self.heads, self.lens, self.d = heads, lens, d
        self.cfg = dict(synth.CONFIGS["tiny"], dtype="bf16", n_layers=1, d_model=d, n_heads=heads, d_ffn=128, vocab=1000, d_rnn=d,
                        max_batch=len(lens), beam_width=beam[0], beam_length=beam[1])
        self.cfg["max_ctx"] = max_ctx or max(lens) + 1 + beam[0] * beam[1] + 8
        gen = torch.Generator(device="cuda").manual_seed(seed)
        w = synth.make_weights(self.cfg, "cuda:0")
        emb = torch.where(torch.rand(1000, d, device="cuda", generator=gen) < 0.5, -1.0, 1.0) / 16
        emb[:, 0] = 1 / 16
        w["tok_emb"] = emb.to(torch.bfloat16)
        qkv = w["wqkv.0"]
        qkv[:2 * d] = 0
        qkv[:d, 0], qkv[d:2 * d, 0] = q.reshape(-1).to(qkv), k_new.reshape(-1).to(qkv)
        qkv[2 * d:] = torch.randn(d, d, device="cuda", generator=gen) / math.sqrt(d)
        w["wo.0"] = (64 * torch.eye(d, device="cuda")).to(torch.bfloat16)
        w["w_down.0"].zero_()
        self.q, self.w = qkv[:d, 0].double().view(heads, HD), w
        monkeypatch.setenv("RD_ATT_KL", str(kl))
        self.eng = ReDrafter(self.cfg, w)
        monkeypatch.delenv("RD_ATT_KL")
        self.kv = self.eng.kv_view()[0]            # [2, batch, heads, max_ctx, 128]
        self.kv[1].normal_(0.0, 1.0, generator=gen)
        self.rng = np.random.default_rng(seed)
        self.roots = dev(self.rng.integers(0, 1000, size=len(lens)))
        self.h = torch.zeros(len(lens), d, device="cuda")
        self.beams = dev(self.rng.integers(0, 1000, size=(len(lens), *beam)))

    def start(self):
        self.eng.set_state(dev(np.asarray(self.lens)), self.roots, self.h, batch=len(self.lens), ctx_bound=max(self.lens))

    def verify(self, change=None):
        """Hidden rows of a verification pass, sequence by sequence; `change` may alter the packed candidates."""
        self.start()
        self.pk = self.eng.pack(self.beams)
        if change:
            change(self.pk)
        hidden = self.eng.verify(self.pk)[1]
        self.eng.poll()
        return [hidden[b, :int(n)] for b, n in enumerate(self.pk.n)]

    def ar(self):
        self.start()
        self.eng.ar_step()
        self.eng.poll()
        return list(self.eng.get_state()[2][:, None])

    def exact(self, b, tokens, pos, keys, see):
        """64 bits: rows of `tokens` at `pos` over the first `keys` slots of sequence b's cache as it lies there; see: [rows, keys]."""
        half = HD // 2
        ang = pos.double()[:, None] * self.cfg["rope_theta"] ** (-torch.arange(half, dtype=torch.float64, device="cuda") / half)
        c, s, q = ang.cos()[:, None], ang.sin()[:, None], self.q
        q = torch.cat([q[:, :half] * c - q[:, half:] * s, q[:, half:] * c + q[:, :half] * s], -1).to(torch.bfloat16).double()
        sc = torch.einsum("rhd,hkd->rhk", q, self.kv[0, b, :, :keys].double()) / math.sqrt(HD)
        sc.masked_fill_(~see[:, None], -math.inf)
        att = torch.einsum("rhk,hkd->rhd", sc.softmax(-1), self.kv[1, b, :, :keys].double())
        x = self.w["tok_emb"][tokens.long()].double() + 64 * att.reshape(len(tokens), -1)
        return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + self.cfg["rms_eps"])

    def exact_verify(self):
        out = []
        for b, n in enumerate(self.pk.n.tolist()):
            c = self.lens[b]
            words = self.pk.mask[b, :n].cpu().numpy().view(np.uint32)
            bits = (words[:, :, None] >> np.arange(32, dtype=np.uint32)) & 1
            see = torch.ones(n, c + n, dtype=torch.bool, device="cuda")
            see[:, c:] = torch.from_numpy(bits.reshape(n, -1)[:, :n].astype(bool)).cuda()
            out.append(self.exact(b, self.pk.tokens[b, :n], self.pk.pos[b, :n], c + n, see))
        return out

    def exact_ar(self):
        return [self.exact(b, self.roots[b:b + 1], torch.tensor([c], device="cuda"), c + 1, torch.ones(1, c + 1, dtype=torch.bool, device="cuda"))
                for b, c in enumerate(self.lens)]

    def errors(self, got, ref):
        """Relative error (2-norm) of every row and head."""
        a, r = (torch.cat(t).double().view(-1, self.heads, HD) for t in (got, ref))
        return (a - r).norm(dim=-1) / r.norm(dim=-1)

    def route(self):
        return {k: v for k, v in self.eng.route_counts().items() if k.startswith("att_") and v}


def slow(heads, size):
    """Vectors along the pair of dimensions that the rotary embedding turns least: the same at every position, nearly."""
    v = torch.zeros(heads, HD, device="cuda")
    v[:, HD // 2 - 1] = size
    return v


def fill_scores(a, b, scores):
    """Cached keys of sequence b whose scores with `slow(heads, 8.0)` are `scores` (base 2) give or take a few."""
    s = torch.as_tensor(scores, dtype=torch.float32, device="cuda") + torch.randn(a.heads, len(scores), device="cuda") * 1.5
    a.kv[0, b, :, :len(scores)] = 0
    a.kv[0, b, :, :len(scores), HD // 2 - 1] = (s / LOG2E * math.sqrt(HD) / 8.0).to(torch.bfloat16)


@pytest.mark.parametrize("level", [-100.0, -126.0, -130.0, -1000.0])
@pytest.mark.parametrize("lens,late", [([3, 5], 0.0), ([40, 150], 0.0), ([300, 420], 0.0), ([300, 700], 60.0), ([300, 700], -60.0),
                                       ([300, 700], 900.0)])
def test_first_chunk_of_low_scores(monkeypatch, level, lens, late):
    """Every score of the first chunk of keys far below zero, so that the rows' reference falls; later chunks alike, or `late` above."""
    torch.manual_seed(3)
    a = Attention(monkeypatch, 4, lens, (5, 3), slow(4, 8.0), slow(4, (level + late) / LOG2E * math.sqrt(HD) / 8.0), 2)
    for b, c in enumerate(lens):
        fill_scores(a, b, [level] * min(c, 128) + [level + late] * max(c - 128, 0))
    assert a.errors(a.verify(), a.exact_verify()).max() < CLOSE
    assert a.errors(a.ar(), a.exact_ar()).max() < CLOSE
    assert a.route() == {"att_keys_on_lanes": 2}


def test_rows_whose_keys_all_lie_behind_the_first_chunk(monkeypatch):
    """Candidates without a context, some of which attend nothing but themselves, as a mask of the caller's own may say: their
    first key lies in the second chunk, far below zero."""
    torch.manual_seed(3)
    a = Attention(monkeypatch, 2, [0, 90], (32, 5), slow(2, 8.0), slow(2, -200 / LOG2E * math.sqrt(HD) / 8.0), 2)
    fill_scores(a, 1, [-3.0] * 90)

    def alone(pk):
        pk.mask[0, 128:] = 0
        for r in range(128, int(pk.n[0])):
            bit = 1 << (r & 31)
            pk.mask[0, r, r >> 5] = bit - (1 << 32) if bit >> 31 else bit

    got = a.verify(alone)
    assert int(a.pk.n[0]) > 130
    assert a.errors(got, a.exact_verify()).max() < CLOSE
    assert a.route() == {"att_keys_on_lanes": 1}


@pytest.mark.parametrize("beam,lens", [((1, 3), [77, 30, 250]), ((9, 5), [100, 30, 129]), ((3, 2), [249, 10, 63])])
def test_nothing_behind_an_extent_reaches_the_output(monkeypatch, beam, lens):
    """Slots behind a sequence's keys, and another sequence's cache, may hold anything: not-a-number and infinities there leave every
    other row's bits alone, also where the last box of keys runs past the last slot into the next head's and sequence's."""
    rows = 1 + beam[0] * beam[1]
    q = torch.randn(3, HD, generator=torch.Generator().manual_seed(5)).cuda()
    a = Attention(monkeypatch, 3, lens, beam, q, torch.ones(3, HD), 2, max_ctx=max(lens) + rows)
    a.beams = dev(np.arange(len(lens) * rows)[:len(lens) * beam[0] * beam[1]].reshape(len(lens), *beam))
    a.roots = dev(np.full(len(lens), 999))
    a.kv[0].normal_()
    clean = a.kv.clone()
    for call in (a.verify, a.ar):
        a.kv.copy_(clean)
        want = [t.clone() for t in call()]
        for bad in (math.nan, math.inf):
            a.kv.copy_(clean)
            for b, c in enumerate(lens):
                a.kv[:, b, :, 0 if b == 1 else c:] = bad
            got = call()
            assert not torch.isfinite(got[1]).all()
            assert torch.equal(got[0], want[0]) and torch.equal(got[2], want[2])
    assert int(a.pk.n.min()) == rows and set(a.route()) == {"att_keys_on_lanes"}


@pytest.mark.parametrize("spread", [0.6, 1.5, 3.0, 5.0])
@pytest.mark.parametrize("lens,beam", [([300, 60], (3, 5)), ([900, 2000], (8, 5)), ([120, 250], (19, 5)), ([1024] * 3, (64, 3))])
def test_no_less_exact_than_the_other_kernels(monkeypatch, spread, lens, beam):
    """Scores of a deviation of `spread` (natural logarithms): the error against 64 bits is at most that of the kernels with the rows
    on the lanes, in which a row's largest weight is exact.  (What is left is the rounding of the output, the same for all; 0.2 and
    1 % are the scatter of the means over thousands of rows and heads and, in autoregressive steps, 24 to 72.)"""
    heads, means = 24, []
    for kl in (0, 2):
        torch.manual_seed(3)
        q = torch.randn(heads, HD, device="cuda")
        a = Attention(monkeypatch, heads, lens, beam, q, torch.randn(heads, HD, device="cuda") * spread, kl)
        a.kv[0].normal_()
        a.kv[0].mul_(spread)
        means.append([a.errors(got(), ref()).mean().item() for got, ref in ((a.verify, a.exact_verify), (a.ar, a.exact_ar))])
        assert ("att_keys_on_lanes" in a.route()) == (kl == 2)
        a.eng.close()
    assert means[1][0] <= 1.002 * means[0][0] and means[1][1] <= 1.01 * means[0][1]
