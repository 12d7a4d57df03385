"""The counter hand-off between launches changes when a kernel may start, never what it computes.

Two engines with the same seeded weights run the same speculative steps, one with the hand-off (the
default) and one created with RD_CHAIN=0, where every launch waits for its predecessor through the grid
dependency alone.  Everything a step produces must be bit-identical: drafted beams, packed tree,
verification logits, greedy tokens, acceptance, the handed-over state and the KV cache.  A race in the
hand-off (a consumer reading before its producer's last store, a counter reused too early) shows up here
as a difference, and repeating the steps makes it likelier to surface.  Sizes: the depth-reduced 7B shape,
whose launches take the tensor-core path and the two-kernel selection.
"""
import os

import numpy as np
import pytest
import torch

from helpers import Rig
from paper_2403_09919_b200 import synth

pytestmark = pytest.mark.gpu


def make_rig(chain):
    cfg = synth.with_layers(dict(synth.CONFIGS["7b"], max_ctx=512), 2)
    old = os.environ.get("RD_CHAIN")
    os.environ["RD_CHAIN"] = "1" if chain else "0"
    try:
        return Rig(cfg=cfg, oracle_dtype=np.float32)
    finally:
        if old is None:
            del os.environ["RD_CHAIN"]
        else:
            os.environ["RD_CHAIN"] = old


def test_hand_off_is_bit_identical_to_grid_dependencies():
    a, b = make_rig(True), make_rig(False)
    rng = np.random.default_rng(5)
    prompts = [rng.integers(0, a.cfg["vocab"], size=150)]
    a.eng.prefill(prompts)
    b.eng.prefill(prompts)
    for sa, sb in zip(a.eng.get_state(), b.eng.get_state()):
        assert torch.equal(sa, sb)
    for step in range(6):
        beams_a, sc_a = a.eng.draft()
        beams_b, sc_b = b.eng.draft()
        assert torch.equal(beams_a, beams_b) and torch.equal(sc_a, sc_b)
        pk_a, pk_b = a.eng.pack(beams_a), b.eng.pack(beams_b)
        assert torch.equal(pk_a.n, pk_b.n) and torch.equal(pk_a.tokens, pk_b.tokens)
        am_a, hid_a, lg_a = a.eng.verify(pk_a, want_logits=True)
        am_b, hid_b, lg_b = b.eng.verify(pk_b, want_logits=True)
        n = int(pk_a.n[0])
        assert torch.equal(lg_a[0, :n], lg_b[0, :n])
        assert torch.equal(hid_a[0, :n], hid_b[0, :n])
        assert torch.equal(am_a, am_b)
        out_a = a.eng.accept(beams_a, pk_a, am_a, hid_a)
        out_b = b.eng.accept(beams_b, pk_b, am_b, hid_b)
        a.eng.poll()
        b.eng.poll()
        assert torch.equal(out_a.n_accept, out_b.n_accept) and torch.equal(out_a.tokens, out_b.tokens)
        for sa, sb in zip(a.eng.get_state(), b.eng.get_state()):
            assert torch.equal(sa, sb)
    assert torch.equal(a.eng.kv_view(), b.eng.kv_view())


def test_fused_steps_repeat_bit_identically():
    """redrafter_step from the same state, twice on each of two engines: four identical token streams."""
    streams = []
    for chain in (True, True, False):
        r = make_rig(chain)
        rng = np.random.default_rng(9)
        r.eng.prefill([rng.integers(0, r.cfg["vocab"], size=97)])
        out = r.binding.AcceptOut(1, r.cfg["beam_length"], "cuda:0")
        toks = []
        for _ in range(8):
            r.eng.step(None, out)
            r.eng.poll()
            toks.append((int(out.n_accept[0]), out.tokens[0].cpu().numpy().copy()))
        streams.append(toks)
    for other in streams[1:]:
        for (na, ta), (nb, tb) in zip(streams[0], other):
            assert na == nb and (ta[:na + 1] == tb[:nb + 1]).all()


def test_a_wait_that_nothing_satisfies_gives_up_and_is_reported():
    """The device-side waits are bounded: one that can never be satisfied returns after about a second, the next
    poll reports RD_ERR_TIMEOUT and clears it, and the engine keeps working."""
    import time
    r = make_rig(True)
    rng = np.random.default_rng(3)
    r.eng.prefill([rng.integers(0, r.cfg["vocab"], size=64)])
    out = r.binding.AcceptOut(1, r.cfg["beam_length"], "cuda:0")
    r.eng.step(None, out)
    r.eng.poll()
    ref_state = [s.clone() for s in r.eng.get_state()]
    t0 = time.time()
    r.eng.selftest_wait()
    with pytest.raises(r.binding.RdError) as e:
        r.eng.poll()
    dt = time.time() - t0
    assert e.value.code == 6 and 0.5 < dt < 10.0          # RD_ERR_TIMEOUT, after the wait's one-second limit
    r.eng.poll()                                          # the status word was cleared
    for a, b in zip(ref_state, r.eng.get_state()):
        assert torch.equal(a, b)                          # nothing of the state was touched
    r.eng.step(None, out)                                 # and the engine still decodes
    r.eng.poll()
    assert int(out.n_accept[0]) >= 0


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_captured_calls_replay_with_new_state(dtype):
    """A drafter call captured into a graph and replayed after the state has changed gives what an eager call gives: under
    capture the launches do not hand over by counters, whose values a replay would find already reached."""
    from paper_2403_09919_b200.binding import ReDrafter
    cfg = dict(synth.CONFIGS["tiny"], dtype=dtype, d_model=256, n_heads=2, max_ctx=200)
    eng = ReDrafter(cfg, synth.make_weights(cfg, "cuda:0"))
    gen = torch.Generator(device="cuda").manual_seed(1)
    states = [(torch.tensor([11 + 7 * i], dtype=torch.int32, device="cuda"), torch.randn(1, 256, device="cuda", generator=gen)) for i in range(4)]
    ctx = torch.tensor([20], dtype=torch.int32, device="cuda")

    def put(i):
        eng.set_state(ctx, states[i][0], states[i][1], ctx_bound=20)

    want = []
    for i in range(4):
        put(i)
        want.append([x.clone() for x in eng.draft()])
    beams, scores = [torch.zeros_like(x) for x in want[0]]
    put(0)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        eng.draft(beams, scores)
    for i in (0, 1, 2, 3, 1):
        put(i)
        g.replay()
        eng.poll()
        assert torch.equal(beams, want[i][0]) and torch.equal(scores, want[i][1])
    put(2)
    again = eng.draft()                     # and eager calls go on as before
    eng.poll()
    assert torch.equal(again[0], want[2][0]) and torch.equal(again[1], want[2][1])
    del g
    eng.close()


def test_a_capture_after_a_wait_that_gave_up_is_refused():
    """After a wait that gave up the next call resets the hand-off counters.  A captured call cannot: its graph would hold the
    reset, while the host already counts from zero.  It is refused until an eager call has been made; eager calls and, from
    then on, captured ones give what they gave before."""
    from paper_2403_09919_b200.binding import RdError, ReDrafter
    cfg = dict(synth.CONFIGS["tiny"], dtype="bf16", d_model=256, n_heads=2, max_ctx=200)
    eng = ReDrafter(cfg, synth.make_weights(cfg, "cuda:0"))
    i32 = dict(dtype=torch.int32, device="cuda")
    eng.set_state(torch.tensor([20], **i32), torch.tensor([11], **i32), torch.ones(1, 256, device="cuda"), ctx_bound=20)
    want = eng.draft()
    eng.poll()
    eng.selftest_wait()
    with pytest.raises(RdError) as e:
        eng.poll()
    assert e.value.code == 6
    beams, scores = [torch.zeros_like(x) for x in want]
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        with pytest.raises(RdError) as e:
            eng.draft(beams, scores)
    assert e.value.code == 4
    got = eng.draft()
    eng.poll()
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        eng.draft(beams, scores)
    for _ in range(2):
        g.replay()
        got = eng.draft()
        eng.poll()
        for a, b, c in zip(want, got, (beams, scores)):
            assert torch.equal(a, b) and torch.equal(a, c)
    del g
    eng.close()


@pytest.mark.parametrize("call", ["step", "ar_step"])
@pytest.mark.parametrize("pending", [True, False])
def test_captured_steps_leave_the_context_feedback_working(call, pending):
    """A step captured while a copy of the context lengths is on its way (after an eager step): its replays give what an
    eager step gives.  A step captured as the call that would enqueue such a copy (the handle's first): the feedback goes
    on -- 48 steps that accept about one token each fit a cache that the bound alone would have run out of."""
    from paper_2403_09919_b200.binding import AcceptOut, ReDrafter
    L = 4
    cfg = dict(synth.CONFIGS["tiny"], beam_width=4, beam_length=L, max_ctx=20 + 48 * 2 + 17 + 10 * L)
    eng = ReDrafter(cfg, synth.make_weights(cfg, "cuda:0"))
    i32 = dict(dtype=torch.int32, device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(3)
    eng.kv_view().normal_(generator=gen)
    kv0 = eng.kv_view().clone()
    ctx, root = torch.tensor([20], **i32), torch.tensor([11], **i32)
    h = torch.randn(1, cfg["d_model"], device="cuda", generator=gen)
    rng = np.random.default_rng(15)
    beams = lambda: torch.from_numpy(rng.integers(0, cfg["vocab"], size=(1, 4, L)).astype(np.int32)).cuda()
    fixed, out, token = beams(), AcceptOut(1, L, "cuda:0"), torch.zeros(1, **i32)

    def one(b=None):
        return eng.step(fixed if b is None else b, out) if call == "step" else eng.ar_step(token)

    def put():
        eng.kv_view().copy_(kv0)
        eng.set_state(ctx, root, h)

    def seen():
        got = [out.n_accept, out.best, out.tokens, token, *eng.get_state(), eng.kv_view()]
        return [x.clone() for x in got]

    eng.set_state(ctx, root, h, ctx_bound=20)
    if pending:
        one()                                # its copy of the context lengths stays pending: nothing polls before the capture
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        one()
    if not pending:
        for i in range(48):
            one(beams())
            if i % 8 == 7:
                eng.poll()
        eng.set_ctx_bound(20)
    put()
    one()
    want = seen()
    for _ in range(2):
        put()
        g.replay()
        eng.poll()
        for a, b in zip(seen(), want):
            assert torch.equal(a, b)
    del g
    eng.close()


def test_a_captured_prompt_is_refused_and_the_capture_goes_on():
    from paper_2403_09919_b200.binding import RdError, ReDrafter
    cfg = dict(synth.CONFIGS["tiny"], max_ctx=200)
    eng = ReDrafter(cfg, synth.make_weights(cfg, "cuda:0"))
    prompt = [np.arange(1, 40)]
    eng.prefill(prompt)
    want = [x.clone() for x in (*eng.get_state(), *eng.draft())]
    beams, scores = [torch.zeros_like(x) for x in want[3:]]
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        with pytest.raises(RdError) as e:
            eng.prefill(prompt)
        eng.draft(beams, scores)
    assert e.value.code == 4
    g.replay()
    eng.poll()
    for a, b in zip(want, (*eng.get_state(), beams, scores)):
        assert torch.equal(a, b)
    del g
    eng.close()
