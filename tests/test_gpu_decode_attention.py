"""The persistent decode step at the edges of its attention phase and of its data
exchange: one page and one split, the step that opens a page, more pages than
splits, the largest group (its states leave room for fewer page sets than warps),
and CTAs that have no rows of a phase.  Against the fp64 oracle with the parity
rules of tests/parity.py.  Its precision over long chains of pages, against 64 bits on
the cache's own K and V.  And a step that gives up half way and is run again."""
import math

import numpy as np
import pytest

import gen
import oracle
from tests.parity import run_teacher_forced

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2608_24204_gb300 import WiciModel, wici  # noqa: E402

GROUP8 = gen.TINY.with_(name="tiny-g8", hidden=512, n_q_heads=8, n_kv_heads=1, vocab=512)
WIDE_GROUP8 = gen.LLAMA_8B.with_(name="8b-g8", n_layers=1, n_kv_heads=4, ffn_dim=12288, vocab=512)


@pytest.mark.parametrize("cfg,prompt,steps", [
    (gen.TINY, 1, 18),          # a single cached key, then the first page fills and the second opens
    (gen.TINY, 509, 6),         # 32 splits: one page each, then two (513 keys)
    (GROUP8, 127, 4),           # group of eight at head_dim 64
    (WIDE_GROUP8, 126, 4),      # group of eight at head_dim 128: five page sets
    (gen.TINY.with_(name="tiny-narrow", ffn_dim=64, vocab=64), 40, 3),   # fewer rows than CTAs in every phase
])
def test_decode_attention_edges(cfg, prompt, steps):
    cfg = cfg.with_(prompt_len=prompt, decode_steps=steps)
    w = gen.make_weights(cfg)
    model = WiciModel(cfg, max_tokens=prompt + steps).load(w)
    ref = oracle.OracleModel(cfg, w, max_tokens=prompt + steps)
    run_teacher_forced(model, ref, [gen.make_prompt(cfg, prompt, seed=1)], steps, {})
    model.close()


def _aligned(t):   # the 256-byte aligned part of a model's buffer, as the library sees it
    return t[(-t.data_ptr()) % 256:]


@pytest.mark.parametrize("base,max_sms", [(gen.LLAMA_8B, 0), (gen.LLAMA_8B, 8), (gen.LLAMA_1B, 8)])
def test_decode_attention_precision_over_many_pages(base, max_sms):
    # 8000 keys on eight SMs: one split a head, 63 pages summed one after the other by each warp.
    # One layer without its MLP (wd = 0) and a large wo, so that the logits show the attention's
    # error; K and V are read from the cache, so their storage rounding drops out.
    # Tolerance: 2^-19, eight times below what operands of two bf16 terms would leave (2^-16).
    # Measured 7.0e-7 at the 8B widths (8.5e-7 for the scalar fp32 code this one replaced).
    ctx, steps, V = 8000, 2, 512
    cfg = base.with_(name="attn", n_layers=1, vocab=V, tied_embeddings=False, max_chunk=2048)
    H, d, nq, nkv = cfg.hidden, cfg.head_dim, cfg.n_q_heads, cfg.n_kv_heads
    g = torch.Generator(device="cuda").manual_seed(1)

    def normal(r, c, std, mean=0.0):
        return (torch.randn((r, c), generator=g, device="cuda") * std + mean).bfloat16()

    p = "layers.0."
    w = {"embed": normal(V, H, 0.02), "lm_head": normal(V, H, 0.02), "final_norm": normal(1, H, 0.1, 1.0),
         p + "attn_norm": normal(1, H, 0.1, 1.0), p + "ffn_norm": normal(1, H, 0.1, 1.0),
         p + "wq": normal(nq * d, H, 0.02), p + "wk": normal(nkv * d, H, 0.02), p + "wv": normal(nkv * d, H, 0.02),
         p + "wo": normal(H, nq * d, 0.2), p + "wg": normal(cfg.ffn_dim, H, 0.02),
         p + "wu": normal(cfg.ffn_dim, H, 0.02), p + "wd": normal(H, cfg.ffn_dim, 0.0)}
    m = WiciModel(cfg, max_tokens=ctx + steps, max_sms=max_sms)
    wici.wici_load_weights(m.ctx, [(n, (t.data_ptr(), 1), *t.shape) for n, t in w.items()])
    rng = np.random.RandomState(1)
    m.prefill(rng.randint(0, V, ctx).astype(np.int32))
    pages = (ctx + steps + 15) // 16
    kv = _aligned(m._kv)[:2 * pages * 2 * nkv * 16 * d].view(torch.bfloat16).view(pages, 2, nkv, 16, d)
    w = {n: t.double() for n, t in w.items()}

    def norm(x, gain):
        return x / torch.sqrt((x * x).mean() + float(np.float32(cfg.rms_eps))) * gain[0]

    for s in range(steps):
        tok, n = int(rng.randint(0, V)), ctx + s + 1
        got, _ = m.decode_step(tok, logits=True)
        k, v = (kv[:, i].permute(0, 2, 1, 3).reshape(-1, nkv, d)[:n].double() for i in (0, 1))
        x = w["embed"][tok]
        q = (w[p + "wq"] @ norm(x, w[p + "attn_norm"])).view(nq, d)
        ang = (n - 1) * cfg.rope_theta ** (-torch.arange(0, d, 2, dtype=torch.float64, device="cuda") / d)
        a, b = q[:, :d // 2], q[:, d // 2:]
        q = torch.cat([a * ang.cos() - b * ang.sin(), b * ang.cos() + a * ang.sin()], 1)
        o = torch.cat([torch.softmax(k[:, j * nkv // nq] @ q[j] / math.sqrt(d), 0) @ v[:, j * nkv // nq]
                       for j in range(nq)])
        want = w["lm_head"] @ norm(x + w[p + "wo"] @ o, w["final_norm"])
        err = float((torch.from_numpy(got).cuda().double() - want).norm() / want.norm())
        assert err <= 2.0 ** -19, f"rel-L2 {err:.2e}"
    m.close()


def test_a_step_that_gave_up_leaves_nothing_to_the_next():
    # Waits also end when an error is on record.  With one planted in the control words the step
    # below gives up half way: one of its two CTAs has two of the three KV heads, and the other
    # waits for them.  The words it had already handed over carry the tags of the step that is run
    # next, with another token, and must not be taken for that step's.
    cfg = gen.TINY.with_(name="tiny-3h", hidden=512, n_q_heads=3, n_kv_heads=3, vocab=512)
    w = gen.make_weights(cfg)
    ctx, epoch = 16000, 4
    prompt = gen.make_prompt(cfg, ctx, seed=1)
    models = [WiciModel(cfg, max_tokens=ctx + 8, max_chunk=2048, max_sms=2).load(w) for _ in range(2)]
    for m in models:
        m.prefill(prompt)
        m.decode_step(3)
    m, fresh = models
    ctrl = _aligned(m._ws)[:64].view(torch.int32)
    before = int(ctrl[epoch])
    ctrl[2] = 1                                           # the error word
    with pytest.raises(wici.WiciError) as e:
        m.decode_step(5)
    assert e.value.status == wici.WICI_E_TIMEOUT
    assert int(ctrl[epoch]) == before == 1, "the step was meant to give up before its end"
    assert int(ctrl[2]) == 0 and m.kv_len == ctx + 1
    for tok in (7, 11):
        want, wtok = fresh.decode_step(tok, logits=True)
        got, gtok = m.decode_step(tok, logits=True)
        np.testing.assert_array_equal(got, want)
        assert gtok == wtok
    m.close()
    fresh.close()
