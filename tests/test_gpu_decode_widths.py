"""The decode step of widths without an instantiation of their own: each phase's shape
is picked at run time from K, so every chunk count that hidden, n_q * head_dim and ffn
can have is met (1 to 4, 1 to 8 and 1 to 8), tails included; and contexts on fewer SMs
than they have KV heads, which run the same kernel (with the q/k norm too) or, in the
8-bit format, their own.  Against the fp64 oracle with the parity rules of tests/parity.py."""
import pytest

import gen
import oracle
from gen import q8 as gq
from tests.parity import run_teacher_forced

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2608_24204_gb300 import WiciModel  # noqa: E402


def _cfg(hidden, nq, nkv, d, ffn):
    return gen.TINY.with_(name="any", n_layers=2, hidden=hidden, n_q_heads=nq, n_kv_heads=nkv, head_dim=d, ffn_dim=ffn,
                          vocab=512, prompt_len=20, decode_steps=3)


@pytest.mark.parametrize("cfg,max_sms", [
    (_cfg(512, 16, 8, 64, 2056), 0),          # chunks per thread: hidden 1, n_q d 1, ffn 2
    (_cfg(3072, 24, 8, 128, 8192), 0),        # 2, 2, 4
    (_cfg(2048, 40, 8, 128, 6000), 0),        # 1, 3, 3
    (_cfg(6144, 16, 4, 128, 10000), 0),       # 3, 1, 5
    (_cfg(8192, 56, 8, 128, 1024), 0),        # 4, 4, 1
    (_cfg(264, 96, 16, 128, 16384), 0),       # 1, 6, 8
    (_cfg(256, 128, 16, 128, 14000), 0),      # 1, 8, 7
    (_cfg(264, 80, 10, 128, 12000), 0),       # 1, 5, 6
    (_cfg(256, 112, 16, 128, 512), 0),        # 1, 7, 1
    (_cfg(512, 16, 8, 64, 704), 3),           # eight KV heads on three SMs
    (gen.TINY.with_(qk_norm=True, decode_steps=3), 1),
    (gen.QWEN3_8B.with_(n_layers=1, vocab=512, prompt_len=20, decode_steps=3), 3),
])
def test_decode_step_of_any_widths(cfg, max_sms):
    w = gen.make_weights(cfg)
    model = WiciModel(cfg, max_tokens=64, max_sms=max_sms).load(w)
    ref = oracle.OracleModel(cfg, w, max_tokens=64)
    run_teacher_forced(model, ref, [gen.make_prompt(cfg, cfg.prompt_len, seed=1)], cfg.decode_steps, {})
    model.close()


def test_decode_step_of_the_8_bit_format_on_fewer_sms_than_kv_heads():
    cfg = gen.TINY.with_(ffn_dim=768, prompt_len=20, decode_steps=3)
    w, q8w = gen.make_weights(cfg), gq.make_q8_weights(cfg)
    model = WiciModel(cfg, max_tokens=64, max_sms=1, q8=True).load(w, q8w)
    ref = oracle.OracleModel(cfg, w, max_tokens=64, q8_weights=q8w)
    run_teacher_forced(model, ref, [gen.make_prompt(cfg, cfg.prompt_len, seed=1)], cfg.decode_steps, {})
    model.close()
