"""The decode step of widths without an instantiation of their own: each phase's shape
is picked at run time from K, so every chunk count of hidden, n_q * head_dim and ffn
is met once, tails included; and a context on fewer SMs than it has KV heads.  Against
the fp64 oracle with the parity rules of tests/parity.py."""
import pytest

import gen
import oracle
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
    (_cfg(512, 16, 8, 64, 704), 3),           # eight KV heads on three SMs
])
def test_decode_step_of_any_widths(cfg, max_sms):
    w = gen.make_weights(cfg)
    model = WiciModel(cfg, max_tokens=64, max_sms=max_sms).load(w)
    ref = oracle.OracleModel(cfg, w, max_tokens=64)
    run_teacher_forced(model, ref, [gen.make_prompt(cfg, cfg.prompt_len, seed=1)], cfg.decode_steps, {})
    model.close()
