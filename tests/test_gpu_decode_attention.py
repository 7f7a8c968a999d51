"""The persistent decode step at the edges of its attention phase and of its data
exchange: one page and one split, the step that opens a page, more pages than
splits, the largest group (its states leave room for fewer page sets than warps),
and CTAs that have no rows of a phase.  Against the fp64 oracle with the parity
rules of tests/parity.py."""
import pytest

import gen
import oracle
from tests.parity import run_teacher_forced

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2608_24204_gb300 import WiciModel  # noqa: E402

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
