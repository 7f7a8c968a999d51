"""Prefill GEMMs over the tile shapes their rule picks for short and ragged chunks:
tiles shared by two and four CTAs, activation boxes of 32 to 96 rows, both terms of up to
64 rows in one tile, pairs of CTAs on
256-row tiles, a chunk that ends one token into a tile, and widths whose last tile is
partly outside the matrix.  Against the fp64 oracle with the parity rules."""
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

W8B = gen.LLAMA_8B.with_(name="8b-1l", n_layers=1, vocab=512)
W1B = gen.LLAMA_1B.with_(name="1b-1l", n_layers=1, vocab=512)
RAGGED = gen.TINY.with_(name="ragged", hidden=512, n_q_heads=12, n_kv_heads=4, ffn_dim=1000, vocab=512)


@pytest.mark.parametrize("cfg,prompt,chunk,q8", [
    (W8B, 1, 2048, False),
    (W8B, 33, 2048, False),
    (W8B, 64, 2048, False),      # the two terms stacked in one tile
    (W8B, 65, 2048, False),
    (W8B, 96, 2048, False),
    (W8B, 97, 2048, False),
    (W8B, 129, 2048, False),
    (W8B, 70, 64, False),        # a full 64-token chunk, then one of six
    (W8B, 61, 2048, True),
    (W1B, 40, 2048, False),
    (W1B, 300, 2048, False),
    (W8B, 257, 2048, False),     # pairs of CTAs: a second 256-row tile of one row
    (W8B, 640, 2048, False),
    (W1B, 1100, 2048, False),
    (W8B, 300, 2048, True),
    (RAGGED, 50, 2048, False),
    (RAGGED, 200, 2048, False),
    (RAGGED, 1500, 2048, False),
])
def test_prefill_tile_choices(cfg, prompt, chunk, q8):
    cfg = cfg.with_(prompt_len=prompt, decode_steps=1)
    w = gen.make_weights(cfg)
    q8w = gq.make_q8_weights(cfg) if q8 else None
    model = WiciModel(cfg, max_tokens=2048, max_chunk=chunk, q8=q8).load(w, q8w)
    ref = oracle.OracleModel(cfg, w, max_tokens=2048, q8_weights=q8w)
    run_teacher_forced(model, ref, [gen.make_prompt(cfg, prompt, seed=1)], 1, {})
    model.close()
