"""Small fp32 models: a pass in one launch per 128 rows, against the oracle, where the row tiles, staged chunks,
head sizes and the vocabulary end."""
import os
import tempfile

import numpy as np
import pytest

from oracle.transformer import Transformer
from paper_2510_19705_b200 import binding, inputs

pytestmark = pytest.mark.gpu


# width, query heads, KV heads, head size, feed-forward width, vocabulary, page, batch, prompt, T_0
@pytest.mark.parametrize("d,nq,nkv,hd,ff,V,page,batch,prompt,T0", [
    (128, 4, 4, 32, 512, 512, 16, 1, 33, 3),       # prompt pass of 32 rows: two row tiles
    (132, 2, 1, 64, 516, 333, 4, 3, 9, 4),         # an odd vocabulary, a second chunk of 4 columns, 15 rows a target pass
    (256, 2, 2, 128, 700, 1000, 64, 4, 7, 6),      # head size 128; 28 rows a target pass
    (96, 6, 2, 32, 300, 64, 16, 1, 300, 2)])       # 300 keys: a warp's second key tile; the prompt in launches per operation
def test_small_fp32_passes_match_oracle(d, nq, nkv, hd, ff, V, page, batch, prompt, T0):
    cfg = inputs.model_cfg(3, d, nq, nkv, ff, V, "fp32", head_dim=hd)
    w = inputs.make_weights(cfg, 13)
    w_gpu = {k: (v.cuda() if k != "layers" else [{a: t.cuda() for a, t in l.items()} for l in v]) for k, v in w.items()}
    prompts = inputs.make_prompts(V, batch, prompt, 4)
    eng = binding.Hsd(cfg, w_gpu, (1, 3), (T0,), max_batch=batch, max_seq=prompt + 40, page_size=page)
    with tempfile.TemporaryDirectory() as tmp:
        path = os.path.join(tmp, "trace.bin")
        eng.set_trace(path, logit_calls=10 ** 6)
        eng.generate(prompts.cuda(), 6, 5)
        eng.set_trace(None)
        recs = binding.read_trace(path)
    eng.close()
    om = Transformer(cfg, inputs.weights_to_numpy(w), (1, 3))
    for b in range(batch):
        rec = next(r for r in recs if r["level"] == 1 and r["seq"] == b)
        om.reset()
        om.rows(1, prompts[b].tolist(), rec["tokens"][:-1].tolist())
        err = float(np.abs(om.last_logits64 - rec["logits"]).max())
        assert err < 1e-5, (b, err)                # the bound of the other fp32 parity tests


@pytest.mark.parametrize("d,nq,nkv,hd,ff,V,prompt", [(128, 4, 4, 32, 512, 512, 16), (256, 4, 2, 64, 700, 1001, 70)])
def test_small_fp32_rows_do_not_depend_on_the_batch(d, nq, nkv, hd, ff, V, prompt):
    """Sequence 0 alone, in a batch whose passes have more than 32 rows, and in one whose passes have more than 128: the
    same logits bit for bit in every pass."""
    cfg = inputs.model_cfg(3, d, nq, nkv, ff, V, "fp32", head_dim=hd)
    w = inputs.make_weights(cfg, 13, device="cuda")
    prompts = inputs.make_prompts(V, 40, prompt, 4)
    seen = []
    for batch in (1, 9, 40):
        eng = binding.Hsd(cfg, w, (1, 3), (4,), max_batch=batch, max_seq=prompt + 40)
        with tempfile.TemporaryDirectory() as tmp:
            path = os.path.join(tmp, "trace.bin")
            eng.set_trace(path, logit_calls=10 ** 6)
            toks, _, _ = eng.generate(prompts[:batch].cuda(), 8, 5)
            eng.set_trace(None)
            recs = [r for r in binding.read_trace(path) if r["seq"] == 0]
        eng.close()
        seen.append((toks[0].cpu().numpy(), [(r["level"], r["logits"]) for r in recs]))
    for toks, recs in seen[1:]:
        assert np.array_equal(toks, seen[0][0]) and len(recs) == len(seen[0][1])
        for (level, a), (want_level, b) in zip(recs, seen[0][1]):
            assert level == want_level and np.array_equal(a, b)
