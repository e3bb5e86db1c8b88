"""Long prompts: the many-row chunk path (tensor-bound GEMMs on CTA pairs, attention on tensor memory) against the
oracle, at the sizes where its tiles, items, pages and chunks end."""
import os
import tempfile

import numpy as np
import pytest
import torch

from oracle.transformer import Transformer
from paper_2510_19705_b200 import binding, inputs

pytestmark = pytest.mark.gpu

# head size, query heads, KV heads, page, batch, prompt length.  Rows of a chunk = prompt - 1 per sequence.
CASES = [
    (128, 4, 1, 16, 1, 130),       # 129 rows: the fewest of this path, one row in the second A half
    (128, 4, 1, 16, 1, 257),       # 256 rows: exactly one token tile
    (128, 4, 1, 32, 3, 150),       # several sequences in one chunk, items that end inside a tile
    (128, 8, 8, 16, 2, 300),       # no grouped heads: 128 tokens per query tile
    (128, 8, 1, 64, 1, 210),       # eight heads to a group
    (128, 6, 2, 16, 1, 345),       # group of three: two rows of every query tile unused
    (64, 8, 4, 16, 1, 391),        # head size 64: two heads per accumulator half
    (64, 4, 2, 32, 2, 1300),       # 2598 rows: two chunks, the second starting inside a sequence
    (64, 4, 2, 16, 1, 2600),       # head size 64 well past 2048 keys
    (128, 4, 1, 16, 1, 2433),      # 2432 rows: a full chunk and one of 128 rows
    (128, 4, 1, 16, 9, 16),        # 135 rows of nine short prompts
]


@pytest.mark.parametrize("hd,nq,nkv,page,batch,prompt", CASES)
def test_prompt_chunks_match_oracle(hd, nq, nkv, page, batch, prompt):
    # 704 = 11 x 64 feed-forward columns: a half-empty last gate / up tile
    cfg = inputs.model_cfg(3, 256, nq, nkv, 704, 1024, "bf16", head_dim=hd)
    w = inputs.make_weights(cfg, 11)
    for layer in w["layers"]:          # scores of unit size: the softmax is not flat
        layer["wq"].mul_(3.0)
        layer["wk"].mul_(3.0)
    w_gpu = {k: (v.cuda() if k != "layers" else [{a: t.cuda() for a, t in l.items()} for l in v]) for k, v in w.items()}
    prompts = inputs.make_prompts(cfg["vocab"], batch, prompt, 3)
    eng = binding.Hsd(cfg, w_gpu, (1, 3), (2,), max_batch=batch, max_seq=prompt + 32, page_size=page)
    with tempfile.TemporaryDirectory() as tmp:
        path = os.path.join(tmp, "trace.bin")
        eng.set_trace(path, logit_calls=2 * batch)
        eng.generate(prompts.cuda(), 2, 5)
        eng.set_trace(None)
        recs = binding.read_trace(path)
    eng.close()
    om = Transformer(cfg, inputs.weights_to_numpy(w), (1, 3))
    for b in range(batch):
        rec = next(r for r in recs if r["level"] == 1 and r["seq"] == b)
        om.reset()
        om.rows(1, prompts[b].tolist(), rec["tokens"][:-1].tolist())
        # the bound of the other bf16 parity tests: 2e-2 on logits of standard deviation 0.02 sqrt(256) = 0.32
        err = float(np.abs(om.last_logits64 - rec["logits"]).max())
        assert err < 2e-2, (b, err)
        # over all logits: the oracle rounds where the kernels do (7 points a layer, the head's two), so at worst every point
        # has tipped independently, 2^-9 / sqrt(3) of its values each: sqrt(23) x 1.13e-3 = 5.4e-3, and half as much again
        rel = float(np.linalg.norm(om.last_logits64 - rec["logits"]) / np.linalg.norm(om.last_logits64))
        assert rel < 8.1e-3, (b, rel)


@pytest.mark.parametrize("hd,nq,nkv,batch,prompt", [
    (128, 4, 1, 8, 300),           # 2392 rows: the last 88 of the last sequence are a chunk of their own
    (64, 8, 4, 2, 2100),           # the second sequence starts in the middle of a chunk: other items, other key ranges
    (128, 4, 1, 2, 2100)])
def test_a_prompt_does_not_depend_on_its_place_in_the_batch(hd, nq, nkv, batch, prompt):
    # the same prompt as every sequence of a batch: the chunks cut each of them somewhere else
    cfg = inputs.model_cfg(3, 256, nq, nkv, 704, 1024, "bf16", head_dim=hd)
    w = inputs.make_weights(cfg, 11, device="cuda")
    prompts = inputs.make_prompts(cfg["vocab"], 1, prompt, 3).repeat(batch, 1)
    eng = binding.Hsd(cfg, w, (1, 3), (2,), max_batch=batch, max_seq=prompt + 32)
    with tempfile.TemporaryDirectory() as tmp:
        path = os.path.join(tmp, "trace.bin")
        eng.set_trace(path, logit_calls=2 * batch)
        eng.generate(prompts.cuda(), 2, 5)
        eng.set_trace(None)
        recs = binding.read_trace(path)
    eng.close()
    rows = [next(r for r in recs if r["level"] == 1 and r["seq"] == b)["logits"][0] for b in range(batch)]
    for b in range(1, batch):
        assert np.array_equal(rows[b], rows[0]), b


@pytest.mark.parametrize("seed", [5, 6])
def test_prompt_residual_sums_are_short_chains(seed):
    """The tensor core drops what lies below its accumulator's last bit at every step of 16 columns.  A down projection whose
    first 16 columns add a large term and whose last 16 take it away again shows how many steps had it in the accumulator: 128
    (a quarter of 8192 columns), half a bit of it each, 0.8 % of the result here (512 in one chain, 3 %); the bf16 roundings of
    the second layer and the logits add 0.5 %, and the two seeds' terms differ by half as much again."""
    cfg = inputs.model_cfg(2, 256, 4, 2, 8192, 1024, "bf16", head_dim=64)
    w = inputs.make_weights(cfg, seed)
    first, second = w["layers"]
    first["wo"].zero_()                                              # layer 1: embedding + down projection
    for name in ("wg", "wu"):
        first[name][-16:] = first[name][:16]                         # the last 16 activations equal the first 16
    first["wd"].mul_(32.0)
    first["wd"][:, :16] = 2.0 ** 15 * torch.sign(first["wd"][:, :16].float()).to(torch.bfloat16)
    first["wd"][:, -16:] = -first["wd"][:, :16]
    second["wo"].mul_(64.0)                                          # layer 2: the attention over the prompt's rows outweighs the row itself
    w_gpu = {k: (v.cuda() if k != "layers" else [{a: t.cuda() for a, t in l.items()} for l in v]) for k, v in w.items()}
    prompts = torch.full((1, 300), 7, dtype=torch.int32)             # equal rows: the attention returns their value
    eng = binding.Hsd(cfg, w_gpu, (1, 2), (1,), max_batch=1, max_seq=332)
    with tempfile.TemporaryDirectory() as tmp:
        path = os.path.join(tmp, "trace.bin")
        eng.set_trace(path, logit_calls=2)
        eng.generate(prompts.cuda(), 1, 5)
        eng.set_trace(None)
        rec = next(r for r in binding.read_trace(path) if r["level"] == 1)
    eng.close()
    om = Transformer(cfg, inputs.weights_to_numpy(w), (1, 2))
    om.rows(1, prompts[0].tolist(), rec["tokens"][:-1].tolist())
    want = om.last_logits64[0]
    rel = float(np.linalg.norm(rec["logits"][0] - want) / np.linalg.norm(want))
    assert rel < 1.5e-2, rel


@pytest.mark.parametrize("hd,nq,nkv,prompt", [(128, 4, 1, 300), (64, 8, 4, 700)])
def test_chains_of_early_launches_follow_the_work_before_them(hd, nq, nkv, prompt):
    """The kernels of a prompt and of layer logits start early, one after the other, but not ahead of what was on the stream
    before the call: tokens and weights that arrive there right before it, behind 50 ms of other work, are the ones it uses."""
    cfg = inputs.model_cfg(3, 256, nq, nkv, 704, 1024, "bf16", head_dim=hd)
    w, other = (inputs.make_weights(cfg, seed, device="cuda") for seed in (11, 12))
    prompts = inputs.make_prompts(cfg["vocab"], 1, prompt, 3).cuda()

    def flat(weights):
        return [t for k, v in sorted(weights.items()) for t in ([v] if k != "layers" else [l[n] for l in v for n in sorted(l)])]

    def calls(eng, tokens):
        return eng.layer_logits(tokens[0, :100].contiguous(), [1, 3]), eng.generate(tokens, 16, 5)[0]

    eng = binding.Hsd(cfg, w, (1, 3), (2,), max_batch=1, max_seq=prompt + 64)
    want = calls(eng, prompts)
    with torch.cuda.stream(torch.cuda.Stream()):
        for late in range(2):                        # before the layer logits, before the prompt
            right = [t.clone() for t in flat(w)]
            tokens = torch.zeros_like(prompts)
            for t, o in zip(flat(w), flat(other)):
                t.copy_(o)
            torch.cuda._sleep(100_000_000)
            for t, r in zip(flat(w), right):
                t.copy_(r)
            tokens.copy_(prompts)
            got = calls(eng, tokens) if late == 0 else (want[0], eng.generate(tokens, 16, 5)[0])
            assert all(torch.equal(a, b) for a, b in zip(got, want)), late
    eng.close()
