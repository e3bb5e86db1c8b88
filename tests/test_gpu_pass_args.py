"""Row lists and decisions of small passes travel in kernel parameters and mapped memory, those of larger ones in copies: the
decision log and the tokens have to tell the same story on either side of the line."""
import numpy as np
import pytest

from paper_2510_19705_b200 import inputs

pytestmark = pytest.mark.gpu


def _run(lib, model, batch, prompt_len, n_new, T, path):
    wl = inputs.WORKLOADS[model]
    cfg = wl["model"]
    w = inputs.make_weights(cfg, wl["weight_seed"], device="cuda")
    eng = lib.Hsd(cfg, w, wl["exits"], T, max_batch=batch, max_seq=prompt_len + n_new + sum(T) + 16)
    prompt = inputs.make_prompts(cfg["vocab"], batch, prompt_len, 3).cuda()
    eng.set_trace(path, 0)
    tokens, stats, _ = eng.generate(prompt, n_new, 11)
    eng.set_trace(None)
    return tokens.cpu().numpy(), stats, lib.read_trace(path)


@pytest.mark.parametrize("model,batch,prompt_len,T", [("tiny3", 1, 5, (1, 1)), ("tiny3", 8, 9, (3, 2)), ("tiny3", 9, 9, (3, 2)), ("tiny3", 2, 150, (15, 3)),
                                                      ("mini3", 8, 24, (1, 1)), ("mini3", 9, 24, (1, 1)), ("mini3", 5, 20, (6, 2))])
def test_log_and_tokens_agree(lib, tmp_path, model, batch, prompt_len, T):
    n_new = 20
    tokens, stats, recs = _run(lib, model, batch, prompt_len, n_new, T, str(tmp_path / "log"))
    again, stats2, recs2 = _run(lib, model, batch, prompt_len, n_new, T, str(tmp_path / "log2"))
    assert np.array_equal(tokens, again) and len(recs) == len(recs2)
    top = len(T)
    for b in range(batch):
        stream = {}                                                    # position -> token, as the records say
        for r in (r for r in recs if r["seq"] == b):
            if r["level"] == 0:
                for j, tok in enumerate(r["tokens"]):
                    stream[r["ctx_len"] + j] = int(tok)
                continue
            t, n = r["t"], r["n"]
            # a verification's drafts are what the level below left there; it keeps n of them and its own token
            assert [stream[r["ctx_len"] + j] for j in range(t)] == [int(v) for v in r["tokens"][:t]]
            stream[r["ctx_len"] + n] = int(r["tokens"][t])
            for pos in [p for p in stream if p > r["ctx_len"] + n]:
                del stream[pos]
        assert [stream[prompt_len + j] for j in range(n_new)] == tokens[b].tolist()
        assert sum(r["n"] for r in recs if r["seq"] == b and r["level"] == top) > 0 or n_new < 5
    for i in range(1, top + 1):
        assert sum(r["n"] for r in recs if r["level"] == i) == stats[i]["accepted"]
