"""The one-launch forward hands partial sums to the next phase as words that are "not written" until they are: every
launch has to leave all of them unwritten again, whatever its rows, its phases and the calls before it."""
import pytest
import torch

from paper_2510_19705_b200 import inputs

pytestmark = pytest.mark.gpu


# residual projections cut into 8 parts (width 256, 2048) and 4 (2304); gate / up in equal parts and dealt out
@pytest.mark.parametrize("d_model,nq,nkv,hd,ff", [(256, 8, 2, 32, 704), (2048, 32, 8, 64, 5632), (2304, 18, 3, 128, 1472)])
def test_calls_do_not_depend_on_the_calls_before(lib, d_model, nq, nkv, hd, ff):
    cfg = inputs.model_cfg(3, d_model, nq, nkv, ff, 2000, "bf16", head_dim=hd)
    w = inputs.make_weights(cfg, 5, device="cuda")
    tokens = inputs.make_prompts(cfg["vocab"], 1, 40, 9)[0].cuda().contiguous()

    def engine(folded=True):
        eng = lib.Hsd(cfg, w, (1, 3), (2,), max_batch=6, max_seq=160)
        if not folded:
            eng.set_phase_folding(False, False, False)
        return eng

    def call(eng, kind, n, batch):
        if kind == "layers":
            return [eng.layer_logits(tokens[:n], [1, 3])]
        toks, stats, _ = eng.generate(inputs.make_prompts(cfg["vocab"], batch, n, n).cuda(), 24, n)
        return [toks, torch.tensor([[s[k] for k in ("calls", "rows", "accepted", "emitted")] for s in stats])]

    # prompts of up to four tokens are a pass without logits of at most three rows; six sequences have more rows than fold
    calls = [("gen", 24, 1), ("gen", 3, 1), ("layers", 40, 1), ("gen", 100, 6), ("gen", 2, 6), ("layers", 1, 1), ("gen", 24, 1), ("gen", 17, 3)]
    used, separate = engine(), engine(folded=False)
    for c in calls:
        alone = engine()
        want = call(alone, *c)
        for eng in (used, separate):
            for a, b in zip(call(eng, *c), want):
                assert torch.equal(a, b), c
        alone.close()
    used.close()
    separate.close()


def test_first_pass_on_another_stream_finds_the_buffers_filled(lib):
    """A context is created on the default stream; its first pass may run on one that does not wait for that stream."""
    cfg = inputs.model_cfg(3, 256, 8, 2, 704, 2000, "bf16", head_dim=32)
    w = inputs.make_weights(cfg, 5, device="cuda")
    prompt = inputs.make_prompts(cfg["vocab"], 1, 24, 24).cuda()
    torch.cuda.synchronize()
    side, outs = torch.cuda.Stream(), []
    for stream in (torch.cuda.current_stream(), side):
        eng = lib.Hsd(cfg, w, (1, 3), (2,), max_batch=6, max_seq=4096)
        with torch.cuda.stream(stream):
            outs.append(eng.generate(prompt, 24, 3)[0])
        stream.synchronize()
        eng.close()
    assert torch.equal(outs[0], outs[1])


# k-blocks of a CTA's part of the down projection, with eight parts of width 256 and a ring of eight slots: some without a
# second one, one turn less one, one, one and one more, several with a remainder
@pytest.mark.parametrize("blocks_of_8_parts", [7, 8, 11, 56, 64, 72, 136])
def test_built_down_projections_of_any_length(lib, blocks_of_8_parts):
    """Passes of up to four rows build the down projection's activations in the ring slots; the activation producer steps over
    as many slots and takes up the next projection's tiles behind them."""
    cfg = inputs.model_cfg(3, 256, 8, 2, 64 * blocks_of_8_parts, 2000, "bf16", head_dim=32)
    w = inputs.make_weights(cfg, 5, device="cuda")
    prompt, outs = inputs.make_prompts(cfg["vocab"], 1, 24, 24).cuda(), []
    for folded in (True, False):
        eng = lib.Hsd(cfg, w, (1, 3), (2,), max_batch=1, max_seq=160)
        eng.set_phase_folding(True, folded, True)
        outs.append(eng.generate(prompt, 100, 3)[0])
        eng.close()
    assert torch.equal(outs[0], outs[1])


def test_thousands_of_passes(lib):
    """Hand-overs that fail once in a million fail in long runs: 3000 tokens through 48 layers, about 4000 passes, 148 CTAs."""
    cfg = inputs.model_cfg(48, 256, 8, 2, 1408, 2000, "bf16", head_dim=32)
    w = inputs.make_weights(cfg, 5, device="cuda")
    prompt, outs = inputs.make_prompts(cfg["vocab"], 1, 24, 24).cuda(), []
    eng = lib.Hsd(cfg, w, (8, 48), (2,), max_batch=1, max_seq=3072)
    for _ in range(2):
        outs.append(eng.generate(prompt, 3000, 3)[0])
    eng.close()
    assert torch.equal(outs[0], outs[1])


def _grid_counters(eng, cfg, max_seq, T, n_levels):
    """The two barrier counters of a context of one sequence (bf16, head size 32, pages of 16): one line of 64 bytes each."""
    from paper_2510_19705_b200 import binding
    up = lambda n: (n + 255) // 256 * 256
    slots = [sum(T[:i + 1]) + 1 for i in range(n_levels)]
    parts = [4 * max_seq, 4 * ((max_seq + 15) // 16)] + [s * cfg["vocab"] * 2 for s in slots]
    parts += [binding.hsd_verify_workspace_bytes(1, sum(T) + 1), 256 + 4, up(128 * 40 + 96 + 40 + 1024) * 48]
    base = (-eng.workspace.data_ptr()) % 256
    off = base + sum(up(n) for n in parts)
    return eng.workspace[off:off + 256].view(torch.int32).view(4, 16)[:2, 0]


def test_a_wait_that_runs_out_ends_with_an_error(lib):
    """Barrier counters far below anything the launch can count up to: the first barrier's waits, and those of the roles behind
    it, run out after two seconds.  The call reports it, and the GPU goes on."""
    cfg = inputs.model_cfg(3, 256, 8, 2, 704, 2000, "bf16", head_dim=32)
    w = inputs.make_weights(cfg, 5, device="cuda")
    prompt = inputs.make_prompts(cfg["vocab"], 1, 24, 24).cuda()
    eng = lib.Hsd(cfg, w, (1, 3), (2,), max_batch=1, max_seq=160)
    want = eng.generate(prompt, 24, 3)[0]
    counters, sms = _grid_counters(eng, cfg, 160, (2,), 2), torch.cuda.get_device_properties(0).multi_processor_count
    seen = sorted(counters.tolist())
    assert seen[0] == 0 and seen[1] > 0 and seen[1] % sms == 0, seen         # these are the counters: cleared, and one pass's arrivals
    counters.fill_(-2 ** 30)
    torch.cuda.synchronize()
    with pytest.raises(lib.HsdError, match="timed out"):
        eng.generate(prompt, 24, 3)
    eng.close()
    eng = lib.Hsd(cfg, w, (1, 3), (2,), max_batch=1, max_seq=160)
    assert torch.equal(eng.generate(prompt, 24, 3)[0], want)
    eng.close()


def test_creation_waits_for_work_on_the_memory_it_is_given(lib):
    """The workspace may be a block whose last user, on a stream the default one does not wait for, is still writing to it."""
    cfg = inputs.model_cfg(3, 256, 8, 2, 704, 2000, "bf16", head_dim=32)
    w = inputs.make_weights(cfg, 5, device="cuda")
    prompt = inputs.make_prompts(cfg["vocab"], 1, 24, 24).cuda()
    eng = lib.Hsd(cfg, w, (1, 3), (2,), max_batch=6, max_seq=160)
    want, size = eng.generate(prompt, 24, 3)[0], eng.workspace.numel()
    eng.close()
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):
        block = torch.empty(size, dtype=torch.uint8, device="cuda")
        where = block.data_ptr()
        torch.cuda._sleep(200_000_000)               # about 0.1 s
        block.zero_()
        del block
        eng = lib.Hsd(cfg, w, (1, 3), (2,), max_batch=6, max_seq=160)
        assert eng.workspace.data_ptr() == where     # the allocator handed the block on
        got = eng.generate(prompt, 24, 3)[0]
    torch.cuda.synchronize()
    assert torch.equal(got, want)
    eng.close()


def test_heads_are_in_place_for_a_pass_on_another_stream(lib):
    """New output heads go up on the default stream; the next pass may run on one that does not wait for that stream."""
    cfg = inputs.model_cfg(3, 256, 8, 2, 704, 2000, "bf16", head_dim=32)
    w, other = (inputs.make_weights(cfg, seed, device="cuda") for seed in (5, 6))
    prompt = inputs.make_prompts(cfg["vocab"], 1, 24, 24).cuda()
    torch.cuda.synchronize()
    eng, side = lib.Hsd(cfg, w, (1, 3), (2,), max_batch=1, max_seq=160), torch.cuda.Stream()
    heads, outs = [[None, None], [{"lm_head": other["lm_head"]}, {"lm_head": other["lm_head"]}]], {}
    for turn in range(6):
        for i, h in enumerate(heads):
            eng.set_exit_heads(h)
            with torch.cuda.stream(side if turn else torch.cuda.current_stream()):
                got = eng.generate(prompt, 24, 3)[0]
            torch.cuda.synchronize()
            assert torch.equal(got, outs.setdefault(i, got)), (turn, i)
    assert not torch.equal(outs[0], outs[1])
    eng.close()
