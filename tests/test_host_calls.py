"""The binding's native calls check their arguments as the C ABI's callers expect, without a GPU; on one, given outputs are
the ones returned."""
import pytest
import torch

from paper_2510_19705_b200 import binding, inputs


def test_arguments_are_checked_without_a_gpu():
    logits = torch.zeros(2, 3, 8)
    for call in (lambda: binding.hsd_draft_sample(logits, 0, 0), lambda: binding.hsd_verify_level(1, logits, logits, None, 0, 0),
                 lambda: binding.hsd_gemm_bf16(torch.zeros(4, 64, dtype=torch.bfloat16), torch.zeros(8, 64, dtype=torch.bfloat16))):
        with pytest.raises(binding.HsdError, match="contiguous CUDA tensor"):
            call()
    with pytest.raises(binding.HsdError, match="unsupported shape R=4 N=8 K=100"):
        binding.hsd_gemm_bf16(torch.zeros(4, 100), torch.zeros(8, 100))
    with pytest.raises(ValueError):
        binding.hsd_draft_sample(logits[0], 0, 0)
    with pytest.raises(TypeError):
        binding.hsd_draft_sample(None, 0, 0)


@pytest.mark.gpu
def test_given_outputs_are_returned_and_errors_raised(lib):
    p, q = inputs.make_accept_logits(2, 2, 512, seed=1, device="cuda", dtype="fp32")
    x = torch.empty(2, 2, dtype=torch.int32, device="cuda")
    assert lib.hsd_draft_sample(q, -1, 0, x) is x                      # seeds are taken modulo 2^64
    assert torch.equal(x, lib.hsd_draft_sample(q, 2 ** 64 - 1, 0))
    out, n = torch.empty(2, 3, dtype=torch.int32, device="cuda"), torch.empty(2, dtype=torch.int32, device="cuda")
    got = lib.hsd_verify_level(1, p, q, x, 7, 0, out_tokens=out, out_n_accepted=n)
    assert got[0] is out and got[1] is n
    want = lib.hsd_verify_level(1, p, q, x, 7, 0)
    assert torch.equal(out, want[0]) and torch.equal(n, want[1])
    with pytest.raises(lib.HsdError, match="contiguous CUDA tensor"):
        lib.hsd_draft_sample(q.transpose(0, 1), 0, 0)
    with pytest.raises(lib.HsdError, match="unsupported logits dtype"):
        lib.hsd_draft_sample(q.half(), 0, 0)
    with pytest.raises(lib.HsdError, match="workspace too small"):
        lib.hsd_verify_level(1, p, q, x, 0, 0, workspace=torch.empty(16, dtype=torch.uint8, device="cuda"))
    with torch.cuda.stream(torch.cuda.Stream()) as s:
        side = lib.hsd_verify_level(1, p, q, x, 7, 0)
        torch.cuda.current_stream().synchronize()
    assert torch.equal(side[0], want[0]) and torch.equal(side[1], want[1])
