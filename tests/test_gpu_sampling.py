"""Parity of the sampling kernels with the oracle on identical logits (decisions are bit-exact)."""
import numpy as np
import pytest
import torch

from oracle import philox, sampling
from paper_2510_19705_b200 import inputs

pytestmark = pytest.mark.gpu


def _oracle_draft(logits_np, seed, serial):
    B, R, V = logits_np.shape
    out = np.empty((B, R), dtype=np.int32)
    for b in range(B):
        for j in range(R):
            out[b, j] = sampling.categorical(logits_np[b, j], philox.uniform24(seed, j, serial, 0, philox.PURPOSE_DRAFT, b))
    return out


def _oracle_verify(level, p_np, q_np, x_np, seed, serial):
    """Algorithm 2's decisions on given rows, per sequence."""
    from oracle.hsd import SpecDecisions
    from oracle.verify import verify

    class Rows:
        def __init__(self, rows):
            self.r = rows

        def rows(self, idx, ctx, draft):
            return list(self.r)

    B, tp1, V = p_np.shape
    t = tp1 - 1
    out = np.full((B, t + 1), -1, dtype=np.int32)
    n_acc = np.empty(B, dtype=np.int32)
    for b in range(B):
        toks, _, _ = verify(level, list(x_np[b]), list(q_np[b]), [0], Rows(p_np[b]), SpecDecisions(seed, b), serial)
        out[b, :len(toks)] = toks
        n_acc[b] = len(toks) - 1
    return out, n_acc


@pytest.mark.parametrize("dtype,V,B,R", [("bf16", 32000, 6, 5), ("fp32", 512, 3, 4), ("bf16", 1000, 2, 3),
                                         ("fp32", 33, 2, 2), ("bf16", 50001, 1, 2)])
def test_draft_sample_matches_oracle(lib, dtype, V, B, R):
    _, q = inputs.make_accept_logits(B, R, V, seed=V + B, device="cuda", dtype=dtype)
    for seed, serial in [(0, 0), (12345678901234, 7)]:
        got = lib.hsd_draft_sample(q, seed, serial).cpu().numpy()
        want = _oracle_draft(inputs.logits_to_numpy(q), seed, serial)
        assert np.array_equal(got, want)


@pytest.mark.parametrize("dtype,V,B,t", [("bf16", 32000, 8, 8), ("fp32", 512, 4, 3), ("bf16", 4097, 3, 5),
                                         ("bf16", 32000, 2, 1), ("fp32", 7, 5, 2)])
def test_verify_level_matches_oracle(lib, dtype, V, B, t):
    p, q = inputs.make_accept_logits(B, t, V, seed=3 * V + t, device="cuda", dtype=dtype)
    x = lib.hsd_draft_sample(q, 99, 0)
    p_np, q_np, x_np = inputs.logits_to_numpy(p), inputs.logits_to_numpy(q), x.cpu().numpy()
    seen_n = set()
    for seed, serial, level in [(0, 0, 1), (5, 3, 2), (2 ** 40 + 17, 1000, 1)]:
        out, n = lib.hsd_verify_level(level, p, q, x, seed, serial)
        want_out, want_n = _oracle_verify(level, p_np, q_np, x_np, seed, serial)
        assert np.array_equal(n.cpu().numpy(), want_n)
        assert np.array_equal(out.cpu().numpy(), want_out)
        seen_n.update(want_n.tolist())
    assert len(seen_n) >= 2          # both accepted and rejected positions were exercised


def test_verify_edge_cases(lib):
    V = 64
    # t = 0: only the bonus draw from the single target row
    p, _ = inputs.make_accept_logits(3, 0, V, seed=1, device="cuda", dtype="fp32")
    out, n = lib.hsd_verify_level(1, p, None, None, 4, 2)
    p_np = inputs.logits_to_numpy(p)
    for b in range(3):
        U = philox.uniform24(4, 0, 2, 1, philox.PURPOSE_FINAL, b)
        assert n[b].item() == 0 and out[b, 0].item() == sampling.categorical(p_np[b, 0], U)
    # identical rows: everything is accepted (ratio 1), the bonus comes from the last target row
    p, _ = inputs.make_accept_logits(2, 4, V, seed=2, device="cuda", dtype="bf16")
    q = p[:, :4].contiguous()
    x = lib.hsd_draft_sample(q, 1, 0)
    out, n = lib.hsd_verify_level(1, p, q, x, 1, 0)
    assert n.tolist() == [4, 4] and torch.equal(out[:, :4], x)
    # a drafted token the target gives (almost) no mass is rejected and never re-emitted
    p = torch.zeros(1, 2, V, device="cuda")
    q = torch.zeros(1, 1, V, device="cuda")
    p[0, 0, 5] = -60.0
    x = torch.tensor([[5]], dtype=torch.int32, device="cuda")
    for seed in range(8):
        out, n = lib.hsd_verify_level(1, p, q, x, seed, 0)
        assert n.item() == 0 and out[0, 0].item() != 5 and out[0, 1].item() == -1


def test_acceptance_frequency_is_one_minus_tv(lib):
    # Section 2: P(accept) = 1 - sum |p - q| / 2 when x ~ q; measured over many sequences of the
    # same pair of rows (sequence index and serial vary the uniforms)
    V, B = 4096, 2048
    p1, q1 = inputs.make_accept_logits(1, 1, V, seed=8, device="cuda", dtype="bf16")
    p, q = p1.expand(B, 2, V).contiguous(), q1.expand(B, 1, V).contiguous()
    x = lib.hsd_draft_sample(q, 3, 0)
    _, n = lib.hsd_verify_level(1, p, q, x, 3, 0)
    alpha = sampling.acceptance_rate(sampling.softmax64(inputs.logits_to_numpy(p1)[0, 0]),
                                     sampling.softmax64(inputs.logits_to_numpy(q1)[0, 0]))
    freq = n.float().mean().item()
    assert abs(freq - alpha) < 4.5 * (alpha * (1 - alpha) / B) ** 0.5 + 1e-3


def test_bad_arguments_are_rejected(lib):
    p, q = inputs.make_accept_logits(2, 2, 32, seed=1, device="cuda", dtype="fp32")
    x = lib.hsd_draft_sample(q, 0, 0)
    small = torch.empty(16, dtype=torch.uint8, device="cuda")
    with pytest.raises(lib.HsdError, match="workspace too small"):
        lib.hsd_verify_level(1, p, q, x, 0, 0, workspace=small)
    with pytest.raises(lib.HsdError, match="invalid argument"):
        lib.hsd_verify_level(300, p, q, x, 0, 0)


@pytest.mark.parametrize("dtype,V,B,t", [("bf16", 4096, 3, 3),       # one CTA a sequence, every thread's eight tokens used
                                         ("bf16", 4098, 2, 2),       # two CTAs, the second with an odd tail of pairs
                                         ("bf16", 32000, 14, 2), ("bf16", 32000, 15, 2),    # clusters of eight / of four
                                         ("bf16", 65538, 1, 1),      # 32 tokens a thread
                                         ("bf16", 1536, 2, 31),      # the most rows a sequence can have here
                                         ("bf16", 512, 128, 16),     # one CTA a sequence, 33 rows each
                                         ("bf16", 2048, 16, 16), ("bf16", 2048, 64, 8),     # statistics of many short rows
                                         ("bf16", 30001, 2, 1), ("fp32", 32769, 1, 8), ("fp32", 24001, 40, 1), ("bf16", 9000, 2, 0)])
def test_cluster_decisions_match_oracle(lib, dtype, V, B, t):
    p, q = inputs.make_accept_logits(B, t, V, seed=V + 7 * t, device="cuda", dtype=dtype)
    p[0, :, V // 2:] = -float("inf")                                  # a mask over half the vocabulary
    x = lib.hsd_draft_sample(q, 5, 0) if t else None
    p_np, q_np = inputs.logits_to_numpy(p), inputs.logits_to_numpy(q)
    x_np = x.cpu().numpy() if t else np.zeros((B, 0), np.int32)
    if t:
        assert np.array_equal(x_np, _oracle_draft(q_np, 5, 0))
    for serial in range(3):
        out, n = lib.hsd_verify_level(1, p, q, x, 17, serial)
        want_out, want_n = _oracle_verify(1, p_np, q_np, x_np, 17, serial)
        assert np.array_equal(n.cpu().numpy(), want_n) and np.array_equal(out.cpu().numpy(), want_out)


@pytest.mark.parametrize("dtype,V,B", [("bf16", 32000, 2), ("bf16", 32000, 37), ("fp32", 32001, 18), ("bf16", 9000, 70)])
def test_cluster_draws_on_a_busy_gpu(lib, dtype, V, B):
    # clusters of eight, four and two whose CTAs start while another stream's kernels occupy SMs and shared memory: the
    # first exchange of a draw needs every CTA of its cluster on the GPU
    _, q = inputs.make_accept_logits(B, 1, V, seed=V + B, device="cuda", dtype=dtype)
    _, other = inputs.make_accept_logits(64, 4, 32000, seed=1, device="cuda", dtype="bf16")
    want = [_oracle_draft(inputs.logits_to_numpy(q), 31, s) for s in range(4)]
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    got = []
    for i in range(64):
        with torch.cuda.stream(side):
            lib.hsd_draft_sample(other, 8, i)
        got.append(lib.hsd_draft_sample(q, 31, i % 4))
    torch.cuda.synchronize()
    for i, x in enumerate(got):
        assert np.array_equal(x.cpu().numpy(), want[i % 4]), i


# Rows of up to 2048 tokens are taken by CTAs of 128 or 256 threads, longer ones by clusters where a cluster a row fits two rounds, else by
# the streaming kernel: its ring holds 229376 bytes; up to 148 rows one group of warps a CTA, three past that.
@pytest.mark.parametrize("dtype,V,B,t,shift", [("bf16", 32000, 19, 4, 0), ("fp32", 32001, 14, 6, 0),  # more rows than SMs
                                               ("bf16", 50000, 16, 5, 0),      # rows of four chunks, CTAs whose third group has no row
                                               ("bf16", 16385, 9, 8, 3),       # a second chunk of a few elements, rows that begin anywhere
                                               ("fp32", 57341, 30, 2, 1), ("fp32", 57345, 25, 3, 1),   # the longest rows in the ring; one element past it: twice through
                                               ("bf16", 114700, 31, 2, 3),     # twice through the ring, three groups, rows that begin anywhere
                                               ("fp32", 60000, 17, 2, 2),      # ... one group
                                               ("fp32", 57347, 1, 2, 0),       # clusters
                                               ("bf16", 65537, 11, 2, 1), ("fp32", 128256, 4, 3, 0), ("bf16", 131072, 8, 3, 0), ("fp32", 131072, 19, 1, 1),   # 32 tokens a
                                                                               # thread of a cluster up to 56 rows, the ring past them
                                               ("bf16", 131080, 2, 1, 0), ("fp32", 131081, 2, 1, 1),   # longer than the clusters of the decision take
                                               ("bf16", 5, 60, 2, 1), ("fp32", 3, 64, 2, 0), ("bf16", 64, 2, 40, 0),     # 128 threads; more drafts than lanes,
                                               ("fp32", 40, 1, 600, 2), ("bf16", 1024, 170, 3, 0), ("fp32", 1024, 3, 2, 1),   # ... than threads; every token
                                               ("bf16", 1025, 90, 3, 1), ("fp32", 1025, 2, 1, 0), ("bf16", 2048, 33, 4, 0),    # 256 threads
                                               ("bf16", 2049, 100, 1, 1), ("fp32", 2049, 60, 2, 0)])     # the shortest rows on the ring
def test_row_statistics_and_decisions_match_oracle(lib, dtype, V, B, t, shift):
    def moved(x):                                                      # the same values from element `shift` of a buffer on
        buf = torch.empty(x.numel() + shift, dtype=x.dtype, device="cuda")
        buf[shift:] = x.reshape(-1)
        return buf[shift:].view(x.shape)
    p, q = inputs.make_accept_logits(B, t, V, seed=V + t, device="cuda", dtype=dtype)
    p[0, :, V // 2:] = -float("inf")
    p, q = moved(p), moved(q)
    x = lib.hsd_draft_sample(q, 5, 0)
    p_np, q_np, x_np = inputs.logits_to_numpy(p), inputs.logits_to_numpy(q), x.cpu().numpy()
    for serial in range(2):
        out, n = lib.hsd_verify_level(1, p, q, x, 23, serial)
        want_out, want_n = _oracle_verify(1, p_np, q_np, x_np, 23, serial)
        assert np.array_equal(n.cpu().numpy(), want_n) and np.array_equal(out.cpu().numpy(), want_out)


def test_verifications_in_a_captured_graph_and_back_to_back(lib):
    # each call's kernels start under the end of the one before it; all share one workspace, and a call drafts from the rows
    # that a kernel of the same stream has just written
    B, t, V = 24, 3, 32000
    sets = [inputs.make_accept_logits(B, t, V, seed=s, device="cuda", dtype="bf16") for s in range(3)]
    p, q = torch.empty_like(sets[0][0]), torch.empty_like(sets[0][1])
    ws = torch.empty(lib.hsd_verify_workspace_bytes(B, t), dtype=torch.uint8, device="cuda")
    want = []
    for i, (pi, qi) in enumerate(sets):
        x = lib.hsd_draft_sample(qi, 3, i)
        want.append([v.cpu() for v in lib.hsd_verify_level(1, pi, qi, x, 9, i)])

    def chain():
        got = []
        for i in range(12):
            p.copy_(sets[i % 3][0])
            q.copy_(sets[i % 3][1])
            got.append(lib.hsd_verify_level(1, p, q, lib.hsd_draft_sample(q, 3, i % 3), 9, i % 3, workspace=ws))
        return got
    runs = [chain()]
    side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=side):
        captured = chain()
    graph.replay()
    torch.cuda.synchronize()
    for got in runs + [captured]:
        for i, (out, n) in enumerate(got):
            assert torch.equal(out.cpu(), want[i % 3][0]) and torch.equal(n.cpu(), want[i % 3][1]), i


@pytest.mark.parametrize("dtype,V,B", [("bf16", 2048, 3), ("fp32", 513, 300),      # one CTA a row; more rows than run at once
                                       ("bf16", 1024, 2400), ("fp32", 1024, 5), ("bf16", 1025, 301), ("fp32", 2048, 3), ("fp32", 2049, 3),    # 128, 256, 512 threads
                                       ("bf16", 32000, 112), ("bf16", 32000, 148), ("fp32", 32001, 75),   # several rounds of clusters, a row a CTA
                                       ("fp32", 9001, 149), ("bf16", 8190, 297)])
def test_draws_of_many_rows_match_oracle(lib, dtype, V, B):
    _, q = inputs.make_accept_logits(B, 1, V, seed=V + B, device="cuda", dtype=dtype)
    want = _oracle_draft(inputs.logits_to_numpy(q), 41, 2)
    got = [lib.hsd_draft_sample(q, 41, 2) for _ in range(3)]
    assert all(np.array_equal(x.cpu().numpy(), want) for x in got)


def _without_weight(kind, row):
    """A row of no finite weight."""
    row.fill_(float("nan") if kind == "nan" else -float("inf"))
    if kind == "+inf":
        row.normal_()
        row[row.numel() // 3] = float("inf")


@pytest.mark.parametrize("kind", ["-inf", "nan", "+inf"])
@pytest.mark.parametrize("dtype,V,B", [("bf16", 2048, 3), ("fp32", 32001, 5),      # clusters
                                       ("bf16", 32000, 148), ("fp32", 9001, 149)])  # a CTA a row, in chunks and not
def test_draws_of_rows_without_weight_give_no_token(lib, dtype, V, B, kind):
    _, q = inputs.make_accept_logits(B, 1, V, seed=V, device="cuda", dtype=dtype)
    want = _oracle_draft(inputs.logits_to_numpy(q), 3, 0)
    for b in (0, B - 1):
        _without_weight(kind, q[b, 0])
        want[b] = -1
    assert np.array_equal(lib.hsd_draft_sample(q, 3, 0).cpu().numpy(), want)


@pytest.mark.parametrize("kind", ["-inf", "nan", "+inf"])
@pytest.mark.parametrize("dtype,V,B,t", [("bf16", 2048, 3, 2), ("fp32", 32001, 4, 3),          # statistics by clusters
                                         ("bf16", 32000, 20, 2), ("fp32", 9001, 49, 3),        # streamed, one group and three
                                         ("fp32", 57345, 30, 2), ("bf16", 131080, 6, 1)])      # twice through the ring; a CTA a decision
def test_verifications_of_rows_without_weight(lib, dtype, V, B, t, kind):
    p, q = inputs.make_accept_logits(B, t, V, seed=V, device="cuda", dtype=dtype)
    q[:2] = p[:2, :t]                                                  # every draft accepted
    x = lib.hsd_draft_sample(q, 5, 0)
    for j in range(t):
        x[2, j] = p[2, j].float().argmax()
    p_np, q_np, x_np = inputs.logits_to_numpy(p), inputs.logits_to_numpy(q), x.cpu().numpy()
    # sequence 0: no weight in its last draft's target row: the draft is rejected and nothing can be drawn.  Sequence 1: in the bonus
    # row.  Sequence 2: in every draft row: q(x) = 0, every draft with weight in the target row is accepted.  For the oracle the first
    # is a target row with all its weight on another token.
    _without_weight(kind, p[0, t - 1])
    p_np[0, t - 1] = -np.inf
    p_np[0, t - 1, (x_np[0, t - 1] + 1) % V] = 0.0
    _without_weight(kind, p[1, t])
    for j in range(t):
        _without_weight(kind, q[2, j])
        q_np[2, j] = -np.inf
        q_np[2, j, (x_np[2, j] + 1) % V] = 0.0
    for serial in range(2):
        out, n = lib.hsd_verify_level(1, p, q, x, 23, serial)
        want_out, want_n = _oracle_verify(1, p_np, q_np, x_np, 23, serial)
        assert want_n[:3].tolist() == [t - 1, t, t]
        want_out[0, t - 1] = want_out[1, t] = -1
        assert np.array_equal(n.cpu().numpy(), want_n) and np.array_equal(out.cpu().numpy(), want_out)


def test_nan_logits_weigh_nothing(lib):
    p, q = inputs.make_accept_logits(9, 2, 32001, seed=2, device="cuda", dtype="bf16")
    p[:, :, 5::7] = float("nan")
    q[:, :, 3::11] = float("nan")
    x = lib.hsd_draft_sample(q, 5, 0)
    p_np, q_np = (np.where(np.isnan(a), -np.inf, a) for a in (inputs.logits_to_numpy(p), inputs.logits_to_numpy(q)))
    assert np.array_equal(x.cpu().numpy(), _oracle_draft(q_np, 5, 0))
    out, n = lib.hsd_verify_level(1, p, q, x, 23, 0)
    want_out, want_n = _oracle_verify(1, p_np, q_np, x.cpu().numpy(), 23, 0)
    assert np.array_equal(n.cpu().numpy(), want_n) and np.array_equal(out.cpu().numpy(), want_out)


@pytest.mark.parametrize("dtype,V,B,t", [("bf16", 2049, 149, 1), ("fp32", 4096, 150, 1), ("bf16", 4098, 149, 2), ("bf16", 8192, 149, 1),   # 256 threads
                                         ("fp32", 4097, 297, 1), ("bf16", 8193, 149, 2), ("fp32", 24576, 149, 1),     # a CTA of 1024
                                         ("bf16", 24577, 149, 1)])                                                    # clusters of two
def test_decisions_of_more_sequences_than_sms_match_oracle(lib, dtype, V, B, t):
    p, q = inputs.make_accept_logits(B, t, V, seed=V + B, device="cuda", dtype=dtype)
    p[0, :, V // 2:] = -float("inf")
    q[1] = p[1, :t]                                                    # an all-zero residual, if it comes to one; else the bonus row
    x = lib.hsd_draft_sample(q, 5, 0)
    p_np, q_np, x_np = inputs.logits_to_numpy(p), inputs.logits_to_numpy(q), x.cpu().numpy()
    out, n = lib.hsd_verify_level(1, p, q, x, 23, 0)
    want_out, want_n = _oracle_verify(1, p_np, q_np, x_np, 23, 0)
    assert np.array_equal(n.cpu().numpy(), want_n) and np.array_equal(out.cpu().numpy(), want_out)
