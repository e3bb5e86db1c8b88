"""The calibration kernels (pairwise acceptance rates between exit layers) against the oracle."""
import numpy as np
import pytest
import torch

from oracle import sampling as S
from paper_2510_19705_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,R,V,dtype", [(3, 5, 777, torch.float32), (4, 9, 2048, torch.bfloat16), (2, 3, 5000, torch.bfloat16),
                                         (8, 4, 1500, torch.float32), (1, 2, 100, torch.float32)])
def test_pairwise_alpha_matches_oracle(lib, L, R, V, dtype):
    g = torch.Generator().manual_seed(L * 1000 + R)
    base = torch.randn(R, V, generator=g) * 2.5
    logits = torch.stack([base + 0.8 * (m + 1) * torch.randn(R, V, generator=g) for m in range(L)]).to(dtype)
    got = lib.hsd_pairwise_alpha(logits.cuda())
    torch.cuda.synchronize()
    want = S.pairwise_acceptance(logits.float().numpy().astype(np.float64))
    got = got.cpu().numpy()
    assert got.shape == (L, L) and np.array_equal(got, got.T) and np.array_equal(np.diag(got), np.ones(L))
    assert np.abs(got - want).max() < 2e-5, np.abs(got - want).max()
    again = lib.hsd_pairwise_alpha(logits.cuda()).cpu().numpy()          # no atomics: repeatable bit for bit
    assert np.array_equal(got, again)


def test_pairwise_alpha_of_a_model_stack(lib):
    """The rates between the exits of one random-init model on its own drafted positions feed the hierarchy
    search: nearer exits accept each other more often, and the search returns a valid chain."""
    from paper_2510_19705_b200 import inputs
    torch.manual_seed(0)
    R, V = 16, 2048
    h = torch.randn(R, V)
    logits = torch.stack([h + s * torch.randn(R, V) for s in (1.5, 1.0, 0.5, 0.0)]).bfloat16().cuda()
    alpha = lib.hsd_pairwise_alpha(logits).cpu().numpy()
    assert alpha[2, 3] > alpha[1, 3] > alpha[0, 3]
    lat, sigma, T = binding.hsd_search_hierarchy([0.1, 0.3, 1.0, 3.0], alpha.tolist(), 8)
    assert sigma[-1] == 3 and len(T) == len(sigma) - 1 and lat <= 3.0


def _engine(lib, name):
    from paper_2510_19705_b200 import inputs
    wl = inputs.WORKLOADS[name]
    cfg = wl["model"]
    w_cpu = inputs.make_weights(cfg, wl["weight_seed"])
    w = {k: (v.cuda() if k != "layers" else [{n: t.cuda() for n, t in l.items()} for l in v]) for k, v in w_cpu.items()}
    eng = lib.Hsd(cfg, w, wl["exits"], wl["T"], max_batch=1, max_seq=160, page_size=wl["page"])
    return wl, cfg, w_cpu, eng


def test_layer_logits_match_the_oracle_fp32(lib):
    """Logits of every exit layer at every position (shared final norm + head): fp32 model, 1e-5 bound."""
    from oracle.transformer import Transformer
    from paper_2510_19705_b200 import inputs
    wl, cfg, w_cpu, eng = _engine(lib, "tiny3")
    toks = inputs.make_prompts(cfg["vocab"], 1, 40, 21)[0]
    layers = [1, 2, 3, 4]
    got = eng.layer_logits(toks.cuda(), layers).cpu().numpy()
    om = Transformer(cfg, inputs.weights_to_numpy(w_cpu), layers)
    for i in range(len(layers)):
        om.reset()
        om.rows(i, toks[:1].tolist(), toks[1:].tolist())              # rows of positions 0 .. n-1
        want = np.asarray(om.last_logits64)
        assert got[i].shape == want.shape
        assert np.abs(got[i] - want).max() < 1e-5, (layers[i], np.abs(got[i] - want).max())
    # a generation afterwards still works on the same context
    out, stats, _ = eng.generate(inputs.make_prompts(cfg["vocab"], 1, wl["prompt"], wl["prompt_seed"]).cuda(), 8, 1)
    assert out.shape == (1, 8)
    eng.close()


def test_calibrate_then_search_end_to_end(lib):
    """bf16 stand-in model: exit-layer logits -> pairwise acceptance rates -> latency-optimal hierarchy."""
    from oracle.transformer import Transformer
    from paper_2510_19705_b200 import inputs
    wl, cfg, w_cpu, eng = _engine(lib, "mini3")
    toks = inputs.make_prompts(cfg["vocab"], 1, 96, 22)[0]
    layers = [1, 2, 3, 4, 5, 6]
    logits = eng.layer_logits(toks.cuda(), layers)
    eng.close()
    alpha = lib.hsd_pairwise_alpha(logits).cpu().numpy()
    # the rates of the library's own logits equal the oracle's formula on those logits
    want = S.pairwise_acceptance(logits.float().cpu().numpy().astype(np.float64))
    assert np.abs(alpha - want).max() < 2e-5
    # and the logits are the oracle's forward (first and last exit; bf16: a few 1e-2 at most on this depth)
    om = Transformer(cfg, inputs.weights_to_numpy(w_cpu), layers)
    for i in (0, len(layers) - 1):
        om.reset()
        om.rows(i, toks[:1].tolist(), toks[1:].tolist())
        ref = np.asarray(om.last_logits64)
        d = np.abs(logits[i].float().cpu().numpy() - ref)
        assert np.sqrt((d ** 2).mean()) < 2e-2 * max(1.0, float(np.std(ref))), (layers[i], float(d.max()))
    costs = [float(l) for l in layers]                              # cost of an exit ~ its depth
    lat, sigma, T = binding.hsd_search_hierarchy(costs, alpha.tolist(), 8)
    assert sigma[-1] == len(layers) - 1 and lat <= costs[-1] and len(T) == len(sigma) - 1
    assert abs(lat - __import__("oracle.latency", fromlist=["x"]).search_hierarchy(costs, alpha.tolist(), 8)[0]) <= 1e-12 * lat


@pytest.mark.parametrize("L,R,V,dtype", [(9, 2, 4104, torch.bfloat16),      # two 8-model blocks, a unit of one 8-token vector
                                         (17, 3, 9001, torch.float32),       # three blocks, rows off the 16-byte grid
                                         (24, 2, 5000, torch.float32), (32, 2, 8200, torch.bfloat16), (32, 1, 255, torch.bfloat16),
                                         # up to eight models: 1024-token tiles, a last one of 904 and of 1 token; up to sixteen: 512
                                         (2, 40, 5000, torch.bfloat16), (8, 3, 3073, torch.float32), (3, 700, 24, torch.float32), (16, 2, 4608, torch.bfloat16)])
def test_pairwise_alpha_block_edges(lib, L, R, V, dtype):
    """Model counts at the ends of the 8-model blocks and vocabularies at the ends of tiles and units."""
    g = torch.Generator().manual_seed(L + V)
    base = torch.randn(R, V, generator=g) * 2.5
    logits = torch.stack([base + 0.1 * (m + 1) * torch.randn(R, V, generator=g) for m in range(L)]).to(dtype)
    logits[0, 0, : V // 2] = -float("inf")                                   # a masked half: weight exactly zero
    got = lib.hsd_pairwise_alpha(logits.cuda()).cpu().numpy()
    p = torch.softmax(logits.double(), -1)
    want = torch.stack([torch.minimum(p[i:i + 1], p).sum(-1).mean(-1) for i in range(L)]).numpy()
    # fp32 sums of at most 128 terms per lane and 8 per warp and slice: about 2^-24 x 136 of a rate, 1e-5 at most
    assert np.array_equal(got, got.T) and np.abs(got - want).max() < 1e-5, np.abs(got - want).max()


@pytest.mark.parametrize("d,nq,nkv,V", [(256, 4, 2, 1000), (256, 4, 2, 1004), (192, 3, 1, 1000)])     # head in one product over all layers / a product per layer
def test_layer_logits_into_any_element_address(lib, d, nq, nkv, V):
    """The output needs the alignment of its elements only, whatever the vocabulary's divisors."""
    import ctypes
    from paper_2510_19705_b200 import inputs
    cfg = inputs.model_cfg(2, d, nq, nkv, 256, V, "bf16", head_dim=64)
    w = inputs.make_weights(cfg, 5)
    w = {k: (v.cuda() if k != "layers" else [{n: t.cuda() for n, t in l.items()} for l in v]) for k, v in w.items()}
    eng = lib.Hsd(cfg, w, (1, 2), (1,), max_batch=1, max_seq=64, page_size=16)
    toks = inputs.make_prompts(V, 1, 21, 3)[0].cuda()
    want = eng.layer_logits(toks, [1, 2])
    for off in (1, 2, 3, 4):
        buf = torch.full((want.numel() + 8,), 7.0, dtype=torch.bfloat16, device="cuda")
        st = lib.library().hsd_layer_logits(eng._ctx, toks.data_ptr(), 21, (ctypes.c_int32 * 2)(1, 2), 2, buf.data_ptr() + 2 * off,
                                            torch.cuda.current_stream().cuda_stream)
        assert st == 0
        assert torch.equal(buf[off:off + want.numel()].view(want.shape), want)
        assert (buf[:off] == 7.0).all() and (buf[off + want.numel():] == 7.0).all()
    eng.close()


@pytest.mark.parametrize("R", [65535, 65536, 65600])
def test_pairwise_alpha_of_many_positions(lib, R):
    """More positions than a grid's second and third dimensions hold."""
    g = torch.Generator().manual_seed(R)
    logits = torch.randn(3, R, 8, generator=g) * 2.0
    got = lib.hsd_pairwise_alpha(logits.cuda()).cpu()
    p = torch.softmax(logits.double(), -1)
    want = torch.stack([torch.minimum(p[i:i + 1], p).sum(-1).mean(-1) for i in range(3)])
    assert torch.equal(got, got.T) and (got - want).abs().max() < 1e-5


@pytest.mark.parametrize("V,dtype", [(2048, torch.bfloat16), (2047, torch.bfloat16), (1000, torch.float32), (1001, torch.float32)])
def test_pairwise_alpha_of_extreme_logits(lib, V, dtype):
    """Rows far from zero, of the type's lowest value only, and half at the highest: what the softmax of the rows gives."""
    g = torch.Generator().manual_seed(V)
    x = torch.randn(4, 9, V, generator=g, dtype=torch.float64) * 2.0
    fi = torch.finfo(dtype)
    x[:, 1] += 3e4
    x[:, 2] = x[:, 2] * 1e9 + 3e12
    x[:, 3] = x[:, 3] * 1e31 - 2e34
    x[:, 4] = fi.min                                     # a fully masked row: uniform
    x[:, 5] = x[:, 5].sign() * 3.0e38
    x[1:, 6] = fi.min                                    # masked under some models only
    x[:, 7, V // 3:] = fi.min
    x[:, 8, ::2] = -float("inf")
    logits = x.to(dtype)
    got = lib.hsd_pairwise_alpha(logits.cuda()).cpu()
    z = logits.double()
    p = torch.softmax(z - z.max(-1, keepdim=True).values, -1)
    want = torch.stack([torch.minimum(p[i:i + 1], p).sum(-1).mean(-1) for i in range(4)])
    assert torch.equal(got, got.T) and (got - want).abs().max() < 1e-5, (got, want)


@pytest.mark.parametrize("dtype,L,R,V", [(torch.bfloat16, 5, 20, 4001), (torch.bfloat16, 24, 30, 2048), (torch.float32, 18, 200, 8192)])
def test_rates_of_calls_back_to_back(lib, dtype, L, R, V):
    # the kernels of a call start under the end of the one before it, and read logits that the stream has just written
    g = torch.Generator(device="cuda").manual_seed(L)
    sets = [(torch.randn(L, R, V, generator=g, device="cuda") * 3).to(dtype) for _ in range(3)]
    want = [lib.hsd_pairwise_alpha(x).clone() for x in sets]
    x = torch.empty_like(sets[0])
    got = []
    for i in range(12):
        x.copy_(sets[i % 3])
        got.append(lib.hsd_pairwise_alpha(x))
        lib.hsd_pairwise_alpha(sets[(i + 1) % 3])
    assert all(torch.equal(a, want[i % 3]) for i, a in enumerate(got))


def test_more_rows_of_all_models_than_fit_one_grid_dimension(lib):
    # 8 models x (2^28 + 3) positions of two tokens: 2^31 rows; 8.6 GB of logits, 47 GB of workspace
    L, R, split = 8, 2 ** 28 + 3, 2 ** 27
    a = torch.tensor([[0.25 * l, 1.0] for l in range(L)], device="cuda").to(torch.bfloat16)
    b = torch.tensor([[-1.0, 0.5 * l] for l in range(L)], device="cuda").to(torch.bfloat16)
    x = torch.empty(L, R, 2, dtype=torch.bfloat16, device="cuda")
    x[:, :split] = a[:, None]
    x[:, split:] = b[:, None]
    got = lib.hsd_pairwise_alpha(x).cpu()
    want = torch.zeros(L, L, dtype=torch.float64)
    for rows, share in ((a, split / R), (b, 1 - split / R)):
        p = torch.softmax(rows.cpu().double(), -1)
        want += share * torch.minimum(p[:, None], p[None]).sum(-1)
    assert (got - want).abs().max() < 1e-5                            # fp32 softmax and sums of two tokens
    del x
    torch.cuda.empty_cache()
