"""The bounded waits of a verification: their limit is for the kernel's own work, and one that runs out is reported.  The kernels
are built here with a limit of a millisecond."""
import ctypes
import os
import subprocess

import pytest
import torch

from paper_2510_19705_b200 import build, inputs

pytestmark = pytest.mark.gpu
vp, i32, u64 = ctypes.c_void_p, ctypes.c_int, ctypes.c_uint64


@pytest.fixture(scope="module")
def waits(tmp_path_factory):
    if not os.path.exists(build.NVCC):
        pytest.skip("no nvcc")
    out = str(tmp_path_factory.mktemp("native") / "verify_waits.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "native", "verify_waits.cu")
    subprocess.run([build.NVCC] + build.FLAGS + ["-DHSD_WAIT_LIMIT_NS=1000000ull", "-shared", "-o", out, src], check=True)
    so = ctypes.CDLL(out)
    so.occupy.argtypes = [u64, vp]
    so.verify_without_data.argtypes = [vp, vp, vp, i32, i32, i32, i32, i32, vp, vp, vp, vp, vp, vp]
    so.hsd_verify_level.argtypes = [i32, vp, vp, vp, i32, i32, i32, i32, u64, u64, vp, ctypes.c_size_t, vp, vp, vp]
    return so


def _inputs(lib, B, t, V, dtype, seed):
    p, q = inputs.make_accept_logits(B, t, V, seed=seed, device="cuda", dtype=dtype)
    ws = torch.zeros(lib.hsd_verify_workspace_bytes(B, t), dtype=torch.uint8, device="cuda")
    out, n = torch.zeros(B, t + 1, dtype=torch.int32, device="cuda"), torch.zeros(B, dtype=torch.int32, device="cuda")
    x = lib.hsd_draft_sample(q, 5, 0) if t else torch.zeros(B, 0, dtype=torch.int32, device="cuda")
    return p, q, x, ws, out, n


# statistics by three groups of warps, by one, by clusters; rows that come through the ring twice
@pytest.mark.parametrize("dtype,V,B,t", [("bf16", 32000, 24, 3), ("fp32", 9001, 60, 2), ("bf16", 32000, 20, 2), ("bf16", 32000, 3, 2),
                                         ("fp32", 60000, 25, 3)])
def test_the_kernel_in_front_may_take_its_time(lib, waits, dtype, V, B, t):
    p, q, x, ws, out, n = _inputs(lib, B, t, V, dtype, 3)
    want = lib.hsd_verify_level(1, p, q, x, 7, 0)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    stream = side.cuda_stream
    assert waits.occupy(20_000_000, stream) == 0                       # twenty limits
    assert waits.hsd_verify_level(1, p.data_ptr(), q.data_ptr(), x.data_ptr(), B, t, V, 1 if dtype == "bf16" else 0, 7, 0, ws.data_ptr(),
                                  ws.numel(), stream, out.data_ptr(), n.data_ptr()) == 0
    torch.cuda.synchronize()
    assert torch.equal(out, want[0]) and torch.equal(n, want[1])


# decisions by clusters of several sizes, of 256 threads; by a CTA a sequence (many sequences, vocabularies past 131072)
@pytest.mark.parametrize("groups", [1, 3])
@pytest.mark.parametrize("dtype,V,B,t", [("bf16", 2050, 3, 2), ("bf16", 32000, 60, 2), ("fp32", 32001, 2, 0), ("bf16", 5000, 149, 1), ("fp32", 20000, 150, 1), ("bf16", 131080, 2, 1), ("fp32", 131073, 1, 1)])
def test_a_wait_that_runs_out_is_reported(lib, waits, dtype, V, B, t, groups):
    p, q, x, _, out, n = _inputs(lib, B, t, V, dtype, 3)
    # statistics that a call before left behind: any would give a plausible decision
    stats = torch.zeros(B * (2 * t + 1), 2, dtype=torch.int64, device="cuda")
    stats[:, 0], stats[:, 1] = 0x41200000, 1 << 40
    host = torch.full((2, B), 9, dtype=torch.int32).pin_memory()
    stream = torch.cuda.current_stream().cuda_stream
    assert waits.verify_without_data(p.data_ptr(), q.data_ptr(), x.data_ptr(), B, t, V, 1 if dtype == "bf16" else 0, groups, stats.data_ptr(), stream,
                                     out.data_ptr(), n.data_ptr(), host[0].data_ptr(), host[1].data_ptr()) == 0
    torch.cuda.synchronize()
    assert (n == -1).all() and (out == -1).all() and (host == -1).all()
