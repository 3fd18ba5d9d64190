"""darkattn_forward_static: the forward pass for hosts that cannot allocate device memory.

A serving process that handed the whole GPU to its own memory pool, or a plug-in that only ever sees
input and output buffers, has no workspace to give and must not call cudaMalloc. The static entry
point keeps its intermediates in an array inside the library instead. These tests call it through
the C ABI and hold it to the ordinary entry point's result and to the float64 oracle, twice in a row
because the array keeps the previous call's contents. The file sorts last on purpose, so a run that stops at the first
failure has already been through every other test.
"""
import numpy as np
import pytest
import torch

from paper_2603_04127_b200 import inputs
from tests.util import TOL, rel_errors, to_dev, torch_dtype


@pytest.fixture(scope="module")
def binding():
    from paper_2603_04127_b200 import build
    build.build()
    from paper_2603_04127_b200 import binding as b
    return b


def _have_library():
    import os
    import shutil
    here = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    return os.path.exists(os.path.join(here, "paper_2603_04127_b200", "libdarkattn.so")) or shutil.which("nvcc") or os.path.exists("/usr/local/cuda/bin/nvcc")


@pytest.mark.skipif(not _have_library(), reason="neither libdarkattn.so nor nvcc to build it")
def test_oversized_problem_is_refused_on_the_host(binding):
    plan = binding.darkattn_plan(4, 16, 8192, 128, 256, dtype=binding.BF16, causal=True)
    assert binding.darkattn_static_scratch_needed(plan) > binding.STATIC_SCRATCH_BYTES
    a = 4096  # never dereferenced: the size check comes before any GPU work
    rc = binding.lib.darkattn_forward_static(plan.handle, a, a, a, a, a, a, None)
    assert rc == binding.ERR_WORKSPACE
    plan.destroy()


@pytest.mark.gpu
@pytest.mark.parametrize("dtype,causal", [("f32", False), ("bf16", True)])
def test_static_scratch_forward_matches_workspace_forward(binding, dtype, causal):
    wl = inputs.small(name="noalloc", wid=41, B=1, H=2, N=300, d=64, m=128, dtype=dtype, causal=causal,
                      backward=False)
    t = inputs.generate(wl)
    dt = torch_dtype(dtype)
    Q, K, V, M, W = (to_dev(x, dt) for x in (t.Q, t.K, t.V, t.M, t.W))
    plan = binding.darkattn_plan(1, 2, 300, 64, 128, dtype=binding.F32 if dtype == "f32" else binding.BF16,
                                 causal=causal, path=binding.PATH_SIMT)
    assert 0 < binding.darkattn_static_scratch_needed(plan) <= binding.STATIC_SCRATCH_BYTES
    ws = plan.alloc_workspace()
    want = torch.empty_like(V)
    binding.darkattn_forward(plan, Q, K, V, M, W, want, ws)
    torch.cuda.synchronize()
    want = want.float().cpu().numpy()
    from oracle import ref
    exact = ref.forward(t.Q, t.K, t.V, t.M, t.W, causal=causal)
    for call in range(2):
        # the second call runs on a different problem's leftovers: swap queries and keys in between
        if call == 1:
            junk = torch.empty_like(V)
            binding.darkattn_forward_static(plan, K, Q, V, M, W, junk)
        got = torch.full_like(V, float("nan"))
        binding.darkattn_forward_static(plan, Q, K, V, M, W, got)
        torch.cuda.synchronize()
        got = got.float().cpu().numpy()
        assert np.isfinite(got).all()
        fro, mx = rel_errors(got.astype(np.float64), want.astype(np.float64))
        assert fro < TOL[dtype] and mx < TOL[dtype], (call, fro, mx)
        fro, mx = rel_errors(got.astype(np.float64), exact)          # and against the oracle, like every other entry point
        assert fro < TOL[dtype] and mx < TOL[dtype], ("oracle", call, fro, mx)
    plan.destroy()


@pytest.mark.gpu
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_static_scratch_takes_the_heads_one_by_one(binding, dtype):
    """A problem whose heads together need more than the array, each alone less: the same rows as with a workspace."""
    wl = inputs.small(name="noalloc_heads", wid=42, B=3, H=4, N=1001, d=48, m=264, dv=40, dtype=dtype, causal=True, backward=False)
    t = inputs.generate(wl)
    dt = torch_dtype(dtype)
    Q, K, V, M, W = (to_dev(x, dt) for x in (t.Q, t.K[:, ::2], t.V[:, ::2], t.M, t.W))       # two query heads per key/value head
    plan = binding.darkattn_plan(3, 4, 1001, 48, 264, dv=40, dtype=binding.F32 if dtype == "f32" else binding.BF16, causal=True,
                                 path=binding.PATH_SIMT, H_kv=2)
    assert plan.workspace_bytes > binding.STATIC_SCRATCH_BYTES >= binding.darkattn_static_scratch_needed(plan)
    want, got = (torch.full((3, 4, 1001, 40), float("nan"), dtype=dt, device="cuda") for _ in range(2))
    binding.darkattn_forward(plan, Q, K, V, M, W, want, plan.alloc_workspace())
    binding.darkattn_forward_static(plan, Q, K, V, M, W, got)
    torch.cuda.synchronize()
    assert torch.equal(got, want)
    plan.destroy()


LEAN = [
    # one pair's bf16 parts (6 bytes an element, inputs among them) need more than the array, its fp32 intermediates less
    dict(B=1, H=1, N=5090, d=429, r=21, m=63, dv=121, causal=False),
    dict(B=1, H=2, N=6923, d=406, r=43, m=86, dv=10, causal=False),
    dict(B=1, H=1, N=3571, d=373, r=106, m=357, dv=11, causal=True),
    dict(B=1, H=1, N=10509, d=116, m=22, dv=9, causal=True, chunk=16),
]


@pytest.mark.skipif(not _have_library(), reason="neither libdarkattn.so nor nvcc to build it")
@pytest.mark.parametrize("i", range(len(LEAN)))
def test_long_sequences_of_wide_queries_are_accepted(binding, i):
    kw = dict(LEAN[i])
    B, H, N, d, m = (kw.pop(k) for k in ("B", "H", "N", "d", "m"))
    plan = binding.darkattn_plan(B, H, N, d, m, dtype=binding.F32, **kw)
    assert 0 < binding.darkattn_static_scratch_needed(plan) <= binding.STATIC_SCRATCH_BYTES // 2
    plan.destroy()


@pytest.mark.gpu
@pytest.mark.parametrize("i", range(len(LEAN)))
def test_static_scratch_forward_of_long_sequences(binding, i):
    kw = dict(LEAN[i])
    chunk = kw.pop("chunk", 0)
    wl = inputs.small(name="noalloc_lean", wid=43 + i, dtype="f32", backward=False, **kw)
    t = inputs.generate(wl)
    Q, K, V, M, W = (to_dev(x, torch.float32) for x in (t.Q, t.K, t.V, t.M, t.W))
    plan = binding.darkattn_plan(wl.B, wl.H, wl.N, wl.d, wl.m, r=wl.r, dv=wl.dv, dtype=binding.F32, causal=wl.causal, chunk=chunk)
    got = torch.full((wl.B, wl.H, wl.N, wl.dv), float("nan"), device="cuda")
    binding.darkattn_forward_static(plan, Q, K, V, M, W, got)
    torch.cuda.synchronize()
    from oracle import ref
    want = ref.forward(t.Q, t.K, t.V, t.M, t.W, causal=wl.causal)
    fro, mx = rel_errors(got.cpu().numpy().astype(np.float64), want)
    assert fro < TOL["f32"] and mx < TOL["f32"], (fro, mx)
    plan.destroy()
