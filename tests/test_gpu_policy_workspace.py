"""policy_forward's workspace (large batches, two kernels): from the handle's
allocator, in the order of the call's stream, handed back by the end of the
call; the one-kernel form, with the same bits, where the allocator has none and
under capture."""
import ctypes

import numpy as np
import pytest
import torch

import synth
from synth import preset

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2505_08222_gb300 as ut  # noqa: E402
from paper_2505_08222_gb300 import _abi, make_config  # noqa: E402

D, L, SLOTS, N = 64, 1, 10, 10100  # 919 tiles of 11 agents: just past three waves


class _Allocator:
    """Torch's caching allocator behind the callback: the streams asked for, the
    blocks handed out, NULL while `empty`."""

    def __init__(self):
        self.streams, self.live, self.empty = [], set(), False
        dev = torch.cuda.current_device()

        def _alloc(nbytes, stream, ctx):
            self.streams.append(int(stream or 0))
            if self.empty:
                return None
            ptr = torch.cuda.caching_allocator_alloc(int(nbytes), dev, int(stream or 0))
            self.live.add(int(ptr))
            return ptr

        def _free(ptr, stream, ctx):
            self.live.discard(int(ptr))
            torch.cuda.caching_allocator_delete(int(ptr))

        self._a, self._f = _abi.ALLOC_FN(_alloc), _abi.FREE_FN(_free)
        self.struct = _abi.Allocator(self._a, self._f, None)


def _handle(alloc):
    p = preset("fleet5", n_envs=4).replace(n_particles=32, d_model=D, n_layers=L, n_heads=D // 16)
    cfg, keep = make_config(p, 0)
    h = ctypes.c_void_p()
    assert ut.lib.env_create(ctypes.byref(cfg), ctypes.byref(alloc.struct) if alloc else None, None,
                             ctypes.byref(h)) == 0
    prm = np.ascontiguousarray(synth.policy_params(synth.PolicyDims(D, L, D // 16), seed=5), np.float32)
    assert ut.lib.env_set_policy(h, prm.ctypes.data_as(ctypes.c_void_p), prm.size) == 0
    return h


def _inputs():
    g = torch.Generator(device="cuda")
    g.manual_seed(6)
    return ((0.4 * torch.randn(N, SLOTS, 8, generator=g, device="cuda")).bfloat16(),
            torch.randint(0, SLOTS + 1, (N,), generator=g, device="cuda", dtype=torch.int32),
            torch.randn(N, D, generator=g, device="cuda").bfloat16())


def _forward(h, stream, x):
    tok, ne, emb = x[0], x[1], x[2].clone()
    logits = torch.full((N, 7), -1.0, device="cuda")
    act = torch.full((N,), -1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    rc = ut.lib.policy_forward(h, *(ctypes.c_void_p(t.data_ptr()) for t in (tok, ne, emb, logits, act)), N, SLOTS, 3,
                               ctypes.c_void_p(stream.cuda_stream))
    assert rc == 0, ut.lib.env_last_error(h)
    torch.cuda.synchronize()
    return logits, act, emb


def test_workspace_comes_from_the_handles_allocator():
    alloc = _Allocator()
    h, x = _handle(alloc), _inputs()
    held = set(alloc.live)
    sides = [torch.cuda.Stream(), torch.cuda.Stream()]
    got = []
    for side in sides:
        alloc.streams.clear()
        got.append(_forward(h, side, x))
        assert alloc.streams == [side.cuda_stream] and alloc.live == held
    alloc.empty = True
    got.append(_forward(h, sides[0], x))
    assert len(alloc.streams) == 2
    own = _handle(None)  # the library's own stream-ordered allocations
    got.append(_forward(own, sides[1], x))
    for other in got[1:]:
        assert all(torch.equal(a, b) for a, b in zip(got[0], other))
    assert int(got[0][1].min()) >= 0
    ut.lib.env_destroy(own)
    ut.lib.env_destroy(h)
    assert not alloc.live


def test_a_captured_call_asks_for_no_memory():
    alloc = _Allocator()
    h, x = _handle(alloc), _inputs()
    want = _forward(h, torch.cuda.current_stream(), x)
    alloc.streams.clear()
    emb, logits, act = x[2].clone(), torch.empty((N, 7), device="cuda"), torch.empty(N, dtype=torch.int32, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        assert ut.lib.policy_forward(h, *(ctypes.c_void_p(t.data_ptr()) for t in (x[0], x[1], emb, logits, act)), N,
                                     SLOTS, 3, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    g.replay()
    torch.cuda.synchronize()
    assert not alloc.streams
    assert all(torch.equal(a, b) for a, b in zip(want, (logits, act, emb)))
    ut.lib.env_destroy(h)
