"""Decode attention (a few query vectors per KV head): how its launches are laid out, and streaming tokens over long lists."""
import ctypes

import pytest
import torch

import paper_2606_10944_b200 as elm
from paper_2606_10944_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype_code", [binding.ELM_F32, binding.ELM_BF16])
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("vectors", [1, 2, 4, 5, 8])
def test_split_grid_is_resident_at_once(dtype_code, d, vectors):
    """A long list is split over as many CTAs as the device holds, not over more (they would be a second wave)."""
    for problems in (1, 8, 64, 296):
        ctas, resident = binding.debug_decode_grid(problems, vectors, 1, 20000, d, 20000, dtype_code=dtype_code)
        assert problems <= ctas <= resident


class _Exact:
    """A stream inside its exact start, rewound to the same token before every call (what a call appends lies behind
    the entries a rewound stream reads)."""

    def __init__(self, dtype, d, rep, hkv, log2_nout, tokens, spare, batch=1):
        g = torch.Generator(device="cuda").manual_seed(3)
        K = torch.randn(batch, hkv, 4 << log2_nout, d, device="cuda", generator=g).to(dtype)
        V = torch.randn(batch, hkv, 4 << log2_nout, d, device="cuda", generator=g).to(dtype)
        self.Q = torch.randn(spare, batch, hkv * rep, 1, d, device="cuda", generator=g).to(dtype)
        self.s = elm.Stream(K, V, hkv * rep, log2_nout, 4)
        while self.s.state.n < tokens:
            self.s.steps(self.Q[:min(spare, tokens - self.s.state.n)])
        self.start = bytes(self.s.state)

    def rewind(self):
        ctypes.memmove(ctypes.byref(self.s.state), self.start, len(self.start))

    def one_call(self, T):
        self.rewind()
        return self.s.steps(self.Q[:T])

    def single_steps(self, T):
        self.rewind()
        return torch.stack([self.s.step(self.Q[t]) for t in range(T)])


def _median_us(f, reps=15):
    times = []
    for i in range(reps + 3):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        f()
        b.record()
        b.synchronize()
        if i >= 3:
            times.append(a.elapsed_time(b) * 1e3)
    return sorted(times)[reps // 2]


@pytest.mark.parametrize("dtype,d,rep,hkv,log2_nout", [
    (torch.bfloat16, 128, 4, 8, 11), (torch.bfloat16, 128, 1, 1, 11), (torch.bfloat16, 64, 8, 2, 11), (torch.float32, 128, 2, 3, 10),
])
def test_short_stream_calls_over_long_lists(dtype, d, rep, hkv, log2_nout):
    """A call of a few tokens over a list of thousands of entries gives what single steps give, bit for bit, and takes
    no longer than they do (with room for noise: spread over too few CTAs it took up to ten times as long)."""
    x = _Exact(dtype, d, rep, hkv, log2_nout, 3 << log2_nout, 1024)
    for T in (2, 3, 8, 40, 330):                      # (clusters, and from 148 or 296 tokens and heads on CTAs that walk the parts)
        assert torch.equal(x.one_call(T), x.single_steps(T))
        if T <= 8:
            assert _median_us(lambda: x.one_call(T)) <= 1.3 * _median_us(lambda: x.single_steps(T)) + 5
