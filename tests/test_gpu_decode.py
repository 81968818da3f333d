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
    """A stream inside its exact start, rewound to the same token before every call: what a call appends lies behind
    the entries a rewound stream reads, as long as it does not reach a multiple of 2**log2_nout tokens."""

    def __init__(self, dtype, d, rep, hkv, log2_nout, tokens, spare, batch=1):
        g = torch.Generator(device="cuda").manual_seed(3)
        K = torch.randn(batch, hkv, tokens + spare, d, device="cuda", generator=g).to(dtype)
        V = torch.randn(batch, hkv, tokens + spare, d, device="cuda", generator=g).to(dtype)
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


def _graph_us(f, calls=10):
    """Device time of a call: many of them replayed as one graph."""
    f()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        for _ in range(calls):
            f()
    return _median_us(g.replay) / calls


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


@pytest.mark.parametrize("largest", [0, 8, 2, 1])
@pytest.mark.parametrize("dtype,d,rep,hkv,batch,log2_nout,start", [
    (torch.bfloat16, 128, 4, 2, 1, 10, 3072),       # sixteen parts: more than 2048 entries
    (torch.float32, 128, 1, 3, 1, 9, 1536),         # sixteen parts: more than 1024 entries of 512 bytes
    (torch.float32, 128, 4, 1, 1, 14, 8150),        # a window that grows past the longest list taken in clusters
    (torch.bfloat16, 64, 2, 2, 32, 11, 1500),       # clusters of four: 64 problems
])
def test_streamed_tokens_over_long_lists_match_exact_attention(dtype, d, rep, hkv, batch, log2_nout, start, largest):
    """Lists long enough for clusters of 16 CTAs, on devices that can place them and on devices that cannot: one call of
    60 tokens and single steps agree bit for bit and equal exact causal attention in 64 bits (the exact start)."""
    lib = binding.load_library()
    assert lib.elm_debug_set(2, largest) == 0
    try:
        x = _Exact(dtype, d, rep, hkv, log2_nout, start, 256, batch)
        got = x.one_call(60)
        assert torch.equal(got, x.single_steps(60))
    finally:
        assert lib.elm_debug_set(2, 0) == 0
    K, V = (t.double().repeat_interleave(rep, dim=1) for t in (x.s.K, x.s.V))
    # fp32 sums of a few thousand positive terms; bf16 outputs are rounded to 8 bits
    bound = 1e-5 if dtype == torch.float32 else 2.0 ** -8
    for t in (0, 42, 43, 59):
        p = torch.softmax(torch.einsum("bhqd,bhnd->bhqn", x.Q[t].double(), K[:, :, :start + t + 1]) / d ** 0.5, dim=-1)
        want = p @ V[:, :, :start + t + 1]
        assert ((got[t].double() - want).abs().amax(-1) / want.abs().amax(-1)).max() <= bound


@pytest.mark.parametrize("d,rep,hkv", [(128, 1, 8), (64, 1, 8), (128, 2, 8), (64, 2, 8), (64, 3, 4), (128, 4, 8), (64, 5, 3), (128, 8, 3), (64, 8, 3)])
@pytest.mark.parametrize("start", [1, 30, 127, 500, 2046, 4090])
def test_bf16_tokens_match_exact_attention(d, rep, hkv, start):
    """Calls of 1 ... 600 tokens whose lists cross the edges of tiles, groups and units, against exact causal attention in 64 bits:
    eight and sixteen query vectors per warp, clusters and, the longest call, CTAs that walk the list.  Infinite values and a NaN
    of four neighbouring tokens, so of one group where tokens share it, reach the tokens that see them, in their columns, as what they are."""
    x = _Exact(torch.bfloat16, d, rep, hkv, 13, start, 604)
    K, V = (t.double().repeat_interleave(rep, dim=1) for t in (x.s.K, x.s.V))
    seen = torch.arange(start + 604, device="cuda")
    for T in (1, 2, 7, 33, 600):
        assert binding.debug_stream_form(1, hkv * rep, hkv, start + 604, d, start + 1, T) == (2 if T == 600 else 1)
        got = x.one_call(T).double()
        s = torch.einsum("tbhqd,bhnd->tbhqn", x.Q[:T].double(), K) / d ** 0.5
        s = s.masked_fill(seen > start + torch.arange(T, device="cuda")[:, None, None, None, None], -torch.inf)
        want = torch.einsum("tbhqn,bhnd->tbhqd", torch.softmax(s, dim=-1), V)
        assert ((got - want).abs().amax(-1) / want.abs().amax(-1)).max() <= 2.0 ** -8          # rounded to 8 bits
        rows = x.s.V[:, :, start + T // 2:start + T // 2 + 4]
        kept, values = rows.clone(), (torch.inf, -torch.inf, torch.nan, torch.inf)
        for i, v in enumerate(values):                 # seen by the tokens from T // 2 + i on
            rows[:, :, i, 3 + i] = v
        after = x.one_call(T).double()
        rows.copy_(kept)
        for i, v in enumerate(values):
            at = after[T // 2 + i:, ..., 3 + i]
            assert (at.isnan() if v != v else at == v).all()
            at.copy_(got[T // 2 + i:, ..., 3 + i])
        # (sums in another order: neighbouring values of 8 bits are up to 2^-7 of the larger apart)
        assert ((after - got).abs() <= 2.0 ** -7 * got.abs().amax(-1, keepdim=True)).all()


@pytest.mark.parametrize("d,B,H,rep,n_core", [(128, 4, 8, 4, 5193), (128, 8, 8, 4, 12288), (64, 8, 8, 8, 12288), (128, 1, 8, 5, 2048)])
def test_partial_results_of_decode_are_as_precise_as_fp32_fma(d, B, H, rep, n_core):
    """The partial results that the split form leaves at the front of the workspace ([problem][split][vector][accumulator, maximum,
    denominator]), put together in 64 bits, against attention in 64 bits."""
    g = torch.Generator(device="cuda").manual_seed(5)
    K, V, Q = (torch.randn(s, device="cuda", generator=g).bfloat16() for s in ((B, H, n_core, d), (B, H, n_core, d), (B, H * rep, 1, d)))
    idx = torch.arange(n_core, device="cuda", dtype=torch.int32).repeat(B, H, 1)
    w = torch.rand(B, H, n_core, device="cuda", generator=g) + 0.05
    ws = torch.zeros(1 << 30, device="cuda", dtype=torch.uint8)
    elm.attend(Q, K, V, idx, w, workspace=ws)
    ctas, _ = binding.debug_decode_grid(B, H * rep, H, n_core, d, n_core)
    splits, vectors = ctas // (B * H), 4 if rep <= 4 else 8
    part = ws.view(torch.float32)[:ctas * vectors * (d + 2)].view(B, H, splits, vectors, d + 2)[:, :, :, :rep].double()
    f = torch.exp2(part[..., d] - part[..., d].amax(2, keepdim=True))
    got = (f.unsqueeze(-1) * part[..., :d]).sum(2) / (f * part[..., d + 1]).sum(2).unsqueeze(-1)
    s = Q.double().view(B, H, rep, d) @ K.double().transpose(-1, -2) / d ** 0.5 + w.double().log().unsqueeze(2)
    want = torch.softmax(s, dim=-1) @ V.double()
    # fp32 sums of terms that mostly cancel: 8 roundings to 24 bits (fp32 fma: 2.1e-7 and, over 12288 entries, 3.6e-7)
    assert (got - want).norm() / want.norm() <= 2.0 ** -21


@pytest.mark.parametrize("d,rep", [(128, 4), (128, 1), (64, 4)])
def test_streamed_bf16_outputs_are_mostly_the_rounded_exact_value(d, rep):
    """Neighbouring bf16 values are 2^-8 to 2^-7 of themselves apart, and outputs are many times smaller than what fp32 sums: errors of 2^-22
    of an output put about one in 2^12 on the other side of a rounding."""
    x = _Exact(torch.bfloat16, d, rep, 8, 11, 6000, 512)
    got = x.one_call(144)
    K, V = (t.double().repeat_interleave(rep, dim=1) for t in (x.s.K, x.s.V))
    wrong = 0
    for t in range(0, 144, 16):
        s = torch.einsum("tbhqd,bhnd->tbhqn", x.Q[t:t + 16].double(), K) / d ** 0.5
        s = s.masked_fill(torch.arange(6512, device="cuda") > 6000 + t + torch.arange(16, device="cuda")[:, None, None, None, None], -torch.inf)
        want = torch.einsum("tbhqn,bhnd->tbhqd", torch.softmax(s, dim=-1), V).bfloat16()
        wrong += (got[t:t + 16] != want).sum().item()
    assert wrong / got.numel() <= 1.2 * 2.0 ** -12


@pytest.mark.parametrize("gap", [6.0, 7.0, 8.0, 8.75])             # the entry's probability: about 2^-101, 2^-117, 2^-134, 2^-146
@pytest.mark.parametrize("d,rep", [(64, 1), (128, 3), (128, 8)])
def test_infinite_values_at_vanishing_probabilities(d, rep, gap):
    """An entry far below the others: its infinite values reach the output as infinities as long as fp32 holds its probability, a value
    of 1e38 with its share, and the other columns as always - in decode, in single tokens and beside tokens that see the entry with
    an ordinary probability."""
    H, at, n = 2, 70, 700
    x = _Exact(torch.bfloat16, d, rep, H, 8, n, 70)
    K, V, Q = x.s.K, x.s.V, x.Q
    K *= 0.125
    K[:, :, at] = -gap * (128 / d) ** 0.5
    V[:, :, at, 3], V[:, :, at, 5], V[:, :, at, 7] = torch.inf, -torch.inf, 1e38
    ordinary = torch.arange(70, device="cuda") % 5 == 2
    Q[~ordinary] = 1.0
    Q[ordinary] *= 0.125
    Kd, Vd = (t.double().repeat_interleave(rep, dim=1) for t in (K, V))
    Vd[..., at, 3] = Vd[..., at, 5] = 0

    def check(got, q, seen):
        s = q.double() @ Kd[:, :, :seen].transpose(-1, -2) / d ** 0.5
        want = torch.softmax(s, dim=-1) @ Vd[:, :, :seen]
        assert (got[..., 3] == torch.inf).all() and (got[..., 5] == -torch.inf).all()
        for c in (slice(0, 3), slice(4, 5), slice(6, 7), slice(7, 8), slice(8, d)):
            # rounded to 8 bits; 2^-20: columns that come out near zero
            assert ((got[..., c].double() - want[..., c]).abs().amax(-1) <= 2.0 ** -8 * want[..., c].abs().amax(-1) + 2.0 ** -20).all()

    together = x.one_call(60)
    assert torch.equal(together, x.single_steps(60))
    for t in (0, 1, 2, 37, 59):
        check(together[t], Q[t], n + t + 1)
    idx = torch.arange(n, device="cuda", dtype=torch.int32).repeat(1, H, 1)
    check(elm.attend(Q[0], K, V, idx, torch.ones(1, H, n, device="cuda")), Q[0], n)


@pytest.mark.parametrize("B,H,rep,log2_nout,start", [(2, 8, 4, 12, 9000), (2, 9, 1, 12, 8300), (9, 4, 2, 11, 4500), (2, 8, 8, 12, 9000)])
def test_streams_of_many_problems_share_their_launches(B, H, rep, log2_nout, start):
    """Problems whose longer clusters the device cannot hold all at once, lists beyond eight rounds of the shorter ones: the tokens
    of a call still take two launches, the list and the attention, and agree with single steps."""
    x = _Exact(torch.bfloat16, 128, rep, H, log2_nout, start, 64, B)
    before = elm.launch_count()
    got = x.one_call(60)
    assert elm.launch_count() - before == 2
    assert torch.equal(got, x.single_steps(60))


def test_debug_limit_of_clusters_refuses_other_sizes():
    lib = binding.load_library()
    assert all(lib.elm_debug_set(2, v) != 0 for v in (-1, 3, 12, 32))


@pytest.mark.parametrize("dtype_code", [binding.ELM_F32, binding.ELM_BF16])
@pytest.mark.parametrize("vectors", [1, 4, 8])
def test_more_problems_than_resident_ctas_fill_their_waves(dtype_code, vectors):
    """512 problems of a long list: no wave that is nearly empty."""
    ctas, resident = binding.debug_decode_grid(64, 8 * vectors, 8, 4096, 128, 4096, dtype_code=dtype_code)
    assert ctas / (-(-ctas // resident) * resident) >= 0.75


@pytest.mark.parametrize("d", [64, 128])
def test_short_lists_are_spread_over_more_ctas(d):
    """200 entries of 8 KV heads: a CTA for every 32 entries (128 per CTA left the SMs idle and its warps with a chain four
    times as long)."""
    for dtype_code in (binding.ELM_F32, binding.ELM_BF16):
        ctas, _ = binding.debug_decode_grid(1, 32, 8, 200, d, 200, dtype_code=dtype_code)
        assert ctas == 8 * 7


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("rep,n_q", [(1, 1), (2, 1), (4, 1), (1, 3), (8, 1)])
def test_decode_of_short_lists(dtype, d, rep, n_q):
    """Lists around the edges of the short tiles (8 per warp, 32 per CTA), of the CTAs (512 entries) and of the next form,
    unequal weights, one of them zero, an infinite row that no list names."""
    g = torch.Generator(device="cuda").manual_seed(7)
    B, H, n = 2, 3, 700
    K, V = (torch.randn(B, H, n, d, device="cuda", generator=g).to(dtype) for _ in range(2))
    K[:, :, n - 1], V[:, :, n - 1] = float("inf"), float("inf")
    Q = torch.randn(B, H * rep, n_q, d, device="cuda", generator=g).to(dtype)
    # fp32 sums of positive terms; bf16 outputs are rounded to 8 bits
    bound = 1e-5 if dtype == torch.float32 else 2.0 ** -8
    for n_core in (1, 2, 7, 8, 9, 16, 31, 32, 33, 64, 65, 100, 128, 129, 511, 512, 513, 650):
        idx = torch.randint(0, n - 1, (B, H, n_core), device="cuda", generator=g, dtype=torch.int32)
        w = torch.rand(B, H, n_core, device="cuda", generator=g) + 0.05
        if n_core > 1:
            w[:, :, n_core // 2] = 0.0
        got = elm.attend(Q, K, V, idx, w)
        gather = idx.long().unsqueeze(-1).expand(-1, -1, -1, d)
        Kc, Vc = (t.double().gather(2, gather).repeat_interleave(rep, dim=1) for t in (K, V))
        s = torch.einsum("bhqd,bhnd->bhqn", Q.double(), Kc) / d ** 0.5 + w.double().log().repeat_interleave(rep, dim=1).unsqueeze(2)
        want = torch.softmax(s, dim=-1) @ Vc
        err = ((got - want).abs().amax(-1) / want.abs().amax(-1)).max()
        assert err <= bound, (n_core, float(err))


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,H,rep,n_q", [(1, 1, 3, 1), (2, 4, 4, 1), (1, 3, 2, 2), (1, 2, 1, 5), (3, 1, 8, 1), (8, 8, 6, 1), (160, 1, 1, 3)])
def test_decode_on_matrix_instructions(d, B, H, rep, n_q):
    """Lists around the lengths where elm_attend's route, the clusters and the warps' tiles change, three to eight query
    vectors per KV head (heads and rows), unequal weights, one of them zero, against 64 bits."""
    g = torch.Generator(device="cuda").manual_seed(11)
    n = 5300
    K, V = (torch.randn(B, H, n, d, device="cuda", generator=g).bfloat16() for _ in range(2))
    Q = torch.randn(B, H * rep, n_q, d, device="cuda", generator=g).bfloat16()
    for n_core in (1, 31, 33, 129, 513, 1025, 2048, 2049, 4096, 4097, 5250) if B * H < 60 else (33, 600, 4097):
        idx = torch.randint(0, n, (B, H, n_core), device="cuda", generator=g, dtype=torch.int32)
        w = torch.rand(B, H, n_core, device="cuda", generator=g) + 0.05
        if n_core > 1:
            w[:, :, n_core // 2] = 0.0
        got = elm.attend(Q, K, V, idx, w)
        gather = idx.long().unsqueeze(-1).expand(-1, -1, -1, d)
        Kc, Vc = (t.double().gather(2, gather).repeat_interleave(rep, dim=1) for t in (K, V))
        s = torch.einsum("bhqd,bhnd->bhqn", Q.double(), Kc) / d ** 0.5 + w.double().log().repeat_interleave(rep, dim=1).unsqueeze(2)
        want = torch.softmax(s, dim=-1) @ Vc
        err = ((got - want).abs().amax(-1) / want.abs().amax(-1)).max()
        assert err <= 2.0 ** -8, (n_core, float(err))                    # rounded to 8 bits


@pytest.mark.parametrize("rep", [1, 4, 8])
@pytest.mark.parametrize("entries", [100, 200, 400])
def test_streamed_token_over_a_short_list_takes_no_longer_than_attend(rep, entries):
    """One streaming token over a few hundred entries: two launches (its list, its attention) that take no longer than
    elm_attend's two over the same list, a tenth and 3.5 us for the list and noise (a token of eight query vectors took
    twice as long)."""
    x = _Exact(torch.bfloat16, 128, rep, 8, 9, entries, 64)
    q, o = x.Q[0], torch.empty_like(x.Q[0])

    def step():
        x.rewind()
        x.s.step(q, out=o)

    idx = torch.arange(entries, device="cuda", dtype=torch.int32).repeat(1, 8, 1)
    w = torch.ones(1, 8, entries, device="cuda")
    ws = torch.empty(64 << 20, device="cuda", dtype=torch.uint8)
    out = torch.empty_like(q)
    assert _graph_us(step) <= 1.1 * _graph_us(lambda: elm.attend(q, x.s.K, x.s.V, idx, w, workspace=ws, out=out)) + 3.5
