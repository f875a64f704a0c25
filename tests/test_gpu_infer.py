"""GPU parity of the inference side: a condensed KV cache grown in uneven steps and decode attention over
it, against the fp64 CPU oracle.  Decoding the token at position t of a cache that holds t + 1 tokens must
give row t of the oracle's forward on the first t + 1 tokens, and the kept positions recorded in the cache
must be the oracle's selection (bit-exact up to counted ties)."""
import numpy as np
import pytest
import torch

from oracle import lrsa_oracle as orc
from paper_2506_11498_b200 import lrsa, workloads
from tests.parity_utils import check_close, compare_idx, f64, host_bits

pytestmark = pytest.mark.gpu

W = workloads.Workload

CASES = [
    (W("i_d128", 2, 4, 2, 4 + 5 * 128 + 77, 128, 128, 32, 4, seed=81), (1, 1, 2, 37, 128, 300, 5, 1)),
    (W("i_d64", 1, 4, 4, 16 + 6 * 64, 64, 64, 16, 16, seed=82), (7, 64, 1, 129)),
    (W("i_gqa7", 1, 7, 1, 3 + 4 * 200 + 50, 128, 200, 50, 3, seed=83, values="channel_offset"), (250, 1, 1, 199, 403)),
    (W("i_nosink", 1, 2, 2, 6 * 96, 64, 96, 24, 0, seed=84), (96, 96, 1, 95, 200)),
    (W("i_prefill_once", 1, 4, 2, 4 + 7 * 128 + 3, 128, 128, 64, 4, seed=85), (4 + 7 * 128 + 3,)),
    # more query heads per KV head than one pass of the decode kernel takes (16): two passes over the keys
    (W("i_gqa20", 1, 20, 1, 4 + 3 * 128 + 50, 128, 128, 32, 4, seed=88), (200, 1, 150, 87)),
    (W("i_gqa40_d64", 2, 40, 1, 2 + 3 * 64 + 9, 64, 64, 16, 2, seed=89), (100, 1, 1, 101)),
    # lag windows beyond 4096 tokens are scored by the one-slice-per-CTA kernel, here on the ring
    (W("i_long_window", 1, 2, 1, 2 + 3 * 4608 + 100, 64, 4608, 100, 2, seed=86), (5000, 4608, 1, 4000)),
]


def _oracle_row(w, bits, gidx_valid, n):
    """Row n-1 of the oracle's forward on the first n tokens, for every (batch, query head)."""
    op = orc.OracleParams(w.B, w.Hq, w.Hkv, n, w.d, w.L, w.K, w.S)
    sub = {k: np.ascontiguousarray(v[:, :, :n]) for k, v in bits.items()}
    oidx, _ = orc.score_select(op, sub["K"], sub["V"])
    nv = min(gidx_valid.shape[2], oidx.shape[2])
    oidx[:, :, :nv] = gidx_valid[:, :, :nv]     # the cache's own selection where it has one (ties are checked apart)
    rows = np.array([[b, h, n - 1] for b in range(w.B) for h in range(w.Hq)], np.int32)
    O, LSE = orc.fwd_rows(op, sub["Q"], sub["K"], sub["V"], oidx, rows)
    return O.reshape(w.B, w.Hq, w.d), LSE.reshape(w.B, w.Hq)


@pytest.mark.parametrize("w,steps", CASES, ids=lambda x: x.name if hasattr(x, "name") else None)
def test_cache_growth_and_decode(w, steps):
    host = workloads.generate(w, ("Q", "K", "V"))
    bits = host_bits(host)
    dev = {k: v.cuda() for k, v in host.items()}
    p = lrsa.Params.from_workload(w)
    cache = lrsa.KVCache(p)
    i = 0
    checked = 0
    while cache.n_tokens < w.N:
        n_new = min(steps[i % len(steps)], w.N - cache.n_tokens)
        i += 1
        lo = cache.n_tokens
        cache.append(dev["K"][:, :, lo:lo + n_new].contiguous(), dev["V"][:, :, lo:lo + n_new].contiguous())
        n = cache.n_tokens
        o, lse = cache.decode(dev["Q"][:, :, n - 1].contiguous())
        assert cache.status() == 0
        wc = cache.windows_compressed()
        gidx = cache.kept()[:, :, :wc].cpu().numpy()
        oO, oL = _oracle_row(w, bits, gidx, n)
        check_close(f"o at {n} tokens", f64(o), oO)
        check_close(f"lse at {n} tokens", f64(lse), oL, max_abs=2e-3, rel_l2=1e-4, ulp=0.0)
        checked += 1
    # the selection recorded in the cache against the oracle's on the whole sequence
    op = orc.OracleParams(w.B, w.Hq, w.Hkv, w.N, w.d, w.L, w.K, w.S)
    oidx, osc = orc.score_select(op, bits["K"], bits["V"])
    wc = cache.windows_compressed()
    assert wc == max((w.N - 1 - w.S) // w.L - 1, 0) and wc <= oidx.shape[2]
    if wc:
        ties = compare_idx(np.ascontiguousarray(cache.kept()[:, :, :wc].cpu().numpy()), oidx[:, :, :wc], osc[:, :, :wc], w.S, w.L)
        print(f"{w.name}: {checked} decode steps checked, {ties} windows differ only at oracle ties")


@pytest.mark.parametrize("B,Hkv,d", [(15, 1, 64), (8, 2, 128), (16, 2, 64), (33, 1, 128)])   # 15, 16, 32, 33 pairs
def test_growth_on_both_sides_of_the_row_copies_rule(B, Hkv, d):
    """For one token of 16 to 32 (batch, KV head) pairs the row copies wait for the kernel in front before they form their indexes."""
    test_cache_growth_and_decode(W("i_wait", B, 2 * Hkv, Hkv, 4 + 4 * 64 + 9, d, 64, 16, 4, seed=97), (1, 2, 70, 1, 64, 90))


def test_decode_equals_forward_row():
    """The decode kernel and the training forward agree on the last row (same mask, different kernels)."""
    w = W("i_vs_fwd", 1, 8, 2, 4 + 6 * 256 + 100, 128, 256, 64, 4, seed=87)
    host = workloads.generate(w, ("Q", "K", "V"))
    dev = {k: v.cuda() for k, v in host.items()}
    p = lrsa.Params.from_workload(w)
    idx, _ = lrsa.lrsa_score_select(p, dev["K"], dev["V"])
    O, LSE = lrsa.lrsa_attn_fwd(p, dev["Q"], dev["K"], dev["V"], idx)
    cache = lrsa.KVCache(p)
    cache.append(dev["K"], dev["V"])
    o, lse = cache.decode(dev["Q"][:, :, -1].contiguous())
    wc = cache.windows_compressed()
    assert torch.equal(cache.kept()[:, :, :wc], idx[:, :, :wc])
    assert (o.float() - O[:, :, -1].float()).abs().max().item() <= 1e-2
    assert (lse - LSE[:, :, -1]).abs().max().item() <= 1e-3


def test_cache_rejects_bad_arguments():
    p = lrsa.Params(1, 4, 2, 1000, 128, 128, 32, 4)
    cache = lrsa.KVCache(p)
    k = torch.zeros((1, 2, 8, 128), dtype=torch.bfloat16, device="cuda")
    cache.n_tokens = 996
    with pytest.raises(lrsa.LrsaError) as e:       # beyond the capacity
        cache.append(k, k)
    assert e.value.status == 1
    with pytest.raises(lrsa.LrsaError) as e:
        lrsa.KVCache(lrsa.Params(1, 4, 2, 1000, 128, 128, 32, 4, n_dense_prev=0))
    assert e.value.status == 2


@pytest.mark.parametrize("d,L,K,S,N,first", [
    (128, 96, 24, 4, 4 + 9 * 96 + 17, 0),          # a prompt at once: every window lies in the new tokens
    (64, 40, 11, 0, 10 * 40, 40 + 13),             # two windows hold earlier tokens, the others do not
    (128, 33, 33, 7, 7 + 6 * 33 + 1, 7 + 33),      # starts and ends at a chunk start, every token kept
    (64, 64, 16, 16, 16 + 2 * 64 + 1, 3),          # starts inside the sinks; one window, complete with the last token
    (64, 4608, 100, 2, 2 + 3 * 4608 + 5, 4000),    # windows of the one-slice-per-CTA scoring kernel
    (64, 4608, 100, 2, 2 + 4 * 4608 + 5, 0),       # several of them in one launch
])
def test_append_at_once_equals_token_ranges(d, L, K, S, N, first):
    """The cache does not depend on how its tokens were cut into calls: one call for everything after `first` leaves
    the bytes that calls of half a window leave (those never see a whole new window)."""
    w = W("i_cuts", 2, 4, 2, N, d, L, K, S, seed=90, values="channel_offset")
    dev = {k: v.cuda() for k, v in workloads.generate(w, ("K", "V")).items()}
    p = lrsa.Params.from_workload(w)
    cuts = {0, N, *(x for x in range(S, N, max(L // 2, 1)))}
    bufs = []
    for ends in (sorted(cuts), sorted({0, first, N})):
        cache = lrsa.KVCache(p)
        for lo, hi in zip(ends[:-1], ends[1:]):
            cache.append(dev["K"][:, :, lo:hi].contiguous(), dev["V"][:, :, lo:hi].contiguous())
            assert cache.status() == 0
        assert cache.n_tokens == N
        bufs.append(cache.buf)
    assert torch.equal(bufs[0], bufs[1])


@pytest.mark.parametrize("G", [1, 8, 9, 16])
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,N", [(1, 1), (1, 17), (3, 700), (40, 2500), (1, 70000)])
def test_decode_against_fp64(G, d, B, N):
    """Decode over caches of one key, a ragged block, a few splits, several blocks per warp (the small-CTA plan) and
    several clusters for a head (long caches of few heads), with one and two groups of eight heads, against fp64 attention over the visible keys.  P is rounded to bf16
    (2^-9 relative, random signs) and so is the output: the contract's bound holds with room."""
    w = W("i_dec", B, 2 * G, 2, N, d, 256, 256 if N > 2500 else 64, min(4, N), seed=91)
    g = torch.Generator(device="cuda").manual_seed(7)
    k = torch.randn((B, 2, N, d), generator=g, device="cuda").bfloat16()
    v = torch.randn((B, 2, N, d), generator=g, device="cuda").bfloat16()
    q = torch.randn((B, 2 * G, d), generator=g, device="cuda").bfloat16()
    cache = lrsa.KVCache(lrsa.Params.from_workload(w))
    cache.append(k, v)
    o, lse = cache.decode(q)
    assert cache.status() == 0
    nc = max(max(N - 1 - w.S, 0) // w.L - 1, 0)
    pos = torch.arange(w.S, device="cuda").expand(B, 2, -1)
    if nc:
        pos = torch.cat([pos, cache.kept()[:, :, :nc].reshape(B, 2, -1).long()], -1)
    pos = torch.cat([pos, torch.arange(w.S + nc * w.L, N, device="cuda").expand(B, 2, -1)], -1)
    ix = pos[..., None].expand(-1, -1, -1, d)
    kk, vv = k.gather(2, ix).double(), v.gather(2, ix).double()
    s = torch.einsum("bhgd,bhkd->bhgk", q.double().view(B, 2, G, d), kk) / d ** 0.5
    want = torch.einsum("bhgk,bhkd->bhgd", s.softmax(-1), vv).reshape(B, 2 * G, d)
    check_close("o", f64(o), want.cpu().numpy())
    check_close("lse", f64(lse), s.logsumexp(-1).reshape(B, 2 * G).cpu().numpy(), max_abs=2e-3, rel_l2=1e-4, ulp=0.0)


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("G", [7, 12])
@pytest.mark.parametrize("S,N", [(32, 33), (32, 700), (1024, 9000), (40000, 70000), (500, 500)])
def test_decode_scores_of_minus_infinity(d, G, S, N):
    """Keys whose scores overflow to -inf have probability zero, also where a warp's block, a CTA or a whole cluster (long
    caches: several for a head) has no other key: the output is that of attention over the remaining keys.  With no other key at all
    (S = N) it is not defined, and lse is -inf."""
    L, K = 256, 256 if N > 2500 else 64
    g = torch.Generator(device="cuda").manual_seed(8)
    k, v = (torch.randn((1, 2, N, d), generator=g, device="cuda").bfloat16() for _ in range(2))
    q = torch.randn((1, 2 * G, d), generator=g, device="cuda").bfloat16()
    q[..., 0] = 4.0
    k[:, :, :S] = 0.0
    k[:, :, :S, 0] = -3e38
    cache = lrsa.KVCache(lrsa.Params(1, 2 * G, 2, N, d, L, K, S))
    cache.append(k, v)
    o, lse = cache.decode(q)
    assert cache.status() == 0
    if S == N:
        assert (lse == -float("inf")).all()
        return
    nc = cache.windows_compressed()
    pos = torch.cat([cache.kept()[0, :, :nc].reshape(2, -1).long(), torch.arange(S + nc * L, N, device="cuda").expand(2, -1)], -1)
    ix = pos[..., None].expand(-1, -1, d)
    kk, vv = k[0].gather(1, ix).double(), v[0].gather(1, ix).double()
    s = torch.einsum("hgd,hkd->hgk", q.double().view(2, G, d), kk) / d ** 0.5
    want = torch.einsum("hgk,hkd->hgd", s.softmax(-1), vv).reshape(1, 2 * G, d)
    check_close("o", f64(o), want.cpu().numpy())
    check_close("lse", f64(lse), s.logsumexp(-1).reshape(1, 2 * G).cpu().numpy(), max_abs=2e-3, rel_l2=1e-4, ulp=0.0)


@pytest.mark.parametrize("G", [17, 24, 40])
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("B,N,launches", [(1, 1, 2), (1, 129, 2), (2, 700, 2), (3, 5000, 2), (40, 2500, 1), (1, 70000, 2)])
def test_decode_of_wide_groups(G, d, B, N, launches):
    """Groups that take two or three passes of 16 query heads, against fp64 attention: the split kernel (one CTA per 128 keys, two launches with
    its merge) on one key, ragged last splits and full ones; clusters of CTAs for large batches (one launch) and long caches
    (several clusters and the merge)."""
    w = W("i_wide", B, 2 * G, 2, N, d, 256, 256 if N > 5000 else 64, min(4, N), seed=92)
    g = torch.Generator(device="cuda").manual_seed(9)
    k, v = (torch.randn((B, 2, N, d), generator=g, device="cuda").bfloat16() for _ in range(2))
    q = torch.randn((B, 2 * G, d), generator=g, device="cuda").bfloat16()
    cache = lrsa.KVCache(lrsa.Params.from_workload(w))
    cache.append(k, v)
    o, lse = cache.decode(q)
    assert lrsa.lrsa_last_launch_count() == launches
    assert cache.status() == 0
    nc = cache.windows_compressed()
    pos = torch.cat([torch.arange(w.S, device="cuda").expand(B, 2, -1), cache.kept()[:, :, :nc].reshape(B, 2, -1).long(),
                     torch.arange(w.S + nc * w.L, N, device="cuda").expand(B, 2, -1)], -1)
    ix = pos[..., None].expand(-1, -1, -1, d)
    s = torch.einsum("bhgd,bhkd->bhgk", q.double().view(B, 2, G, d), k.gather(2, ix).double()) / d ** 0.5
    want = torch.einsum("bhgk,bhkd->bhgd", s.softmax(-1), v.gather(2, ix).double()).reshape(B, 2 * G, d)
    check_close("o", f64(o), want.cpu().numpy())
    check_close("lse", f64(lse), s.logsumexp(-1).reshape(B, 2 * G).cpu().numpy(), max_abs=2e-3, rel_l2=1e-4, ulp=0.0)


@pytest.mark.parametrize("G", [1, 8])
@pytest.mark.parametrize("d", [64, 128])
def test_decode_on_small_ctas(G, d):
    """Enough blocks of keys for the plan of four-warp CTAs (more than two per warp of the whole GPU) with one group of heads."""
    B, N = 100, 2500
    keys = 4 + (N - 1 - 4) // 256 * 64 - 64 + N - 4 - ((N - 1 - 4) // 256 - 1) * 256
    assert 2 * B * -(-keys // (2048 // d)) > 2 * 148 * 16
    test_decode_against_fp64(G, d, B, N)
