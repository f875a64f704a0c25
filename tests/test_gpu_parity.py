"""GPU parity: the CUDA path, called through the C ABI, against the fp64 CPU oracle on the same
seeded inputs.  Indices bit-exact up to counted oracle ties; O, dQ, dK, dV within max-abs 2e-2
and relative L2 1e-2."""
import numpy as np
import pytest
import torch

from oracle import lrsa_oracle as orc
from paper_2506_11498_b200 import lrsa, workloads
from tests.parity_utils import (REPORT, check_close, gradient_error_terms, compare_idx, error_stats, f64, host_bits, oparams, to_dev)

pytestmark = pytest.mark.gpu

W = workloads.Workload

SCORE_CASES = [
    W("s_d128", 2, 4, 2, 2048 + 4 + 77, 128, 256, 64, 4, seed=11),
    W("s_d64", 1, 4, 4, 4096, 64, 512, 128, 16, seed=12),
    W("s_ragged128", 1, 2, 2, 3 + 7 * 100 + 5, 128, 100, 30, 3, seed=13),
    W("s_ragged64", 2, 2, 2, 9 * 72, 64, 72, 9, 0, seed=14),
    W("s_keepall", 1, 2, 2, 5 * 128 + 2, 128, 128, 128, 2, seed=15),
    W("s_keep1", 1, 2, 2, 5 * 128 + 2, 64, 128, 1, 2, seed=16),
    W("s_offsets", 1, 4, 2, 4 + 8 * 1024, 128, 1024, 256, 4, seed=17, values="channel_offset"),
    W("s_salient", 1, 2, 2, 4 + 4 * 2048 + 9, 128, 2048, 512, 4, seed=18, values="salient"),
    W("s_tiny_window", 1, 1, 1, 70, 64, 8, 3, 1, seed=19),
    # lag windows beyond 4096 tokens take the one-slice-per-CTA kernel with global statistics
    W("s_long_window", 1, 1, 1, 2 + 3 * 4608 + 11, 64, 4608, 100, 2, seed=42),
    W("s_long_window128", 1, 2, 1, 4 * 4160, 128, 4160, 4000, 0, seed=43),
]


@pytest.mark.parametrize("w", SCORE_CASES, ids=lambda w: w.name)
@pytest.mark.parametrize("ddof", [1, 0])
def test_score_select(w, ddof):
    if ddof == 0 and w.name not in ("s_d128", "s_d64"):
        pytest.skip("ddof=0 covered on two cases")
    host = workloads.generate(w, ("K", "V"))
    bits = host_bits(host)
    op = oparams(w, ddof=ddof)
    oidx, osc = orc.score_select(op, bits["K"], bits["V"])
    dev = to_dev(host)
    p = lrsa.Params.from_workload(w, std_ddof=ddof)
    ws = lrsa.new_workspace(lrsa.lrsa_workspace_bytes(p)[0])
    idx, sc = lrsa.lrsa_score_select(p, dev["K"], dev["V"], workspace=ws, want_score=True)
    assert lrsa.lrsa_workspace_status(ws) == 0
    np.testing.assert_allclose(f64(sc), osc, rtol=2e-5, atol=0)
    ties = compare_idx(idx.cpu().numpy(), oidx, osc, w.S, w.L)
    print(f"{w.name}: windows differing only at oracle ties: {ties}")
    # a second call on the same workspace gives the same bits
    idx2, _ = lrsa.lrsa_score_select(p, dev["K"], dev["V"], workspace=ws)
    assert torch.equal(idx, idx2)


@pytest.mark.parametrize("B,Hkv,N,d,L,cuts", [
    (1, 8, 16384, 64, 333, ()),              # d = 64, two windows a CTA
    (2, 8, 33000, 64, 500, ()),              # four
    (1, 8, 16384, 64, 333, (5000, 5001, 11000)),   # the same over the sequences of a packed row
    (1, 8, 33000, 128, 512, ()),
    (1, 8, 33000, 128, 512, (700, 9000, 25000)),
    (1, 4, 2100 * 9, 64, 2100, ()),          # long windows at d = 64: one window a CTA, or a cluster's
])
def test_selection_with_several_windows_per_cta(B, Hkv, N, d, L, cuts):
    """Enough windows that a CTA walks a run of them and folds the statistics of each while it is scored, against the oracle."""
    w = W("s_runs", B, Hkv, Hkv, N, d, L, L // 4, 4, seed=45, values="channel_offset")
    host = workloads.generate(w, ("K", "V"))
    bits = host_bits(host)
    op = oparams(w)
    cu = (0, *cuts, N)
    oidx, osc = orc.score_select_packed(op, bits["K"], bits["V"], cu)
    dev = to_dev(host)
    p = lrsa.Params.from_workload(w, cu_seqlens=cu if cuts else ())
    idx, sc = lrsa.lrsa_score_select(p, dev["K"], dev["V"], want_score=True)
    np.testing.assert_allclose(f64(sc), osc, rtol=2e-5, atol=0)
    got = idx.cpu().numpy()
    for t0, n, wsel, woff in orc.packed_windows(op, cu):
        if wsel:
            compare_idx(got[:, :, woff:woff + wsel] - t0, oidx[:, :, woff:woff + wsel] - t0, osc[:, :, woff:woff + wsel],
                        min(w.S, n), w.L)


def test_longest_window_that_is_scored():
    """25 448 tokens is the longest lag window of the selection (its scores lie in shared memory); one more is refused."""
    w = W("s_longest", 1, 1, 1, 2 * 25448 + 1, 64, 25448, 700, 1, seed=44)
    host = workloads.generate(w, ("K", "V"))
    bits = host_bits(host)
    oidx, osc = orc.score_select(oparams(w), bits["K"], bits["V"])
    dev = to_dev(host)
    p = lrsa.Params.from_workload(w)
    ws = lrsa.new_workspace(lrsa.lrsa_workspace_bytes(p)[0])
    idx, sc = lrsa.lrsa_score_select(p, dev["K"], dev["V"], workspace=ws, want_score=True)
    assert lrsa.lrsa_workspace_status(ws) == 0
    np.testing.assert_allclose(f64(sc), osc, rtol=2e-5, atol=0)
    compare_idx(idx.cpu().numpy(), oidx, osc, w.S, w.L)
    longer = lrsa.Params(1, 1, 1, 2 * 25449, 64, 25449, 700, 0)
    with pytest.raises(lrsa.LrsaError) as e:
        lrsa.lrsa_score_select(longer, dev["K"], dev["V"])
    assert e.value.status == 2


def test_score_zero_range_channel():
    w = W("s_const", 1, 2, 2, 2 + 4 * 128, 128, 128, 32, 2, seed=20)
    host = workloads.generate(w, ("K", "V"))
    host["K"][..., 5] = 1.5
    host["V"][:, 0, :, 100] = -2.0
    bits = host_bits(host)
    oidx, osc = orc.score_select(oparams(w), bits["K"], bits["V"])
    dev = to_dev(host)
    idx, sc = lrsa.lrsa_score_select(lrsa.Params.from_workload(w), dev["K"], dev["V"], want_score=True)
    np.testing.assert_allclose(f64(sc), osc, rtol=2e-5)
    compare_idx(idx.cpu().numpy(), oidx, osc, w.S, w.L)


ATTN_CASES = [
    # name, B, Hq, Hkv, N, d, L, K, S ; then ndp
    (W("a_d128", 1, 4, 2, 4 + 5 * 256 + 77, 128, 256, 64, 4, seed=21), 1),
    (W("a_d64", 2, 4, 4, 16 + 6 * 128, 64, 128, 32, 16, seed=22), 1),           # T = 0
    (W("a_gqa7", 1, 7, 1, 3 + 4 * 200 + 50, 128, 200, 50, 3, seed=23), 1),      # L, S not tile multiples
    (W("a_nosink", 1, 2, 2, 5 * 128 + 1, 64, 128, 100, 0, seed=24), 1),         # S = 0, T = 1
    (W("a_keepall", 1, 2, 1, 4 + 4 * 128 + 30, 128, 128, 128, 4, seed=25), 1),  # K = L: dense causal
    (W("a_ndp0", 1, 4, 2, 4 + 5 * 256 + 77, 128, 256, 64, 4, seed=26), 0),
    (W("a_short", 1, 2, 2, 300, 128, 256, 64, 4, seed=27), 1),                  # W = 1: plain causal
    (W("a_two", 1, 2, 2, 4 + 2 * 256 + 10, 64, 256, 16, 4, seed=28), 1),        # one scored window, unused
    (W("a_ndp0_two", 1, 2, 2, 4 + 2 * 256 + 10, 64, 256, 16, 4, seed=29), 0),
    (W("a_one_token", 1, 1, 1, 1, 64, 8, 2, 0, seed=30), 1),
    (W("a_sinks_only", 1, 2, 1, 5, 64, 8, 2, 5, seed=31), 1),
    (W("a_offsets", 1, 4, 2, 4 + 5 * 256 + 77, 128, 256, 64, 4, seed=32, values="channel_offset"), 1),
    (W("a_salient64", 1, 4, 1, 16 + 5 * 128 + 40, 64, 128, 32, 16, seed=33, values="salient"), 1),
]


def _run_attention(w, ndp, idx_np, host, impl=0):
    """impl 0: the tensor-core kernels; 1: the CUDA-core validation kernels (fp32 throughout)."""
    dev = to_dev(host)
    p = lrsa.Params.from_workload(w, n_dense_prev=ndp)
    idx = torch.from_numpy(idx_np).cuda()
    wf, wb = lrsa.lrsa_workspace_bytes(p)[1:]
    wsf, wsb = lrsa.new_workspace(wf), lrsa.new_workspace(wb)
    lrsa.lrsa_debug_set_impl(impl)
    try:
        O, LSE = lrsa.lrsa_attn_fwd(p, dev["Q"], dev["K"], dev["V"], idx, workspace=wsf)
        dQ, dK, dV = lrsa.lrsa_attn_bwd(p, dev["Q"], dev["K"], dev["V"], O, dev["dO"], LSE, idx, workspace=wsb)
    finally:
        lrsa.lrsa_debug_set_impl(0)
    assert lrsa.lrsa_workspace_status(wsf) == 0 and lrsa.lrsa_workspace_status(wsb) == 0
    return O, LSE, dQ, dK, dV


@pytest.mark.parametrize("w,ndp", ATTN_CASES, ids=lambda x: x.name if hasattr(x, "name") else str(x))
def test_attention_fwd_bwd(w, ndp):
    host = workloads.generate(w)
    bits = host_bits(host)
    op = oparams(w, n_dense_prev=ndp)
    oidx, _ = orc.score_select(op, bits["K"], bits["V"])
    oO, oL = orc.attn_fwd(op, bits["Q"], bits["K"], bits["V"], oidx)
    odQ, odK, odV = orc.attn_bwd(op, bits["Q"], bits["K"], bits["V"], bits["dO"], oidx)
    O, LSE, dQ, dK, dV = _run_attention(w, ndp, oidx, host)
    check_close("O", f64(O), oO)
    check_close("LSE", f64(LSE), oL, max_abs=2e-3, rel_l2=1e-4, ulp=0.0)
    if w.values == "salient":
        # The deliberately ill-conditioned case (700 tokens, d = 64, a handful of keys scaled by 8): its
        # gradient elements are cancelling sums of large terms, and the bound follows the terms.
        e = gradient_error_terms(w, op, bits, oidx, oO, oL)
        check_close("dQ", f64(dQ), odQ, terms=e["mQ"])
        check_close("dK", f64(dK), odK, terms=e["mK"], extra=e["dK_from_D"])
        check_close("dV", f64(dV), odV, terms=e["mV"])
    else:
        check_close("dQ", f64(dQ), odQ)
        check_close("dK", f64(dK), odK)
        check_close("dV", f64(dV), odV)


@pytest.mark.parametrize("S", [1, 16, 17, 80])
@pytest.mark.parametrize("d,B", [(64, 1), (128, 1), (64, 20)])
def test_last_list_tile_of_few_keys(d, B, S):
    """K = 128 leaves S keys for the last tile of the sinks + kept list: the short form of the tile takes up to 16 (in the dQ
    kernel, whose tiles hold 64 keys, S = 80 is 64 + 16).  Batch 20: the dQ kernel's form for many CTAs at d = 64."""
    w = W(f"a_tail{S}", B, 2, 1, S + 900, d, 256, 128, S, seed=35)
    host = workloads.generate(w)
    bits = host_bits(host)
    op = oparams(w, n_dense_prev=1)
    oidx, _ = orc.score_select(op, bits["K"], bits["V"])
    oO, oL = orc.attn_fwd(op, bits["Q"], bits["K"], bits["V"], oidx)
    odQ, odK, odV = orc.attn_bwd(op, bits["Q"], bits["K"], bits["V"], bits["dO"], oidx)
    O, LSE, dQ, dK, dV = _run_attention(w, 1, oidx, host)
    check_close("O", f64(O), oO)
    check_close("LSE", f64(LSE), oL, max_abs=2e-3, rel_l2=1e-4, ulp=0.0)
    check_close("dQ", f64(dQ), odQ)
    check_close("dK", f64(dK), odK)
    check_close("dV", f64(dV), odV)


@pytest.mark.parametrize("S", [1, 4, 16, 40])
@pytest.mark.parametrize("d,B,L,n", [(64, 1, 256, 700), (128, 1, 256, 700), (128, 30, 1024, 2100)])
def test_sinks_with_scores_of_minus_infinity(d, B, L, n, S):
    """A score that overflows to -inf has probability zero, also where the sinks are all that a query's first list tile
    holds (up to 16 of them: the short tile; batch 30: two query tiles per CTA).  The queries at the sinks see nothing else
    and have no defined output."""
    w = W(f"a_inf{S}", B, 2, 1, S + n, d, L, 64, S, seed=37)
    host = workloads.generate(w, ("Q", "K", "V"))
    host["Q"][..., 0] = 4.0
    host["K"][:, :, :S] = 0.0
    host["K"][:, :, :S, 0] = -3e38
    dev = to_dev(host)
    p = lrsa.Params.from_workload(w)
    idx, _ = lrsa.lrsa_score_select(p, dev["K"], dev["V"])
    O, LSE = lrsa.lrsa_attn_fwd(p, dev["Q"], dev["K"], dev["V"], idx)
    one = w.with_(B=1)
    bits = host_bits({k: v[:1] for k, v in host.items()})
    oO, oL = orc.attn_fwd(oparams(one), bits["Q"], bits["K"], bits["V"], idx[:1].cpu().numpy())
    check_close("O", f64(O[:1, :, S:]), oO[:, :, S:])
    check_close("LSE", f64(LSE[:1, :, S:]), oL[:, :, S:], max_abs=2e-3, rel_l2=1e-4, ulp=0.0)
    assert torch.isfinite(O[:, :, S:].float()).all() and torch.isfinite(LSE[:, :, S:]).all()


@pytest.mark.parametrize("S,N", [(1, 2949), (17, 3300)])
def test_one_and_two_query_tiles_per_cta_agree(S, N):
    """The forward of four sequences runs with two query tiles per CTA, that of one with one (fewer CTAs): every row does the
    same arithmetic in the same order, so the results are the same bits."""
    w = W(f"a_tiles{S}", 4, 28, 4, N, 128, 512, 128, S, seed=36)
    dev = to_dev(workloads.generate(w))
    p = lrsa.Params.from_workload(w, n_dense_prev=1)
    idx = lrsa.lrsa_score_select(p, dev["K"], dev["V"])[0]
    O, LSE = lrsa.lrsa_attn_fwd(p, dev["Q"], dev["K"], dev["V"], idx)
    p1 = lrsa.Params.from_workload(W(f"a_tiles{S}", 1, 28, 4, N, 128, 512, 128, S, seed=36), n_dense_prev=1)
    for b in range(4):
        part = [t[b:b + 1].contiguous() for t in (dev["Q"], dev["K"], dev["V"], idx)]
        o, lse = lrsa.lrsa_attn_fwd(p1, *part)
        assert torch.equal(o, O[b:b + 1]) and torch.equal(lse, LSE[b:b + 1])


@pytest.mark.parametrize("name", ["a_salient64", "a_offsets", "a_gqa7", "a_ndp0"])
def test_cuda_core_validation_kernels_against_oracle(name):
    """The slow CUDA-core kernels (fp32 P and dS, no tensor cores) against the oracle at the same
    element-wise bound: they share the bf16 inputs and outputs with the tensor-core path but none of its
    bf16 rounding of P and dS, so their error is the floor set by the I/O format alone."""
    w, ndp = next(c for c in ATTN_CASES if c[0].name == name)
    host = workloads.generate(w)
    bits = host_bits(host)
    op = oparams(w, n_dense_prev=ndp)
    oidx, _ = orc.score_select(op, bits["K"], bits["V"])
    oO, oL = orc.attn_fwd(op, bits["Q"], bits["K"], bits["V"], oidx)
    odQ, odK, odV = orc.attn_bwd(op, bits["Q"], bits["K"], bits["V"], bits["dO"], oidx)
    O, LSE, dQ, dK, dV = _run_attention(w, ndp, oidx, host, impl=1)
    check_close("ref-kernel O", f64(O), oO)
    check_close("ref-kernel LSE", f64(LSE), oL, max_abs=2e-3, rel_l2=1e-4, ulp=0.0)
    check_close("ref-kernel dV", f64(dV), odV)
    if name == "a_salient64":
        # These kernels take D = rowsum(dO * O) from the bf16 O, as the textbook backward does.  With a few
        # dominant keys of large norm that D is not accurate enough for dQ and dK, fp32 arithmetic or not:
        # the error is recorded (it is why the tensor-core path sums P * dP instead), not bounded.
        for nm, got, want in (("dQ", dQ, odQ), ("dK", dK, odK)):
            st = error_stats(f64(got), want)
            REPORT.append({"test": "textbook D, fp32 CUDA-core kernels, a_salient64", "tensor": nm, **st})
            print(f"ref-kernel {nm} with the textbook D: max|err| {st['max_abs']:.3g}, rel L2 {st['rel_l2']:.3g}")
            assert st["rel_l2"] < 2e-2
        assert error_stats(f64(dQ), odQ)["max_abs"] > 2e-2
    else:
        check_close("ref-kernel dQ", f64(dQ), odQ)
        check_close("ref-kernel dK", f64(dK), odK)


def test_end_to_end_and_determinism():
    w = W("e2e", 2, 8, 2, 4 + 6 * 256 + 100, 128, 256, 64, 4, seed=40, values="channel_offset")
    host = workloads.generate(w)
    bits = host_bits(host)
    op = oparams(w)
    oidx, osc = orc.score_select(op, bits["K"], bits["V"])
    dev = to_dev(host)
    p = lrsa.Params.from_workload(w)
    idx, _ = lrsa.lrsa_score_select(p, dev["K"], dev["V"])
    assert compare_idx(idx.cpu().numpy(), oidx, osc, w.S, w.L) == 0
    outs = []
    for _ in range(2):
        O, LSE = lrsa.lrsa_attn_fwd(p, dev["Q"], dev["K"], dev["V"], idx)
        dQ, dK, dV = lrsa.lrsa_attn_bwd(p, dev["Q"], dev["K"], dev["V"], O, dev["dO"], LSE, idx)
        outs.append((O, LSE, dQ, dK, dV))
    rows = orc.all_rows(op)[:: 37]
    oO, oL = orc.fwd_rows(op, bits["Q"], bits["K"], bits["V"], oidx, rows)
    got = np.stack([f64(outs[0][0][b, h, t]) for b, h, t in rows])
    check_close("O rows", got, oO)
    # run-to-run: forward bitwise, backward within accumulation-order noise
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])
    for a, b in zip(outs[0][2:], outs[1][2:]):
        assert (a.float() - b.float()).abs().max().item() <= 2e-2


def test_unkept_rows_get_no_gradient_from_later_chunks():
    """Static-mask invariant: with dO zero before chunk 2, un-kept rows of window 0 get exactly zero
    dK and dV while its kept rows and the sinks do not."""
    w = W("p11", 1, 4, 2, 4 + 5 * 256, 128, 256, 64, 4, seed=41)
    host = workloads.generate(w)
    host["dO"][:, :, : w.S + 2 * w.L] = 0
    bits = host_bits(host)
    oidx, _ = orc.score_select(oparams(w), bits["K"], bits["V"])
    O, LSE, dQ, dK, dV = _run_attention(w, 1, oidx, host)
    kept = np.zeros(w.N, bool)
    kept[oidx[0, 0, 0]] = True
    win0 = np.arange(w.S, w.S + w.L)
    un = win0[~kept[win0]]
    assert dK[0, 0, un].abs().max().item() == 0 and dV[0, 0, un].abs().max().item() == 0
    assert dV[0, 0, oidx[0, 0, 0]].abs().min(dim=0).values.max().item() > 0
    assert dV[0, 0, : w.S].abs().max().item() > 0


# ---- packed variable-length batches and query chunks of several lag windows ----

PACKED_CASES = [
    # workload (N = last boundary), boundaries, ndp
    (W("p_two", 1, 4, 2, 1500, 128, 128, 32, 4, seed=51), (0, 4 + 5 * 128 + 77, 1500), 1),     # unequal, both with tails
    (W("p_three64", 2, 4, 4, 1200, 64, 64, 16, 16, seed=52), (0, 16 + 8 * 64, 16 + 8 * 64 + 10, 1200), 1),  # T = 0; shorter than S
    (W("p_gqa7", 1, 7, 1, 1000, 128, 100, 30, 3, seed=53, values="channel_offset"), (0, 333, 334, 1000), 1),  # one-token sequence
    (W("p_ndp0", 1, 2, 2, 900, 64, 128, 32, 4, seed=54), (0, 500, 900), 0),
    # more sequences than one launch takes (16): two batches, the last of one sequence
    (W("p_17", 1, 2, 1, 1700, 128, 32, 8, 4, seed=55), (0, 90, 93, *range(200, 1600, 100), 1700), 1),
    (W("p_20", 2, 2, 2, 1300, 64, 24, 5, 2, seed=56), (0, *range(17, 1000, 53), 1300), 1),
]


@pytest.mark.parametrize("w,cu,ndp", PACKED_CASES, ids=lambda x: x.name if hasattr(x, "name") else None)
def test_packed_sequences(w, cu, ndp):
    """Several sequences back to back on the token axis: every stage against the oracle applied to
    each sequence on its own."""
    host = workloads.generate(w)
    bits = host_bits(host)
    op = oparams(w, n_dense_prev=ndp)
    oidx, osc = orc.score_select_packed(op, bits["K"], bits["V"], cu)
    dev = to_dev(host)
    p = lrsa.Params.from_workload(w, n_dense_prev=ndp, cu_seqlens=cu)
    assert lrsa.lrsa_num_sel_windows(p) == oidx.shape[2]
    sizes = lrsa.lrsa_workspace_bytes(p)
    ws = [lrsa.new_workspace(s) for s in sizes]
    idx, sc = lrsa.lrsa_score_select(p, dev["K"], dev["V"], workspace=ws[0], want_score=True)
    np.testing.assert_allclose(f64(sc), osc, rtol=2e-5, atol=0)
    got = idx.cpu().numpy()
    for t0, n, wsel, woff in orc.packed_windows(op, cu):      # per sequence: window numbering restarts
        if wsel:
            compare_idx(got[:, :, woff:woff + wsel] - t0, oidx[:, :, woff:woff + wsel] - t0,
                        osc[:, :, woff:woff + wsel], min(w.S, n), w.L)
    idx = torch.from_numpy(oidx).cuda()
    O, LSE = lrsa.lrsa_attn_fwd(p, dev["Q"], dev["K"], dev["V"], idx, workspace=ws[1])
    dQ, dK, dV = lrsa.lrsa_attn_bwd(p, dev["Q"], dev["K"], dev["V"], O, dev["dO"], LSE, idx, workspace=ws[2])
    for s in ws:
        assert lrsa.lrsa_workspace_status(s) == 0
    oO, oL = orc.attn_fwd_packed(op, bits["Q"], bits["K"], bits["V"], oidx, cu)
    odQ, odK, odV = orc.attn_bwd_packed(op, bits["Q"], bits["K"], bits["V"], bits["dO"], oidx, cu)
    check_close("O", f64(O), oO)
    check_close("LSE", f64(LSE), oL, max_abs=2e-3, rel_l2=1e-4, ulp=0.0)
    check_close("dQ", f64(dQ), odQ)
    check_close("dK", f64(dK), odK)
    check_close("dV", f64(dV), odV)


@pytest.mark.parametrize("N,d,L,K,S", [(700, 64, 40, 13, 5), (2048, 128, 64, 64, 16), (1500, 128, 600, 100, 40), (333, 64, 8, 3, 0)])
def test_one_workspace_for_every_packing_of_a_row(N, d, L, K, S):
    """The workspace of the unpacked row, between margins that must stay untouched, through packings of a few sequences to
    very many (several batches of sequences, the compact buffers and launch tables used again by each), the shortest ones all sinks.  O is
    bit-equal to that of each sequence on its own."""
    w = W("p_ws", 1, 4, 2, N, d, L, K, S, seed=57)
    dev = to_dev(workloads.generate(w))
    sizes = lrsa.lrsa_workspace_bytes(lrsa.Params.from_workload(w))
    bufs = [torch.full((n + 8192,), 0xA5, dtype=torch.uint8, device="cuda") for n in sizes]
    ws = [b[4096:4096 + n] for b, n in zip(bufs, sizes)]
    rng = np.random.default_rng(N)
    packings = [[], range(max(S, 1), N, max(S, 1)), range(S + 2 * L, N, S + 2 * L)]
    packings += [sorted(rng.choice(np.arange(1, N), int(k), replace=False).tolist()) for k in (1, 5, 14, 15, 16, 40)]
    for cuts in packings:
        cu = (0, *[c for c in cuts][:300], N)
        p = lrsa.Params.from_workload(w, cu_seqlens=cu)
        idx, _ = lrsa.lrsa_score_select(p, dev["K"], dev["V"], workspace=ws[0])
        O, LSE = lrsa.lrsa_attn_fwd(p, dev["Q"], dev["K"], dev["V"], idx, workspace=ws[1])
        grads = lrsa.lrsa_attn_bwd(p, dev["Q"], dev["K"], dev["V"], O, dev["dO"], LSE, idx, workspace=ws[2])
        assert all(lrsa.lrsa_workspace_status(x) == 0 for x in ws)
        assert all(torch.isfinite(t.float()).all() for t in (O, LSE, *grads))
        for b, n in zip(bufs, sizes):
            assert (b[:4096] == 0xA5).all() and (b[4096 + n:] == 0xA5).all()
        for i in rng.choice(len(cu) - 1, min(4, len(cu) - 1), replace=False):
            lo, hi = cu[i], cu[i + 1]
            one = W("p_ws1", 1, 4, 2, hi - lo, d, L, K, min(S, hi - lo))
            q, k, v = (dev[x][:, :, lo:hi].contiguous() for x in "QKV")
            p1 = lrsa.Params.from_workload(one)
            i1, _ = lrsa.lrsa_score_select(p1, k, v)
            o1, l1 = lrsa.lrsa_attn_fwd(p1, q, k, v, i1)
            assert torch.equal(o1, O[:, :, lo:hi]) and torch.equal(l1, LSE[:, :, lo:hi])


@pytest.mark.parametrize("heads,d,L,K,S,lens", [
    ((28, 4), 128, 512, 128, 4, (3000, 3100, 2901)),           # forward of two query tiles per CTA, packed
    ((8, 8), 64, 256, 64, 16, (1800, 2100, 77, 2500, 2523)),   # dQ with one score buffer per CTA, packed
])
def test_packed_forms_for_many_ctas(heads, d, L, K, S, lens):
    """Packed rows large enough for the forms that only large grids take, against each sequence on its own (the forms for small
    grids, which the oracle cases cover): O and LSE bit-equal, gradients within the bound of two bf16 results."""
    N, cu = sum(lens), (0, *np.cumsum(lens).tolist())
    w = W("p_many", 1, *heads, N, d, L, K, S, seed=58, values="channel_offset")

    def blocks(n, rows):       # query blocks of a sequence: sinks, full windows, tail
        wins, tail = (n - S) // L, (n - S) % L
        return -(-S // rows) + wins * -(-L // rows) + -(-tail // rows)
    if d == 128:
        keys = sum(n * (S + max(-(-(n - S) // L) - 2, 0) * K // 2 + min(n // 2, L + L // 2)) for n in lens)
        assert sum(blocks(n, 256) for n in lens) * heads[0] > 4 * 148 and 2 * keys > 15 * 128 * N
    else:
        assert sum(blocks(n, 128) for n in lens) * heads[0] > 2 * 148
    dev = to_dev(workloads.generate(w))
    p = lrsa.Params.from_workload(w, cu_seqlens=cu)
    ws = [lrsa.new_workspace(n) for n in lrsa.lrsa_workspace_bytes(p)]
    idx, _ = lrsa.lrsa_score_select(p, dev["K"], dev["V"], workspace=ws[0])
    O, LSE = lrsa.lrsa_attn_fwd(p, dev["Q"], dev["K"], dev["V"], idx, workspace=ws[1])
    grads = lrsa.lrsa_attn_bwd(p, dev["Q"], dev["K"], dev["V"], O, dev["dO"], LSE, idx, workspace=ws[2])
    assert all(lrsa.lrsa_workspace_status(x) == 0 for x in ws)
    woff = 0
    for lo, hi in zip(cu[:-1], cu[1:]):
        one = w.with_(N=hi - lo)
        q, k, v, do = (dev[x][:, :, lo:hi].contiguous() for x in ("Q", "K", "V", "dO"))
        p1 = lrsa.Params.from_workload(one)
        i1, _ = lrsa.lrsa_score_select(p1, k, v)
        assert torch.equal(i1 + lo, idx[:, :, woff:woff + i1.shape[2]])
        woff += i1.shape[2]
        o1, l1 = lrsa.lrsa_attn_fwd(p1, q, k, v, i1)
        assert torch.equal(o1, O[:, :, lo:hi]) and torch.equal(l1, LSE[:, :, lo:hi])
        for name, a, b in zip(("dQ", "dK", "dV"), grads, lrsa.lrsa_attn_bwd(p1, q, k, v, o1, do, l1, i1)):
            check_close(name, f64(a[:, :, lo:hi]), f64(b))


@pytest.mark.parametrize("B,heads,N,d,L,K,S", [
    (37, (1, 1), 304, 64, 128, 32, 4), (149, (1, 1), 100, 64, 128, 32, 0), (74, (1, 1), 304, 64, 128, 32, 4),   # forward and dQ: 148, 149, 296 blocks
    (75, (1, 1), 304, 64, 128, 32, 4), (150, (1, 1), 304, 128, 128, 32, 4),   # 300; dK/dV of more than 592 CTAs
    (2, (14, 2), 2500, 128, 256, 64, 4), (9, (14, 2), 2500, 128, 256, 64, 4),   # tiles of several segments, in both orders
])
def test_launch_orders_of_small_and_large_grids(B, heads, N, d, L, K, S):
    """The launch order of dK/dV (longest segments first, or segment-major) follows the size of the grid: every sequence of a batch
    as on its own.  O and LSE bit-equal, gradients (sums in another order) within the bound of two bf16 results."""
    w = W("a_order", B, *heads, N, d, L, K, S, seed=61, values="channel_offset")
    dev = to_dev(workloads.generate(w))

    def run(p, t):
        ws = [lrsa.new_workspace(n) for n in lrsa.lrsa_workspace_bytes(p)]
        idx, _ = lrsa.lrsa_score_select(p, t["K"], t["V"], workspace=ws[0])
        O, LSE = lrsa.lrsa_attn_fwd(p, t["Q"], t["K"], t["V"], idx, workspace=ws[1])
        grads = lrsa.lrsa_attn_bwd(p, t["Q"], t["K"], t["V"], O, t["dO"], LSE, idx, workspace=ws[2])
        assert all(lrsa.lrsa_workspace_status(x) == 0 for x in ws)
        return idx, O, LSE, *grads
    whole = run(lrsa.Params.from_workload(w), dev)
    for b in (0, B // 2, B - 1):
        one = run(lrsa.Params.from_workload(w.with_(B=1)), {x: dev[x][b:b + 1].contiguous() for x in dev})
        for t, o in zip(whole[:3], one[:3]):
            assert torch.equal(t[b:b + 1], o)
        for name, t, o in zip(("dQ", "dK", "dV"), whole[3:], one[3:]):
            check_close(name, f64(t[b:b + 1]), f64(o))


@pytest.mark.parametrize("B,heads,N,d,L,S", [(1, (28, 4), 6000, 128, 512, 4), (4, (28, 4), 3000, 128, 512, 17), (2, (8, 8), 8000, 64, 256, 16)])
def test_forward_gives_the_same_bits_every_time(B, heads, N, d, L, S):
    """P is overwritten by the next scores as soon as the product that reads it has been issued, on the order in which the tensor
    core runs one thread's products.  An overlap of the two would depend on timing and show between repeats."""
    w = W("a_repeat", B, *heads, N, d, L, L // 4, S, seed=59)
    dev = to_dev(workloads.generate(w, ("Q", "K", "V")))
    p = lrsa.Params.from_workload(w)
    idx, _ = lrsa.lrsa_score_select(p, dev["K"], dev["V"])
    O, LSE = lrsa.lrsa_attn_fwd(p, dev["Q"], dev["K"], dev["V"], idx)
    for _ in range(20):
        o, lse = lrsa.lrsa_attn_fwd(p, dev["Q"], dev["K"], dev["V"], idx)
        assert torch.equal(o, O) and torch.equal(lse, LSE)


def _backward(w):
    """Inputs of a backward call, and the call."""
    dev = to_dev(workloads.generate(w))
    p = lrsa.Params.from_workload(w)
    idx, _ = lrsa.lrsa_score_select(p, dev["K"], dev["V"])
    O, LSE = lrsa.lrsa_attn_fwd(p, dev["Q"], dev["K"], dev["V"], idx)
    return lambda: lrsa.lrsa_attn_bwd(p, dev["Q"], dev["K"], dev["V"], O, dev["dO"], LSE, idx)


@pytest.mark.parametrize("d", [64, 128])
def test_dk_and_dv_have_the_same_bits_every_time(d):
    """The same order of products, S^T over P^T and dP^T over dS^T.  No window is compressed here and a key tile is one CTA's (16 pairs
    of head and query tile at most), so that every row of dK and dV is one sum of one thread block, added to zero."""
    call = _backward(W("a_repeat_kv", 4, 16, 8, 1024, d, 512, 128, 0, seed=67))
    _, dK, dV = call()
    for _ in range(20):
        _, dk, dv = call()
        assert torch.equal(dk, dK) and torch.equal(dv, dV)


@pytest.mark.parametrize("B,heads,N,d,L,S", [(1, (28, 4), 6000, 128, 512, 4), (2, (8, 8), 8000, 64, 256, 16)])
def test_dq_is_the_same_every_time_but_for_roundings(B, heads, N, d, L, S):
    """dS overwritten by the next scores, as above.  The rows' D is added up in any order, which moves it by fp32 roundings and with it
    some bf16 roundings of dS and dQ: by 2^-7 of an element each, so by no more than that of a block's norm.  A product that
    read a tile's next scores instead would move a whole block by a part of its own size."""
    call = _backward(W("a_repeat_q", B, *heads, N, d, L, L // 4, S, seed=71))
    blocks = lambda t: t.float().view(-1, 100 * d)   # 100 rows of one head
    dQ = blocks(call()[0])
    worst = 0.0
    for _ in range(20):
        worst = max(worst, float(((blocks(call()[0]) - dQ).norm(dim=1) / dQ.norm(dim=1)).max()))
    assert worst <= 2.0 ** -7, worst


def test_packed_single_sequence_equals_unpacked():
    w = W("p_one", 1, 4, 2, 4 + 5 * 256 + 77, 128, 256, 64, 4, seed=55)
    dev = to_dev(workloads.generate(w))
    a = lrsa.Params.from_workload(w)
    b = lrsa.Params.from_workload(w, cu_seqlens=(0, w.N))
    ia, _ = lrsa.lrsa_score_select(a, dev["K"], dev["V"])
    ib, _ = lrsa.lrsa_score_select(b, dev["K"], dev["V"])
    assert torch.equal(ia, ib)
    Oa, La = lrsa.lrsa_attn_fwd(a, dev["Q"], dev["K"], dev["V"], ia)
    Ob, Lb = lrsa.lrsa_attn_fwd(b, dev["Q"], dev["K"], dev["V"], ia)
    assert torch.equal(Oa, Ob) and torch.equal(La, Lb)


@pytest.mark.parametrize("m", [2, 4])
def test_query_chunk_of_several_lag_windows(m):
    """chunk = m * lag: the mask does not depend on how many windows are filled at a time, so the
    results are those of chunk = lag (and match the oracle, which has no chunk parameter)."""
    w = W("c_multi", 1, 4, 2, 4 + 6 * 128 + 50, 128, 128, 32, 4, seed=56)
    host = workloads.generate(w)
    bits = host_bits(host)
    op = oparams(w)
    oidx, _ = orc.score_select(op, bits["K"], bits["V"])
    oO, _ = orc.attn_fwd(op, bits["Q"], bits["K"], bits["V"], oidx)
    dev = to_dev(host)
    p1 = lrsa.Params.from_workload(w)
    pm = lrsa.Params.from_workload(w, chunk=m * w.L)
    i1, _ = lrsa.lrsa_score_select(p1, dev["K"], dev["V"])
    im, _ = lrsa.lrsa_score_select(pm, dev["K"], dev["V"])
    assert torch.equal(i1, im) and np.array_equal(im.cpu().numpy(), oidx)
    O1, L1 = lrsa.lrsa_attn_fwd(p1, dev["Q"], dev["K"], dev["V"], i1)
    Om, Lm = lrsa.lrsa_attn_fwd(pm, dev["Q"], dev["K"], dev["V"], im)
    assert torch.equal(O1, Om) and torch.equal(L1, Lm)
    check_close("O", f64(Om), oO)
    g1 = lrsa.lrsa_attn_bwd(p1, dev["Q"], dev["K"], dev["V"], O1, dev["dO"], L1, i1)
    gm = lrsa.lrsa_attn_bwd(pm, dev["Q"], dev["K"], dev["V"], Om, dev["dO"], Lm, im)
    odQ, odK, odV = orc.attn_bwd(op, bits["Q"], bits["K"], bits["V"], bits["dO"], oidx)
    for name, a, b, ref in zip(("dQ", "dK", "dV"), g1, gm, (odQ, odK, odV)):
        check_close(name, f64(b), ref)
        assert (a.float() - b.float()).abs().max().item() <= 2e-2


def test_expired_wait_is_reported_and_the_next_call_is_clean():
    """The bounded wait of the long-window scoring kernel, made to give up at once through the test hook:
    the call returns, the workspace reports LRSA_ERR_TIMEOUT, and an ordinary call on the same workspace
    afterwards is clean and correct."""
    w = W("s_timeout", 1, 1, 1, 2 + 3 * 4608 + 11, 64, 4608, 100, 2, seed=42)
    host = workloads.generate(w, ("K", "V"))
    dev = to_dev(host)
    p = lrsa.Params.from_workload(w)
    ws = lrsa.new_workspace(lrsa.lrsa_workspace_bytes(p)[0])
    want, _ = lrsa.lrsa_score_select(p, dev["K"], dev["V"], workspace=ws)
    assert lrsa.lrsa_workspace_status(ws) == 0
    lrsa.lrsa_debug_set_wait_limit(-1)
    try:
        lrsa.lrsa_score_select(p, dev["K"], dev["V"], workspace=ws)
        assert lrsa.lrsa_workspace_status(ws) == 5      # LRSA_ERR_TIMEOUT
    finally:
        lrsa.lrsa_debug_set_wait_limit(0)
    again, _ = lrsa.lrsa_score_select(p, dev["K"], dev["V"], workspace=ws)
    assert lrsa.lrsa_workspace_status(ws) == 0
    assert torch.equal(again, want)


def _padded(shape, dtype, fill, pad=4096):
    """A tensor of `shape` carved out of a larger buffer whose margins hold a sentinel."""
    n = int(np.prod(shape))
    buf = torch.full((n + 2 * pad,), fill, dtype=dtype, device="cuda")
    return buf, buf[pad:pad + n].view(shape)


def _margins_intact(buf, n, fill, pad=4096):
    ref = torch.full((pad,), fill, dtype=buf.dtype, device="cuda")
    return torch.equal(buf[:pad], ref) and torch.equal(buf[pad + n:], ref)


@pytest.mark.parametrize("w", [
    W("canary_ragged", 1, 7, 1, 3 + 4 * 200 + 50, 128, 200, 50, 3, seed=61),      # nothing is a tile multiple
    W("canary_d64", 2, 4, 2, 16 + 6 * 128 + 1, 64, 128, 32, 16, seed=62),
], ids=lambda w: w.name)
def test_outputs_never_written_outside_their_tensors(w):
    """Every output tensor sits inside a larger buffer with sentinel margins: after the three calls the
    margins are untouched (a stray store of a ragged tile, a bulk copy of a partial row or a reduction onto a
    wrong row would show) and every element inside has been overwritten."""
    host = workloads.generate(w)
    dev = to_dev(host)
    p = lrsa.Params.from_workload(w)
    wsel = lrsa.lrsa_num_sel_windows(p)
    bf, f32 = torch.bfloat16, torch.float32
    bi, idx = _padded((w.B, w.Hkv, wsel, w.K), torch.int32, -7)
    bs, sc = _padded((w.B, w.Hkv, wsel, w.L), f32, -7.0)
    bO, O = _padded((w.B, w.Hq, w.N, w.d), bf, 777.0)
    bL, LSE = _padded((w.B, w.Hq, w.N), f32, 777.0)
    bQ, dQ = _padded((w.B, w.Hq, w.N, w.d), bf, 777.0)
    bK, dK = _padded((w.B, w.Hkv, w.N, w.d), bf, 777.0)
    bV, dV = _padded((w.B, w.Hkv, w.N, w.d), bf, 777.0)
    lrsa.lrsa_score_select(p, dev["K"], dev["V"], idx=idx, score=sc)
    lrsa.lrsa_attn_fwd(p, dev["Q"], dev["K"], dev["V"], idx, O=O, LSE=LSE)
    lrsa.lrsa_attn_bwd(p, dev["Q"], dev["K"], dev["V"], O, dev["dO"], LSE, idx, dQ=dQ, dK=dK, dV=dV)
    torch.cuda.synchronize()
    for name, buf, t, fill in (("idx", bi, idx, -7), ("score", bs, sc, -7.0), ("O", bO, O, 777.0), ("LSE", bL, LSE, 777.0),
                               ("dQ", bQ, dQ, 777.0), ("dK", bK, dK, 777.0), ("dV", bV, dV, 777.0)):
        assert _margins_intact(buf, t.numel(), fill), f"{name}: a margin was written"
        assert not (t == fill).any(), f"{name}: an element was left unwritten"


@pytest.mark.parametrize("L,K,n_win", [(4096, 1000, 6), (1024, 1024, 5), (333, 1, 9), (8, 3, 40)])
@pytest.mark.parametrize("values", ["normal", "few"])
def test_selection_of_the_returned_scores(L, K, n_win, values):
    """The kept positions are exactly the top_k of the returned scores, equal scores to the lower position: windows whose
    keys need one to four digits of the search ("few": rows from a set of seven, so that most scores tie)."""
    w = W("sel", 2, 2, 2, 5 + n_win * L + 3, 64, L, K, 5, seed=61)
    g = torch.Generator(device="cuda").manual_seed(L + K)
    kv = [torch.randn((w.B, w.Hkv, w.N, w.d), generator=g, device="cuda").bfloat16() for _ in range(2)]
    if values == "few":
        pick = torch.randint(0, 7, (w.N,), generator=g, device="cuda")
        kv = [t[:, :, pick].contiguous() for t in kv]
    p = lrsa.Params.from_workload(w)
    idx, sc = lrsa.lrsa_score_select(p, kv[0], kv[1], want_score=True)
    order = torch.argsort(sc, dim=-1, descending=True, stable=True)[..., :K].sort(-1).values
    base = w.S + torch.arange(n_win - 1, device="cuda").view(1, 1, -1, 1) * L
    assert torch.equal(idx.long(), order + base)
