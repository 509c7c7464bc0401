"""The row walk of the aggregations (agg.cuh) where its layout changes: feature
counts on both sides of every lanes-per-row and features-per-lane choice, rows
that end inside, at and after a 32-edge window, empty rows, a row shared by all
warps of a CTA, and weights with an infinity in a row that no edge names."""
import numpy as np
import pytest
import torch

import oracle
from _helpers import (KAPPA_GAT, TOL_F32, assert_alpha_close, assert_exact_f32, assert_scaled_close,
                      csr_rows, dev, dot_logit_mag, features, gat_logit_mag, host_features, kappa_dot)
from paper_2101_11552_gb300 import graphgen as gg
from paper_2101_11552_gb300 import tfg

pytestmark = pytest.mark.gpu

# degrees around the 32-edge window, runs of empty rows, one hub
DEGREES = [0, 1, 31, 32, 33, 0, 0, 64, 5, 3, 9000, 2, 0, 95, 96, 97] + [3, 0, 7] * 40


def graph(seed, more=0):
    rng = np.random.default_rng(seed)
    deg = np.array(DEGREES + [3, 0, 7] * more)
    n = len(deg)
    dst = np.repeat(np.arange(n), deg)
    src = rng.integers(0, n - 1, size=dst.size)      # the last node is nobody's source
    order = rng.permutation(dst.size)
    return np.ascontiguousarray(np.stack([src[order], dst[order]]).astype(np.int64)), n


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("f", [2, 7, 8, 9, 16, 17, 31, 32, 33, 41, 48, 49, 64, 65, 96, 97, 100, 128,
                               129, 132, 200, 256, 257, 264, 392])
def test_widths(f, dtype):
    ei, n = graph(f)
    rng = np.random.default_rng(1000 + f)
    x = rng.standard_normal((n, f), dtype=np.float32)
    x[-1] = np.inf                                    # reaches no row but its own
    wl = gg.Workload("walk", n, ei, x, x_bf16=gg.bf16_bits_rne(x))
    ew = rng.uniform(-1.5, 1.5, ei.shape[1]).astype(np.float32)
    csr = tfg.tfg_build_csr(dev(ei), n)
    xd = features(wl, dtype)
    finite = host_features(wl, dtype).copy()
    finite[-1] = 0
    for w in (None, ew):
        wd = None if w is None else dev(w).index_select(0, csr.perm)
        for reduce, fn in (("sum", tfg.tfg_aggregate_sum), ("mean", tfg.tfg_aggregate_mean),
                           ("max", tfg.tfg_aggregate_max)):
            got = fn(csr.rowptr, csr.col, xd, wd).cpu().numpy()
            ref, scale = oracle.aggregate(ei, n, finite, reduce, w=w)
            if reduce == "max":
                assert_exact_f32(got, ref, f"max F={f}")
            else:
                assert_scaled_close(got, ref, scale, TOL_F32, f"{reduce} F={f}")
        dinv, w_csr = tfg.tfg_gcn_norm(csr.rowptr, csr.col, csr.perm, n,
                                       None if w is None else dev(np.abs(w)), 1, 1.0,
                                       want_w_csr=w is not None)
        got = tfg.tfg_gcn_aggregate_sum(csr.rowptr, csr.col, dinv, xd, w_csr, 1, 1.0).cpu().numpy()
        ref, scale = oracle.gcn_aggregate(ei, n, finite, None if w is None else np.abs(w), 1, 1.0)
        assert np.isinf(got[-1]).all()
        assert_scaled_close(got[:-1], ref[:-1], scale[:-1], TOL_F32, f"gcn F={f}")
    # dinv is that of the weighted graph, so the weights are read from w_csr
    x0 = dev(finite) if dtype == "f32" else dev(finite.view(np.int16)).view(torch.bfloat16)
    out = tfg.tfg_appnp_propagate(csr.rowptr, csr.col, dinv, x0, 3, 0.1, w_csr, add_self_loops=1).cpu().numpy()
    ref, scale = oracle.appnp(ei, n, finite, 3, 0.1, np.abs(ew), add_self_loops=1)
    assert_scaled_close(out, ref, scale, TOL_F32, f"appnp F={f}")
    dinv, _ = tfg.tfg_gcn_norm(csr.rowptr, csr.col, csr.perm, n, None, 1, 1.0, want_w_csr=False)
    out = tfg.tfg_appnp_propagate(csr.rowptr, csr.col, dinv, x0, 3, 0.1, add_self_loops=1).cpu().numpy()
    ref, scale = oracle.appnp(ei, n, finite, 3, 0.1, add_self_loops=1)
    assert_scaled_close(out, ref, scale, TOL_F32, f"appnp, weights on the fly, F={f}")


# layouts of one slice per lane, several features per lane (one head and many),
# and more than one feature tile; backward where the layout has one
LAYOUTS = [(1, 3), (1, 41), (1, 100), (3, 5), (2, 9), (5, 13), (1, 130), (7, 20), (8, 16), (4, 8),
           (1, 32), (2, 64), (3, 4), (16, 4), (6, 32), (12, 4), (1, 4), (1, 8), (4, 4), (5, 4)]


@pytest.mark.parametrize("more", [0, 1000])     # mean in-degree 72 and 6
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("heads,channels", LAYOUTS)
def test_gat_layouts(heads, channels, dtype, more):
    f = heads * channels
    ei, n = graph(f, more)
    rng = np.random.default_rng(2000 + f)
    x = rng.standard_normal((n, f), dtype=np.float32)
    wl = gg.Workload("walk", n, ei, x, x_bf16=gg.bf16_bits_rne(x))
    a_s, a_d = (0.5 * rng.standard_normal((2, f))).astype(np.float32)
    csr = tfg.tfg_build_csr(dev(ei), n)
    xd, xh = features(wl, dtype), host_features(wl, dtype)
    out, alpha = tfg.tfg_edge_softmax_aggregate(csr.rowptr, csr.col, xd, heads, channels, dev(a_s),
                                                dev(a_d), 0.2, want_alpha=True)
    ref, ref_alpha, scale = oracle.edge_softmax(ei, n, xh, heads, channels, a_s, a_d, 0.2)
    what = f"{dtype} H={heads} C={channels} more={more}"
    assert_scaled_close(out.cpu().numpy(), ref, scale, TOL_F32, "out " + what)
    rowptr, col, perm, _ = oracle.build_csr(ei, n)
    row = csr_rows(rowptr)
    lam = gat_logit_mag(oracle.widen(xh), col, row, heads, channels, a_s, a_d)
    assert_alpha_close(alpha.cpu().numpy(), ref_alpha[perm], lam, row, KAPPA_GAT, "alpha " + what)
    if f > 256 or not (32 % channels == 0 if channels <= 32 else channels % 32 == 0):
        return
    src = tfg.tfg_build_csr_by_source(dev(ei), n)
    g = rng.standard_normal((n, f)).astype(np.float32)
    got = tfg.tfg_edge_softmax_aggregate_backward(csr.rowptr, csr.col, src.rowptr, src.col, xd, heads,
                                                  channels, dev(a_s), dev(a_d), 0.2, out, dev(g))
    want = oracle.edge_softmax_backward(ei, n, xh, heads, channels, a_s, a_d, 0.2, g)
    lam_max = np.zeros((n, heads))
    np.maximum.at(lam_max, row, lam)
    tol = TOL_F32 + KAPPA_GAT * float(np.max(lam + lam_max[row]))
    for name, a, b, sc in zip(("grad_x", "grad_a_src", "grad_a_dst"), got, want[:3], want[3]):
        assert_scaled_close(a.cpu().numpy(), b, sc, tol, f"{name} {what}")


@pytest.mark.parametrize("more", [0, 1000])     # softmax_fast, the walk
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("heads,channels", [(8, 16), (1, 64), (4, 8), (3, 32)])
def test_gat_infinity_in_a_node_without_edges(heads, channels, dtype, more):
    """Slots of a window without an edge hold id 0; node 0 has no edges, so an infinity in
    its features reaches no output but its own gradient's vectors."""
    f = heads * channels
    ei, n = graph(f + 5, more)
    ei = ei[:, (ei != 0).all(0)]
    rng = np.random.default_rng(2500 + f)
    x = rng.standard_normal((n, f)).astype(np.float32)
    a_s, a_d = (dev((0.5 * rng.standard_normal(f)).astype(np.float32)) for _ in range(2))
    g = dev(rng.standard_normal((n, f)).astype(np.float32))
    csr, src = tfg.tfg_build_csr(dev(ei), n), tfg.tfg_build_csr_by_source(dev(ei), n)
    got = []
    for first in (0.0, np.inf):
        x[0] = first
        xd = dev(x).to(torch.bfloat16 if dtype == "bf16" else torch.float32)
        out, alpha = tfg.tfg_edge_softmax_aggregate(csr.rowptr, csr.col, xd, heads, channels, a_s, a_d, 0.2,
                                                    want_alpha=True)
        gx, _, _ = tfg.tfg_edge_softmax_aggregate_backward(csr.rowptr, csr.col, src.rowptr, src.col, xd, heads,
                                                           channels, a_s, a_d, 0.2, out, g)
        got.append((out, alpha, gx))
    for name, a, b in zip(("out", "alpha", "grad_x"), *got):
        assert torch.isfinite(a).all() and torch.equal(a, b), name


@pytest.mark.parametrize("more", [0, 1000])     # mean in-degree 72 and 6
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("heads,channels", [(1, 8), (4, 8), (5, 8), (2, 16), (8, 16), (3, 32), (2, 64),
                                            (1, 128), (1, 256), (16, 16)])
def test_dot_layouts(heads, channels, dtype, more):
    f = heads * channels
    ei, n = graph(f + 1, more)
    rng = np.random.default_rng(3000 + f)
    wls = [gg.Workload("walk", n, ei, x, x_bf16=gg.bf16_bits_rne(x))
           for x in rng.standard_normal((3, n, f), dtype=np.float32)]
    (q, k, v), (qh, kh, vh) = ([features(w, dtype) for w in wls], [host_features(w, dtype) for w in wls])
    scale = float(np.float32(1.0 / np.sqrt(channels)))
    csr = tfg.tfg_build_csr(dev(ei), n)
    out, alpha = tfg.tfg_dot_edge_softmax_aggregate(csr.rowptr, csr.col, q, k, v, heads, channels, scale,
                                                    want_alpha=True)
    ref, ref_alpha, sc = oracle.dot_softmax(ei, n, qh, kh, vh, heads, channels, scale)
    what = f"{dtype} H={heads} C={channels} more={more}"
    assert_scaled_close(out.cpu().numpy(), ref, sc, TOL_F32, "out " + what)
    rowptr, col, perm, _ = oracle.build_csr(ei, n)
    row = csr_rows(rowptr)
    lam = dot_logit_mag(oracle.widen(qh), oracle.widen(kh), col, row, heads, channels, scale)
    assert_alpha_close(alpha.cpu().numpy(), ref_alpha[perm], lam, row, kappa_dot(channels), "alpha " + what)
    if not (32 % channels == 0 if channels <= 32 else channels % 32 == 0):
        return
    src = tfg.tfg_build_csr_by_source(dev(ei), n)
    g = rng.standard_normal((n, f)).astype(np.float32)
    got = tfg.tfg_dot_edge_softmax_aggregate_backward(csr.rowptr, csr.col, src.rowptr, src.col, q, k, v,
                                                      heads, channels, scale, out, dev(g))
    want = oracle.dot_softmax_backward(ei, n, qh, kh, vh, heads, channels, scale, g)
    lam_max = np.zeros((n, heads))
    np.maximum.at(lam_max, row, lam)
    tol = TOL_F32 + kappa_dot(channels) * float(np.max(lam + lam_max[row]))
    for name, a, b, s in zip(("grad_q", "grad_k", "grad_v"), got, want[:3], want[3]):
        assert_scaled_close(a.cpu().numpy(), b, s, tol, f"{name} {what}")


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("f", [3, 8, 16, 24, 40, 41, 64, 72, 100, 128, 136, 256, 264])
def test_max_argmax_widths(f, dtype):
    """Argmax where the layout changes, weighted and not, with values that tie."""
    ei, n = graph(f + 2, 300)
    rng = np.random.default_rng(4000 + f)
    x = np.round(rng.standard_normal((n, f), dtype=np.float32) * 4) / 4
    wl = gg.Workload("walk", n, ei, x, x_bf16=gg.bf16_bits_rne(x))
    csr = tfg.tfg_build_csr(dev(ei), n)
    for ew in (None, rng.uniform(-1.5, 1.5, ei.shape[1]).astype(np.float32)):
        w = None if ew is None else dev(ew).index_select(0, csr.perm)
        out, arg = tfg.tfg_aggregate_max_argmax(csr, features(wl, dtype), w)
        ref, ref_arg = oracle.max_argmax(ei, n, host_features(wl, dtype), ew)
        assert np.array_equal(arg.cpu().numpy(), ref_arg), f"argmax F={f}"
        assert_exact_f32(out.cpu().numpy(), ref, f"max F={f}")


@pytest.mark.parametrize("f", [8, 64, 72, 128, 136, 264])
def test_plain_bf16_max_of_special_values(f):
    """The packed bf16 max passes over NaN and knows the infinities, as the fp32 kernel
    does on the same values: rows of one value, of NaN only, of -infinity only, a NaN first,
    last and between, signed zeros, the largest and smallest finite values."""
    ei, n = graph(f + 3, 300)
    rng = np.random.default_rng(4500 + f)
    special = np.array([np.nan, np.inf, -np.inf, 0.0, -0.0, 3.3895e38, -3.3895e38, 1.0, -2.0], np.float32)
    x = rng.choice(special, size=(n, f), p=[.4, .05, .25, .05, .05, .05, .05, .05, .05])
    x[:, :2] = np.nan                                  # NaN only
    x[:, 2:4] = -np.inf
    xb = torch.from_numpy(x).cuda().to(torch.bfloat16)
    csr = tfg.tfg_build_csr(dev(ei), n)
    got = tfg.tfg_aggregate_max(csr.rowptr, csr.col, xb)
    assert torch.equal(got, tfg.tfg_aggregate_max(csr.rowptr, csr.col, xb.float()))
    seen = np.where(np.isnan(x), -np.inf, xb.float().cpu().numpy())
    ref, _ = oracle.aggregate(ei, n, seen.astype(np.float32), "max")
    assert_exact_f32(got.cpu().numpy(), ref, f"max F={f}")


@pytest.mark.parametrize("f", [33, 64, 65, 97, 128, 129, 132, 264])
def test_max_backward_walk_widths(f):
    """The backward's row walk where its lanes and feature tiles change, weighted and not,
    with a source of 9,000 edges that the warps of a CTA share and sources of none."""
    ei, n = graph(f + 4, 1000)
    ei = np.ascontiguousarray(ei[::-1])                # the degrees are the sources'
    rng = np.random.default_rng(4700 + f)
    x = np.round(rng.standard_normal((n, f), dtype=np.float32) * 4) / 4
    g = rng.standard_normal((n, f)).astype(np.float32)
    csr, src = tfg.tfg_build_csr(dev(ei), n), tfg.tfg_build_csr_by_source(dev(ei), n)
    for ew in (None, rng.uniform(-1.5, 1.5, ei.shape[1]).astype(np.float32)):
        w = None if ew is None else dev(ew).index_select(0, csr.perm)
        _, arg = tfg.tfg_aggregate_max_argmax(csr, dev(x), w)
        got = tfg.tfg_aggregate_max_backward(src, arg, dev(g), None if ew is None else dev(ew))
        ref, scale = oracle.max_backward(ei, n, arg.cpu().numpy(), g, ew)
        assert_scaled_close(got.cpu().numpy(), ref, scale, TOL_F32, f"max backward F={f}")


def test_max_argmax_of_a_row_past_16_bit_positions():
    """A target of 3,000,000 edges: each warp's share exceeds the 65,000 edges that
    16-bit positions cover; the maximum sits first, last and twice in the row."""
    n, e, f = 40, 3_000_000, 24
    rng = np.random.default_rng(5)
    ei = np.stack([rng.integers(8, n, size=e), np.zeros(e, np.int64)])
    ei[0, [0, e // 3, e - 1]] = [1, 2, 3]
    x = rng.standard_normal((n, f), dtype=np.float32)
    x[1, :6], x[2, 4:12], x[3, 8:18] = 9.0, 9.0, 9.0
    wl = gg.Workload("star", n, ei, x, x_bf16=gg.bf16_bits_rne(x))
    csr = tfg.tfg_build_csr(dev(ei), n)
    out, arg = tfg.tfg_aggregate_max_argmax(csr, features(wl, "bf16"))
    ref, ref_arg = oracle.max_argmax(ei, n, host_features(wl, "bf16"), None)
    assert np.array_equal(arg.cpu().numpy(), ref_arg)
    assert_exact_f32(out.cpu().numpy(), ref)


@pytest.mark.parametrize("offset", [0, 4, 8])   # floats before grad_out: 32-byte aligned, 16, 32
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("heads,channels", [(4, 8), (5, 8), (8, 8), (3, 16), (8, 16), (1, 64), (1, 128)])
def test_gradient_slices_of_32_bytes(heads, channels, dtype, offset):
    """Backward by source of both attentions on rows of mean degree 206, with
    gradients that 32-byte loads may and may not read."""
    f = heads * channels
    rng = np.random.default_rng(6000 + f)
    deg = np.array(DEGREES[:16] + [3, 0, 7] * 10)
    n = len(deg)
    ei = np.stack([np.repeat(np.arange(n), deg), rng.integers(0, n, size=deg.sum())]).astype(np.int64)
    wls = [gg.Workload("walk", n, ei, x, x_bf16=gg.bf16_bits_rne(x))
           for x in rng.standard_normal((3, n, f), dtype=np.float32)]
    (q, k, v), (qh, kh, vh) = ([features(w, dtype) for w in wls], [host_features(w, dtype) for w in wls])
    a_s, a_d = (0.5 * rng.standard_normal((2, f))).astype(np.float32)
    g = rng.standard_normal((n, f)).astype(np.float32)
    gd = torch.empty(offset + n * f, device="cuda")[offset:].view(n, f)
    gd.copy_(dev(g))
    csr, src = tfg.tfg_build_csr(dev(ei), n), tfg.tfg_build_csr_by_source(dev(ei), n)
    rowptr, col, _, _ = oracle.build_csr(ei, n)
    row = csr_rows(rowptr)

    def check(names, got, want, lam, kappa):
        lam_max = np.zeros((n, heads))
        np.maximum.at(lam_max, row, lam)
        tol = TOL_F32 + kappa * float(np.max(lam + lam_max[row]))
        for name, a, b, s in zip(names, got, want[:3], want[3]):
            assert_scaled_close(a.cpu().numpy(), b, s, tol, f"{name} {dtype} H={heads} C={channels}")

    out, _ = tfg.tfg_edge_softmax_aggregate(csr.rowptr, csr.col, q, heads, channels, dev(a_s), dev(a_d), 0.2,
                                            want_alpha=True)
    got = tfg.tfg_edge_softmax_aggregate_backward(csr.rowptr, csr.col, src.rowptr, src.col, q, heads,
                                                  channels, dev(a_s), dev(a_d), 0.2, out, gd)
    check(("grad_x", "grad_a_src", "grad_a_dst"), got,
          oracle.edge_softmax_backward(ei, n, qh, heads, channels, a_s, a_d, 0.2, g),
          gat_logit_mag(oracle.widen(qh), col, row, heads, channels, a_s, a_d), KAPPA_GAT)
    scale = float(np.float32(1.0 / np.sqrt(channels)))
    out, _ = tfg.tfg_dot_edge_softmax_aggregate(csr.rowptr, csr.col, q, k, v, heads, channels, scale,
                                                want_alpha=True)
    got = tfg.tfg_dot_edge_softmax_aggregate_backward(csr.rowptr, csr.col, src.rowptr, src.col, q, k, v,
                                                      heads, channels, scale, out, gd)
    check(("grad_q", "grad_k", "grad_v"), got,
          oracle.dot_softmax_backward(ei, n, qh, kh, vh, heads, channels, scale, g),
          dot_logit_mag(oracle.widen(qh), oracle.widen(kh), col, row, heads, channels, scale), kappa_dot(channels))


# One row of 32 edges: 2^24, then 31 ones.  A one added to 2^24 in fp32 is lost (half a
# unit in the last place, ties to even), so one chain over a 32-edge window ends 31 short.
# With a second lane group or a second chain at most 15 ones meet the large term and the
# two sums' own addition rounds by at most 1: |error| <= 16.  Rows of 17 and more slices
# have one lane group.  Enough rows that windows begin at every place in a row.
BIG, CHAIN_BOUND = 2.0 ** 24, 16.0


def chain_graph(rows):
    src = np.ones((rows, 32), np.int64) + rows        # node rows: the large term, rows + 1: one
    src[:, 0] = rows
    return np.stack([src.reshape(-1), np.repeat(np.arange(rows), 32)]), rows + 2


def chain_values(n, f, dtype):
    x = torch.ones(n, f, device="cuda")
    x[n - 2] = BIG
    return x.to(torch.bfloat16 if dtype == "bf16" else torch.float32)


def assert_short_chains(got, want, bound, what):
    worst = float((got.double() - want).abs().max())
    assert worst <= bound, f"{what}: {worst} > {bound}"


@pytest.mark.parametrize("f,dtype", [(68, "f32"), (100, "f32"), (124, "f32"), (136, "bf16"), (200, "bf16"),
                                     (248, "bf16")])
def test_sums_of_17_to_31_slices_keep_two_chains(f, dtype):
    rows = 20000
    ei, n = chain_graph(rows)
    csr = tfg.tfg_build_csr(dev(ei), n)
    x = chain_values(n, f, dtype)
    assert_short_chains(tfg.tfg_aggregate_sum(csr.rowptr, csr.col, x)[:rows], BIG + 31, CHAIN_BOUND, "sum")
    one = torch.ones(n, device="cuda")                # dinv: the edges' weights and the row's factor
    gcn = tfg.tfg_gcn_aggregate_sum(csr.rowptr, csr.col, one, x, None, 0, 1.0)[:rows]
    assert_short_chains(gcn, BIG + 31, CHAIN_BOUND, "gcn")
    hop = tfg.tfg_sgc_propagate(csr.rowptr, csr.col, one, x, 1)[:rows]
    assert_short_chains(hop, BIG + 31, CHAIN_BOUND, "hop")


@pytest.mark.parametrize("heads,channels,dtype", [(8, 16, "f32"), (4, 32, "f32"), (1, 128, "f32"), (4, 64, "bf16"),
                                                  (2, 128, "f32")])
def test_gat_over_32_slices_keeps_two_chains(heads, channels, dtype):
    f = heads * channels
    ei, n = chain_graph(20000)
    csr = tfg.tfg_build_csr(dev(ei), n)
    zero = torch.zeros(f, device="cuda")
    out, _ = tfg.tfg_edge_softmax_aggregate(csr.rowptr, csr.col, chain_values(n, f, dtype), heads, channels, zero,
                                            zero, 0.2)
    assert_short_chains(out[:n - 2], (BIG + 31) / 32, CHAIN_BOUND / 32, "gat")


@pytest.mark.parametrize("heads,channels,dtype", [(3, 32, "f32"), (5, 16, "f32"), (7, 16, "f32"), (1, 100, "f32"),
                                                  (3, 64, "bf16"), (5, 32, "bf16")])
def test_attention_over_17_to_31_slices_keeps_two_chains(heads, channels, dtype):
    f = heads * channels
    ei, n = chain_graph(20000)
    rows = n - 2
    csr = tfg.tfg_build_csr(dev(ei), n)
    x, zero = chain_values(n, f, dtype), torch.zeros(f, device="cuda")
    # equal logits: every weight is 1 / 32, and the division is exact
    out, _ = tfg.tfg_edge_softmax_aggregate(csr.rowptr, csr.col, x, heads, channels, zero, zero, 0.2)
    assert_short_chains(out[:rows], (BIG + 31) / 32, CHAIN_BOUND / 32, "gat")
    if channels & (channels - 1):
        return
    none = torch.zeros_like(x)
    out, _ = tfg.tfg_dot_edge_softmax_aggregate(csr.rowptr, csr.col, none, none, x, heads, channels, 1.0)
    assert_short_chains(out[:rows], (BIG + 31) / 32, CHAIN_BOUND / 32, "dot")
    # by target: dalpha = 0 and beta = -1, so grad_q = sum of k / 32
    src = tfg.tfg_build_csr_by_source(dev(ei), n)
    g = torch.zeros(n, heads, channels, device="cuda")
    g[:, :, 0] = 1
    g = g.view(n, f)
    gq, _, _ = tfg.tfg_dot_edge_softmax_aggregate_backward(csr.rowptr, csr.col, src.rowptr, src.col, none, x, none,
                                                           heads, channels, 1.0, -g, g)
    assert_short_chains(gq[:rows], (BIG + 31) / 32, CHAIN_BOUND / 32, "grad_q")
    # by source: 32 out-edges, each the only in-edge of its target, so alpha = 1
    rows = 4000
    n = 33 * rows
    ei = np.stack([np.tile(np.arange(rows), 32), np.arange(rows, n)])
    csr, src = tfg.tfg_build_csr(dev(ei), n), tfg.tfg_build_csr_by_source(dev(ei), n)
    none = torch.zeros(n, f, device="cuda", dtype=x.dtype)
    g = torch.ones(n, f, device="cuda")
    g[rows:2 * rows] = BIG
    _, _, gv = tfg.tfg_dot_edge_softmax_aggregate_backward(csr.rowptr, csr.col, src.rowptr, src.col, none, none, none,
                                                           heads, channels, 1.0, none.float(), g)
    assert_short_chains(gv[:rows], BIG + 31, CHAIN_BOUND, "grad_v")
