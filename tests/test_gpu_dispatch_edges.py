"""Every branch that the dispatch on sizes and alignment can take, at the sizes where its kernel can go wrong: block-tiled forward and
reverse pass, two-CTA clusters of the fused MLP forward, narrow state accesses, streamed decode."""
import numpy as np
import pytest
import torch

from paper_2608_21308_b200 import binding as E
from paper_2608_21308_b200 import inputs
from tests import util
from tests.test_gpu_apply import gpu_apply, oracle_apply
from tests.test_gpu_normed import gpu_backward_normed, gpu_forward_normed, oracle_bwd, oracle_fwd, targets
from tests.test_gpu_parity import TOL_BF16, check_backward, check_forward

pytestmark = pytest.mark.gpu
MLP, SWIGLU = inputs.KIND_MLP, inputs.KIND_SWIGLU


def _inputs(N, L, d, h, C, kind, **kw):
    r = inputs.paper_regime(inputs.Recipe(B=N, H=1, L=L, d=d, h=h, C=C, kind=kind, io="bf16", seed=31, m_std=0.002))
    return inputs.generate(r, **kw), dict(d=d, h=h, C=C, kind=kind, io="bf16")


def check_fp32(got, ref, what):
    """What is returned in fp32.  Every product takes both operands as two bf16 terms (2^-17 of a value is left over); over the few chunks
    here that comes to 1e-4 at most, where an operand without its second term is off by 2^-9 and shows as 4e-3."""
    errs = {}
    for n in ("W", "M", "dW", "dM", "drow_norm", "deta", "dbeta", "dgamma"):
        if n in got:
            pairs = zip(got[n], ref[n]) if isinstance(got[n], list) else [(got[n], ref[n])]
            errs.update({f"{n}{i}": util.rel_l2(a, b) for i, (a, b) in enumerate(pairs)})
    assert all(e <= 1e-3 for e in errs.values()), f"{what}: {errs}"


@pytest.mark.parametrize("normed", [False, True], ids=["plain", "normed"])
@pytest.mark.parametrize("kind", [MLP, SWIGLU])
@pytest.mark.parametrize("d,h,C,L", [
    (8, 64, 24, 30),      # one block in every direction
    (64, 72, 64, 65),     # a hidden block of 8 units; a chunk of one token
    (72, 640, 65, 66),    # five CTAs in the reverse chain; two token blocks, the second of one token
    (128, 1024, 16, 20),  # the most CTAs the chain takes
    (128, 1088, 16, 20),  # more hidden units than it takes
    (128, 136, 512, 520), # the longest chunks
])
def test_block_tiled_edges(d, h, C, L, kind, normed):
    x, shape = _inputs(1, L, d, h, C, kind, with_d_o=True, with_dstate=True)
    if normed:
        tgt = targets(x)
        got = gpu_forward_normed(x, tgt, impl=E.E2TTT_IMPL_TILED, **shape)
        ref = oracle_fwd(x, tgt, C, kind)
        check_forward(got, ref, TOL_BF16, "block-tiled normed forward")
        check_fp32(got, ref, "block-tiled normed forward")
        got = gpu_backward_normed(x, tgt, impl=E.E2TTT_IMPL_TILED, via_saved_states=True, **shape)
        ref = oracle_bwd(x, tgt, C, kind)
        check_backward(got, ref, 2 * TOL_BF16, "block-tiled normed backward")
        check_fp32(got, ref, "block-tiled normed backward")
    else:
        got, hd = util.gpu_forward(x, impl=E.E2TTT_IMPL_TILED, **shape)
        assert E.e2ttt_device_status(hd["ws"]) == 0
        ref = util.oracle_forward(x, C, kind)
        check_forward(got, ref, TOL_BF16, "block-tiled forward")
        check_fp32(got, ref, "block-tiled forward")
        got, ref = util.gpu_backward(x, impl=E.E2TTT_IMPL_TILED, **shape), util.oracle_backward(x, C, kind)
        check_backward(got, ref, 2 * TOL_BF16, "block-tiled backward")
        check_fp32(got, ref, "block-tiled backward")


@pytest.mark.parametrize("N,ckpt", [(1, 0), (1, 5), (40, 0), (40, 5)])
def test_block_tiled_reverse_over_groups_of_chunks(N, ckpt):
    """23 chunks: groups of 9 of them per launch (of 3 or 4 with 40 sequences), the last shorter; segments of an odd number of chunks."""
    x, shape = _inputs(N, 23 * 16 - 3, 64, 192, 16, MLP, with_d_o=True, with_dstate=True)
    got = util.gpu_backward(x, impl=E.E2TTT_IMPL_TILED, via_saved_states=ckpt > 0, ckpt_every=ckpt, **shape)
    ref = util.gpu_backward(x, impl=E.E2TTT_IMPL_SIMT, **shape)
    check_backward(got, ref, TOL_BF16, f"groups N={N} ckpt={ckpt}")
    check_fp32(got, ref, f"groups N={N} ckpt={ckpt}")


@pytest.mark.parametrize("kind", [MLP, SWIGLU])
@pytest.mark.parametrize("d,h", [(64, 192), (128, 1088)], ids=["chain", "wide"])
@pytest.mark.parametrize("how", ["plain", "checkpoints", "normed"])
def test_both_reverse_chains_pass_their_state_from_group_to_group(how, d, h, kind):
    """11 chunks, groups of 9 at most: the adjoints of the state, those of the row targets (summed over all chunks) and dk's last shares go from
    one launch to the next, for up to 1024 hidden units and for more; with checkpoints the launches are segments of 4 chunks."""
    x, shape = _inputs(1, 11 * 16 - 3, d, h, 16, kind, with_d_o=True, with_dstate=True)
    if how == "normed":
        tgt = targets(x)
        got, ref = (gpu_backward_normed(x, tgt, impl=i, via_saved_states=True, **shape) for i in (E.E2TTT_IMPL_TILED, E.E2TTT_IMPL_SIMT))
    else:
        ckpt = 4 if how == "checkpoints" else 0
        got, ref = (util.gpu_backward(x, impl=i, via_saved_states=True, ckpt_every=ckpt, **shape) for i in (E.E2TTT_IMPL_TILED, E.E2TTT_IMPL_SIMT))
    check_backward(got, ref, TOL_BF16, how)
    check_fp32(got, ref, how)


@pytest.mark.parametrize("normed", [False, True], ids=["plain", "normed"])
@pytest.mark.parametrize("N,d,h,C,L", [(34, 64, 256, 64, 130), (74, 128, 256, 16, 50), (75, 64, 128, 32, 64), (34, 128, 128, 128, 300)])
def test_two_cta_clusters_of_the_fused_forward(N, d, h, C, L, normed):
    """Copies of two sequences: all copies equal, the first two against the oracle."""
    if normed and C > 64:
        pytest.skip("normalised chunks of several blocks run on the block-tiled kernels")
    x, shape = _inputs(2, L, d, h, C, MLP)
    rep = lambda a: np.concatenate([a] * ((N + 1) // 2))[:N]
    xs = {n: [rep(w) for w in a] if isinstance(a, list) else rep(a) for n, a in x.items()}
    if normed:
        got = gpu_forward_normed(xs, targets(xs), impl=E.E2TTT_IMPL_TCGEN05, **shape)
        ref = oracle_fwd(x, targets(x), C, MLP)
    else:
        got, hd = util.gpu_forward(xs, impl=E.E2TTT_IMPL_TCGEN05, **shape)
        assert E.e2ttt_device_status(hd["ws"]) == 0
        ref = util.oracle_forward(x, C, MLP)
    cut = lambda a: [w[:2] for w in a] if isinstance(a, list) else a[:2]
    for a in [got["o"]] + got["W"] + got["M"]:
        assert all(np.array_equal(a[n], a[n % 2]) for n in range(N))
    check_forward({n: cut(a) for n, a in got.items()}, ref, TOL_BF16, "two-CTA clusters")


@pytest.mark.parametrize("kind,h", [(MLP, 512), (SWIGLU, 384)])
def test_states_off_the_32_byte_grid_give_the_same_result(kind, h):
    x, shape = _inputs(2, 100, 128, h, 64, kind)
    ref, _ = util.gpu_forward(x, impl=E.E2TTT_IMPL_TCGEN05, **shape)
    p = E.make_params(2, 1, 100, 128, h, 64, kind, E.E2TTT_BF16, 1e-5, E.E2TTT_IMPL_TCGEN05)
    dev = lambda a, t=torch.float32: torch.tensor(a, dtype=torch.float32).to(t).cuda()
    q, k, v = (dev(x[n], torch.bfloat16).view(2, 1, 100, 128) for n in ("q", "k", "v"))
    gates = [dev(x[n]).view(2, 1, 100) for n in ("eta", "beta", "gamma")]

    def off16(a):  # a copy 16 bytes past a 32-byte boundary
        t = torch.empty(a.size + 4, dtype=torch.float32, device="cuda")[4:].view((2, 1) + a.shape[1:])
        t.copy_(dev(a).view(t.shape))
        return t

    W, M = [off16(w) for w in x["W"]], [off16(m) for m in x["M"]]
    Wf, Mf = [off16(w) for w in x["W"]], [off16(m) for m in x["M"]]
    o = torch.empty_like(q)
    ws = torch.empty(E.e2ttt_workspace_bytes(p, 0), dtype=torch.uint8, device="cuda")
    E.e2ttt_chunk_fwd(p, q, k, v, *gates, W, M, o, Wf, Mf, ws, 0)
    torch.cuda.synchronize()
    assert np.array_equal(o.float().cpu().numpy()[:, 0], ref["o"])
    for a, b in zip(Wf + Mf, ref["W"] + ref["M"]):
        assert np.array_equal(a.cpu().numpy()[:, 0], b)


@pytest.mark.parametrize("kind", [MLP, SWIGLU])
@pytest.mark.parametrize("io", ["f32", "bf16"])
@pytest.mark.parametrize("d,h,N", [(4, 4, 1), (8, 260, 3), (132, 256, 2), (256, 4096, 1), (256, 4100, 1), (128, 510, 2), (260, 64, 1), (64, 256, 300)])
def test_one_token_decode(kind, io, d, h, N):
    """Rows of less than a piece and of several, the widest that is streamed, and neighbours that are not."""
    r = inputs.Recipe(B=N, H=1, L=1, d=d, h=h, C=1, kind=kind, io=io, seed=22, w_std=0.05)
    x = inputs.generate(r)
    got = gpu_apply(x["q"], x["W"], d=d, h=h, kind=kind, io=io)
    assert util.rel_err(got, oracle_apply(x["q"], x["W"], kind)) <= (1e-5 if io == "f32" else TOL_BF16)


@pytest.mark.parametrize("io", ["f32", "bf16"])
@pytest.mark.parametrize("T", [1, 3, 9])
def test_decode_with_ctas_that_own_no_hidden_unit(T, io):
    """Four hidden units in a cluster of eight: seven CTAs do nothing but store their zero partial sums."""
    r = inputs.Recipe(B=3, H=1, L=T, d=4, h=4, C=T, kind=MLP, io=io, seed=23, w_std=0.5)
    x = inputs.generate(r)
    for _ in range(20):
        got = gpu_apply(x["q"], x["W"], d=4, h=4, kind=MLP, io=io)
        assert util.rel_err(got, oracle_apply(x["q"], x["W"], MLP)) <= (1e-5 if io == "f32" else TOL_BF16)


@pytest.mark.parametrize("N,d,h,C,L", [
    (15, 64, 64, 129, 260), (16, 64, 64, 129, 260), (2, 72, 72, 129, 260),    # forward: 64 hidden units or more, 15 sequences or more
    (33, 64, 64, 385, 400), (34, 64, 64, 385, 400),                           # forward: clusters of 4 that fit together, and not
    (75, 64, 64, 4, 10), (149, 96, 128, 16, 20), (149, 64, 200, 16, 20),      # forward: many sequences of short chunks
    (8, 64, 128, 257, 520), (9, 64, 128, 257, 520), (15, 48, 64, 385, 400),   # reverse pass: 8 and 15 sequences
    (19, 16, 32, 193, 200),                                                   # reverse pass: small states
])
def test_few_hidden_units_or_tokens(N, d, h, C, L):
    """Either side of the lines between the block-tiled kernels and the others, on copies of two sequences.  Forward and reverse pass
    need not be on the same side, nor the reverse pass of a checkpointed call and the forward that saved its states."""
    x, shape = _inputs(2, L, d, h, C, MLP, with_d_o=True, with_dstate=True)
    rep = lambda a: np.concatenate([a] * ((N + 1) // 2))[:N]
    xs = {n: [rep(w) for w in a] if isinstance(a, list) else rep(a) for n, a in x.items()}
    cut = lambda a: [w[:2] for w in a] if isinstance(a, list) else a[:2]
    got, hd = util.gpu_forward(xs, impl=E.E2TTT_IMPL_TILED, **shape)
    assert E.e2ttt_device_status(hd["ws"]) == 0
    check_forward({n: cut(a) for n, a in got.items()}, util.oracle_forward(x, C, MLP), TOL_BF16, "forward")
    ref = util.oracle_backward(x, C, MLP)
    plans = [util.gpu_backward(xs, impl=E.E2TTT_IMPL_TILED, via_saved_states=saved, ckpt_every=ckpt, **shape)
             for saved, ckpt in ((True, 0), (True, 2), (False, 0), (False, 2))]
    check_backward({n: cut(a) for n, a in plans[0].items()}, ref, 2 * TOL_BF16, "backward")
    for got in plans[1:]:  # every memory plan: the same bits
        for n, a in got.items():
            assert all(np.array_equal(v, w) for v, w in (zip(a, plans[0][n]) if isinstance(a, list) else [(a, plans[0][n])])), n


@pytest.mark.parametrize("saved", [True, False], ids=["saved", "recomputed"])
@pytest.mark.parametrize("d,h,C,L", [(64, 64, 129, 260), (64, 128, 257, 520), (48, 64, 400, 450)], ids=["forward", "reverse", "both"])
def test_normed_calls_off_the_block_tiled_kernels(d, h, C, L, saved):
    """Forward, reverse pass or both on the other kernels: the row norms and the states pass from one kind to the other."""
    x, shape = _inputs(2, L, d, h, C, MLP, with_d_o=True, with_dstate=True)
    tgt = targets(x)
    got, ref = gpu_forward_normed(x, tgt, impl=E.E2TTT_IMPL_TILED, **shape), oracle_fwd(x, tgt, C, MLP)
    check_forward(got, ref, TOL_BF16, "normed forward")
    check_fp32(got, ref, "normed forward")
    got, ref = gpu_backward_normed(x, tgt, impl=E.E2TTT_IMPL_TILED, via_saved_states=saved, **shape), oracle_bwd(x, tgt, C, MLP)
    check_backward(got, ref, 2 * TOL_BF16, "normed backward")
    check_fp32(got, ref, "normed backward")


@pytest.mark.parametrize("kind,N,h,C,L", [(SWIGLU, 2, 384, 128, 200), (MLP, 2, 512, 96, 100), (SWIGLU, 2, 384, 256, 256)])
def test_noalloc_forward_where_the_block_tiled_layout_does_not_fit(kind, N, h, C, L):
    """The last one fits neither layout and is refused.  The others run on the kernels for wider heads: the same two-term products and fp32
    sums in another order.  A product's operands are off by 2^-17 each at most, so both sides are within a few 1e-5 of the exact result;
    1e-4 leaves room for the amplification over two chunks.  A lost term of an operand would show as 4e-3."""
    x, shape = _inputs(N, L, 128, h, C, kind)
    ref, hd = util.gpu_forward(x, impl=E.E2TTT_IMPL_AUTO, **shape)
    p = hd["p"]
    assert E.e2ttt_workspace_bytes(p, 0) > E.E2TTT_NOALLOC_SCRATCH_BYTES
    o = torch.empty_like(hd["q"])
    Wf, Mf = [torch.empty_like(w) for w in hd["W"]], [torch.empty_like(w) for w in hd["W"]]
    args = (p, hd["q"], hd["k"], hd["v"], hd["eta"], hd["beta"], hd["gamma"], hd["W"], hd["M"], o, Wf, Mf)
    simt = E.make_params(N, 1, L, 128, h, C, kind, E.E2TTT_BF16, 1e-5, E.E2TTT_IMPL_SIMT)
    if E.e2ttt_workspace_bytes(simt, 0) > E.E2TTT_NOALLOC_SCRATCH_BYTES:
        with pytest.raises(E.E2TTTError) as ei:
            E.e2ttt_chunk_fwd_noalloc(*args)
        assert ei.value.status == -5
        return
    E.e2ttt_chunk_fwd_noalloc(*args)
    assert E.e2ttt_device_status(None) == 0
    for a, b in zip(Wf + Mf, ref["W"] + ref["M"]):
        assert util.rel_l2(a.cpu().numpy()[:, 0], b) <= 1e-4
    assert util.rel_l2(o.float().cpu().numpy()[:, 0], ref["o"]) <= 1e-3  # bf16: a few values round to the other neighbour


@pytest.mark.parametrize("kind", [MLP, SWIGLU])
@pytest.mark.parametrize("N,d,h,C,L", [
    (1, 72, 840, 65, 131), (15, 128, 1088, 128, 257),   # two blocks of tokens, the second of one token and full; a chunk of one token
    (2, 128, 1600, 130, 261), (1, 64, 2112, 200, 450),  # three and four blocks, the last ones ragged
])
def test_wide_networks_on_clusters_with_several_blocks_of_tokens(N, d, h, C, L, kind):
    """Few sequences of wide networks stay off the work items; their chunks have several blocks of tokens.  Plain, with saved states, normalised."""
    U = min(N, 2)
    x, shape = _inputs(U, L, d, h, C, kind)
    rep = lambda a: np.concatenate([a] * ((N + U - 1) // U))[:N]
    xs = {n: [rep(w) for w in a] if isinstance(a, list) else rep(a) for n, a in x.items() if a is not None}
    cut = lambda got: {n: [w[:U] for w in a] if isinstance(a, list) else a[:U] for n, a in got.items()}
    got, hd = util.gpu_forward(xs, impl=E.E2TTT_IMPL_TILED, **shape)
    assert E.e2ttt_device_status(hd["ws"]) == 0
    ref = util.oracle_forward(x, C, kind)
    check_forward(cut(got), ref, TOL_BF16, "forward on clusters")
    check_fp32(cut(got), ref, "forward on clusters")
    saved, _ = util.gpu_forward(xs, impl=E.E2TTT_IMPL_TILED, save_states=True, **shape)
    assert all(np.array_equal(a, b) for a, b in zip([got["o"], *got["W"], *got["M"]], [saved["o"], *saved["W"], *saved["M"]]))
    tgt = targets(x)
    got, ref = gpu_forward_normed(xs, [rep(t) for t in tgt], impl=E.E2TTT_IMPL_TILED, **shape), oracle_fwd(x, tgt, C, kind)
    check_forward(cut(got), ref, TOL_BF16, "normed forward on clusters")
    check_fp32(cut(got), ref, "normed forward on clusters")


# (The ids and comments of test_few_hidden_units_or_tokens name lines of the forward as they were before it ran on work items: of its rows the
# forwards are all block-tiled now, the reverse passes on either side.)
@pytest.mark.parametrize("normed", [False, True], ids=["plain", "normed"])
@pytest.mark.parametrize("N,d,h,C", [(79, 64, 64, 4), (80, 64, 64, 4), (148, 64, 64, 4), (148, 64, 64, 5), (149, 64, 64, 4), (228, 64, 64, 4), (229, 64, 64, 4), (100, 64, 72, 4),
                                     (101, 64, 72, 4), (148, 8, 512, 1), (122, 128, 64, 4), (123, 128, 64, 4), (221, 16, 16, 16), (222, 16, 16, 16), (243, 8, 8, 32),
                                     (601, 16, 64, 17)])
def test_many_sequences_of_short_chunks(N, d, h, C, normed):
    """Either side of the lines that take a forward of many small sequences off the block-tiled kernels; its states and row norms pass to their
    reverse pass.  Six chunks, checkpoints of two."""
    x, shape = _inputs(2, 5 * C + 1, d, h, C, MLP, with_d_o=True, with_dstate=True)
    rep = lambda a: np.concatenate([a] * ((N + 1) // 2))[:N]
    xs = {n: [rep(w) for w in a] if isinstance(a, list) else rep(a) for n, a in x.items()}
    cut = lambda got: {n: [w[:2] for w in a] if isinstance(a, list) else a[:2] for n, a in got.items()}
    if normed:
        tgt = targets(x)
        got, ref = gpu_forward_normed(xs, [rep(t) for t in tgt], impl=E.E2TTT_IMPL_TILED, **shape), oracle_fwd(x, tgt, C, MLP)
        refb = oracle_bwd(x, tgt, C, MLP)
        plans = [gpu_backward_normed(xs, [rep(t) for t in tgt], impl=E.E2TTT_IMPL_TILED, via_saved_states=saved, **shape) for saved in (True, False)]
    else:
        got, ref, refb = util.gpu_forward(xs, impl=E.E2TTT_IMPL_TILED, **shape)[0], util.oracle_forward(x, C, MLP), util.oracle_backward(x, C, MLP)
        plans = [util.gpu_backward(xs, impl=E.E2TTT_IMPL_TILED, via_saved_states=saved, ckpt_every=ckpt, **shape)
                 for saved, ckpt in ((True, 0), (True, 2), (False, 0), (False, 2))]
    for a in [got["o"], *got["W"], *got["M"]]:
        assert all(np.array_equal(a[n], a[n % 2]) for n in range(N))
    check_forward(cut(got), ref, TOL_BF16, "forward")
    check_fp32(cut(got), ref, "forward")
    check_backward(cut(plans[0]), refb, 2 * TOL_BF16, "backward")
    check_fp32(cut(plans[0]), refb, "backward")
    for got in plans[1:]:  # every memory plan: the same bits
        for n, a in got.items():
            assert all(np.array_equal(v, w) for v, w in (zip(a, plans[0][n]) if isinstance(a, list) else [(a, plans[0][n])])), n
