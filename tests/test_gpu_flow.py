"""The forward on work items (csrc/tile_flow.cu) against the fp64 oracle, at the edges of its tiles and of its dispatch: one block of hidden units
and an odd number, one and two blocks of d and of tokens, ragged chunks, several sets of sequences."""
import numpy as np
import pytest

from paper_2608_21308_b200 import binding as E
from paper_2608_21308_b200 import inputs
from tests import util
from tests.test_gpu_dispatch_edges import check_fp32
from tests.test_gpu_normed import gpu_backward_normed, gpu_forward_normed, oracle_bwd, oracle_fwd, targets
from tests.test_gpu_parity import TOL_BF16, check_backward

pytestmark = pytest.mark.gpu
MLP, SWIGLU = inputs.KIND_MLP, inputs.KIND_SWIGLU
# Operands are hi + lo of bf16: what a product drops is 2^-16 of it, the state sums up to 512 of them and carries them over three chunks
# that amplify a perturbation by up to 1.8 each (GELU) or, with the product of two projections, twice that
TOL = {MLP: 6 * 2.0**-16 * 5, SWIGLU: 40 * 2.0**-16 * 5}


@pytest.mark.parametrize("kind", [MLP, SWIGLU])
@pytest.mark.parametrize("d,h,C,L,N", [(8, 8, 65, 131, 1), (64, 64, 128, 300, 2), (72, 200, 200, 450, 3), (128, 384, 512, 1100, 2), (128, 128, 65, 66, 150),
                                       (16, 16, 80, 250, 170), (96, 296, 64, 150, 3), (128, 520, 24, 60, 16), (33, 50, 70, 150, 2),
                                       (127, 131, 65, 70, 1)])
def test_states_and_outputs(kind, d, h, C, L, N):
    r = inputs.paper_regime(inputs.Recipe(B=N, H=1, L=L, d=d, h=h, C=C, kind=kind, io="bf16", seed=7, m_std=0.002))
    x = inputs.generate(r)
    heads = sorted({0, N // 2, N - 1})
    ref = util.oracle_forward({k: [m[heads] for m in v] if isinstance(v, list) else v[heads] for k, v in x.items() if v is not None}, C, kind)
    got, hd = util.gpu_forward(x, d=d, h=h, C=C, kind=kind, io="bf16", impl=E.E2TTT_IMPL_TILED)
    assert E.e2ttt_device_status(hd["ws"]) == 0
    errs = {"o": util.rel_err(got["o"][heads], ref["o"])}
    assert errs["o"] <= 1e-2  # bf16 outputs
    for name in ("W", "M"):
        for i, m in enumerate(ref[name]):
            errs[f"{name}{i + 1}"] = util.rel_err(got[name][i][heads], m)
    bad = {k: v for k, v in errs.items() if k != "o" and not v <= TOL[kind]}
    assert not bad, errs
    again, _ = util.gpu_forward(x, d=d, h=h, C=C, kind=kind, io="bf16", impl=E.E2TTT_IMPL_TILED)
    assert all(np.array_equal(a, b) for a, b in zip([got["o"], *got["W"], *got["M"]], [again["o"], *again["W"], *again["M"]]))


def copies_of_two(d, h, C, L, N, kind, change=lambda x: None):
    """N sequences, copies of two: all copies equal.  Returns the result and the oracle's for the two."""
    x = inputs.generate(inputs.paper_regime(inputs.Recipe(B=2, H=1, L=L, d=d, h=h, C=C, kind=kind, io="bf16", seed=11, m_std=0.002)))
    change(x)
    ref = util.oracle_forward(x, C, kind)
    rep = lambda a: np.concatenate([a] * ((N + 1) // 2))[:N]
    xs = {n: [rep(w) for w in a] if isinstance(a, list) else rep(a) for n, a in x.items() if a is not None}
    got, hd = util.gpu_forward(xs, d=d, h=h, C=C, kind=kind, io="bf16", impl=E.E2TTT_IMPL_TILED)
    assert E.e2ttt_device_status(hd["ws"]) == 0
    for a in [got["o"], *got["W"], *got["M"]]:
        assert all(np.array_equal(a[n], a[n % 2]) for n in range(N))
    assert util.rel_err(got["o"][:2], ref["o"]) <= 1e-2  # bf16 outputs
    return got, ref


# A product's operands, two bf16 terms each, are off by 2^-17 / sqrt 3 = 4.4e-6 of their size (rms).  An MMA truncates the sum it adds to, by 2^-24 of it on
# average and always towards zero: 64 of them, one sum of u over 1024 hidden units, come to less than 64 * 2^-24 = 3.8e-6 of u.  Chunk-end states
# of two chunks: within sqrt(4.4^2 + 3.8^2) = 5.8e-6, a fifth more for the second chunk.  512 MMAs in one sum (8192 hidden units): 9e-6 measured
@pytest.mark.parametrize("d,h,C,L,N", [(128, 8192, 64, 128, 40), (64, 1160, 64, 100, 40), (128, 2048, 24, 48, 40), (72, 3200, 64, 128, 40)])
def test_u_of_many_hidden_units_is_as_exact_as_that_of_few(d, h, C, L, N):
    got, ref = copies_of_two(d, h, C, L, N, MLP)
    errs = {f"{name}{i + 1}": util.rel_l2(got[name][i][:2], m) for name in ("W", "M") for i, m in enumerate(ref[name])}
    assert all(e <= 7e-6 for e in errs.values()), errs


# Operands are off by 2^-17 / sqrt 3 = 4.4e-6 (rms) in each of the four products from a chunk's keys to its aggregates, 9e-6 together; two more chunks that
# amplify it by up to 2 each stay below 1e-4.  An operand without its second term is off by 2^-9 / sqrt 3 = 1.1e-3
@pytest.mark.parametrize("normed", [False, True], ids=["plain", "normed"])
@pytest.mark.parametrize("kind", [MLP, SWIGLU])
@pytest.mark.parametrize("d,h,C,L,N", [(128, 384, 512, 1025, 67), (72, 200, 512, 1100, 101), (64, 64, 512, 600, 131)])
def test_sequences_in_several_sets_of_which_the_last_is_short(d, h, C, L, N, kind, normed):
    """Tokens, weights and norm items of several sequences and sets in work at a time; the last set has places without a sequence."""
    if not normed:
        got, ref = copies_of_two(d, h, C, L, N, kind)
    else:
        x = inputs.generate(inputs.paper_regime(inputs.Recipe(B=2, H=1, L=L, d=d, h=h, C=C, kind=kind, io="bf16", seed=12, m_std=0.002)))
        tgt = targets(x)
        ref = oracle_fwd(x, tgt, C, kind)
        rep = lambda a: np.concatenate([a] * ((N + 1) // 2))[:N]
        xs = {n: [rep(w) for w in a] if isinstance(a, list) else rep(a) for n, a in x.items() if a is not None}
        got = gpu_forward_normed(xs, [rep(t) for t in tgt], d=d, h=h, C=C, kind=kind, io="bf16", impl=E.E2TTT_IMPL_TILED)
        for a in [got["o"], *got["W"], *got["M"]]:
            assert all(np.array_equal(a[n], a[n % 2]) for n in range(N))
        assert util.rel_err(got["o"][:2], ref["o"]) <= 1e-2  # bf16 outputs
    errs = {f"{name}{i + 1}": util.rel_l2(got[name][i][:2], m) for name in ("W", "M") for i, m in enumerate(ref[name])}
    assert all(e <= 1e-4 for e in errs.values()), errs


@pytest.mark.parametrize("kind", [MLP, SWIGLU])
@pytest.mark.parametrize("d,h,C,L", [(4, 8, 64, 70), (36, 144, 40, 75), (68, 72, 65, 130), (100, 400, 64, 129), (124, 64, 128, 200)])
def test_rows_of_8_bytes_alignment(d, h, C, L, kind):
    """Head dimensions that are multiples of four and not of eight; the bound as above, two chunks of several at most."""
    got, ref = copies_of_two(d, h, C, L, 3, kind)
    errs = {f"{name}{i + 1}": util.rel_l2(got[name][i][:2], m) for name in ("W", "M") for i, m in enumerate(ref[name])}
    assert all(e <= 1e-4 for e in errs.values()), errs


@pytest.mark.parametrize("kind", [MLP, SWIGLU])
@pytest.mark.parametrize("N,d,h,C", [(8, 128, 384, 64), (16, 64, 320, 48), (24, 128, 1024, 16), (19, 128, 768, 64), (16, 128, 1600, 128), (3, 128, 512, 512)])
def test_a_sequence_in_several_calls_has_the_bits_of_one(N, d, h, C, kind):
    """Chunk by chunk, and in calls of one and two chunks, on either side of the lines between work items and clusters."""
    L = 3 * C
    x = inputs.generate(inputs.paper_regime(inputs.Recipe(B=2, H=1, L=L, d=d, h=h, C=C, kind=kind, io="bf16", seed=13, m_std=0.002)))
    rep = lambda a: np.concatenate([a] * ((N + 1) // 2))[:N]
    x = {n: [rep(w) for w in a] if isinstance(a, list) else rep(a) for n, a in x.items() if a is not None}
    run = lambda y: util.gpu_forward(y, d=d, h=h, C=C, kind=kind, io="bf16", impl=E.E2TTT_IMPL_TILED)[0]
    whole = run(x)
    for cuts in ((0, C, 2 * C, L), (0, C, L)):
        W, M, o = x["W"], x["M"], []
        for a, b in zip(cuts, cuts[1:]):
            part = run({**{n: np.ascontiguousarray(v[:, a:b]) for n, v in x.items() if n not in ("W", "M")}, "W": W, "M": M})
            W, M = part["W"], part["M"]
            o.append(part["o"])
        assert np.array_equal(np.concatenate(o, 1), whole["o"])
        assert all(np.array_equal(a, b) for a, b in zip([*W, *M], [*whole["W"], *whole["M"]]))


def test_normalised_swiglu_training_step_of_four_long_chunks():
    """2048 tokens in chunks of 512, d = 128, h = 384, saved states.  The bound as above for what is returned in fp32 of the state and its adjoints."""
    shape = dict(d=128, h=384, C=512, kind=SWIGLU, io="bf16", impl=E.E2TTT_IMPL_TILED)
    x = inputs.generate(inputs.paper_regime(inputs.Recipe(B=2, H=1, L=2048, d=128, h=384, C=512, kind=SWIGLU, io="bf16", seed=14, m_std=0.002)), with_d_o=True, with_dstate=True)
    tgt = targets(x)
    got, ref = gpu_forward_normed(x, tgt, **shape), oracle_fwd(x, tgt, 512, SWIGLU)
    gotb, refb = gpu_backward_normed(x, tgt, via_saved_states=True, **shape), oracle_bwd(x, tgt, 512, SWIGLU)
    assert util.rel_err(got["o"], ref["o"]) <= 1e-2  # bf16 outputs
    errs = {f"{n}{i + 1}": util.rel_l2(a, b) for g, r, names in ((got, ref, ("W", "M")), (gotb, refb, ("dW", "dM"))) for n in names for i, (a, b) in enumerate(zip(g[n], r[n]))}
    assert all(e <= 1e-4 for e in errs.values()), errs
    check_backward(gotb, refb, 2 * TOL_BF16, "backward")
    check_fp32(gotb, refb, "backward")
