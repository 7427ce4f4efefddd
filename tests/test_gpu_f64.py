"""fp32 I/O on the fp64 kernels (csrc/f64_*.cu) at the edges of their tiles, parts and groups of chunks, against the oracle."""
import numpy as np
import pytest

from paper_2608_21308_b200 import binding as E
from paper_2608_21308_b200 import inputs
from tests import util
from tests.test_gpu_normed import gpu_backward_normed, gpu_forward_normed, oracle_bwd, oracle_fwd, targets
from tests.test_gpu_parity import check_backward, check_forward

pytestmark = pytest.mark.gpu
MLP, SWIGLU = inputs.KIND_MLP, inputs.KIND_SWIGLU
# fp64 inside, rounded once to fp32 (2^-24 of a value); the oracle's sums are in another order, which in fp64 does not show
TOL = 1e-6


def _inputs(N, L, d, h, C, kind):
    r = inputs.paper_regime(inputs.Recipe(B=N, H=1, L=L, d=d, h=h, C=C, kind=kind, io="f32", seed=17, m_std=0.002))
    return inputs.generate(r, with_d_o=True, with_dstate=True), dict(d=d, h=h, C=C, kind=kind, io="f32")


@pytest.mark.parametrize("kind", [MLP, SWIGLU])
@pytest.mark.parametrize("N,d,h,C,L", [
    (1, 1, 1, 1, 3),        # a value in every direction
    (2, 16, 16, 16, 33),    # whole tiles; a chunk of one token
    (8, 17, 33, 15, 40),    # one past a tile; clusters of 8
    (1, 48, 336, 24, 31),   # 63 tiles of 16 x 16: the last with narrow tiles
    (3, 64, 256, 16, 50),   # 64: wide tiles of the state, narrow ones of the tokens
    (1, 40, 130, 65, 130),  # contractions of two slices and a remainder, in three parts
    (75, 33, 70, 33, 66),   # one CTA per sequence
    (1, 128, 136, 300, 310),# [tokens x d] results uncut
    (9, 128, 384, 64, 300), # groups of three chunks (SwiGLU two), the last shorter
])
def test_forward_and_reverse_pass(N, d, h, C, L, kind):
    x, shape = _inputs(N, L, d, h, C, kind)
    got, hd = util.gpu_forward(x, **shape)
    assert E.e2ttt_device_status(hd["ws"]) == 0
    check_forward(got, util.oracle_forward(x, C, kind), TOL, "fp64 forward")
    check_backward(util.gpu_backward(x, via_saved_states=True, **shape), util.oracle_backward(x, C, kind), TOL, "fp64 reverse pass")


@pytest.mark.parametrize("kind", [MLP, SWIGLU])
def test_normalised_reverse_pass_over_groups_of_chunks(kind):
    x, shape = _inputs(9, 5 * 64 - 20, 128, 384, 64, kind)
    tgt = targets(x)
    check_backward(gpu_backward_normed(x, tgt, impl=E.E2TTT_IMPL_AUTO, via_saved_states=True, **shape), oracle_bwd(x, tgt, 64, kind), 1e-5, "fp64 normed reverse pass")


@pytest.mark.parametrize("kind", [MLP, SWIGLU])
def test_results_do_not_depend_on_the_cluster(kind):
    """One sequence (a cluster of 16) and the same one among 80 (a CTA each): the same bits."""
    x, shape = _inputs(1, 70, 40, 130, 16, kind)
    many = {n: [np.concatenate([w] * 80) for w in a] if isinstance(a, list) else np.concatenate([a] * 80) for n, a in x.items()}
    one, all_ = util.gpu_backward(x, **shape), util.gpu_backward(many, **shape)
    for n, a in one.items():
        for p, q in zip(a, all_[n]) if isinstance(a, list) else [(a, all_[n])]:
            assert np.array_equal(np.asarray(p)[0], np.asarray(q)[0]) and np.array_equal(np.asarray(p)[0], np.asarray(q)[79]), n


@pytest.mark.parametrize("kind", [MLP, SWIGLU])
@pytest.mark.parametrize("d,h,C,L", [
    (828, 1, 365, 400),  # compact layout (f64_compact): the widest head of one hidden unit that fits the fixed scratch; a short last chunk
    (256, 1, 126, 253),  # the first chunk length that takes it, a last chunk of one token
    (256, 1, 125, 251),  # the last one that does not
    (300, 40, 256, 512), # several tiles of hidden units
])
def test_wide_heads_with_few_hidden_units(d, h, C, L, kind):
    import torch

    x, shape = _inputs(1, L, d, h, C, kind)
    got, hd = util.gpu_forward(x, **shape)
    check_forward(got, util.oracle_forward(x, C, kind), TOL, "fp64 forward")
    if h > 1:  # (a row of one weight is +-n: where the weight crosses zero, n w / (|w| + eps) magnifies its error by n / |w|)
        tgt = targets(x)
        check_forward(gpu_forward_normed(x, tgt, impl=E.E2TTT_IMPL_AUTO, **shape), oracle_fwd(x, tgt, C, kind), 1e-5, "fp64 normed forward")
    # the same call in the fixed scratch: the same bits
    o, Wf, Mf = torch.empty_like(hd["q"]), [torch.empty_like(w) for w in hd["W"]], [torch.empty_like(w) for w in hd["W"]]
    E.e2ttt_chunk_fwd_noalloc(hd["p"], hd["q"], hd["k"], hd["v"], hd["eta"], hd["beta"], hd["gamma"], hd["W"], hd["M"], o, Wf, Mf)
    torch.cuda.synchronize()
    assert np.array_equal(o.cpu().numpy().reshape(1, L, d), got["o"])
    for w, m, w0, m0 in zip(Wf, Mf, got["W"], got["M"]):
        assert np.array_equal(w.cpu().numpy()[:, 0], w0) and np.array_equal(m.cpu().numpy()[:, 0], m0)


@pytest.mark.parametrize("kind", [MLP, SWIGLU])
@pytest.mark.parametrize("d,h,C,L", [
    (40, 130, 16, 37),   # narrow tiles
    (16, 16, 446, 450),  # the longest chunk with two CTAs on an SM, and the next one
    (16, 16, 447, 450),
    (64, 256, 215, 220), # the same with wide tiles
    (64, 256, 216, 220),
    (64, 256, 16, 1),    # a token
])
def test_forward_of_more_sequences_than_sms(d, h, C, L, kind):
    """150 copies of a sequence on kernels that share an SM (f64_fwd_two): the bits of the one that has a cluster, which match the oracle."""
    x, shape = _inputs(1, L, d, h, C, kind)
    many = {n: [np.concatenate([w] * 150) for w in a] if isinstance(a, list) else np.concatenate([a] * 150) for n, a in x.items()}
    one, _ = util.gpu_forward(x, **shape)
    check_forward(one, util.oracle_forward(x, C, kind), TOL, "one sequence")
    all_, _ = util.gpu_forward(many, **shape)
    for n in ("o", "W", "M"):
        for p, q in zip(one[n], all_[n]) if n != "o" else [(one[n], all_[n])]:
            assert all(np.array_equal(p[0], q[i]) for i in (0, 75, 149)), n
