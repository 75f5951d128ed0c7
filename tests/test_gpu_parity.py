"""GPU parity: the CUDA path, called through the C ABI, against the float64 oracle on the same
seeded inputs, element by element."""
import threading

import numpy as np
import pytest
import torch

from paper_1805_10032_b200 import synthetic as syn
from paper_1805_10032_b200 import zeno

import parity as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _library():
    from paper_1805_10032_b200 import build as zbuild
    zbuild.build()
    assert torch.cuda.is_available(), "these tests need a CUDA device"
    zeno.load_library()


# ---------------------------------------------------------------- shrunk versions of the five workloads
# sizes chosen to span several row tiles / k stages and to leave ragged tails in every dimension

SHRUNK = {
    "cfg1": (1, dict()),                                                   # full size (d = 7850)
    "cfg1_nr7": (1, dict(n_r=7, m=11, b=4, faults=[(4, "signflip")])),
    "cfg2_small": (2, dict(dims=(300, 72, 40, 10), n_r=9)),
    "cfg2_wide_k": (2, dict(dims=(1028, 36, 68, 10), n_r=33, m=7, b=3, faults=[(3, "noise200")])),
    # hidden layers wide enough for the tensor-core stream: ragged row tiles and k tails in both
    "cfg2_mid_layers": (2, dict(dims=(520, 200, 136, 10), n_r=21, m=6, b=2, faults=[(2, "noise200")])),
    "cfg3_mid_layers": (3, dict(dims=(520, 136, 200, 10), m=11, b=4, n_r=40,
                                faults=[(2, "signflip"), (2, "omniscient")])),
    # the streamed tensor-core layer kernel: 128 samples (N = 256) on a bfloat16 model, a padded
    # sample count above 64 on an fp32 model, and an fp32 first layer with a tile for every SM
    "cfg4_128_samples": (4, dict(dims=(136, 200, 72, 50), m=4, b=1, n_r=128, faults=[(1, "signflip")])),
    "cfg3_100_samples": (3, dict(dims=(200, 136, 130, 10), m=7, b=2, n_r=100,
                                 faults=[(1, "signflip"), (1, "omniscient")])),
    "cfg3_many_tiles": (3, dict(dims=(132, 384, 10), m=100, b=40, n_r=5,
                                faults=[(20, "signflip"), (20, "omniscient")])),
    "cfg3_small": (3, dict(dims=(260, 44, 36, 10), m=37, b=15, n_r=70,
                           faults=[(7, "signflip"), (8, "omniscient")])),
    "cfg4_small": (4, dict(dims=(264, 136, 72, 50), m=9, b=3, n_r=19, faults=[(3, "signflip")])),
    # a small last layer folded into the tensor-core layer before it, bfloat16 and fp32 (ragged tiles,
    # several tiles per model, an odd number of classes)
    "cfg4_ten_classes": (4, dict(dims=(264, 136, 200, 10), m=9, b=3, n_r=19, faults=[(3, "signflip")])),
    "cfg2_seven_classes": (2, dict(dims=(520, 200, 300, 7), n_r=30, m=12, b=5, faults=[(5, "noise200")])),
    # more tiles than SMs, not a multiple of the SM count (several rounds of tiles per block, the last one
    # partly empty): the linear fp32 first layer, a later fp32 layer, and a bfloat16 model -- ragged row
    # tiles and a ragged last k-block in each
    "cfg3_ragged_rounds_first_layer": (3, dict(dims=(200, 384, 10), m=100, b=40, n_r=5,
                                              faults=[(20, "signflip"), (20, "omniscient")])),
    "cfg3_ragged_rounds_later_layer": (3, dict(dims=(136, 264, 330, 10), m=100, b=40, n_r=9,
                                              faults=[(20, "signflip"), (20, "omniscient")])),
    "cfg4_ragged_rounds": (4, dict(dims=(392, 264, 50), m=100, b=30, n_r=7, faults=[(30, "signflip")])),
    "cfg5_small": (5, dict(d=70000, m=13, b=5, n_r=16, n_noise=5)),
    "cfg5_nr5": (5, dict(d=33333 * 4, m=70, b=30, n_r=5, n_noise=30)),
    # d a multiple of 32: the tensor-core stream fetches both k-blocks of a pair with one copy per operand
    "cfg5_d_mult_32": (5, dict(d=69632 + 32, m=37, b=12, n_r=16, n_noise=12)),
    "cfg5_d_mult_32_nr30": (5, dict(d=40960, m=64, b=20, n_r=30, n_noise=20)),
    "cfg5_nr40": (5, dict(d=9000, m=6, b=2, n_r=40, n_noise=2)),
    # the tensor-core least-squares stream with 32 padded samples (N = 128) and all 64 candidate lanes in use,
    # a parameter count that leaves a ragged last k-block pair
    # (at the configuration's own gamma = 0.01 one honest score is a 1e-6 difference of terms near 0.6: that
    # candidate is held to the conditioning-aware bound and its condition number is printed)
    "cfg5_nr24_m64": (5, dict(d=50004, m=64, b=20, n_r=24, n_noise=20)),
}


# the small last layer over its limits: one to eight blocks a model, slices with remainders, rows of any alignment,
# every compiled number of classes and samples; candidates up to and beyond what the averaging kernel ranks itself
@pytest.mark.parametrize("dims,n_r,m,dtype,pad", [
    ((33, 2), 1, 5, "f32", 1), ((250, 10), 9, 7, "f32", 0), ((517, 16), 33, 20, "bf16", 0), ((1028, 17), 8, 9, "f32", 0),
    ((1029, 32), 32, 37, "f32", 1), ((4100, 10), 16, 20, "bf16", 4), ((4100, 16), 64, 20, "f32", 4), ((784, 31), 17, 36, "bf16", 1),
    ((784, 10), 4, 149, "f32", 0), ((60, 10), 4, 256, "f32", 0), ((60, 10), 4, 257, "f32", 0)])
def test_small_last_layer_over_its_limits(oracle, dims, n_r, m, dtype, pad):
    d = dims[0] * dims[1] + dims[1]
    b = m // 3
    w = syn.make_config(1, dims=dims, n_r=n_r, m=m, b=b, dtype=dtype, ldv=d + pad, faults=[(b, "signflip")])
    P.run_step_parity(oracle, w)


# the same by what a cluster stages at once and by its classes and samples: slices in several turns, twelve rows, thirteen and
# more, samples of a last half warp, one sample more than the warps take
@pytest.mark.parametrize("dims,n_r,m,dtype,pad", [
    ((2600, 32), 7, 120, "f32", 0), ((9000, 12), 9, 70, "f32", 1), ((7001, 13), 33, 40, "f32", 0), ((8200, 10), 63, 75, "bf16", 4), ((2051, 11), 1, 9, "bf16", 1)])
def test_small_last_layer_in_turns(oracle, dims, n_r, m, dtype, pad):
    d = dims[0] * dims[1] + dims[1]
    b = m // 3
    P.run_step_parity(oracle, syn.make_config(1, dims=dims, n_r=n_r, m=m, b=b, dtype=dtype, ldv=d + pad, faults=[(b, "signflip")]))


# the layer kernel for rows of any alignment: one row tile and several, slices with remainders, one to eight blocks a tile,
# every compiled number of samples, several sample tiles, no bias
@pytest.mark.parametrize("dims,n_r,m,dtype,bias", [
    ((65, 3, 2), 1, 3, "f32", True), ((63, 64, 5), 8, 4, "f32", False), ((1029, 65, 11), 9, 5, "f32", True),
    ((2051, 37, 129, 10), 19, 6, "f32", True), ((515, 301, 40), 25, 37, "f32", True), ((130, 131, 33), 33, 20, "bf16", True),
    ((4100, 43, 43), 70, 7, "bf16", True), ((257, 67, 101), 128, 5, "f32", True)])
def test_layers_of_unaligned_rows(oracle, dims, n_r, m, dtype, bias):
    d = syn.param_count("mlp", dims, bias)
    b = m // 3
    w = syn.make_config(2, dims=dims, n_r=n_r, m=m, b=b, dtype=dtype, has_bias=bias, ldv=d + (d + 1) % 2, faults=[(b, "signflip")] if b else [])
    P.run_step_parity(oracle, w)


# layers by columns: one row and one column short of and beyond a warp's and a block's share, the last stretch of one column
# and of all but one, every compiled number of samples and tiles of them, both ways the weights are fetched, clusters of
# blocks, rows of every alignment, bfloat16 rows that start at an odd entry, no bias
@pytest.mark.parametrize("dims,n_r,m,bias", [
    ((128, 31, 2), 1, 3, True), ((257, 33, 5), 2, 4, True), ((255, 64, 65, 3), 4, 5, True), ((513, 129, 10), 8, 21, True),
    ((129, 32, 40), 12, 6, False), ((383, 97, 10), 13, 9, True), ((1025, 161, 10), 17, 5, True), ((767, 45, 131, 7), 24, 37, True),
    ((640, 100, 9), 25, 4, True), ((2049, 34, 10), 20, 2, False), ((300, 260, 44), 40, 5, True), ((1028, 36, 4), 33, 6, True)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("pad", [0, 1])
def test_layers_by_columns(oracle, dims, n_r, m, bias, dtype, pad):
    b = m // 3
    w = syn.make_config(2, dims=dims, n_r=n_r, m=m, b=b, dtype=dtype, has_bias=bias, ldv=syn.param_count("mlp", dims, bias) + pad,
                        faults=[(b, "signflip")] if b else [])
    P.run_step_parity(oracle, w)


# many binary32 samples of unaligned rows, either side of the rule that takes a layer by columns or by tiles: 20 and 24, 28, 40 and 41
# samples, narrow layers of 48 and 49, one wave of blocks and several, tiles of twelve to 24 samples
@pytest.mark.parametrize("dims,n_r,m", [
    ((129, 33, 34, 3), 40, 4), ((129, 33, 34, 3), 41, 4), ((244, 20, 9), 48, 5), ((244, 20, 9), 49, 5), ((200, 120, 10), 95, 30), ((200, 330, 10), 95, 30),
    ((150, 70, 10), 103, 5), ((131, 270, 10), 84, 21), ((150, 300, 10), 20, 70), ((150, 300, 10), 24, 70), ((150, 300, 10), 28, 100), ((150, 300, 10), 28, 130)])
def test_layers_of_many_samples_of_unaligned_rows(oracle, dims, n_r, m):
    b = m // 3
    P.run_step_parity(oracle, syn.make_config(2, dims=dims, n_r=n_r, m=m, b=b, ldv=syn.param_count("mlp", dims, True) + 1, faults=[(b, "signflip")]))


@pytest.mark.parametrize("cols,rows,dtype", [(40001, 33, "f32"), (40001, 33, "bf16"), (40004, 36, "f32")])
def test_sums_of_long_rows_are_short_sums(cols, rows, dtype):
    """A logit of 40,000 products of random signs against 64 bits, the layer in as many tiles as leave a lane every 32nd
    column of whole rows.  An addition to a partial sum of k products errs by 0.41 x 2^-24 of it in the root mean square and
    the partial sum grows as sqrt(k): a chain of n products is off by 0.41 x 2^-24 sqrt(n / 2) of the result, 6e-7 with all
    1,250 of a lane and 1.4e-7 with runs of 64, to which the additions of the 32 lanes and of the runs add about as much."""
    m, n_r, size, gamma = 12, 128, 3e4, 0.125
    g = torch.Generator().manual_seed(cols + rows)
    store = torch.bfloat16 if dtype == "bf16" else torch.float32
    d = rows * cols + rows
    x = (torch.randn(d, generator=g) * (size / cols ** 0.5)).to(store)
    V = torch.randn((m, d), generator=g).mul_(0.5 * size / cols ** 0.5 / gamma).to(store)
    feats = torch.randn((n_r, cols), generator=g)
    feats[1:] *= 1e-9                                # the first sample's loss is all there is to see
    labels = torch.randint(0, rows, (n_r,), generator=g, dtype=torch.int32)
    with zeno.Zeno(zeno.LOSS_SOFTMAX_MLP, zeno.BF16 if dtype == "bf16" else zeno.F32, (cols, rows), True, m, n_r) as z:
        _, losses, _ = z.score(x.cuda(), V.cuda(), feats.cuda(), labels.cuda(), gamma, 0.0)
        got = losses.double().cpu()
    for c in range(m + 1):
        w = x.double() if c == 0 else x.double() - gamma * V[c - 1].double()
        w = w.float().to(store).double() if dtype == "bf16" else w
        z64 = feats.double() @ w[:rows * cols].view(rows, cols).t() + w[rows * cols:]
        got[c] -= torch.nn.functional.cross_entropy(z64, labels.long())
    # a loss is the difference of two logits of this size, times 1 / n_r
    assert (got.square().mean().sqrt() / (size * 2 ** 0.5 / n_r)).item() <= 3.5e-7


# the same kernel on rows aligned to four elements (four columns a load), and with half its rows a tile (layers of up to 32
# rows, up to 64 samples a tile): columns that end inside a slice and inside a load's reach, one and several slices, one
# row, 32 and 33, every compiled number of samples, clusters
@pytest.mark.parametrize("dims,n_r,m", [((4, 36, 4), 1, 3), ((68, 100, 4), 8, 4), ((324, 148, 100), 16, 5), ((260, 68, 36), 24, 21),
                                        ((132, 132, 64), 33, 20), ((516, 4, 4), 9, 7), ((136, 20, 4), 33, 20), ((1028, 32, 4), 65, 5), ((60, 28, 8), 64, 30),
                                        ((2052, 12, 4), 31, 4)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("pad", [0, 1])
def test_layers_of_rows_aligned_to_four(oracle, dims, n_r, m, dtype, pad):
    d = syn.param_count("mlp", dims, True)
    assert d % 4 == 0                                   # pad = 0: the aligned kernel, 1: that for any rows
    b = m // 3
    w = syn.make_config(2, dims=dims, n_r=n_r, m=m, b=b, dtype=dtype, ldv=d + pad, faults=[(b, "signflip")])
    P.run_step_parity(oracle, w)


def test_small_last_layer_with_huge_logits(oracle):
    """Noise candidates of a deep model whose logits reach 1e10, where neighbouring binary32 values are 1,024 apart:
    their losses stay finite and they are dropped."""
    w = syn.make_config(2, dims=(432, 448, 280, 834, 10), m=64, b=25, n_r=3, faults=[(25, "noise200")])
    P.run_step_parity(oracle, w)
    x, V, feats, tgt = P.to_device(w)
    with zeno.from_workload(w) as z:
        _, scores, idx = z.step(x, V, feats, tgt, w.gamma, w.rho, w.b)
        _, losses, _ = z.score(x, V, feats, tgt, w.gamma, w.rho)
    assert torch.isfinite(scores).all() and losses.max().item() > 1e9
    assert w.honest[idx.cpu().long()].all()


# padded sample counts that would leave the layer kernel an odd ring of weight stages shorter than its A buffers and
# two, on which a converter set could overtake the other one's load
@pytest.mark.parametrize("n_r", [17, 33, 64, 83, 100, 128])
def test_weight_rings_of_every_padded_sample_count(oracle, n_r):
    w = syn.make_config(2, dims=(400, 160, 632, 368, 10), m=32, b=12, n_r=n_r, faults=[(12, "noise200")])
    P.run_step_parity(oracle, w)
    x, V, feats, tgt = P.to_device(w)
    with zeno.from_workload(w) as z:
        first = z.step(x, V, feats, tgt, w.gamma, w.rho, w.b)
        for _ in range(50):
            again = z.step(x, V, feats, tgt, w.gamma, w.rho, w.b)
            assert all(torch.equal(a, b) for a, b in zip(first, again))
        z.check_device_status()


@pytest.mark.parametrize("name", sorted(SHRUNK))
def test_step_matches_oracle_on_shrunk_workloads(oracle, name):
    index, ov = SHRUNK[name]
    w = syn.make_config(index, **ov)
    res = P.run_step_parity(oracle, w)
    assert res["launches"] >= 2


def kernels_of_a_step(w):
    """Names of the kernels one zeno_step launches on this workload, in launch order."""
    x, V, feats, tgt = P.to_device(w)
    with zeno.from_workload(w) as z:
        z.profile(True)
        z.step(x, V, feats, tgt, w.gamma, w.rho, w.b)
        torch.cuda.synchronize()
        return [name for name, _ in z.profile_read(0)]


@pytest.mark.parametrize("name,expected", [
    ("cfg2_mid_layers", ["stream_tf32x3", "stream_combine", "layer_tc_head", "aggregate"]),
    ("cfg4_ten_classes", ["split_acts", "layer_tc", "layer_tc_head", "aggregate"]),
    ("cfg3_many_tiles", ["split_acts", "layer_tc", "stream_combine", "mlp_head_loss_tail", "aggregate"]),
    ("cfg4_128_samples", ["split_acts", "layer_tc", "layer_tc", "layer_tc", "mlp_loss_tail", "aggregate"]),
    ("cfg4_small", ["split_acts", "layer_tc", "layer_tc", "layer_tc", "mlp_loss_tail", "aggregate"]),
    ("cfg3_ragged_rounds_first_layer", ["split_acts", "layer_tc", "stream_combine", "mlp_head_loss_tail", "aggregate"]),
    ("cfg4_ragged_rounds", ["split_acts", "layer_tc", "layer_tc", "mlp_loss_tail", "aggregate"]),
    ("cfg5_nr24_m64", ["lsq_tc", "lsq_finish", "select", "aggregate"]),
    ("cfg5_small", ["lsq_tc", "lsq_finish", "select", "aggregate"]),
])
def test_which_kernels_serve_a_workload(name, expected):
    """The parity cases above exercise the kernels they were written for (no quiet detour)."""
    index, ov = SHRUNK[name]
    assert kernels_of_a_step(syn.make_config(index, **ov)) == expected


def test_config2_full_size(oracle):
    w = syn.make_config(2)
    assert w.d == 1841162 and w.m == 20 and w.n_r == 32
    res = P.run_step_parity(oracle, w)
    assert res["exact_set"]


# ---------------------------------------------------------------- odd shapes, unaligned rows (scalar path)

@pytest.mark.parametrize("dims,n_r,m,pad", [
    ((7, 5, 4, 3), 3, 6, 0),        # nothing aligned
    ((13, 3), 1, 2, 5),             # softmax regression, one sample
    ((129, 33, 2), 17, 5, 1),
    ((130, 66, 10), 8, 33, 3),
    ((260, 10), 32, 4, 2),
])
def test_unaligned_layouts(oracle, dims, n_r, m, pad):
    d = syn.param_count("mlp", dims)
    w = syn.make_config(2, dims=dims, n_r=n_r, m=m, b=m // 3, faults=[(m // 3, "noise200")],
                        ldv=d + pad)
    P.run_step_parity(oracle, w)


def test_unaligned_base_pointers(oracle):
    # x and V start 4 bytes into an allocation: every vector path must be refused
    w = syn.make_config(1, dims=(64, 12), m=6, b=2, faults=[(2, "signflip")])
    xs = torch.empty(w.d + 1, device="cuda"); xs[1:] = w.x.cuda()
    Vs = torch.empty(w.m * w.ldv + 1, device="cuda"); Vs[1:] = w.V.cuda().reshape(-1)
    x, V = xs[1:], Vs[1:].view(w.m, w.ldv)
    s_orc, _, _ = P.oracle_score(oracle, w)
    with zeno.from_workload(w) as z:
        out, scores, idx = z.step(x, V, w.features.cuda(), w.targets.cuda(), w.gamma, w.rho, w.b,
                                  ldv=w.ldv)
    P.assert_scores_close(scores.cpu().numpy(), s_orc)
    o = P.oracle_inputs(w)
    ref = oracle.aggregate(0, o["V"], w.ldv, w.d, w.m, idx.cpu().numpy())
    assert P.rel_l2(out.cpu().numpy(), ref) <= P.AGG_RTOL


def test_lsq_unaligned(oracle):
    w = syn.make_config(5, d=4099, m=5, b=2, n_r=3, n_noise=2, ldv=4101)
    P.run_step_parity(oracle, w)


# the finish: one block or many, one lane or four per model, fewer and more models than a block's lanes
@pytest.mark.parametrize("d,n_r,m", [(500, 1, 1), (500, 8, 300), (3001, 9, 260), (20000, 8, 257), (20000, 33, 65), (70001, 9, 70)])
def test_lsq_finish_over_its_splits(oracle, d, n_r, m):
    w = syn.make_config(5, d=d, m=m, b=m // 3, n_r=n_r, n_noise=m // 3)
    P.run_step_parity(oracle, w)


def test_no_bias_model(oracle):
    w = syn.make_config(2, dims=(96, 24, 10), n_r=6, m=5, b=1, faults=[(1, "noise200")],
                        has_bias=False)
    P.run_step_parity(oracle, w)


# ---------------------------------------------------------------- properties on the GPU output

def _small():
    return syn.make_config(2, dims=(132, 40, 24, 10), n_r=12, m=10, b=4, faults=[(4, "noise200")])


def test_zero_update_scores_exactly_zero():
    w = _small()
    w.V[3, :w.d] = 0.0
    x, V, f, t = P.to_device(w)
    with zeno.from_workload(w) as z:
        s, losses, norms = z.score(x, V, f, t, w.gamma, w.rho)
    assert s[3].item() == 0.0 and norms[3].item() == 0.0 and losses[4].item() == losses[0].item()
    wl = syn.make_config(5, d=5000, m=4, b=1, n_r=16, n_noise=1)
    wl.V[2, :wl.d] = 0.0
    x, V, f, t = P.to_device(wl)
    with zeno.from_workload(wl) as z:
        s, losses, norms = z.score(x, V, f, t, wl.gamma, wl.rho)
    assert s[2].item() == 0.0


def test_b_zero_is_the_mean_and_b_m_minus_1_is_one_row():
    w = _small()
    x, V, f, t = P.to_device(w)
    with zeno.from_workload(w) as z:
        out0, _, idx0 = z.step(x, V, f, t, w.gamma, w.rho, 0)
        out1, s1, idx1 = z.step(x, V, f, t, w.gamma, w.rho, w.m - 1)
    assert sorted(idx0.tolist()) == list(range(w.m))
    mean = w.V[:, :w.d].double().mean(0).numpy()
    assert P.rel_l2(out0.cpu().numpy(), mean) <= P.AGG_RTOL
    best = int(torch.argmax(s1))
    assert idx1.tolist() == [best]
    assert torch.equal(out1.cpu(), w.V[best, :w.d])      # bit-exact copy of one input row


def test_permutation_invariance_and_duplicates():
    w = _small()
    w.V[7] = w.V[2]
    x, V, f, t = P.to_device(w)
    perm = torch.randperm(w.m, generator=torch.Generator().manual_seed(1))
    with zeno.from_workload(w) as z:
        out, s, idx = z.step(x, V, f, t, w.gamma, w.rho, w.b)
        out_p, s_p, idx_p = z.step(x, V[perm.cuda()].contiguous(), f, t, w.gamma, w.rho, w.b)
    assert s[7].item() == s[2].item()                    # duplicates score bit-identically
    assert torch.equal(s_p.cpu(), s.cpu()[perm])         # scores do not depend on the row position
    sel, sel_p = set(idx.tolist()), set(perm[idx_p.cpu().long()].tolist())
    # the two copies are interchangeable; everything else must agree
    canon = lambda S: {2 if i == 7 else i for i in S}
    assert canon(sel) == canon(sel_p)
    assert P.rel_l2(out_p.cpu().numpy(), out.cpu().numpy()) <= 1e-6


def test_lemma1_on_gpu_ranking():
    # Lemma 1: the k-th best score overall is at least the k-th best score inside any subset
    g = torch.Generator().manual_seed(5)
    s = torch.randn(200, generator=g)
    with zeno.Zeno(0, 0, (8, 4), m_max=256, n_r_max=4) as z:
        idx = z.select(s.cuda(), 0).cpu().long()
    ranked = s[idx]
    assert torch.all(ranked[:-1] >= ranked[1:])
    for size in (1, 17, 100, 200):
        sub = s[torch.randperm(200, generator=g)[:size]].sort(descending=True).values
        assert torch.all(ranked[:size] >= sub)


def test_jensen_step_on_gpu_outputs(oracle):
    # convex loss: f_r(x - gamma * Zeno_b(V)) <= mean of the selected candidates' losses
    w = syn.make_config(1)
    x, V, f, t = P.to_device(w)
    with zeno.from_workload(w) as z:
        out, s, idx = z.step(x, V, f, t, w.gamma, w.rho, w.b)
        _, losses, _ = z.score(x, V, f, t, w.gamma, w.rho)
        # evaluate f_r at x - gamma * out by presenting `out` as a single candidate
        V1 = torch.zeros(1, w.ldv, device="cuda"); V1[0, :w.d] = out
        _, l1, _ = z.score(x, V1, f, t, w.gamma, w.rho)
    assert l1[1].item() <= losses[1 + idx.long()].mean().item() + 1e-6


# ---------------------------------------------------------------- ranking alone: integer work, bit-exact

@pytest.mark.parametrize("m", [1, 2, 31, 32, 33, 100, 513, 1024])
def test_select_matches_oracle_bit_exactly(oracle, m):
    g = np.random.default_rng(m)
    s = g.standard_normal(m).astype(np.float32)
    if m >= 31:
        s[g.integers(0, m, m // 4)] = s[0]                 # exact ties
        s[g.integers(0, m, 3)] = np.nan
        s[g.integers(0, m, 2)] = -np.inf
        s[g.integers(0, m, 2)] = np.inf
        s[5], s[6] = 0.0, -0.0
    with zeno.Zeno(0, 0, (8, 4), m_max=1024, n_r_max=4) as z:
        for b in sorted({0, m // 3, m - 1}):
            idx = z.select(torch.from_numpy(s).cuda(), b).cpu().numpy()
            assert np.array_equal(idx, oracle.select(s.astype(np.float64), b))


# ---------------------------------------------------------------- faulty values stay contained

def test_non_finite_candidates_are_ranked_last_and_do_not_leak(oracle):
    w = _small()
    w.V[0, 5] = float("nan")
    w.V[4, 100] = float("inf")
    w.V[6, :w.d] = 1e30
    x, V, f, t = P.to_device(w)
    with zeno.from_workload(w) as z:
        out, s, idx = z.step(x, V, f, t, w.gamma, w.rho, 3)
    s_orc, _, _ = P.oracle_score(oracle, w)
    assert not set(idx.tolist()) & {0, 4, 6}
    assert torch.isfinite(out).all()
    good = [i for i in range(w.m) if i not in (0, 4, 6)]
    P.assert_scores_close(s.cpu().numpy()[good], s_orc[good])
    # NaN / Inf entries make the score non-finite on both sides; the 1e30 row overflows binary32
    # (score -inf) where float64 still holds -3e60: both rank it last
    assert not np.isfinite(s.cpu().numpy()[[0, 4, 6]]).any()
    assert not np.isfinite(s_orc[[0, 4]]).any() and s_orc[6] < -1e59


def test_aggregate_skips_out_of_range_indices():
    w = _small()
    V = w.V.cuda()
    idx = torch.tensor([1, -3, 2, 99], dtype=torch.int32, device="cuda")
    with zeno.from_workload(w) as z:
        out = z.aggregate(V, idx)
    ref = (w.V[1, :w.d].double() + w.V[2, :w.d].double()) / 4
    assert P.rel_l2(out.cpu().numpy(), ref.numpy()) <= P.AGG_RTOL


# ---------------------------------------------------------------- argument errors are status codes

def test_argument_errors():
    w = _small()
    x, V, f, t = P.to_device(w)
    with zeno.from_workload(w) as z:
        for kwargs in (dict(b=w.m), dict(b=-1)):
            with pytest.raises(zeno.ZenoError) as e:
                z.step(x, V, f, t, w.gamma, w.rho, **kwargs)
            assert e.value.status == zeno.ERR_INVALID_ARG
        for bad in (dict(gamma=float("nan")), dict(rho=-1.0), dict(rho=float("inf"))):
            args = dict(gamma=w.gamma, rho=w.rho); args.update(bad)
            with pytest.raises(zeno.ZenoError) as e:
                z.score(x, V, f, t, args["gamma"], args["rho"])
            assert e.value.status == zeno.ERR_INVALID_ARG
        with pytest.raises(zeno.ZenoError):
            z.score(x, V, f, t, w.gamma, w.rho, ldv=w.d - 1)
        with pytest.raises(zeno.ZenoError):
            z.score(x, V, f, t, w.gamma, w.rho, m=w.m + 1)          # beyond m_max
        # the handle still works after rejected calls
        out, s, idx = z.step(x, V, f, t, w.gamma, w.rho, w.b)
        assert torch.isfinite(out).all()


def test_host_entry_point_matches_device_entry_point():
    w = _small()
    x, V, f, t = P.to_device(w)
    out_h = torch.empty(w.d, dtype=torch.float32).pin_memory()
    s_h = torch.empty(w.m, dtype=torch.float32).pin_memory()
    i_h = torch.empty(w.m - w.b, dtype=torch.int32).pin_memory()
    with zeno.from_workload(w) as z:
        out, s, idx = z.step(x, V, f, t, w.gamma, w.rho, w.b)
        z.step_host(w.x.pin_memory(), w.V.pin_memory(), w.features.pin_memory(),
                    w.targets.pin_memory(), w.gamma, w.rho, w.b, out_h, s_h, i_h)
    assert torch.equal(out.cpu(), out_h) and torch.equal(s.cpu(), s_h) and torch.equal(idx.cpu(), i_h)


# Handles are independent of one another: two host threads run the server loops of two models whose last layers (and,
# with rows of no alignment, whose dense layers) are served by one kernel with different amounts of shared memory.
@pytest.mark.parametrize("dims,n_r", [(((3000, 10), (4096, 10)), 4), (((1029, 40), (300, 40)), 32)])
def test_two_handles_on_two_host_threads(dims, n_r):
    failures = []
    ready = threading.Barrier(2)

    def loops(one, steps=100):
        try:
            w = syn.make_config(2, dims=one, m=4, b=1, n_r=n_r, faults=[(1, "signflip")])
            with torch.cuda.stream(torch.cuda.Stream()), zeno.from_workload(w) as z:
                x, V, f, t = (v.repeat(steps, *([1] * v.dim())) if k else v for k, v in enumerate(P.to_device(w)))
                want = z.run(x, V, f, t, 0.0, w.rho, w.b)           # gamma = 0: x stays as it is
                ready.wait(60)
                for i in range(40):
                    got = z.run(x, V, f, t, 0.0, w.rho, w.b)
                    if not all(torch.equal(a, b) for a, b in zip(got, want)):
                        failures.append((one, i))
        except Exception as e:
            failures.append((one, e))
            ready.abort()

    threads = [threading.Thread(target=loops, args=(one,)) for one in dims]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not failures, failures


# more candidates than the averaging kernel ranks, and least squares: both passes end in the block that takes the last
# ticket, which the workspace has to hold zero for
@pytest.mark.parametrize("index,ov", [(1, dict(m=300, b=8)), (5, dict(d=20000, m=12, b=4, n_r=16, n_noise=4))])
def test_a_new_handle_is_ready_for_any_stream(index, ov):
    """zeno_create has cleared its workspace when it returns: calls on a stream that waits for no other are right while
    the default stream still has work ahead of anything queued there, and when that work ends."""
    w = syn.make_config(index, **ov)
    x, V, f, t = (v.repeat(4, *([1] * v.dim())) if k else v for k, v in enumerate(P.to_device(w)))
    with zeno.from_workload(w) as z:
        want, _ = z.run(x, V, f, t, 0.0, w.rho, w.b)                # gamma = 0: x stays as it is
    side = torch.cuda.Stream()
    scores = [torch.empty_like(want) for _ in range(200)]
    for _ in range(10):
        for s in scores:
            s.fill_(-1)
        torch.cuda.synchronize()
        torch.cuda._sleep(20_000_000)                               # some 10 ms
        with zeno.from_workload(w) as z, torch.cuda.stream(side):
            for s in scores:
                z.run(x, V, f, t, 0.0, w.rho, w.b, scores=s)
            torch.cuda.synchronize()
        assert all(torch.equal(s, want) for s in scores)
