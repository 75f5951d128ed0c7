"""GPU parity of the baseline aggregation rules (Experiments, "Baselines": marginal Median, Krum_b) against
the float64 oracle, through the C ABI, on the same seeded candidate matrices the Zeno tests use."""
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


CASES = {
    "cfg1": (1, dict()),                                                       # m = 20: one lane a column
    "cfg2_small_odd_m": (2, dict(dims=(300, 72, 40, 10), n_r=9, m=7, b=2, faults=[(2, "noise200")])),
    "cfg3_m37": (3, dict(dims=(260, 44, 36, 10), m=37, b=15, n_r=7, faults=[(7, "signflip"), (8, "omniscient")])),  # two lanes a column
    "cfg3_m100": (3, dict(dims=(132, 40, 10), m=100, b=40, n_r=5, faults=[(20, "signflip"), (20, "omniscient")])),  # four lanes a column
    "cfg4_bf16": (4, dict(dims=(264, 136, 72, 50), m=9, b=3, n_r=19, faults=[(3, "signflip")])),
    "cfg5_small": (5, dict(d=70001, m=13, b=5, n_r=16, n_noise=5, ldv=70003)),   # unaligned rows
}


# every compiled variant of the sorting network (columns of 8 .. 32 slots in one lane, then 2 .. 32 lanes a
# column) at, below and above its limits, in both storage types; d leaves a ragged last group of columns
MEDIAN_M = [1, 2, 3, 4, 7, 8, 9, 12, 13, 16, 17, 20, 21, 24, 25, 28, 29, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255,
            256, 257, 500, 512, 513, 1000, 1024]


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_median_every_network(oracle, dtype):
    for m in MEDIAN_M:
        if dtype == "fp32":
            w = syn.make_config(5, d=301, m=m, b=0, n_r=4, n_noise=0, ldv=307, seed=1000 + m)
            dt = 0
        else:
            w = syn.make_config(4, dims=(10, 13, 10), m=m, b=0, n_r=4, faults=[], seed=1000 + m)
            dt = 1
        if m >= 5:                                  # ties and special values in some columns
            w.V[1, 0] = w.V[0, 0]
            w.V[m - 1, 1] = float("inf")
            w.V[m // 2, 2] = float("-inf")
            w.V[2, 3] = float("nan")
        want = oracle.median(dt, syn.to_numpy_params(w.V), w.ldv, w.d, w.m)
        with zeno.from_workload(w) as z:
            got = z.median(w.V.cuda()).cpu().numpy().astype(np.float64)
        fin = np.isfinite(want)
        assert np.array_equal(got[~fin], want[~fin]), m
        if m % 2 == 1:
            assert np.array_equal(got, want), (m, np.flatnonzero(got != want)[:5])     # a selection, exactly
        else:                                       # the mean of two stored values formed in binary32: one rounding
            assert np.all(np.abs(got[fin] - want[fin]) <= 1.2e-7 * np.maximum(np.abs(want[fin]), 1e-30) + 1e-45), m


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("ldv_pad", [0, 1])         # rows of an odd pitch: bfloat16 columns are read one by one
def test_median_padded_halves(oracle, dtype, ldv_pad):
    """Columns of 34 .. 126 candidates, padded to the next compiled size by up to seven infinities of both signs,
    with real infinities and NaN beside the padding; d = 515 and 516 leave an odd and an even last tile."""
    for m in (34, 36, 39, 40, 41, 47, 50, 57, 72, 73, 90, 99, 105, 112, 113, 120, 121, 126):
        d = 515 + m % 2
        w = syn.make_config(5, d=d, m=m, b=0, n_r=4, n_noise=0, ldv=d + (d + ldv_pad) % 2, seed=3000 + m)
        V = w.V.to(torch.bfloat16) if dtype == "bf16" else w.V
        V[:, 7] = float("inf")
        V[: m // 2 + 1, 8] = float("-inf")
        V[::3, 9] = float("nan")
        V[:, d - 1] = torch.arange(m).to(V.dtype)
        want = oracle.median(int(dtype == "bf16"), syn.to_numpy_params(V), w.ldv, d, m)
        kind, desc = (0, ((d - 2) // 2, 2) if d % 2 == 0 else (d - 1, 1)) if dtype == "bf16" else (1, (d, 1))
        with zeno.Zeno(kind, int(dtype == "bf16"), desc, True, m, 4) as z:
            assert z.d == d
            got = z.median(V.cuda()).cpu().numpy().astype(np.float64)
        fin = np.isfinite(want)
        assert np.array_equal(got[~fin], want[~fin]), m
        if m % 2 == 1:
            assert np.array_equal(got, want), m
        else:                                       # the mean of two stored values formed in binary32: one rounding
            assert np.all(np.abs(got[fin] - want[fin]) <= 1.2e-7 * np.maximum(np.abs(want[fin]), 1e-30) + 1e-45), m


@pytest.mark.parametrize("name", sorted(CASES))
def test_median_matches_oracle(oracle, name):
    index, ov = CASES[name]
    w = syn.make_config(index, **ov)
    dt = P.DTYPE[w.dtype]
    want = oracle.median(dt, syn.to_numpy_params(w.V), w.ldv, w.d, w.m)
    with zeno.from_workload(w) as z:
        got = z.median(w.V.cuda()).cpu().numpy().astype(np.float64)
    if w.m % 2 == 1:
        assert np.array_equal(got, want)            # a selection: the value of one input entry, exactly
    else:
        # the mean of two stored values, formed in binary32: one rounding
        assert np.all(np.abs(got - want) <= 1.2e-7 * np.maximum(np.abs(want), 1e-30) + 1e-45)
    assert P.rel_l2(got, want) <= 1e-6


def test_median_special_values(oracle):
    w = syn.make_config(1, dims=(64, 12), m=5, b=1, faults=[(1, "signflip")])
    w.V[0, 3] = float("nan")
    w.V[1, 3] = float("nan")
    w.V[2, 3] = float("nan")                        # three of five are NaN: the median is +inf
    w.V[4, 7] = float("inf")
    w.V[3, 9] = -float("inf")
    want = oracle.median(0, syn.to_numpy_params(w.V), w.ldv, w.d, w.m)
    with zeno.from_workload(w) as z:
        got = z.median(w.V.cuda()).cpu().numpy().astype(np.float64)
    assert np.array_equal(got, want) and got[3] == np.inf


@pytest.mark.parametrize("name", sorted(CASES))
def test_krum_matches_oracle(oracle, name):
    index, ov = CASES[name]
    w = syn.make_config(index, **ov)
    dt = P.DTYPE[w.dtype]
    b = min(w.b, w.m - 3)
    k_orc, sums_orc, _ = oracle.krum(dt, syn.to_numpy_params(w.V), w.ldv, w.d, w.m, b)
    with zeno.from_workload(w) as z:
        out, k, sums = z.krum(w.V.cuda(), b)
        torch.cuda.synchronize()
    sums = sums.cpu().numpy().astype(np.float64)
    k = int(k.item())
    assert np.allclose(sums, sums_orc, rtol=2e-5, atol=0)
    # the arg min decides an integer: identical wherever the oracle's best two sums are clearly apart,
    # otherwise any candidate whose sum is the minimum up to the tolerance (identical rows tie exactly)
    order = np.argsort(sums_orc, kind="stable")
    if sums_orc[order[1]] - sums_orc[order[0]] > 1e-4 * abs(sums_orc[order[0]]):
        assert k == k_orc
    else:
        assert sums_orc[k] <= sums_orc[order[0]] * (1 + 1e-4)
    assert k == int(np.argmin(sums))                # on its own sums the choice is exact, lowest index first
    assert torch.equal(out.cpu(), w.V[k, :w.d].float())


# one tile in flight and two, the last size of either, the first with several pair tiles a thread, the most candidates;
# ties of identical rows, a row of infinite distances, odd pitches
@pytest.mark.parametrize("m,b,dtype", [(3, 0, "f32"), (5, 1, "f32"), (64, 20, "f32"), (65, 20, "f32"), (88, 3, "f32"), (89, 30, "f32"),
                                       (128, 50, "f32"), (20, 8, "bf16"), (128, 50, "bf16")])
def test_krum_over_its_sizes(oracle, m, b, dtype):
    w = syn.make_config(1, dims=(333, 7), m=m, b=b, dtype=dtype, ldv=2351, faults=[(b, "noise200")] if b else [], seed=77 + m)
    assert w.ldv >= w.d
    w.V[1] = w.V[0]
    if m > 5:
        w.V[4, 11] = float("nan")
    k_orc, sums_orc, _ = oracle.krum(P.DTYPE[dtype], syn.to_numpy_params(w.V), w.ldv, w.d, m, b)
    with zeno.from_workload(w) as z:
        out, k, sums = z.krum(w.V.cuda(), b)
        none, k2, _ = z.krum(w.V.cuda(), b, want_out=False)
    assert none is None and k2.item() == k.item()
    sums = sums.cpu().numpy().astype(np.float64)
    fin = np.isfinite(sums_orc)
    assert np.array_equal(sums[~fin], sums_orc[~fin])
    assert np.allclose(sums[fin], sums_orc[fin], rtol=2e-5, atol=0)
    assert k.item() == int(np.argmin(sums))
    assert torch.equal(out.cpu(), w.V[k.item(), :w.d].float())


# the last size of every block of rows and the first of the next, one stretch of columns and several, copies of 16 and of 4
# bytes, bfloat16 rows that start in either half of 4 bytes
@pytest.mark.parametrize("m", [3, 6, 7, 10, 11, 14, 15, 16, 17, 20, 21, 28, 29, 40, 42, 43, 70, 71, 96, 97, 100, 112, 113, 120, 121])
@pytest.mark.parametrize("dtype,d,pad", [("f32", 2346, 2), ("f32", 515, 0), ("bf16", 2346, 6), ("bf16", 515, 0), ("bf16", 1026, 0)])
def test_krum_over_its_tiles(oracle, m, dtype, d, pad):
    w = syn.make_config(5, d=d, m=m, b=0, n_r=2, n_noise=0, ldv=d + pad, seed=500 + m)
    V = w.V.to(torch.bfloat16) if dtype == "bf16" else w.V
    V[:, d:] = float("nan")
    V[m - 1] = V[0]                                 # identical rows of two blocks: equal distances, the lower index wins
    V[m // 2, d - 1] += 3
    b = min(m // 3, m - 3)
    _, sums_orc, _ = oracle.krum(int(dtype == "bf16"), syn.to_numpy_params(V), w.ldv, d, m, b)
    kind, desc = (0, ((d - 2) // 2, 2) if d % 2 == 0 else (d - 1, 1)) if dtype == "bf16" else (1, (d, 1))
    with zeno.Zeno(kind, int(dtype == "bf16"), desc, True, m, 4) as z:
        assert z.d == d
        out, k, sums = z.krum(V.cuda(), b)
    sums = sums.cpu().numpy().astype(np.float64)
    # sums of d squares in binary32: relative error below d / lanes * 2^-24, far within
    assert np.allclose(sums, sums_orc, rtol=2e-5, atol=0)
    assert k.item() == int(np.argmin(sums))
    assert sums[0] == sums[m - 1]
    assert torch.equal(out.cpu(), V[k.item(), :d].float())


# every stage of the ring of staged columns used again and again, the last one ragged: at least five stretches a block, of 64 to
# 256 columns; few candidates and many; copies of 16 and of 4 bytes, rows of odd pitch and rows that start at an odd entry (bfloat16:
# in the second half of 4 bytes, in turn or all of them).  Two identical rows are the best ones: the first of them wins
@pytest.mark.parametrize("m,d,b", [(20, 400004, 6), (42, 130004, 20), (48, 40004, 10), (64, 100004, 21), (96, 60004, 8), (128, 24004, 50)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("pad,start", [(4, 0), (5, 0), (4, 1), (5, 1)])
def test_krum_of_many_columns(oracle, m, d, b, dtype, pad, start):
    krum_with_two_best_rows(oracle, m, d, b, dtype, pad, start)


# the last sizes 4 x 4 pairs a thread take, and the first beyond, either way: 96 columns for every SM (128 where rows are not aligned,
# 48 with 49 to 88 candidates; 768 for many), 12, 42, 48, 56, 88, 97, 124 candidates and their neighbours, one and two tiles a thread,
# stretches with a remainder, one and several groups of threads
@pytest.mark.parametrize("m,d,pad,start", [(m, *shape) for m in (12, 13, 24, 42, 43, 48, 49) for shape in
                                           ((300, 0, 0), (1027, 0, 1), (14208, 0, 0), (14216, 0, 0), (18943, 0, 0), (18945, 0, 0))] +
                         [(m, d, 1, 0) for m in (49, 88, 89) for d in (7104, 7106)] +
                         [(m, d, 1, 0) for m in (57, 60, 61, 69, 88, 89, 97, 98, 112, 124, 125) for d in (113664, 113666)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_krum_by_either_kernel(oracle, m, dtype, d, pad, start):
    krum_with_two_best_rows(oracle, m, d, m // 3, dtype, pad, start)


# the same for the fewest candidates, for 43 to 89 of them, where few columns go back to the register tiles, and for about 100: the
# numbers of columns for every SM at which the kernels take turns
@pytest.mark.parametrize("m,d,pad,start", [(m, d, pad, 0) for m in (6, 7, 10, 11, 12) for d, pad in ((2368, 0), (2376, 0), (7103, 0), (7105, 0), (11839, 0), (11841, 0))] +
                         [(m, d, pad, 0) for m in (43, 49, 60, 61) for d, pad in ((6512, 0), (6520, 0), (14800, 0), (14808, 0))] +
                         [(m, d, 1, 0) for m, lo, hi in ((49, 32, 88), (56, 32, 88), (57, 0, 112), (60, 0, 112), (64, 36, 84), (65, 36, 84), (72, 36, 84), (73, 40, 64),
                                                         (88, 40, 64), (89, 40, 64)) for d in (148 * lo, 148 * lo + 2, 148 * hi, 148 * hi + 2) if d >= 4] +
                         [(m, d, 1, 0) for m in (96, 97, 102, 108, 109) for d in (94720, 94722)] + [(m, d, 1, 0) for m in (57, 88, 109) for d in (151552, 151554)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_krum_by_either_kernel_with_few_and_many_candidates(oracle, m, dtype, d, pad, start):
    krum_with_two_best_rows(oracle, m, d, m // 3, dtype, pad, start)


def krum_with_two_best_rows(oracle, m, d, b, dtype, pad, start):
    store = torch.bfloat16 if dtype == "bf16" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(m + d)
    ldv = d + pad
    room = torch.full((start + m * ldv,), float("nan"), dtype=store, device="cuda")
    V = room[start:].view(m, ldv)
    V[:, :d] = torch.randn(d, generator=g, device="cuda").to(store)
    V[1:m - 1, :d] += (torch.randn((m - 2, d), generator=g, device="cuda") * torch.linspace(0.5, 0.8, m - 2, device="cuda")[:, None]).to(store)
    kind, dims = (0, ((d - 2) // 2, 2) if d % 2 == 0 else (d - 1, 1)) if dtype == "bf16" else (1, (d, 1))
    _, sums_orc, _ = oracle.krum(int(dtype == "bf16"), syn.to_numpy_params(V.cpu()), ldv, d, m, b)
    with zeno.Zeno(kind, int(dtype == "bf16"), dims, True, m, 1) as z:
        assert z.d == d
        out, k, sums = z.krum(V, b, ldv=ldv)
    sums = sums.cpu().numpy().astype(np.float64)
    # chains of up to d / 32 squares of one sign in binary32: far within
    assert np.allclose(sums, sums_orc, rtol=2e-5, atol=0)
    assert sums[0] == sums[m - 1] and k.item() == 0
    assert torch.equal(out, V[0, :d].float())


def test_krum_toy_example_on_the_gpu():
    # Discussion, the one-dimensional toy example: Krum_2({-1, -1, 0.2, 0.4, 1.6, 1.8}) = -1
    V = torch.tensor([[-1.0], [-1.0], [0.2], [0.4], [1.6], [1.8]])
    with zeno.Zeno(1, 0, (1, 1), m_max=6, n_r_max=1) as z:
        out, k, sums = z.krum(V.cuda(), 2)
    assert out.item() == -1.0 and k.item() == 0
    assert sums[0].item() == pytest.approx(1.44, rel=1e-6)


def test_krum_argument_errors_and_limits():
    w = syn.make_config(1, dims=(64, 12), m=6, b=2, faults=[(2, "signflip")])
    V = w.V.cuda()
    with zeno.from_workload(w) as z:
        with pytest.raises(zeno.ZenoError) as e:
            z.krum(V, 4)                            # m - b - 2 = 0 neighbours
        assert e.value.status == zeno.ERR_INVALID_ARG
        with pytest.raises(zeno.ZenoError) as e:
            z.krum(V, -1)
        assert e.value.status == zeno.ERR_INVALID_ARG
    w2 = syn.make_config(1, dims=(16, 4), m=130, b=8, faults=[(8, "signflip")])
    with zeno.from_workload(w2) as z:
        with pytest.raises(zeno.ZenoError) as e:
            z.krum(w2.V.cuda(), 8)
        assert e.value.status == zeno.ERR_UNSUPPORTED
        assert torch.isfinite(z.median(w2.V.cuda())).all()      # the median has no such limit
