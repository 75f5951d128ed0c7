"""GPU parity of the convolutional loss (ZENO_LOSS_SOFTMAX_CNN: the model family of the paper's own
experiment, a CNN of four convolutional layers and a dense one) against the float64 oracle, through the
C ABI: whole steps (score, ranking, trimmed mean), the pieces, shapes that leave ragged blocks (planes that
do not fill a block, channel counts that are no multiples of the block's sixteen planes or of the eight
staged at a time, a last group of samples that is not full), both storage types."""
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
    # the experiment's shape at a size the oracle finishes in seconds
    "paper_shape_small": dict(dims=(32, 3, 32, 32, 64, 64, 10), m=6, b=2, n_r=3, faults=[(2, "signflip")]),
    "two_layers": dict(dims=(8, 2, 5, 7, 4), m=7, b=3, n_r=5, faults=[(3, "noise200")]),
    "odd_channels_16x16": dict(dims=(16, 3, 9, 17, 20, 33, 10), m=5, b=2, n_r=6, faults=[(2, "signflip")]),
    "side_12_six_layers": dict(dims=(24, 1, 4, 4, 6, 6, 8, 8, 5), m=4, b=1, n_r=9, faults=[(1, "omniscient")]),
    "many_samples": dict(dims=(8, 3, 8, 8, 12, 12, 10), m=9, b=3, n_r=37, faults=[(3, "signflip")]),
    "no_bias": dict(dims=(16, 3, 8, 8, 10), m=5, b=1, n_r=4, faults=[(1, "signflip")], has_bias=False),
    "bf16": dict(dims=(16, 3, 16, 16, 24, 24, 10), m=6, b=2, n_r=5, faults=[(2, "signflip")], dtype="bf16"),
    "wide_head": dict(dims=(8, 3, 8, 8, 40), m=5, b=2, n_r=4, faults=[(2, "signflip")]),     # 40 classes: separate loss kernel
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_step_matches_oracle(oracle, name):
    w = syn.make_config(6, **CASES[name])
    r = P.run_step_parity(oracle, w)
    assert r["agg_err"] <= P.AGG_RTOL


# one tile and many, a pair of tiles half empty, more than 64 output planes (two items), up to four input planes (paired
# taps) and more, sides whose lines end inside a tile, planes that are no multiple of a group, unaligned rows
@pytest.mark.parametrize("dims,n_r,dtype", [((2, 1, 1, 1, 2), 1, "f32"), ((4, 5, 3, 70, 3), 2, "bf16"), ((28, 1, 5, 13, 10), 3, "f32"),
                                            ((32, 4, 66, 130, 7), 2, "f32"), ((14, 3, 33, 10, 10), 17, "f32"),
                                            ((30, 2, 8, 20, 11), 5, "bf16"), ((16, 9, 16, 16, 40, 40, 43), 6, "f32")])
def test_tensor_core_layers_over_their_limits(oracle, dims, n_r, dtype):
    d = syn.param_count("cnn", dims)
    w = syn.make_config(6, dims=dims, n_r=n_r, dtype=dtype, m=5, b=2, faults=[(2, "signflip")], ldv=d + (d + 1) % 2)
    P.run_step_parity(oracle, w)


def test_fewer_samples_and_candidates_than_the_handle_was_made_for(oracle):
    """The padding stays zero and nothing of a larger call is read by a smaller one."""
    w = syn.make_config(6, dims=(16, 3, 8, 8, 12, 12, 10), m=9, b=3, n_r=11, faults=[(3, "signflip")])
    x, V, f, t = P.to_device(w)
    with zeno.from_workload(w) as z, zeno.Zeno(zeno.LOSS_SOFTMAX_CNN, zeno.F32, w.dims, True, 4, 3) as small:
        z.score(x, V * float("nan"), f, t, w.gamma, w.rho)
        got = z.score(x, V[:4], f[:3].contiguous(), t[:3], w.gamma, w.rho)
        want = small.score(x, V[:4], f[:3].contiguous(), t[:3], w.gamma, w.rho)
        assert all(torch.equal(a, b) for a, b in zip(got, want))


def test_models_in_groups():
    """More models than the convolutional workspace holds (4 GiB) are taken in groups: every candidate's loss, norm and
    score as a handle for fewer candidates gives them; and what the two handles take of the device's memory."""
    w = syn.make_config(6, dims=(32, 3, 32, 32, 10), m=99, b=4, n_r=128, faults=[(4, "signflip")])
    x, V, f, t = P.to_device(w)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    with zeno.from_workload(w) as z, zeno.Zeno(zeno.LOSS_SOFTMAX_CNN, zeno.F32, w.dims, True, 25, 128) as few:
        used = free - torch.cuda.mem_get_info()[0]
        scores, losses, norms = z.score(x, V, f, t, w.gamma, w.rho)
        for i in range(0, 99, 25):
            part = few.score(x, V[i:i + 25], f, t, w.gamma, w.rho)
            # the dense layer deals its 8,192 inputs out to more blocks where there are fewer models: other partial sums
            for got, want in zip(part, (scores[i:i + 25], torch.cat([losses[:1], losses[1 + i:26 + i]]), norms[i:i + 25])):
                assert torch.allclose(got, want, rtol=2e-6, atol=0)
        z.check_device_status()
    # all models at once: 5.3 GB and 1.4 GB, beside them 0.5 GB of the dense layer's input
    assert used < 4 * 2 ** 30 + 2.1e9, used


# the first pixel of a sample is read, with zero weights, by the paired taps of the sample before it (one to four input
# planes); five planes: no paired taps
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("planes", [1, 3, 4, 5])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_a_smaller_batch_reads_no_pixel_of_a_larger_one(dtype, planes, value):
    w = syn.make_config(6, dims=(8, planes, 8, 8, 10), m=4, b=1, n_r=5, faults=[(1, "signflip")], dtype=dtype)
    x, V, f, t = P.to_device(w)
    bad = f.clone().view(5, planes, 8, 8)
    with zeno.from_workload(w) as z, zeno.from_workload(w) as fresh:
        for n in (1, 2, 4):
            bad[n, :, 0, 0] = value
            z.score(x, V, bad.view_as(f), t, w.gamma, w.rho)
            got = z.score(x, V, f[:n].contiguous(), t[:n], w.gamma, w.rho)
            want = fresh.score(x, V, f[:n].contiguous(), t[:n], w.gamma, w.rho)
            assert all(torch.isfinite(v).all() for v in want)
            assert all(torch.equal(a, b) for a, b in zip(got, want))


# Both convolution kernels against 64 bits.  A loss is rounded to binary32 (up to 6e-8 of it) after some thousand binary32
# roundings per logit whose signs are random; measured rms 3e-8 to 7e-8 and mean up to 3e-8 over networks and inputs.
# A systematic error shows in the mean: the truncation of the tensor core's sums alone, not added back, is 2.4e-7 (binary32
# weights) and 1.3e-7 (bfloat16) for these four layers.
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("images", ["both signs", "positive", "large mean"])
@pytest.mark.parametrize("cuda_cores", [False, True])
def test_losses_against_64_bits(oracle, monkeypatch, dtype, images, cuda_cores):
    if cuda_cores:
        monkeypatch.setenv("ZENO_DISABLE_TENSOR_CORES", "1")
    errors = []
    for dims in [(16, 3, 16, 16, 32, 32, 10), (16, 1, 24, 24, 40, 40, 10)]:
        w = syn.make_config(6, dims=dims, m=12, b=4, n_r=16, dtype=dtype, faults=[(4, "signflip")], seed=5 + dims[2])
        if images != "both signs":
            w.features = w.features.abs() if images == "positive" else w.features + 3.0
        _, f_orc, _ = P.oracle_score(oracle, w)
        with zeno.from_workload(w) as z:
            _, losses, _ = z.score(*P.to_device(w), w.gamma, w.rho)
        errors.append((losses.cpu().numpy().astype(np.float64) - f_orc) / f_orc)
    errors = np.concatenate(errors)
    assert np.sqrt((errors ** 2).mean()) <= 1.2e-7 and abs(errors.mean()) <= 7e-8, (errors.mean(), errors)


def test_cuda_core_layers(oracle, monkeypatch):
    """The kernel that serves without tensor cores."""
    monkeypatch.setenv("ZENO_DISABLE_TENSOR_CORES", "1")
    w = syn.make_config(6, dims=(16, 3, 9, 17, 20, 33, 10), m=5, b=2, n_r=6, faults=[(2, "signflip")])
    P.run_step_parity(oracle, w)


def test_kernels_of_the_step():
    w = syn.make_config(6, dims=(16, 3, 8, 8, 12, 12, 10), m=5, b=2, n_r=4, faults=[(2, "signflip")])
    x, V, f, t = P.to_device(w)
    with zeno.from_workload(w) as z:
        z.profile(True)
        z.step(x, V, f, t, w.gamma, w.rho, w.b)
        names = [n for n, _ in z.profile_read(0)]
        z.profile(False)
    assert names == ["cnn_conv3x3"] * 4 + ["mlp_head_loss_tail", "aggregate"], names


def test_description_errors():
    ok = (16, 3, 8, 8, 10)
    for dims in [(16, 3, 8, 10),              # an odd number of convolutional layers
                 (34, 3, 8, 8, 10),           # planes larger than 32 x 32
                 (6, 3, 8, 8, 8, 8, 10),      # 6 -> 3: odd before the second pooling
                 (15, 3, 8, 8, 10)]:          # an odd side
        with pytest.raises(zeno.ZenoError) as e:
            zeno.Zeno(zeno.LOSS_SOFTMAX_CNN, zeno.F32, dims, True, 4, 4)
        assert e.value.status == zeno.ERR_INVALID_ARG, dims
    z = zeno.Zeno(zeno.LOSS_SOFTMAX_CNN, zeno.F32, ok, True, 4, 4)
    assert z.d == syn.param_count("cnn", ok)
    z.close()


def test_nan_pixel_and_nan_candidate(oracle):
    w = syn.make_config(6, dims=(8, 2, 4, 4, 5), m=5, b=2, n_r=3, faults=[(2, "signflip")])
    w.V[1, 7] = float("nan")                         # a candidate with a NaN entry ranks last
    s_orc, f_orc, n_orc = P.oracle_score(oracle, w)
    x, V, f, t = P.to_device(w)
    with zeno.from_workload(w) as z:
        out, scores, idx = z.step(x, V, f, t, w.gamma, w.rho, w.b)
    s = scores.cpu().numpy()
    assert np.isnan(s[1]) and np.isnan(s_orc[1])
    assert 1 not in idx.cpu().tolist()
    ok = ~np.isnan(s_orc)
    assert np.allclose(s[ok], s_orc[ok], rtol=1e-3, atol=1e-6)


def test_host_buffers(oracle):
    """zeno_step_host with the convolutional model: the batch is [n_r][C_0][S][S] values per step."""
    w = syn.make_config(6, dims=(8, 3, 8, 8, 10), m=5, b=2, n_r=3, faults=[(2, "signflip")])
    out = torch.empty(w.d, dtype=torch.float32).pin_memory()
    scores = torch.empty(w.m, dtype=torch.float32).pin_memory()
    idx = torch.empty(w.m - w.b, dtype=torch.int32).pin_memory()
    with zeno.from_workload(w) as z:
        z.step_host(w.x.pin_memory(), w.V.pin_memory(), w.features.contiguous().pin_memory(), w.targets.pin_memory(),
                    w.gamma, w.rho, w.b, out, scores=scores, idx=idx)
        x, V, f, t = P.to_device(w)
        out_d, scores_d, idx_d = z.step(x, V, f, t, w.gamma, w.rho, w.b)
    assert torch.equal(out, out_d.cpu()) and torch.equal(scores, scores_d.cpu()) and torch.equal(idx, idx_d.cpu())
