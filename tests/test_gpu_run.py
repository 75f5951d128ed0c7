"""zeno_run, Algorithm 1's server loop on the device, against the oracle's step and update chained on
the host: T iterations, each with its own candidates and its own batch, x carried from one to the next."""
import numpy as np
import pytest
import torch

from paper_1805_10032_b200 import synthetic as syn
from paper_1805_10032_b200 import zeno

import parity as P

pytestmark = pytest.mark.gpu

T = 3


@pytest.fixture(scope="module", autouse=True)
def _library():
    from paper_1805_10032_b200 import build as zbuild
    zbuild.build()
    assert torch.cuda.is_available(), "these tests need a CUDA device"
    zeno.load_library()


CASES = {
    "cfg1": (1, dict()),
    "cfg2_mid_layers": (2, dict(dims=(520, 200, 136, 10), n_r=21, m=6, b=2, faults=[(2, "noise200")])),
    "cfg4_small": (4, dict(dims=(264, 136, 72, 50), m=9, b=3, n_r=19, faults=[(3, "signflip")])),
    "cfg5_small": (5, dict(d=70000, m=13, b=5, n_r=16, n_noise=5)),
    "cfg6_cnn_small": (6, dict(dims=(8, 3, 8, 8, 12, 12, 10), m=7, b=2, n_r=5, faults=[(2, "signflip")])),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_server_loop_matches_the_chained_oracle(oracle, name):
    index, ov = CASES[name]
    ws = [syn.make_config(index, seed=syn.BASE_SEED + 31 * t + index, **ov) for t in range(T)]
    w = ws[0]
    V = torch.stack([s.V for s in ws]).cuda()
    feats = torch.stack([s.features for s in ws]).cuda()
    tgts = torch.stack([s.targets for s in ws]).cuda()
    x = w.x.cuda().clone()
    with zeno.from_workload(w) as z:
        scores, idx = z.run(x, V, feats, tgts, w.gamma, w.rho, w.b)
        launches = z.last_launch_count
        # the same loop, one call per iteration
        x2 = w.x.cuda().clone()
        for t in range(T):
            _, s2, i2 = z.step_update(x2, V[t], feats[t], tgts[t], w.gamma, w.rho, w.b, want_out=False)
            assert torch.equal(s2, scores[t]) and torch.equal(i2, idx[t])
        torch.cuda.synchronize()
        z.check_device_status()
    assert torch.equal(x, x2)
    assert launches >= 2 * T

    # the oracle's chain: the stored parameter vector is rounded to its storage type between iterations
    kind, dt = P.KIND[w.kind], P.DTYPE[w.dtype]
    gamma, rho = float(np.float32(w.gamma)), float(np.float32(w.rho))
    x_orc = syn.to_numpy_params(w.x)
    for t in range(T):
        Vt = syn.to_numpy_params(ws[t].V)
        f, tg = ws[t].features.numpy(), ws[t].targets.numpy()
        s_orc, f_orc, n_orc = oracle.score(kind, dt, w.dims, w.has_bias, x_orc, Vt, w.ldv, w.m, f, tg, gamma, rho)
        P.assert_scores_close(scores[t].cpu().numpy(), s_orc, f_orc, n_orc, rho)
        got_idx = idx[t].cpu().numpy()
        P.assert_selection_valid(got_idx, s_orc, w.b)
        vbar = oracle.aggregate(dt, Vt, w.ldv, w.d, w.m, got_idx)
        x_new = oracle.update(dt, x_orc, vbar, gamma)
        if w.dtype == "bf16":
            x_orc = syn.to_numpy_params(torch.from_numpy(x_new).to(torch.bfloat16))    # exact: already bfloat16 values
        else:
            x_orc = x_new.astype(np.float32)
    got = x.float().double().cpu().numpy()
    want = (torch.from_numpy(x_orc.view("int16")).view(torch.bfloat16).float().double().numpy()
            if w.dtype == "bf16" else x_orc.astype(np.float64))
    if w.dtype == "f32":
        assert P.rel_l2(got, want) <= T * 1e-6
    else:
        # a bfloat16 parameter may land on the neighbouring number at a rounding boundary, once per iteration
        ulp = np.maximum(np.abs(want), 2.0 ** -126) * 2.0 ** -7
        assert np.all(np.abs(got - want) <= T * ulp)
        assert np.mean(got == want) >= 0.99
    assert not torch.equal(x.cpu(), w.x)


# the loop of a small binary32 softmax regression: features staged whole and by stretch, a stretch with several classes and a
# class over several stretches, one and two copies of the candidates, more candidates than warps, one class and the most,
# samples of one and several passes, rows of every alignment, no bias, more iterations than the products of one launch
@pytest.mark.parametrize("dims,n_r,m,bias,pad,steps", [
    ((784, 10), 4, 20, True, 2, 5), ((33, 2), 1, 1, True, 1, 4), ((32, 32), 9, 5, True, 0, 4), ((40, 3), 64, 12, False, 0, 4),
    ((517, 16), 13, 31, True, 1, 4), ((600, 11), 5, 70, True, 3, 4), ((1023, 31), 4, 7, True, 1, 4), ((300, 1), 2, 16, True, 0, 4),
    ((4096, 4), 8, 15, True, 0, 4), ((20, 32), 6, 200, True, 0, 30), ((20, 5), 3, 200, True, 0, 4)])
def test_two_launch_loop_over_its_limits(oracle, dims, n_r, m, bias, pad, steps):
    b = m // 3
    ov = dict(dims=dims, n_r=n_r, m=m, b=b, has_bias=bias, ldv=syn.param_count("mlp", dims, bias) + pad, faults=[(b, "signflip")] if b else [])
    ws = [syn.make_config(1, seed=900 + t, **ov) for t in range(steps)]
    w = ws[0]
    x = w.x.cuda().clone()
    with zeno.from_workload(w) as z:
        scores, idx = z.run(x, torch.stack([s.V for s in ws]).cuda(), torch.stack([s.features for s in ws]).cuda(),
                            torch.stack([s.targets for s in ws]).cuda(), w.gamma, w.rho, w.b)
        assert z.last_launch_count == (4 if steps == 30 else 2)
    gamma, rho = float(np.float32(w.gamma)), float(np.float32(w.rho))
    x_orc = syn.to_numpy_params(w.x)
    for t in range(steps):
        Vt = syn.to_numpy_params(ws[t].V)
        s_orc, f_orc, n_orc = oracle.score(0, 0, w.dims, bias, x_orc, Vt, w.ldv, m, ws[t].features.numpy(), ws[t].targets.numpy(), gamma, rho)
        P.assert_scores_close(scores[t].cpu().numpy(), s_orc, f_orc, n_orc, rho)
        got_idx = idx[t].cpu().numpy()
        P.assert_selection_valid(got_idx, s_orc, b)
        x_orc = oracle.update(0, x_orc, oracle.aggregate(0, Vt, w.ldv, w.d, m, got_idx), gamma).astype(np.float32)
    assert P.rel_l2(x.cpu().numpy(), x_orc.astype(np.float64)) <= steps * 1e-6


@pytest.mark.parametrize("dims,n_r,m,pad", [((784, 10), 4, 20, 2), ((517, 16), 13, 31, 1), ((1023, 31), 4, 7, 0)])
def test_two_launch_loop_agrees_with_as_many_steps(dims, n_r, m, pad):
    """Scores to rounding: a tenth of what the oracle's comparison allows.  The average and the update are the same sums in rank
    order, so x differs by an addition's rounding where two rows of nearly equal scores change places, and no more."""
    steps, b = 6, m // 3
    ov = dict(dims=dims, n_r=n_r, m=m, b=b, ldv=syn.param_count("mlp", dims, True) + pad, faults=[(b, "signflip")])
    ws = [syn.make_config(1, seed=700 + t, **ov) for t in range(steps)]
    w = ws[0]
    x, y = w.x.cuda().clone(), w.x.cuda().clone()
    V, f, t = (torch.stack([getattr(s, k) for s in ws]).cuda() for k in ("V", "features", "targets"))
    with zeno.from_workload(w) as z:
        scores, idx = z.run(x, V, f, t, w.gamma, w.rho, b)
        assert z.last_launch_count == 2
        for i in range(steps):
            _, losses, norms = z.score(y, V[i], f[i], t[i], w.gamma, w.rho)
            _, want, want_idx = z.step_update(y, V[i], f[i], t[i], w.gamma, w.rho, b, want_out=False)
            assert torch.all((scores[i] - want).abs() <= 1e-5 * (losses[0].abs() + losses[1:].abs() + w.rho * norms))
            assert set(idx[i].tolist()) == set(want_idx.tolist())
    assert P.rel_l2(x.cpu().numpy(), y.double().cpu().numpy()) <= steps * 1e-7


def test_two_launch_loop_with_candidates_and_logits_that_overflow():
    """A candidate of NaN, one of infinities and one of 1e30 rank last in every iteration; logits of 1e10 keep a finite loss."""
    w = syn.make_config(1, dims=(50, 10), n_r=4, m=9, b=3, faults=[(3, "signflip")])
    bad = torch.nonzero(~w.honest).flatten().tolist()
    w.V[bad[0], 3], w.V[bad[1], 4], w.V[bad[2], :w.d] = float("nan"), float("inf"), 1e30
    V, f, t = w.V.repeat(5, 1, 1).cuda(), w.features.repeat(5, 1, 1).cuda(), w.targets.repeat(5, 1).cuda()
    for scale in (1.0, 1e10):
        x = (w.x * scale).cuda()
        with zeno.from_workload(w) as z:
            scores, idx = z.run(x, V, f, t, w.gamma, w.rho, 3)
            assert z.last_launch_count == 2
        assert not any(set(row) & set(bad) for row in idx.tolist())
        assert torch.isfinite(x).all() and torch.isfinite(scores[:, w.honest.cuda()]).all()


def test_run_argument_errors():
    w = syn.make_config(1)
    x, V, f, t = P.to_device(w)
    V3 = torch.stack([V, V]).contiguous()
    f3, t3 = torch.stack([f, f]).contiguous(), torch.stack([t, t]).contiguous()
    with zeno.from_workload(w) as z:
        lib = zeno.load_library()
        st = lib.zeno_run(z._h, x.data_ptr(), V3.data_ptr(), w.ldv, w.m * w.ldv - 1, w.m, f3.data_ptr(),
                          t3.data_ptr(), w.n_r, 2, 0.1, 5e-4, w.b, None, None, None)
        assert st == zeno.ERR_INVALID_ARG                      # iterations would overlap
        st = lib.zeno_run(z._h, x.data_ptr(), V3.data_ptr(), w.ldv, w.m * w.ldv, w.m, f3.data_ptr(),
                          t3.data_ptr(), w.n_r, 0, 0.1, 5e-4, w.b, None, None, None)
        assert st == zeno.ERR_INVALID_ARG                      # no iterations
        scores, idx = z.run(x.clone(), V3, f3, t3, w.gamma, w.rho, w.b)
        assert scores.shape == (2, w.m) and idx.shape == (2, w.m - w.b)


@pytest.mark.parametrize("cols,classes,m", [(20001, 2, 4), (9000, 3, 8)])
def test_loop_of_a_wide_model_adds_up_short_sums(cols, classes, m):
    """The products of a wide model's candidates against 64 bits: scores that are made of them (x is small beside gamma v).  A
    chain of n products of random signs is off by 0.41 x 2^-24 sqrt(n / 2) of its result in the root mean square: 4.5e-7 with
    all 625 of a lane's columns of 20,001, 1.4e-7 with 64 of them; the lanes' and the parts' additions, the rounding of x
    and of the score to binary32 add as much again."""
    steps, gamma = 12, 0.5
    g = torch.Generator().manual_seed(cols)
    d = cols * classes
    x = torch.randn(d, generator=g) * (1.0 / cols ** 0.5)
    V = torch.randn((steps, m, d), generator=g) * (3e4 / cols ** 0.5 / gamma)
    V[:, 0] = 0                                      # scores higher than candidates with losses of thousands
    feats = torch.randn((steps, 1, cols), generator=g)
    labels = torch.zeros((steps, 1), dtype=torch.int32)
    for t in range(steps):                           # the label: where the candidates' logits are small
        labels[t] = int((feats[t] @ V[t, 1:].sum(0).view(classes, cols).t()).argmax())
    xg = x.cuda()
    with zeno.Zeno(zeno.LOSS_SOFTMAX_MLP, zeno.F32, (cols, classes), False, m, 1) as z:
        scores, idx = z.run(xg, V.cuda(), feats.cuda(), labels.cuda(), gamma, 0.0, m - 1)
        assert z.last_launch_count == 2
    scores, idx = scores.double().cpu(), idx.cpu()
    err, count = 0.0, 0
    for t in range(steps):
        def loss(w):
            return torch.nn.functional.cross_entropy(feats[t].double() @ w.view(classes, cols).t(), labels[t].long())
        f0 = loss(x.double())
        for i in range(1, m):
            err += (scores[t, i] - (f0 - loss(x.double() - gamma * V[t, i].double()))).item() ** 2
            count += 1
        x = (x.double() - gamma * V[t, idx[t, 0]].double()).float()
    assert torch.allclose(xg.cpu(), x, rtol=1e-6, atol=1e-3)
    # a loss is the difference of two logits of 3e4, or nothing
    assert (err / count) ** 0.5 / (3e4 * 2 ** 0.5) <= 3.2e-7


def test_handles_of_small_models_are_small():
    """The loop's products have no room of their own beyond a few iterations': 64 handles of the smallest model."""
    handles = [zeno.Zeno(zeno.LOSS_SOFTMAX_MLP, zeno.F32, (784, 10), True, 20, 4)]
    before = torch.cuda.mem_get_info()[0]
    handles += [zeno.Zeno(zeno.LOSS_SOFTMAX_MLP, zeno.F32, (784, 10), True, 20, 4) for _ in range(64)]
    used = before - torch.cuda.mem_get_info()[0]
    for z in handles:
        z.close()
    assert used <= 64 * (2 << 20)


FIRST_CALL = """
import sys, torch
sys.path[:0] = [{root!r}, {tests!r}]
from paper_1805_10032_b200 import synthetic as syn, zeno
w = syn.make_config(1)
V, f, t = (v.repeat(6, *([1] * v.dim())).cuda() for v in (w.V, w.features, w.targets))
with zeno.from_workload(w) as z, zeno.from_workload(w) as other:
    x, y = w.x.cuda(), w.x.cuda()
    scores, idx = torch.zeros((6, w.m), device="cuda"), torch.zeros((6, w.m - w.b), dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        z.run(x, V, f, t, w.gamma, w.rho, w.b, scores=scores, idx=idx)
    assert z.last_launch_count == 2
    g.replay()
    want, want_idx = other.run(y, V, f, t, w.gamma, w.rho, w.b)
    torch.cuda.synchronize()
    assert torch.equal(x, y) and torch.equal(scores, want) and torch.equal(idx, want_idx)
    # Krum in between uses the same room
    other.krum(w.V.cuda(), w.b)
    y = w.x.cuda()
    again, _ = other.run(y, V, f, t, w.gamma, w.rho, w.b)
    assert torch.equal(x, y) and torch.equal(scores, again)
print("captured")
"""


def test_the_first_loop_of_a_process_can_be_captured():
    import os
    import subprocess
    import sys
    tests = os.path.dirname(os.path.abspath(__file__))
    out = subprocess.run([sys.executable, "-c", FIRST_CALL.format(root=os.path.dirname(tests), tests=tests)], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and "captured" in out.stdout, out.stderr[-2000:]
