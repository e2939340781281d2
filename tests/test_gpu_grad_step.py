"""GPU parity: the worker gradient step against the CPU oracle, through the C ABI."""
import numpy as np
import pytest

from paper_2406_05546_b200 import synth
from tests.parity import (TOL_FP32, TOL_TENSOR, assert_argmax_valid, assert_params_close,
                          assert_params_close_up_to_unit_flips, assert_sum_close, tensor_rel_errors)

pytestmark = pytest.mark.gpu

SEED = 0x5EED


def _setup(W, b, n_versions=1, drop_p=0.25, precision=0):
    import torch
    from paper_2406_05546_b200 import ps
    theta0 = synth.init_params(seed=1, bias_scale=0.05)
    srv = ps.ParameterServer(theta0, max_workers=W, max_batch=b, ring_depth=max(1, n_versions),
                             queue_slots=max(W, n_versions), dropout_p=drop_p, precision=precision)
    return torch, ps, srv, theta0


def _conv1_allowance(theta, x, y, keep, drop_p):
    """Per channel of the first convolution: the sum of |dL/dp1| over the pooling windows whose decision (which element
    wins, or whether any is above zero) single precision can take either way.  A sum of ten rounded products is off by at
    most 10 x 2^-24 x (sum of their magnitudes), so a decision between two of them is open below twice that; taken the
    other way it moves a filter tap by at most |dL/dp1| times a pixel (<= 1) and the bias by |dL/dp1|.  float64 on the CPU."""
    import torch
    import torch.nn.functional as F
    p = {n: torch.from_numpy(theta[o:o + int(np.prod(s))].astype(np.float64).reshape(s)) for n, o, s in synth.layout()}
    xx = torch.from_numpy(x.astype(np.float64))[:, None]
    a1 = F.conv2d(xx, p["conv1.w"], p["conv1.b"], padding=1)
    mag = F.conv2d(xx.abs(), p["conv1.w"].abs(), p["conv1.b"].abs(), padding=1)
    win = lambda t: t.unfold(2, 2, 2).unfold(3, 2, 2).reshape(*t.shape[:2], 14, 14, 4)
    top = win(a1).topk(2, dim=-1).values
    margin = torch.where(top[..., 0] > 0, torch.minimum(top[..., 0] - top[..., 1], top[..., 0]), -top[..., 0])
    still_open = margin <= 20 * 2.0 ** -24 * win(mag).amax(-1)
    p1 = F.max_pool2d(F.relu(a1), 2).requires_grad_(True)
    h = F.max_pool2d(F.relu(F.conv2d(p1, p["conv2.w"], p["conv2.b"], padding=1)), 2).flatten(1)
    h = F.relu(F.linear(h, p["fc1.w"], p["fc1.b"])) * torch.from_numpy(keep.astype(np.float64)) / (1 - drop_p)
    F.cross_entropy(F.linear(h, p["fc2.w"], p["fc2.b"]), torch.from_numpy(y).long()).backward()
    return (p1.grad.abs() * still_open).sum(dim=(0, 2, 3)).numpy()


def _run_and_compare(W, b, lags=None, n_versions=1, step=3, drop_p=0.25, worker_ids=None, in_slots=False,
                     precision=0, check=None):
    from oracle import cnn
    tol = TOL_TENSOR if precision else TOL_FP32
    torch, ps, srv, theta0 = _setup(W, b, n_versions, drop_p, precision)
    versions = {0: theta0}
    # produce older/newer versions with async applies of random "gradients" so that snapshots differ
    for v in range(1, n_versions):
        g = np.zeros((1, ps.P_PAD), dtype=np.float32)
        g[0, :ps.P] = synth.random_gradients(1, seed=50 + v, scale=2.0)[0]
        srv.ps_enqueue([0], [v - 1], 0, grads_dev=torch.from_numpy(g).cuda())
        srv.ps_apply(ps.ASYNC, 0.01)
        versions[v], ver = srv.ps_export_params(0)
        assert ver == v
    rng = np.random.default_rng(7)
    x = rng.random((W, b, 28, 28), dtype=np.float32)
    y = rng.integers(0, 10, (W, b)).astype(np.int32)
    lags = [0] * W if lags is None else lags
    ids = list(range(W)) if worker_ids is None else worker_ids
    snaps = [srv.ps_pull_snapshot(w, lags[w]) for w in range(W)]
    xd, yd = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    if in_slots:
        slots = srv.ps_queue_reserve(W)
        loss, am = srv.workers_grad_step(snaps, ids, xd, yd, SEED, step, slot_ids=slots)
        grads = torch.stack([srv.slot_tensor(s) for s in slots]).cpu().numpy()
    else:
        gd = torch.full((W, ps.P_PAD), float("nan"), device="cuda")
        loss, am = srv.workers_grad_step(snaps, ids, xd, yd, SEED, step, grads_dev=gd)
        grads = gd.cpu().numpy()
    srv.ps_stats()
    thetas = [versions[s.version] for s in snaps]
    og, ol, oa, oz = cnn.workers_grad_step(thetas, ids, x, y, SEED, step, drop_p, precision=precision)
    for w in range(W):
        assert (grads[w, ps.P:] == 0).all()
        if check is not None:
            if w in check:
                allowed = _conv1_allowance(thetas[w], x[w], y[w], cnn.dropout_keep(SEED, ids[w], step, b, drop_p), drop_p)
                got = grads[w, :ps.P].astype(np.float64)
                for off, n in ((0, 9), (144, 1)):      # the first convolution's filters, then its biases, channel by channel
                    d = (got[off:off + 16 * n] - og[w][off:off + 16 * n]).reshape(16, n)
                    lim = tol * np.abs(og[w][off:off + 16 * n]).max() + allowed
                    assert (np.abs(d).max(axis=1) <= lim).all(), f"worker {w}: first convolution off by {np.abs(d).max(axis=1)}, allowed {lim}"
                got[:160] = og[w][:160]
                assert_params_close(got, og[w], tol, f"gradient of worker {w}")
            continue
        if precision and W * b > 500:
            # several hundred thousand ReLU decisions: a hidden unit within rounding distance of zero may come out the
            # other way; the helper admits that, and only that (see its docstring), so the oracle's intermediates of
            # this worker are needed whenever a row is off
            errs = tensor_rel_errors(grads[w, :ps.P], og[w])
            if max(errs.values()) > tol:
                g1, _, _, _, diag = cnn.worker_grad_step_diag(thetas[w], ids[w], x[w], y[w], SEED, step, drop_p, precision)
                assert np.array_equal(g1, og[w])
                redo = lambda fl, w=w: cnn.worker_grad_step_diag(thetas[w], ids[w], x[w], y[w], SEED, step, drop_p, precision, flips=fl)[0]
                flips = assert_params_close_up_to_unit_flips(grads[w, :ps.P], og[w], tol, thetas[w], diag, f"gradient of worker {w}", recompute=redo)
                print(f"worker {w}: hidden units decided differently within the rounding bound of zero: {flips}")
            continue
        errs = assert_params_close(grads[w, :ps.P], og[w], tol, f"gradient of worker {w}")
        if precision and w == 0:
            print("tensor-path relative errors:", {k: f"{v:.1e}" for k, v in errs.items()})
    np.testing.assert_allclose(loss.cpu().numpy(), ol, rtol=3e-3 if precision else 1e-5, atol=1e-6)
    assert_argmax_valid(am.cpu().numpy(), oz, tol)
    srv.close()
    return grads


def test_config1_shape_two_workers_batch8():
    _run_and_compare(2, 8, in_slots=True)


def test_ragged_batch_and_worker_ids():
    _run_and_compare(3, 5, worker_ids=[11, 4, 200], step=(1 << 33) + 5)


def test_batch_spanning_several_tiles_with_tail():
    _run_and_compare(2, 70)


def test_stale_snapshots_grouped_over_three_versions():
    # five workers over three distinct weight versions, interleaved so that grouping must reorder
    _run_and_compare(5, 6, lags=[2, 0, 1, 2, 0], n_versions=3)


# 128 / 129 and 1,536 / 1,547 rows, batches that leave one sample over, ranges of rows that cross workers, two weight versions.  At the
# larger sizes two or three workers spread over the blocks are compared, and the first convolution's gradient is allowed
# what pooling decisions within single-precision rounding of a tie can move it by (there are millions of them).
@pytest.mark.parametrize("W,b,kw", [(2, 64, {}), (3, 43, {"lags": [1, 0, 1], "n_versions": 2}), (16, 96, {"check": (0, 8, 15)}),
                                     (17, 91, {"check": (0, 8, 16)}),
                                     # 32 / 33, 64 / 65, 448 / 450, 1,020 / 1,025, 1,280 / 1,290 rows and two sizes beyond,
                                     # where the dense layer's products and the blocks of the first convolution change
                                     # form; groups of rows that leave remainders in every tile
                                     (4, 16, {}), (5, 13, {"lags": [0, 1, 1, 0, 1], "n_versions": 2}), (4, 112, {}), (9, 50, {"check": (0, 4, 8)}),
                                     (10, 128, {"check": (0, 9)}), (10, 129, {"check": (0, 9)}),
                                     (4, 8, {"lags": [0, 1, 1, 0], "n_versions": 2}), (3, 11, {}), (12, 85, {"check": (0, 6, 11)}),
                                     (41, 25, {"check": (0, 20, 40), "lags": [w % 2 for w in range(41)], "n_versions": 2}),
                                     (40, 103, {"check": (0, 39)}), (50, 60, {"check": (0, 49)})])
def test_fp32_path_at_the_edges_of_its_kernel_choices(W, b, kw):
    _run_and_compare(W, b, **kw)


# One row; one row more than a 128-row tile; 18 / 19 and 4 / 5 tiles of rows, where fewer CTAs share a tile's k; 11 / 12 and 37 / 38
# tiles, beyond which one CTA does; k of the weight gradient just below, at and above a stage of 32 samples and a sum of 128;
# three weight groups whose rows end inside a tile.
@pytest.mark.parametrize("W,b,n_versions", [(1, 1, 1), (1, 31, 1), (1, 129, 1), (2, 256, 1), (3, 171, 1), (11, 128, 1), (11, 129, 1), (18, 128, 1), (19, 127, 1),
                                             (37, 128, 1), (38, 127, 1), (70, 33, 3)])
def test_fp32_dense_layer_at_the_edges_of_its_tiles(W, b, n_versions):
    """What the three products of the dense layer give, through the tensors that a pooling decision of a convolution hardly moves
    (of the millions of windows here some lie within rounding distance of a tie, and the filters' gradients depend on it), against
    float64, first, middle and last worker:
      - the output layer's gradients (forward product; a unit at zero adds nothing to them) within the path's tolerance;
      - fc1.w and fc1.b (weight gradient) within it in all units but two: of a worker's 512 b decisions whether a unit is above zero
        a few in ten million lie within rounding distance, so that one falls the other way in one worker of thirty, and moves its
        unit's row; a wrong tile moves 128 units, or some columns of all;
      - conv2.b, the sum of what the input gradient passes back through the windows above zero, within 1e-3 of its 2-norm: a window at
        zero is one of its 49 b terms (1.2e-4 of the largest element in the worst worker seen), a wrong tile a thirteenth of all."""
    torch, ps, srv, theta0 = _setup(W, b, n_versions)
    thetas = {0: theta0}
    for v in range(1, n_versions):
        g = np.zeros((1, ps.P_PAD), dtype=np.float32)
        g[0, :ps.P] = synth.random_gradients(1, seed=50 + v, scale=2.0)[0]
        srv.ps_enqueue([0], [v - 1], 0, grads_dev=torch.from_numpy(g).cuda())
        srv.ps_apply(ps.ASYNC, 0.01)
        thetas[v], _ = srv.ps_export_params(0)
    gen = torch.Generator(device="cuda").manual_seed(W + b)
    x = torch.rand((W, b, 28, 28), generator=gen, device="cuda")
    y = torch.randint(0, 10, (W, b), generator=gen, device="cuda", dtype=torch.int32)
    snaps = [srv.ps_pull_snapshot(w, w % n_versions) for w in range(W)]
    grads = torch.full((W, ps.P_PAD), float("nan"), device="cuda")
    srv.workers_grad_step(snaps, range(W), x, y, SEED, 2, grads_dev=grads)
    assert srv.ps_stats()["device_status"] == 0 and torch.isfinite(grads).all()
    for w in sorted({0, W // 2, W - 1}):
        want = _float64_gradient(thetas[snaps[w].version], x[w], y[w], srv.ps_dropout_mask(SEED, w, 2, b))
        for name, off, shape in synth.layout():
            got = grads[w, off:off + int(np.prod(shape))].double()
            ref, tol = want[name], TOL_FP32 * want[name].abs().max()
            if name == "conv2.b":
                assert (got - ref).norm() <= 1e-3 * ref.norm(), w
            elif name in ("fc1.w", "fc1.b"):
                assert int(((got - ref).abs() > tol).view(512, -1).any(dim=1).sum()) <= 2, (w, name)
            elif name in ("fc2.w", "fc2.b"):
                assert (got - ref).abs().max() <= tol, (w, name)
    srv.close()


@pytest.mark.parametrize("W,b", [(1, 3), (5, 1000)])
def test_fp32_dense_layer_keeps_an_infinite_sum(W, b):
    """A hidden unit whose weights are all infinite, over inputs that are all positive, is infinite (and not NaN, which ReLU
    would turn into zero): the loss cannot be finite."""
    from paper_2406_05546_b200 import ps
    import torch
    theta = np.abs(synth.init_params(1, bias_scale=0.05))
    off = next(o for n, o, _ in synth.layout() if n == "fc1.w")
    theta[off + 7 * 1568:off + 8 * 1568] = np.inf
    srv = ps.ParameterServer(theta, max_workers=W, max_batch=b, queue_slots=1)
    x = torch.rand((W, b, 28, 28), device="cuda") + 0.5
    loss, *_ = srv.workers_eval([srv.ps_pull_snapshot(0)] * W, x, torch.zeros((W, b), dtype=torch.int32, device="cuda"))
    assert not torch.isfinite(loss).any()
    srv.close()


# One sample (half a forward tile, one sample per filter-gradient CTA); one tile; an odd last tile in every weight group; one row per SM
# of 148 and one more; ranges of two and three rows that leave a worker in the middle of one; sums of sixteen rows and seventeen.
@pytest.mark.parametrize("W,b,n_versions", [(1, 1, 1), (1, 2, 1), (5, 3, 3), (4, 37, 1), (1, 149, 1), (7, 43, 2), (3, 149, 3), (1, 2400, 1)])
def test_fp32_second_convolution_at_the_edges_of_its_tiles(W, b, n_versions):
    """The gradients of both convolutions against float64, first, middle and last worker: the second's within 1e-3 in 2-norm, which a decision
    of its pooling that is within rounding distance of a tie may use up and a tile, a range or a shift gone wrong exceeds a
    hundredfold; the first's, which show the input gradient, within the path's tolerance and what its own open decisions allow
    (one of them, in three samples of the case of 5 x 3, moves conv1.w by 7e-3 whatever computes the rest)."""
    from oracle import cnn
    torch, ps, srv, theta0 = _setup(W, b, n_versions)
    thetas = {0: theta0}
    for v in range(1, n_versions):
        g = np.zeros((1, ps.P_PAD), dtype=np.float32)
        g[0, :ps.P] = synth.random_gradients(1, seed=50 + v, scale=2.0)[0]
        srv.ps_enqueue([0], [v - 1], 0, grads_dev=torch.from_numpy(g).cuda())
        srv.ps_apply(ps.ASYNC, 0.01)
        thetas[v], _ = srv.ps_export_params(0)
    gen = torch.Generator(device="cuda").manual_seed(W + b)
    x = torch.rand((W, b, 28, 28), generator=gen, device="cuda")
    y = torch.randint(0, 10, (W, b), generator=gen, device="cuda", dtype=torch.int32)
    snaps = [srv.ps_pull_snapshot(w, w % n_versions) for w in range(W)]
    grads = torch.full((W, ps.P_PAD), float("nan"), device="cuda")
    srv.workers_grad_step(snaps, range(W), x, y, SEED, 2, grads_dev=grads)
    assert srv.ps_stats()["device_status"] == 0 and torch.isfinite(grads).all()
    allowed = {}
    for w in sorted({0, W // 2, W - 1}):
        want = _float64_gradient(thetas[snaps[w].version], x[w], y[w], srv.ps_dropout_mask(SEED, w, 2, b))
        for name, off, shape in synth.layout():
            got = grads[w, off:off + int(np.prod(shape))].double()
            if name.startswith("conv2"):
                assert (got - want[name]).norm() <= 1e-3 * want[name].norm(), (w, name)
            elif name.startswith("conv1"):
                if w not in allowed:
                    allowed[w] = _conv1_allowance(thetas[snaps[w].version], x[w].cpu().numpy(), y[w].cpu().numpy(), cnn.dropout_keep(SEED, w, 2, b, 0.25), 0.25)
                off_by = (got - want[name]).abs().view(16, -1).amax(1).cpu().numpy()
                assert (off_by <= TOL_FP32 * float(want[name].abs().max()) + allowed[w]).all(), (w, name)
    srv.close()


@pytest.mark.parametrize("W,b,n_versions", [(1, 1, 1), (2, 8, 1), (3, 1, 3), (5, 37, 2)])
def test_fp32_evaluation_lays_out_the_weights_of_every_version_in_its_first_kernel(W, b, n_versions):
    """Five launches, and the losses of float64 for workers on different versions (one sample per worker: all spare blocks in one column of
    the first kernel's grid)."""
    import torch.nn.functional as F
    torch, ps, srv, theta0 = _setup(W, b, n_versions, drop_p=0.0)
    thetas = {0: theta0}
    for v in range(1, n_versions):
        g = np.zeros((1, ps.P_PAD), dtype=np.float32)
        g[0, :ps.P] = synth.random_gradients(1, seed=50 + v, scale=2.0)[0]
        srv.ps_enqueue([0], [v - 1], 0, grads_dev=torch.from_numpy(g).cuda())
        srv.ps_apply(ps.ASYNC, 0.01)
        thetas[v], _ = srv.ps_export_params(0)
    gen = torch.Generator(device="cuda").manual_seed(b)
    x = torch.rand((W, b, 28, 28), generator=gen, device="cuda")
    y = torch.randint(0, 10, (W, b), generator=gen, device="cuda", dtype=torch.int32)
    snaps = [srv.ps_pull_snapshot(w, w % n_versions) for w in range(W)]
    before = srv.ps_stats()["kernel_launches"]
    loss, *_ = srv.workers_eval(snaps, x, y)
    assert srv.ps_stats()["kernel_launches"] - before == 5
    for w in range(W):
        p = {n: torch.from_numpy(thetas[snaps[w].version][o:o + int(np.prod(s))].astype(np.float64).reshape(s)).cuda() for n, o, s in synth.layout()}
        h = F.max_pool2d(F.relu(F.conv2d(x[w].double()[:, None], p["conv1.w"], p["conv1.b"], padding=1)), 2)
        h = F.max_pool2d(F.relu(F.conv2d(h, p["conv2.w"], p["conv2.b"], padding=1)), 2).flatten(1)
        want = F.cross_entropy(F.linear(F.relu(F.linear(h, p["fc1.w"], p["fc1.b"])), p["fc2.w"], p["fc2.b"]), y[w].long())
        assert abs(float(loss[w]) - float(want)) <= 1e-5 * float(want), w
    srv.close()


def test_fp32_second_convolution_keeps_an_infinite_sum():
    """An output channel whose filters are all infinite, over inputs that are all positive, is infinite inside the map."""
    from paper_2406_05546_b200 import ps
    import torch
    theta = np.abs(synth.init_params(1, bias_scale=0.05))
    off = next(o for n, o, _ in synth.layout() if n == "conv2.w")
    theta[off + 5 * 144:off + 6 * 144] = np.inf
    srv = ps.ParameterServer(theta, max_workers=3, max_batch=3, queue_slots=1)
    loss, *_ = srv.workers_eval([srv.ps_pull_snapshot(0)] * 3, torch.rand((3, 3, 28, 28), device="cuda") + 0.5,
                                torch.zeros((3, 3), dtype=torch.int32, device="cuda"))
    assert not torch.isfinite(loss).any()
    srv.close()


# Pixels that are not finite, in the first, a middle and the last sample of a worker and beside samples without any; (8, 130) has several samples
# per block of the first convolution's filter gradient.
@pytest.mark.parametrize("value", [float("nan"), float("-inf")])
@pytest.mark.parametrize("W,b", [(1, 1), (2, 7), (8, 130)])
def test_fp32_pixel_that_no_winner_reads_leaves_the_gradient_finite(W, b, value):
    """A window element that reads a NaN loses against ReLU's zero, and so does one that reads minus infinity through positive filters:
    such a pixel is in no winner's patch, and the filter gradient of the first convolution, a sum over the winners' patches, does not
    see it.  Against float64 with the elements that read the pixel taken out, within the path's tolerance (and, at 8 x 130, what its own
    open decisions allow)."""
    import torch.nn.functional as F
    from oracle import cnn
    from paper_2406_05546_b200 import ps
    import torch
    theta = synth.init_params(seed=1, bias_scale=0.05)
    theta[:144] = np.abs(theta[:144])
    theta[144:160] = -0.1
    srv = ps.ParameterServer(theta, max_workers=W, max_batch=b, queue_slots=W)
    gen = torch.Generator(device="cuda").manual_seed(W + b)
    x = torch.rand((W, b, 28, 28), generator=gen, device="cuda")
    y = torch.randint(0, 10, (W, b), generator=gen, device="cuda", dtype=torch.int32)
    odd = torch.zeros((W, b, 28, 28), dtype=torch.bool, device="cuda")
    for i, (r, c) in zip((0, b // 2, b - 1), ((0, 0), (13, 6), (27, 27))):
        odd[0, i, r, c] = odd[W - 1, i, c, r] = True
    grads = torch.full((W, ps.P_PAD), float("nan"), device="cuda")
    srv.workers_grad_step([srv.ps_pull_snapshot(w) for w in range(W)], range(W), torch.where(odd, value, x), y, SEED, 2, grads_dev=grads)
    assert torch.isfinite(grads).all()
    for w in sorted({0, W - 1}):
        keep = srv.ps_dropout_mask(SEED, w, 2, b)
        p = {n: torch.from_numpy(theta[o:o + int(np.prod(s))].astype(np.float64).reshape(s)).cuda().requires_grad_(True) for n, o, s in synth.layout()}
        reads = F.max_pool2d(odd[w].double()[:, None], 3, 1, 1) > 0
        a1 = F.conv2d(torch.where(odd[w], 0.0, x[w].double())[:, None], p["conv1.w"], p["conv1.b"], padding=1).masked_fill(reads, -1.0)
        h = F.max_pool2d(F.relu(a1), 2)
        h = F.max_pool2d(F.relu(F.conv2d(h, p["conv2.w"], p["conv2.b"], padding=1)), 2).flatten(1)
        h = F.relu(F.linear(h, p["fc1.w"], p["fc1.b"])) * keep.double() / 0.75
        F.cross_entropy(F.linear(h, p["fc2.w"], p["fc2.b"]), y[w].long()).backward()
        allowed = _conv1_allowance(theta, x[w].cpu().numpy(), y[w].cpu().numpy(), cnn.dropout_keep(SEED, w, 2, b, 0.25), 0.25) if b > 7 else np.zeros(16)
        for name, off, shape in synth.layout()[:2]:
            want = p[name].grad.flatten()
            off_by = (grads[w, off:off + want.numel()].double() - want).abs().view(16, -1).amax(1).cpu().numpy()
            assert (off_by <= TOL_FP32 * float(want.abs().max()) + allowed).all(), (w, name)
    srv.close()


# The first and the last column of the map, in one, some and all samples of a range of rows
@pytest.mark.parametrize("W,b,samples", [(1, 1, (0,)), (1, 3, (1,)), (2, 300, (0, 1, 2, 3, 4, 150, 299)), (3, 20, tuple(range(20)))])
@pytest.mark.parametrize("col", [0, 13])
def test_fp32_infinite_activation_reaches_only_the_filter_taps_that_read_it(W, b, samples, col):
    """An infinite activation at an end of a row of the second convolution's input, under filters that make every window above it lose:
    the gradients passed back there are zeros, and zero times infinity is NaN, in the taps (of that input channel) that take the activation from
    some position of the map.  The other taps, those that would take it from a column outside of it among them, are finite and, like
    the bias, within 1e-3 of float64 in 2-norm (the bound of the tiles' edges)."""
    import torch.nn.functional as F
    from paper_2406_05546_b200 import ps
    import torch
    theta = synth.init_params(seed=1, bias_scale=0.05)
    rng = np.random.default_rng(3)
    theta[:144] = -0.1 * rng.random(144)        # channels 1 .. 15: minus infinity where they read the pixel
    theta[:9] = 0.1                             # channel 0: infinite there
    theta[144:160] = 0.2
    off = next(o for n, o, _ in synth.layout() if n == "conv2.w")
    taps = theta[off:off + 4608].reshape(32, 16, 9)
    taps[:, 0] = -np.abs(taps[:, 0])
    srv = ps.ParameterServer(theta, max_workers=W, max_batch=b, queue_slots=W)
    gen = torch.Generator(device="cuda").manual_seed(b)
    x = torch.rand((W, b, 28, 28), generator=gen, device="cuda")
    y = torch.randint(0, 10, (W, b), generator=gen, device="cuda", dtype=torch.int32)
    x[0, list(samples), 0, 0 if col == 0 else 27] = float("inf")
    grads = torch.zeros((W, ps.P_PAD), device="cuda")
    loss, _ = srv.workers_grad_step([srv.ps_pull_snapshot(w) for w in range(W)], range(W), x, y, SEED, 2, grads_dev=grads)
    assert torch.isfinite(loss).all() and srv.ps_stats()["device_status"] == 0
    for w in sorted({0, W - 1}):
        p = {n: torch.from_numpy(theta[o:o + int(np.prod(s))].astype(np.float64).reshape(s)).cuda().requires_grad_(not n.startswith("conv1")) for n, o, s in synth.layout()}
        # the pixel stands for 1e30, which decides every window alike and reaches nothing above
        p1 = F.max_pool2d(F.relu(F.conv2d(x[w].double().clamp(max=1e30)[:, None], p["conv1.w"], p["conv1.b"], padding=1)), 2)
        a2 = F.conv2d(p1, p["conv2.w"], p["conv2.b"], padding=1)
        a2.retain_grad()
        h = F.max_pool2d(F.relu(a2), 2).flatten(1)
        h = F.relu(F.linear(h, p["fc1.w"], p["fc1.b"])) * srv.ps_dropout_mask(SEED, w, 2, b).double() / 0.75
        F.cross_entropy(F.linear(h, p["fc2.w"], p["fc2.b"]), y[w].long()).backward()
        # a tap's sum over the positions of the map that it reads a position of the map from
        p1 = torch.where(p1 > 1e20, float("inf"), p1)
        want = torch.zeros((32, 16, 3, 3), dtype=torch.float64, device="cuda")
        for ky in range(3):
            for kx in range(3):
                ys, xs = slice(max(0, 1 - ky), min(14, 15 - ky)), slice(max(0, 1 - kx), min(14, 15 - kx))
                yi, xi = slice(ys.start + ky - 1, ys.stop + ky - 1), slice(xs.start + kx - 1, xs.stop + kx - 1)
                for ic in range(16):
                    want[:, ic, ky, kx] = (a2.grad[:, :, ys, xs] * p1[:, ic:ic + 1, yi, xi]).sum((0, 2, 3))
        got, want = grads[w, off:off + 4608].double(), want.flatten()
        assert int(want.isnan().sum()) == (32 * 4 if w == 0 else 0) and torch.equal(got.isnan(), want.isnan())
        fine = ~want.isnan()
        assert (got - want)[fine].norm() <= 1e-3 * want[fine].norm()
        db = a2.grad.sum((0, 2, 3))
        assert (grads[w, off + 4608:off + 4640].double() - db).norm() <= 1e-3 * db.norm()
    srv.close()


def _float64_gradient(theta, x, y, keep, drop_p=0.25):
    """One worker's gradient in float64 on the device: {tensor name: flat gradient}."""
    import torch
    import torch.nn.functional as F
    p = {n: torch.from_numpy(theta[o:o + int(np.prod(s))].astype(np.float64).reshape(s)).cuda().requires_grad_(True) for n, o, s in synth.layout()}
    h = F.max_pool2d(F.relu(F.conv2d(x.double()[:, None], p["conv1.w"], p["conv1.b"], padding=1)), 2)
    h = F.max_pool2d(F.relu(F.conv2d(h, p["conv2.w"], p["conv2.b"], padding=1)), 2).flatten(1)
    h = F.relu(F.linear(h, p["fc1.w"], p["fc1.b"])) * keep.double() / (1 - drop_p)
    F.cross_entropy(F.linear(h, p["fc2.w"], p["fc2.b"]), y.long()).backward()
    return {n: v.grad.flatten() for n, v in p.items()}


# One sample; a few; the dense layer's products with k split over eight and fewer CTAs; its input gradient without; all without
@pytest.mark.parametrize("W,b,seeds", [(1, 1, (5, 6, 7, 8, 9, 10, 11)), (2, 8, (5, 6, 7)), (3, 37, (5, 6)), (12, 128, (5,)), (38, 128, (5,))])
def test_fp32_gradients_are_as_near_to_float64_as_single_precision(W, b, seeds):
    """Relative 2-norm error of every gradient tensor, median over workers and inputs (a worker in which a pooling or ReLU decision
    within rounding distance of a tie falls the other way counts no more than another).  Any one of the six products of pieces
    left out or taken with another's operand is four times the bound or more off (test_bf16_pieces.py)."""
    from tests.test_bf16_pieces import PRECISION_FP32
    from paper_2406_05546_b200 import ps
    import torch
    errs = {}
    for seed in seeds:
        theta = synth.init_params(seed=seed, bias_scale=0.05)
        srv = ps.ParameterServer(theta, max_workers=W, max_batch=b, queue_slots=W)
        gen = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.rand((W, b, 28, 28), generator=gen, device="cuda")
        y = torch.randint(0, 10, (W, b), generator=gen, device="cuda", dtype=torch.int32)
        grads = torch.zeros((W, ps.P_PAD), device="cuda")
        srv.workers_grad_step([srv.ps_pull_snapshot(w) for w in range(W)], range(W), x, y, SEED, 1, grads_dev=grads)
        for w in range(0, W, max(1, W // 7)):
            want = _float64_gradient(theta, x[w], y[w], srv.ps_dropout_mask(SEED, w, 1, b))
            for name, off, shape in synth.layout():
                got = grads[w, off:off + int(np.prod(shape))].double()
                errs.setdefault(name, []).append(float((got - want[name]).norm() / want[name].norm()))
        srv.close()
    median = {name: float(np.median(e)) for name, e in errs.items()}
    assert max(median.values()) <= PRECISION_FP32, median


@pytest.mark.parametrize("W,b", [(1, 3), (5, 1000)])
def test_fp32_weights_above_the_largest_bf16_stay_finite(W, b):
    """3.4e38 is a float and rounds to no BF16: its first piece is cut off instead.  One weight of a hidden unit that the output layer does not
    listen to (0 x infinity would be NaN there); the unit shows in the gradient of its output weights."""
    from paper_2406_05546_b200 import ps
    import torch
    import torch.nn.functional as F
    theta = synth.init_params(seed=1, bias_scale=0.05)
    at = {n: o for n, o, _ in synth.layout()}
    theta[160:4768] = 0.05 * np.abs(theta[160:4768])       # activations above zero and well below one
    theta[at["fc1.w"] + 7 * 1568:at["fc1.w"] + 8 * 1568] = 0
    theta[at["fc1.w"] + 7 * 1568 + 700] = 3.4e38
    theta[at["fc2.w"]:at["fc2.w"] + 5120].reshape(10, 512)[:, 7] = 0
    srv = ps.ParameterServer(theta, max_workers=W, max_batch=b, queue_slots=W, dropout_p=0.0)
    gen = torch.Generator(device="cuda").manual_seed(b)
    x = 0.1 * torch.rand((W, b, 28, 28), generator=gen, device="cuda")
    y = torch.randint(0, 10, (W, b), generator=gen, device="cuda", dtype=torch.int32)
    grads = torch.zeros((W, ps.P_PAD), device="cuda")
    loss, _ = srv.workers_grad_step([srv.ps_pull_snapshot(w) for w in range(W)], range(W), x, y, SEED, 1, grads_dev=grads)
    assert torch.isfinite(loss).all() and torch.isfinite(grads).all()
    for w in sorted({0, W - 1}):
        want = _float64_gradient(theta, x[w], y[w], torch.ones((b, 512), device="cuda"), drop_p=0.0)["fc2.w"].view(10, 512)[:, 7]
        got = grads[w, at["fc2.w"]:at["fc2.w"] + 5120].double().view(10, 512)[:, 7]
        assert float(want.abs().max()) > 1e35 and (got - want).norm() <= 1e-5 * want.norm()
    srv.close()


def test_fp32_forward_pass_loses_nothing_that_adds_up_over_samples():
    """The tensor cores' accumulators truncate.  What that takes from a forward sum is alike in every sample, so that it stays in a sum over
    samples in which rounding averages out, first of all in the output layer's gradient, which is proportional to the hidden units:
    over 992 samples the 2-norm error of fc2.w against float64 was 1.9e-7 with it and 1.2e-7 with multiply-adds that round.  1.4e-7
    is the bound: rounding and 2^-24 of every hidden unit.  Median over four sets of weights and inputs."""
    from paper_2406_05546_b200 import ps
    import torch
    off, n = next((o, int(np.prod(s))) for name, o, s in synth.layout() if name == "fc2.w")
    errs = []
    for seed in (5, 6, 7, 8):
        theta = synth.init_params(seed=seed, bias_scale=0.05)
        srv = ps.ParameterServer(theta, max_workers=31, max_batch=32, queue_slots=31)
        gen = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.rand((31, 32, 28, 28), generator=gen, device="cuda")
        y = torch.randint(0, 10, (31, 32), generator=gen, device="cuda", dtype=torch.int32)
        grad, *_ = srv.workers_grad_step_summed([srv.ps_pull_snapshot(w) for w in range(31)], range(31), x, y, SEED, 1)
        keep = torch.cat([srv.ps_dropout_mask(SEED, w, 1, 32) for w in range(31)])
        want = 31 * _float64_gradient(theta, x.flatten(0, 1), y.flatten(), keep)["fc2.w"]      # of the mean over all samples
        errs.append(float((grad.flatten()[off:off + n].double() - want).norm() / want.norm()))
        srv.close()
    assert np.median(errs) <= 1.4e-7, errs


def test_fp32_filter_gradient_is_as_precise_in_a_large_call_as_in_a_small_one():
    """Rows of a call are summed in ranges that grow with the call, and what single precision loses grows as the root of a
    sum's length.  At 16 x 128 rows a thread of conv2's filter gradient adds the 49 / 4 winners of its positions over 7
    samples, and 20 such sums make a worker's gradient; at 128 x 128 it is 14 samples and 11 sums.  The errors of the first
    sixteen workers may differ by sqrt((14 * 12.25 + 11) / (7 * 12.25 + 20)) = 1.32 then (median: a worker in which a pooling
    decision fell the other way counts no more than another)."""
    torch, ps, srv, theta = _setup(128, 128)
    gen = torch.Generator(device="cuda").manual_seed(5)
    x = torch.rand((128, 128, 28, 28), generator=gen, device="cuda")
    y = torch.randint(0, 10, (128, 128), generator=gen, device="cuda", dtype=torch.int32)
    off, n = next((o, int(np.prod(s))) for name, o, s in synth.layout() if name == "conv2.w")
    exact = [_float64_gradient(theta, x[w], y[w], srv.ps_dropout_mask(SEED, w, 1, 128))["conv2.w"] for w in range(16)]
    median = {}
    for W in (16, 128):
        grads = torch.zeros((W, ps.P_PAD), device="cuda")
        srv.workers_grad_step([srv.ps_pull_snapshot(w) for w in range(W)], range(W), x[:W], y[:W], SEED, 1, grads_dev=grads)
        median[W] = float(np.median([float((grads[w, off:off + n].double() - e).norm() / e.norm()) for w, e in enumerate(exact)]))
    srv.close()
    assert median[128] <= 1.32 * median[16], median


@pytest.mark.parametrize("b", [64, 65, 1040])
def test_output_layer_split_over_blocks(b):
    # eight blocks per worker with eight samples each, with nine and a short last one, and with 130 each (two chunks of
    # samples in a block).  Only what the output layer itself sums is compared: the gradients below also depend on three
    # million pooling windows of the second convolution, of which a few lie within single-precision rounding of a tie.
    from oracle import cnn
    torch, ps, srv, theta = _setup(2, b)
    rng = np.random.default_rng(11)
    x, y = rng.random((2, b, 28, 28), dtype=np.float32), rng.integers(0, 10, (2, b)).astype(np.int32)
    gd = torch.full((2, ps.P_PAD), float("nan"), device="cuda")
    loss, am = srv.workers_grad_step([srv.ps_pull_snapshot(0)] * 2, [0, 1], torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda(),
                                     SEED, 5, grads_dev=gd)
    og, ol, _, oz = cnn.workers_grad_step([theta] * 2, [0, 1], x, y, SEED, 5)
    for w in range(2):
        errs = tensor_rel_errors(gd[w, :ps.P].cpu().numpy(), og[w])
        assert max(errs[k] for k in ("fc1.b", "fc2.w", "fc2.b")) <= TOL_FP32, errs
    np.testing.assert_allclose(loss.cpu().numpy(), ol, rtol=1e-5)
    assert_argmax_valid(am.cpu().numpy(), oz, TOL_FP32)
    srv.close()


@pytest.mark.parametrize("W,b,kw", [(2, 8, {}), (3, 5, {"worker_ids": [11, 4, 200]}), (2, 150, {}),
                                     (5, 6, {"lags": [2, 0, 1, 2, 0], "n_versions": 3}), (1, 1, {}),
                                     (2, 4, {"drop_p": 0.0}),
                                     # 777 rows over two weight versions: the persistent convolution kernels take
                                     # ranges of several rows that cross worker boundaries inside a version group
                                     (7, 111, {"lags": [1, 0, 1, 1, 0, 0, 1], "n_versions": 2}),
                                     # 896 rows: the first convolution takes two samples per block; 6 rows: ranges of
                                     # the filter gradients shorter than four rows
                                     (8, 112, {}), (3, 2, {}),
                                     # three and four, 37 and 38 128-row tiles, eighteen and nineteen 64-row tiles: where the dense
                                     # layer's products change form; ragged last tiles, two weight versions (tiles never cross them)
                                     (3, 100, {}), (5, 101, {"lags": [1, 0, 0, 1, 0], "n_versions": 2}), (9, 128, {}), (9, 130, {}), (37, 128, {}), (38, 128, {})])
def test_tensor_core_path(W, b, kw):
    _run_and_compare(W, b, precision=2, **kw)


@pytest.mark.parametrize("precision", [0, 2])
def test_maximum_number_of_workers_with_an_odd_batch(precision):
    # 256 workers (the library's limit) of three samples: every worker's last sample has no partner in the first
    # convolution's filter-gradient kernel, and ranges of the persistent kernels cross many worker boundaries
    _run_and_compare(256, 3, precision=precision, worker_ids=[(7 * w + 3) % 1000 for w in range(256)])


def test_tensor_core_path_repeatable_bit_for_bit():
    a = _run_and_compare(3, 9, precision=2)
    b = _run_and_compare(3, 9, precision=2)
    assert (a == b).all()


@pytest.mark.parametrize("W,b", [(2, 32), (5, 13), (7, 73), (8, 64)])
def test_filter_gradient_in_line_and_on_its_own_stream(W, b):
    """64, 65, 511 and 512 rows: the choice changes where the kernel runs, never a bit of what it gives.  The profiled
    call runs the same kernels one at a time in one stream."""
    torch, ps, srv, _ = _setup(W, b, precision=2)
    rng = np.random.default_rng(W)
    x = torch.from_numpy(rng.random((W, b, 28, 28), dtype=np.float32)).cuda()
    y = torch.from_numpy(rng.integers(0, 10, (W, b), dtype=np.int32)).cuda()
    snaps = [srv.ps_pull_snapshot(w) for w in range(W)]
    grads = torch.zeros((4, W, ps.P_PAD), device="cuda")
    for k in range(4):
        srv.ps_profile(1 if k == 3 else 0)
        srv.workers_grad_step(snaps, range(W), x, y, SEED, 1, grads_dev=grads[k])
    srv.ps_profile(0)
    assert (grads[0] != 0).any() and all(torch.equal(grads[0], g) for g in grads[1:])
    srv.close()


@pytest.mark.parametrize("W,b", [(2, 8), (3, 40)])
def test_tensor_core_path_against_the_plain_definition(W, b):
    """The tensor-core path against the oracle with EVERY decision taken on exact values (precision 0): what the
    benchmarked path's error is against the definition, and that it comes from decisions inside the
    operand-rounding bound and from nothing else.
      - output layer: within the tolerance as it stands (a ReLU that flips at zero changes no forward value);
      - 512-unit layer: every row is within the tolerance after removing the contributions of samples whose exact
        pre-activation is inside the bound (least-squares explanation, coefficients -1 / 0 / +1);
      - convolutions: pooling winners inside the bound re-route gradient between neighbouring positions; their
        error is reported and must not exceed what the oracle itself shows between exact and rounded decisions
        plus the tolerance (every such difference lies inside the bound: tests/test_margins.py)."""
    from oracle import cnn
    import torch
    from paper_2406_05546_b200 import ps
    from tests import margins
    torch_, ps_, srv, theta0 = _setup(W, b, 1, 0.25, 2)
    rng = np.random.default_rng(21)
    x = rng.random((W, b, 28, 28), dtype=np.float32)
    y = rng.integers(0, 10, (W, b)).astype(np.int32)
    snaps = [srv.ps_pull_snapshot(w) for w in range(W)]
    gd = torch.full((W, ps.P_PAD), float("nan"), device="cuda")
    srv.workers_grad_step(snaps, list(range(W)), torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda(), SEED, 4, grads_dev=gd)
    srv.ps_stats()
    grads = gd.cpu().numpy()
    srv.close()
    n_flips = n_pool_unc = n_relu_unc = 0
    for w in range(W):
        g0, _, _, _, d0 = cnn.worker_grad_step_diag(theta0, w, x[w], y[w], SEED, 4, 0.25, precision=0)
        g2 = cnn.worker_grad_step_diag(theta0, w, x[w], y[w], SEED, 4, 0.25, precision=2)[0]
        m = margins.decision_margins(theta0, d0)
        n_pool_unc += int(m["pool_uncertain"].sum()); n_relu_unc += int(m["relu_uncertain"].sum())
        e_kernel = tensor_rel_errors(grads[w, :ps.P], g0)
        e_oracle = tensor_rel_errors(g2, g0)
        print(f"worker {w}: kernel vs exact decisions", {k: f"{v:.1e}" for k, v in e_kernel.items()})
        print(f"worker {w}: oracle with rounded decisions vs exact decisions", {k: f"{v:.1e}" for k, v in e_oracle.items()})
        for name in ("fc2.w", "fc2.b"):
            assert e_kernel[name] <= TOL_TENSOR, (name, e_kernel[name])
        for name in ("conv1.w", "conv1.b", "conv2.w", "conv2.b"):
            assert e_kernel[name] <= e_oracle[name] + TOL_TENSOR, (name, e_kernel[name], e_oracle[name])
        # the 512-unit layer, row by row: got = exact-decision gradient + flips of samples inside the bound.  The
        # convolution tensors are excluded from this call's tolerance check by comparing them in a copy.
        probe = g0.copy()
        probe[4800:808128] = grads[w, 4800:808128]
        flips = assert_params_close_up_to_unit_flips(probe, g0, TOL_TENSOR, theta0, d0, f"worker {w} vs exact decisions")
        n_flips += sum(len(f) for _, f in flips)
    print(f"{n_flips} ReLU decisions of the 512-unit layer differ from the exact ones; all inside the bound "
          f"({n_relu_unc} of {W * b * 512} decisions are; pooling: {n_pool_unc} of {W * b * 1568})")


def test_no_dropout():
    _run_and_compare(2, 4, drop_p=0.0)


def test_single_sample_single_worker():
    _run_and_compare(1, 1)


def test_repeatable_bit_for_bit():
    a = _run_and_compare(3, 9)
    b = _run_and_compare(3, 9)
    assert (a == b).all()


def test_dropout_mask_bit_exact():
    from oracle import cnn
    torch, ps, srv, _ = _setup(1, 1)
    for seed, worker, step, b in [(SEED, 0, 0, 1), (SEED, 3, 7, 64), (0xDEADBEEFCAFEF00D, 255, (5 << 32) | 9, 129)]:
        got = srv.ps_dropout_mask(seed, worker, step, b).cpu().numpy()
        assert (got == cnn.dropout_keep(seed, worker, step, b, 0.25)).all()
    srv.close()


def test_grad_step_uses_that_mask():
    # fc1 weights zero and bias one: the hidden layer is 1 before dropout, so with one sample the
    # fc2 weight gradient is dz[c] * keep[j] / (1-p): its zero pattern is exactly the mask.
    from oracle import cnn
    import torch
    from paper_2406_05546_b200 import ps
    theta = synth.init_params(seed=1)
    theta[4800:807616] = 0
    theta[807616:808128] = 1
    srv = ps.ParameterServer(theta, max_workers=4, max_batch=1, queue_slots=4)
    x = np.random.default_rng(0).random((4, 1, 28, 28), dtype=np.float32)
    y = np.array([[1], [2], [3], [4]], dtype=np.int32)
    ids = [9, 0, 77, 3]
    snaps = [srv.ps_pull_snapshot(w) for w in range(4)]
    gd = torch.zeros((4, ps.P_PAD), device="cuda")
    srv.workers_grad_step(snaps, ids, torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda(), SEED, 21, grads_dev=gd)
    g = gd.cpu().numpy()
    for w in range(4):
        keep = cnn.dropout_keep(SEED, ids[w], 21, 1, 0.25)[0]
        gw2 = g[w, 808128:813248].reshape(10, 512)
        assert ((gw2 != 0).all(axis=0) == (keep == 1)).all()
        assert ((gw2 == 0).all(axis=0) == (keep == 0)).all()
    srv.close()


def test_bad_label_is_reported_not_trapped():
    torch, ps, srv, _ = _setup(1, 2)
    x = torch.zeros((1, 2, 28, 28), device="cuda")
    y = torch.tensor([[3, 12]], dtype=torch.int32, device="cuda")
    gd = torch.zeros((1, ps.P_PAD), device="cuda")
    srv.workers_grad_step([srv.ps_pull_snapshot(0)], [0], x, y, SEED, 0, grads_dev=gd)
    with pytest.raises(ps.PSError) as e:
        srv.ps_stats()
    assert e.value.name == "PS_ERR_DEVICE_STATUS"
    srv.close()


def test_argument_errors():
    torch, ps, srv, _ = _setup(2, 4)
    x = torch.zeros((3, 4, 28, 28), device="cuda")
    y = torch.zeros((3, 4), dtype=torch.int32, device="cuda")
    snaps = [srv.ps_pull_snapshot(0)] * 3
    with pytest.raises(ps.PSError) as e:
        srv.workers_grad_step(snaps, [0, 1, 2], x, y, SEED, 0, grads_dev=torch.zeros((3, ps.P_PAD), device="cuda"))
    assert e.value.name == "PS_ERR_BAD_ARG"
    with pytest.raises(ps.PSError):
        srv.workers_grad_step(snaps[:2], [0, 1], x[:2], y[:2], SEED, 0, slot_ids=[0, 1])   # not reserved
    with pytest.raises(ps.PSError) as e:
        srv.ps_pull_snapshot(0, lag=1)
    assert e.value.name == "PS_ERR_VERSION_EVICTED"
    srv.close()


@pytest.mark.parametrize("W", [257, 300])
def test_more_workers_than_any_server_takes_are_refused_by_the_library(W):
    torch, ps, srv, _ = _setup(2, 1)
    x, y = torch.zeros((W, 1, 28, 28), device="cuda"), torch.zeros((W, 1), dtype=torch.int32, device="cuda")
    snaps = [srv.ps_pull_snapshot(0)] * W
    for call in (lambda: srv.workers_grad_step(snaps, list(range(W)), x, y, SEED, 0, grads_dev=torch.zeros((W, ps.P_PAD), device="cuda")),
                 lambda: srv.workers_grad_step_summed(snaps, list(range(W)), x, y, SEED, 0), lambda: srv.workers_eval(snaps, x, y)):
        with pytest.raises(ps.PSError) as e:
            call()
        assert e.value.name == "PS_ERR_BAD_ARG" and "outside" in str(e.value)
    srv.close()


def test_snapshots_of_a_call_in_every_form():
    """A generator, an array of structures and plain pairs are snapshots; too few of them leave workers without weights, which
    the library refuses; too many, and what is no snapshot although it has a snapshot's size, are refused by ctypes."""
    torch, ps, srv, _ = _setup(2, 1)
    x, y = torch.rand((2, 1, 28, 28), device="cuda"), torch.zeros((2, 1), dtype=torch.int32, device="cuda")
    s = srv.ps_pull_snapshot(0)
    want = srv.workers_eval([s, s], x, y)[0]
    for form in ((s, s), iter([s, s]), (ps.Snapshot * 2)(s, s), [(s.version, s.dev_ptr)] * 2):
        assert torch.equal(srv.workers_eval(form, x, y)[0], want)
    with pytest.raises(ps.PSError) as e:
        srv.workers_eval([s], x, y)
    assert e.value.name == "PS_ERR_BAD_ARG" and "no weights" in str(e.value)
    with pytest.raises(IndexError):
        srv.workers_eval([s] * 3, x, y)
    for other in (np.array([s.version, s.dev_ptr], dtype=np.uint64), bytes(s)):
        with pytest.raises(TypeError):
            srv.workers_eval([other, other], x, y)
    srv.close()


# 1,026 rows: two chunks on the FP32 path; 12,480 rows: four, the last of one worker
@pytest.mark.parametrize("precision,W,b", [(0, 3, 4), (0, 9, 5), (2, 9, 5), (2, 8, 16), (0, 9, 114), (2, 13, 960)])
def test_tick_from_host_buffers_matches_the_oracle(precision, W, b):
    """ps_tick_host: inputs copied in by worker chunks (several from a thousand rows on), snapshots
    with lags, grad step into reserved slots, enqueue, sync apply, losses and labels copied out."""
    from oracle import cnn, ps as ops
    import torch
    from paper_2406_05546_b200 import ps
    tol = TOL_TENSOR if precision else TOL_FP32
    theta0 = synth.init_params(seed=1, bias_scale=0.05)
    srv = ps.ParameterServer(theta0, max_workers=W, max_batch=b, ring_depth=2, queue_slots=W, dropout_p=0.25,
                             precision=precision)
    o = ops.OraclePS(theta0, ring_depth=2)
    # one async update first, so that lag 1 reads different weights than lag 0
    g = np.zeros((1, ps.P_PAD), dtype=np.float32)
    g[0, :ps.P] = synth.random_gradients(1, seed=61, scale=2.0)[0]
    srv.ps_enqueue([0], [0], 0, grads_dev=torch.from_numpy(g).cuda())
    srv.ps_apply(ps.ASYNC, 0.01)
    o.enqueue(g[:, :ps.P], [0], [0], 0)
    o.apply(ops.ASYNC, 0.01)
    rng = np.random.default_rng(11)
    x = rng.random((W, b, 28, 28), dtype=np.float32)
    y = rng.integers(0, 10, (W, b)).astype(np.int32)
    lags = [(w * 3) % 2 for w in range(W)]
    am = np.zeros((W, b), dtype=np.int32)
    loss, res = srv.ps_tick_host(x, y, SEED, 5, ps.SYNC, 0.01, lags=lags, argmax_host=am)
    theta, version = srv.ps_export_params()
    srv.ps_stats()
    srv.close()
    thetas = [o.pull_snapshot(w, l)[1] for w, l in enumerate(lags)]
    og, ol, oa, oz = cnn.workers_grad_step(thetas, list(range(W)), x, y, SEED, 5, 0.25, precision=precision)
    o.enqueue(og.astype(np.float32), range(W), [1 - l for l in lags], 5)
    o.apply(ops.SYNC, 0.01)
    assert res["applied"] == W and version == res["new_version"] == 2
    np.testing.assert_allclose(loss, ol, rtol=3e-3 if precision else 1e-5, atol=1e-6)
    assert_argmax_valid(am, oz, tol if precision else 10 * TOL_FP32)
    assert_params_close(theta, o.head(), tol, "parameters after the tick")
    # the tick moves the head by lr * mean gradient: compare that step too, which the parameters' size would hide
    before = o.ring[1].astype(np.float64)
    assert_params_close(theta - before, o.head() - before, max(tol, 10 * TOL_FP32), "the tick's update")


@pytest.mark.parametrize("precision", [0, 2])
def test_pipelined_ticks_equal_sequential_ticks(precision):
    """Two ticks in flight (ps_tick_host_submit / ps_tick_host_wait) leave the same weights, losses, labels and
    versions, bit for bit, as the same ticks run one by one through ps_tick_host."""
    import torch
    from paper_2406_05546_b200 import ps
    W, b, T = 9, 6, 5
    theta0 = synth.init_params(seed=1, bias_scale=0.05)
    rng = np.random.default_rng(3)
    xs = [torch.from_numpy(rng.random((W, b, 28, 28), dtype=np.float32)).pin_memory() for _ in range(T)]
    ys = [torch.from_numpy(rng.integers(0, 10, (W, b)).astype(np.int32)).pin_memory() for _ in range(T)]
    out = []
    for pipelined in (False, True):
        srv = ps.ParameterServer(theta0, max_workers=W, max_batch=b, ring_depth=2, queue_slots=W, precision=precision)
        loss = [np.zeros(W, dtype=np.float32) for _ in range(T)]
        am = [np.zeros((W, b), dtype=np.int32) for _ in range(T)]
        results = []
        if pipelined:
            srv.ps_tick_host_submit(xs[0], ys[0], SEED, 0, ps.SYNC, 0.01, loss_host=loss[0], argmax_host=am[0])
            for t in range(1, T):
                srv.ps_tick_host_submit(xs[t], ys[t], SEED, t, ps.SYNC, 0.01, loss_host=loss[t], argmax_host=am[t])
                results.append(srv.ps_tick_host_wait())
            with pytest.raises(ps.PSError):          # the synchronous form refuses to run while a tick is in flight
                srv.ps_tick_host(xs[0], ys[0], SEED, 99, ps.SYNC, 0.01)
            results.append(srv.ps_tick_host_wait())
            with pytest.raises(ps.PSError):
                srv.ps_tick_host_wait()
        else:
            for t in range(T):
                results.append(srv.ps_tick_host(xs[t], ys[t], SEED, t, ps.SYNC, 0.01, loss_host=loss[t], argmax_host=am[t])[1])
        theta, version = srv.ps_export_params()
        srv.ps_stats()
        srv.close()
        out.append((theta, version, np.stack(loss), np.stack(am), [r["new_version"] for r in results]))
    a, p = out
    assert a[1] == p[1] == T and a[4] == p[4] == list(range(1, T + 1))
    assert (a[0] == p[0]).all() and (a[2] == p[2]).all() and (a[3] == p[3]).all()


@pytest.mark.parametrize("precision,W,b", [(0, 9, 114), (2, 13, 960)])
def test_pipelined_ticks_in_several_chunks_equal_resident_ones(precision, W, b):
    """Two and four chunks, two ticks in flight: copies run beside the kernels of the chunk, and of the tick, before.  Every
    chunk is a grad step of its own, so the resident ticks take the same workers in the same calls."""
    import torch
    from paper_2406_05546_b200 import ps
    theta0, T = synth.init_params(seed=1, bias_scale=0.05), 3
    gen = torch.Generator().manual_seed(3)
    xs = [torch.rand((W, b, 28, 28), generator=gen).pin_memory() for _ in range(T)]
    ys = [torch.randint(0, 10, (W, b), generator=gen, dtype=torch.int32).pin_memory() for _ in range(T)]
    per = -(-W // (4 if W * b >= 12288 else 2))
    out = []
    for host in (True, False):
        srv = ps.ParameterServer(theta0, max_workers=W, max_batch=b, queue_slots=W, precision=precision)
        loss, am = torch.zeros((T, W)).pin_memory(), torch.zeros((T, W, b), dtype=torch.int32).pin_memory()
        if host:
            for t in range(T):
                if t >= 2:
                    srv.ps_tick_host_wait()
                srv.ps_tick_host_submit(xs[t], ys[t], SEED, t, ps.SYNC, 0.01, loss_host=loss[t], argmax_host=am[t])
            srv.ps_tick_host_wait(); srv.ps_tick_host_wait()
        else:
            for t in range(T):
                x, y, snap, slots = xs[t].cuda(), ys[t].cuda(), srv.ps_pull_snapshot(0), srv.ps_queue_reserve(W)
                for w0 in range(0, W, per):
                    part = slice(w0, min(W, w0 + per))
                    l, a = srv.workers_grad_step([snap] * len(range(W)[part]), range(W)[part], x[part], y[part], SEED, t, slot_ids=slots[part])
                    loss[t, part], am[t, part] = l.cpu(), a.cpu()
                srv.ps_enqueue(range(W), [snap.version] * W, t, slot_ids=slots)
                srv.ps_apply(ps.SYNC, 0.01)
        out.append((srv.ps_export_params()[0], loss.numpy().copy(), am.numpy().copy()))
        srv.ps_stats()
        srv.close()
    for h, r in zip(*out):
        assert (h == r).all()


@pytest.mark.parametrize("precision", [0, 2])
def test_a_grad_step_behind_a_wait_for_another_stream_reads_what_that_stream_wrote(precision):
    """The images are still on their way, on another stream, when the grad step is enqueued right behind an update: the
    stream's wait for them holds its first kernel back too, which is launched to overlap the kernel before it."""
    import torch
    W, b = 4, 32
    _, ps, srv, _ = _setup(W, b, precision=precision)
    gen = torch.Generator(device="cuda").manual_seed(9)
    y = torch.randint(0, 10, (W, b), generator=gen, device="cuda", dtype=torch.int32)
    new = torch.rand((W, b, 28, 28), generator=gen, device="cuda")
    x, other = torch.zeros_like(new), torch.cuda.Stream()
    update = torch.zeros((1, ps.P_PAD), device="cuda")
    grads = torch.zeros((2, W, ps.P_PAD), device="cuda")
    torch.cuda.synchronize()
    for late in (1, 0):
        srv.ps_enqueue([0], [0], 0, grads_dev=update)
        if late:
            with torch.cuda.stream(other):
                torch.cuda._sleep(20_000_000)      # about ten milliseconds
                x.copy_(new)
        srv.ps_apply(ps.SYNC, 0.01)
        torch.cuda.current_stream().wait_stream(other)
        srv.workers_grad_step([srv.ps_pull_snapshot(w) for w in range(W)], range(W), x, y, SEED, 1, grads_dev=grads[late])
    assert (grads[0] != 0).any() and torch.equal(grads[0], grads[1])
    srv.close()


@pytest.mark.parametrize("precision,W,b,lags", [(0, 3, 17, None), (2, 3, 17, None), (2, 4, 150, [1, 0, 0, 1]), (0, 1, 1, None)])
def test_evaluation_pass_matches_the_oracle(precision, W, b, lags):
    """workers_eval: forward only, no dropout; loss, labels and the count of correct labels per group."""
    from oracle import cnn
    n_versions = 2 if lags else 1
    torch, ps, srv, theta0 = _setup(W, b, n_versions, 0.25, precision)      # the context's dropout rate must not matter
    versions = {0: theta0}
    if lags:
        g = np.zeros((1, ps.P_PAD), dtype=np.float32)
        g[0, :ps.P] = synth.random_gradients(1, seed=51, scale=2.0)[0]
        srv.ps_enqueue([0], [0], 0, grads_dev=torch.from_numpy(g).cuda())
        srv.ps_apply(ps.ASYNC, 0.01)
        versions[1] = srv.ps_export_params(0)[0]
    rng = np.random.default_rng(8)
    x = rng.random((W, b, 28, 28), dtype=np.float32)
    y = rng.integers(0, 10, (W, b)).astype(np.int32)
    snaps = [srv.ps_pull_snapshot(w, lags[w] if lags else 0) for w in range(W)]
    before = srv.ps_stats()
    loss, am, correct = srv.workers_eval(snaps, torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda())
    after = srv.ps_stats()
    assert after["queue_len"] == before["queue_len"] == 0 and after["version"] == before["version"]
    ol, oa, oc, oz = cnn.workers_eval([versions[s.version] for s in snaps], x, y, precision=precision)
    tol = TOL_TENSOR if precision else TOL_FP32
    np.testing.assert_allclose(loss.cpu().numpy(), ol, rtol=3e-3 if precision else 1e-5, atol=1e-6)
    am = am.cpu().numpy()
    n_amb = assert_argmax_valid(am, oz, tol)
    # the count is exact given the labels the kernel chose; it equals the oracle's where no row is ambiguous
    assert (correct.cpu().numpy() == (am == y).sum(axis=1)).all()
    if n_amb == 0:
        assert (correct.cpu().numpy() == oc).all()
    srv.close()


@pytest.mark.parametrize("precision,W,b", [(0, 3, 5), (0, 8, 9), (2, 2, 8), (2, 8, 24), (2, 17, 6), (2, 6, 70)])
def test_summed_step_equals_the_sum_of_the_workers_gradients_and_the_sync_update(precision, W, b):
    """workers_grad_step_summed + ps_apply_summed: the one vector equals the sum of the oracle's per-worker gradients,
    and the update equals the oracle's synchronous step over those gradients (W = 17 has no divisor up to 16 but 1:
    the whole batch goes through one product; W = 8: eight groups; W = 6: six)."""
    from oracle import cnn, ps as ops
    tol = TOL_TENSOR if precision else TOL_FP32
    torch, ps, srv, theta0 = _setup(W, b, 1, 0.25, precision)
    rng = np.random.default_rng(31)
    x = rng.random((W, b, 28, 28), dtype=np.float32)
    y = rng.integers(0, 10, (W, b)).astype(np.int32)
    ids = [(5 * w + 2) % 251 for w in range(W)]
    snaps = [srv.ps_pull_snapshot(w) for w in range(W)]
    xd, yd = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    gsum = torch.full((ps.P_PAD,), float("nan"), device="cuda")
    _, loss, am = srv.workers_grad_step_summed(snaps, ids, xd, yd, SEED, 6, grad_sum_dev=gsum)
    srv.ps_stats()
    og, ol, oa, oz = cnn.workers_grad_step([theta0] * W, ids, x, y, SEED, 6, 0.25, precision=precision)
    got = gsum.cpu().numpy()
    assert (got[ps.P:] == 0).all()
    assert_sum_close(got[:ps.P], og, tol, "summed gradient")
    np.testing.assert_allclose(loss.cpu().numpy(), ol, rtol=3e-3 if precision else 1e-5, atol=1e-6)
    assert_argmax_valid(am.cpu().numpy(), oz, tol)
    # the per-worker path gives the same sum (another order of additions)
    gd = torch.zeros((W, ps.P_PAD), device="cuda")
    srv.workers_grad_step(snaps, ids, xd, yd, SEED, 6, grads_dev=gd)
    assert_params_close(got[:ps.P], gd.sum(dim=0).cpu().numpy()[:ps.P], 1e-5 if precision == 0 else 1e-4, "summed vs per-worker path")
    # the server step
    o = ops.OraclePS(theta0)
    o.enqueue(og.astype(np.float32), ids, [0] * W, 6)
    ro = o.apply(ops.SYNC, 0.01)
    rg = srv.ps_apply_summed(gsum, W, 0.01)
    assert ro == rg
    th, v = srv.ps_export_params()
    assert v == 1
    assert_params_close(th, o.head(), tol, "parameters after the summed step")
    assert_params_close(th.astype(np.float64) - theta0, o.head().astype(np.float64) - theta0, max(tol, 1e-3), "the summed step's update")
    # errors: stale readers need the per-worker path; a non-empty queue must be applied first
    g = torch.zeros((1, ps.P_PAD), device="cuda")
    srv.ps_enqueue([0], [1], 7, grads_dev=g)
    with pytest.raises(ps.PSError) as e:
        srv.ps_apply_summed(gsum, W, 0.01)
    assert e.value.name == "PS_ERR_BAD_ARG"
    srv.close()


@pytest.mark.parametrize("precision", [0, 2])
def test_summed_step_adds_the_workers_in_pairs(precision):
    """128 workers' gradients of the output layer are added up within the root of 1 + 1/2 + 1/4 + ... < 2 of one rounding's
    root mean square, 2^-24 / sqrt(3), as sums in pairs are: the last rounding counts in full, those of the two halves by
    half each, and so on."""
    W = b = 128
    torch, ps, srv, _ = _setup(W, b, precision=precision)
    gen = torch.Generator(device="cuda").manual_seed(W * b)
    x = torch.rand((W, b, 28, 28), generator=gen, device="cuda")
    y = torch.randint(0, 10, (W, b), generator=gen, device="cuda", dtype=torch.int32)
    snaps = [srv.ps_pull_snapshot(w) for w in range(W)]
    grads = torch.zeros((W, ps.P_PAD), device="cuda")
    srv.workers_grad_step(snaps, range(W), x, y, SEED, 1, grads_dev=grads)
    got = srv.workers_grad_step_summed(snaps, range(W), x, y, SEED, 1)[0].double()
    want = grads.double().sum(0)
    for name, o, shape in synth.layout():
        if name in ("fc1.b", "fc2.w"):
            part = slice(o, o + int(np.prod(shape)))
            error = float((got[part] - want[part]).norm() / want[part].norm())
            assert error <= 2.0 ** -24 * (2 / 3) ** 0.5, (name, error)
    srv.close()


def test_summed_step_refuses_mixed_snapshots():
    torch, ps, srv, theta0 = _setup(2, 4, 2, 0.25, 0)
    g = np.zeros((1, ps.P_PAD), dtype=np.float32)
    g[0, :ps.P] = synth.random_gradients(1, seed=52, scale=2.0)[0]
    srv.ps_enqueue([0], [0], 0, grads_dev=torch.from_numpy(g).cuda())
    srv.ps_apply(ps.ASYNC, 0.01)
    snaps = [srv.ps_pull_snapshot(0, 0), srv.ps_pull_snapshot(1, 1)]
    x = torch.zeros((2, 4, 28, 28), device="cuda")
    y = torch.zeros((2, 4), dtype=torch.int32, device="cuda")
    with pytest.raises(ps.PSError) as e:
        srv.workers_grad_step_summed(snaps, [0, 1], x, y, SEED, 0)
    assert e.value.name == "PS_ERR_BAD_ARG"
    srv.close()
