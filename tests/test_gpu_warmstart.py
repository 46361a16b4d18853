"""The learned warm start: the tensor-core network against the CPU
reference network, training, and what the trained network gains over the
method without it on a demagnetisation curve."""
import numpy as np
import pytest

import synth
from oracle import mlp as omlp

pytestmark = pytest.mark.gpu


def _params_list(flat):
    sizes = omlp.SIZES
    out, o = [], 0
    for n_in, n_out in zip(sizes[:-1], sizes[1:]):
        W = flat[o:o + n_in * n_out].reshape(n_out, n_in).astype(np.float64)
        o += n_in * n_out
        b = flat[o:o + n_out].astype(np.float64)
        o += n_out
        out.append((W, b))
    return out


def test_forward_matches_reference():
    import torch
    from paper_1801_03690_gb300 import MLP
    net = MLP(seed=3)
    p = net.get_params()
    p[16 * 128:16 * 128 + 128] = np.random.default_rng(0).normal(size=128) * 0.1   # nonzero b1
    net.set_params(p)
    rng = np.random.default_rng(1)
    X = rng.normal(size=(301, 16)).astype(np.float32)          # ragged tail
    Y = net.forward(torch.tensor(X, device="cuda")).cpu().numpy()
    Yr, _ = omlp.forward(_params_list(p), X.astype(np.float64), round_bf16=True)
    scale = np.abs(Yr).max()
    np.testing.assert_allclose(Y, Yr, rtol=0, atol=1e-2 * scale)


def test_gradient_matches_reference():
    import torch
    from paper_1801_03690_gb300 import MLP
    net = MLP(seed=5)
    p = net.get_params()
    rng = np.random.default_rng(2)
    X = rng.normal(size=(517, 16)).astype(np.float32)
    T = rng.normal(size=(517, 4)).astype(np.float32)
    g, loss = net.gradient(torch.tensor(X, device="cuda"), torch.tensor(T, device="cuda"))
    lr, gr = omlp.loss_and_grads(_params_list(p), X.astype(np.float64), T.astype(np.float64),
                                 round_bf16=True)
    assert loss == pytest.approx(lr, rel=1e-2)
    gflat = _params_list(g)
    for l, ((gw, gb), (rw, rb)) in enumerate(zip(gflat, gr)):
        sw, sb = np.abs(rw).max(), np.abs(rb).max()
        np.testing.assert_allclose(gw, rw, rtol=0, atol=3e-2 * sw, err_msg=f"W{l + 1}")
        np.testing.assert_allclose(gb, rb, rtol=0, atol=3e-2 * sb, err_msg=f"b{l + 1}")


def test_training_fits_a_smooth_map():
    import torch
    from paper_1801_03690_gb300 import MLP
    net = MLP(seed=7)
    rng = np.random.default_rng(3)
    X = torch.tensor(rng.normal(size=(20000, 16)), dtype=torch.float32, device="cuda")
    R = torch.tensor(rng.normal(size=(16, 4)) / 4, dtype=torch.float32, device="cuda")
    T = torch.tanh(X @ R).contiguous()
    first = net.train_step(X[:4096].contiguous(), T[:4096].contiguous(), 1e-3, want_loss=True)
    for i in range(400):
        j = (i * 4096) % (20000 - 4096)
        net.train_step(X[j:j + 4096].contiguous(), T[j:j + 4096].contiguous(), 1e-3)
    _, last = net.gradient(X, T)
    assert last < 0.2 * first


def test_warm_start_gain_on_a_demag_curve():
    """Train on the method's own trajectory of one jittered hard-magnetic
    cube, then run the curve of another jitter of it with and without the
    warm start: the corrected starts must not change the curve (NCG runs to
    t1-t3 either way) and must save NCG iterations."""
    import torch
    from paper_1801_03690_gb300 import MLP, Magnet, Params, warmstart
    prm = Params(jmax=4, precision=1)
    train_wl = synth.hard_cube(n_mag=10, seed=2, n_fields=40)
    test_wl = synth.hard_cube(n_mag=10, seed=9, n_fields=40)
    fields = train_wl.fields[:16]                 # 0 .. -3.1 T: reversible part of the curve
    mag = Magnet()
    mag.upload_workload(train_wl)
    n_mag = mag.sizes()["n_mag"]
    net = MLP(seed=11)
    X, T, _ = warmstart.collect(mag, net, train_wl.m0, fields, n_mag, prm)
    s_m, s_p, _ = warmstart.train(net, X, T, steps=600, batch=8192, lr=2e-3)
    mag.close()
    mag = Magnet()
    mag.upload_workload(test_wl)
    base, nli_base = warmstart.curve(mag, test_wl.m0, fields, prm)
    warm, nli_warm = warmstart.curve(mag, test_wl.m0, fields, prm, mlp=net, scales=(s_m, s_p),
                                     max_change=0.0)          # reversible segment: no cap needed
    assert all(s["status"] == "ok" for s in base + warm)
    Mb = np.array([s["M"] for s in base])
    Mw = np.array([s["M"] for s in warm])
    np.testing.assert_allclose(Mw, Mb, atol=1e-4)
    print(f"NCG iterations without / with the warm start: {nli_base} / {nli_warm}")
    assert nli_warm < nli_base


def test_library_training_statistics_match_their_definitions():
    """The warm start's data arithmetic runs in the library: the input
    standardisation (mean and unbiased standard deviation per feature; a
    constant feature is only centred), the target scales (standard
    deviation of the m columns together and of the potential column) with
    the scaled targets, and a field step's targets ((after - before) / |dh|
    and the largest nodal change), against numpy in FP64."""
    import torch
    from paper_1801_03690_gb300 import MLP
    net = MLP(seed=3)
    rng = np.random.default_rng(12)
    n = 50000
    Xh = rng.normal(size=(n, 16)) * rng.uniform(0.1, 5.0, 16) + rng.uniform(-3, 3, 16)
    Xh[:, 4] = 0.75                                   # constant feature
    Xh[:, 5] = 0.999 + 1e-3 * rng.normal(size=n)      # small spread on a large mean
    Xh = Xh.astype(np.float32)
    X = torch.tensor(Xh, device="cuda")
    net.fit_input_norm(X)
    mean, inv_sd = net.input_norm()
    x64 = Xh.astype(np.float64)
    mu, sd = x64.mean(0), x64.std(0, ddof=1)
    sd = np.where(sd > 1e-6 * (np.abs(mu) + 1.0), sd, 1.0)
    np.testing.assert_allclose(mean, mu, rtol=1e-6, atol=1e-7)
    np.testing.assert_allclose(inv_sd, 1.0 / sd, rtol=1e-6)
    assert inv_sd[4] == 1.0

    Th = (rng.normal(size=(n, 4)) * np.array([0.01, 0.02, 0.03, 5.0])).astype(np.float32)
    T = torch.tensor(Th, device="cuda")
    Tn, s_m, s_p = net.fit_target_scales(T)
    t64 = Th.astype(np.float64)
    assert s_m == pytest.approx(t64[:, :3].reshape(-1).std(ddof=1), rel=1e-9)
    assert s_p == pytest.approx(t64[:, 3].std(ddof=1), rel=1e-9)
    ref = np.concatenate([Th[:, :3] / np.float32(s_m), Th[:, 3:] / np.float32(s_p)], axis=1)
    np.testing.assert_allclose(Tn.cpu().numpy(), ref, rtol=1e-6)

    X1h = Xh.copy()
    X1h[:, 0:3] += (1e-3 * rng.normal(size=(n, 3))).astype(np.float32)
    X1h[:, 15] += (0.1 * rng.normal(size=n)).astype(np.float32)
    X1h[777, 0:3] += np.float32(0.3)                 # one node turns further
    X0 = X.clone()
    X0[:, 12:15] = torch.tensor([0.02, -0.01, -0.05], device="cuda")   # field increment
    X1 = torch.tensor(X1h, device="cuda")
    T2, dh, change = net.step_targets(X0.contiguous(), X1.contiguous())
    dh_ref = np.linalg.norm(np.array([0.02, -0.01, -0.05], dtype=np.float32).astype(np.float64))
    assert dh == pytest.approx(dh_ref, rel=1e-6)
    d = X1h.astype(np.float64) - Xh.astype(np.float64)
    np.testing.assert_allclose(T2.cpu().numpy(), np.concatenate([d[:, :3], d[:, 15:16]], 1) / dh_ref,
                               rtol=1e-4, atol=1e-6)
    assert change == pytest.approx(np.linalg.norm(d[:, :3], axis=1).max(), rel=1e-5)
    X0[:, 12:15] = 0.0
    T3, dh0, _ = net.step_targets(X0.contiguous(), X1.contiguous())
    assert T3 is None and dh0 == 0.0


def _deviation_stats(Y, Yr):
    d = np.abs(Y - Yr) / np.abs(Yr).max()
    return float(d.max()), float(np.quantile(d, 0.5)), float(np.quantile(d, 0.9))


@pytest.mark.parametrize("n", [128, 301, 20000])
def test_tcgen05_forward_matches_reference_and_mma_sync(n):
    """The tcgen05 forward pass (default) against the oracle's network and
    against the warp-level mma.sync path, on full tiles, a ragged tail and
    many tiles.  All three round at the same points (BF16 inputs, weights,
    hidden activations); they differ in FP32 (GPU) vs FP64 (oracle)
    accumulation order, which moves an output by ~1e-6 of the largest and,
    where a hidden activation lies within that of a BF16 rounding boundary,
    flips it by one BF16 unit (2^-8 relative) -- measured: median 5e-9 and
    largest 9e-4 of the largest output over 20,000 rows; the bound on the
    largest is 2e-3.  The two GPU paths accumulate the same products in the
    same order (measured bitwise equal)."""
    import torch
    from paper_1801_03690_gb300 import MLP
    net = MLP(seed=4)
    p = net.get_params()
    rng = np.random.default_rng(9)
    for off in (16 * 128, 16 * 128 + 128 + 128 * 128, 16 * 128 + 2 * (128 + 128 * 128)):
        p[off:off + 128] = rng.normal(size=128) * 0.1                  # nonzero biases
    net.set_params(p)
    X = rng.normal(size=(n, 16)).astype(np.float32)
    Xd = torch.tensor(X, device="cuda")
    Y_tc = net.forward(Xd).cpu().numpy()
    net.set_tensor_path(1)
    Y_ms = net.forward(Xd).cpu().numpy()
    net.set_tensor_path(0)
    Yr, _ = omlp.forward(_params_list(p), X.astype(np.float64), round_bf16=True)
    for name, Y in (("tcgen05", Y_tc), ("mma.sync", Y_ms)):
        mx, med, q90 = _deviation_stats(Y, Yr)
        print(f"{name} vs oracle, n={n}: max {mx:.2e} median {med:.2e} q90 {q90:.2e} (of the largest output)")
        assert mx <= 2e-3 and med <= 1e-5, (name, mx, med)        # measured: max 9e-4, median 5e-9
    mx, med, q90 = _deviation_stats(Y_tc, Y_ms)
    print(f"tcgen05 vs mma.sync, n={n}: max {mx:.2e} median {med:.2e} q90 {q90:.2e}")
    assert mx <= 1e-6                                             # measured: bitwise equal
    assert np.isfinite(Y_tc).all()


@pytest.mark.parametrize("n", [517, 4096])
def test_tcgen05_weight_gradient_matches_mma_sync_and_reference(n):
    """The weight gradients on tcgen05 (one M = 128, K = 128-row MMA product
    per chunk of rows, default) against the mma.sync path on the same
    activations (the same FP32 sums of BF16 products) and against the
    oracle's network gradients."""
    import torch
    from paper_1801_03690_gb300 import MLP
    net = MLP(seed=6)
    p = net.get_params()
    rng = np.random.default_rng(8)
    X = torch.tensor(rng.normal(size=(n, 16)).astype(np.float32), device="cuda")
    T = torch.tensor(rng.normal(size=(n, 4)).astype(np.float32), device="cuda")
    g_tc, loss_tc = net.gradient(X, T)
    net.set_tensor_path(1)
    g_ms, loss_ms = net.gradient(X, T)
    net.set_tensor_path(0)
    assert loss_tc == loss_ms
    scale = np.abs(g_ms).max()
    err = np.abs(g_tc - g_ms).max() / scale
    print(f"tcgen05 vs mma.sync weight gradients, n={n}: max deviation {err:.2e} of the largest")
    assert err <= 1e-5
    lr, gr = omlp.loss_and_grads(_params_list(p), X.cpu().numpy().astype(np.float64),
                                 T.cpu().numpy().astype(np.float64), round_bf16=True)
    for (gw, gb), (rw, rb) in zip(_params_list(g_tc), gr):
        np.testing.assert_allclose(gw, rw, rtol=0, atol=3e-2 * np.abs(rw).max())


@pytest.mark.parametrize("n", [1, 127, 128, 129, 152 * 128 + 1, 8 * 152 * 128 + 300])
def test_training_pass_edges(n):
    """The fused tcgen05 training pass at the edges of its tiles (128 rows), of
    its grid (152 SMs) and of the tiles it accumulates before a flush (8), on
    aligned and on odd addresses, against the mma.sync path: the same products
    of the same BF16 values in FP32, summed in another order.  Rounding errors
    of n / 128 partial sums of either sign grow like 2^-24 sqrt(n / 128) of the
    largest partial: 2e-6 at the largest n, bound 1e-5."""
    import torch
    from paper_1801_03690_gb300 import MLP
    net = MLP(seed=6)
    g = torch.Generator(device="cuda").manual_seed(n)
    buf = torch.randn(20 * n + 1, generator=g, device="cuda")
    X, T = buf[:16 * n].view(n, 16), buf[16 * n:20 * n].view(n, 4)
    g_tc, loss_tc = net.gradient(X, T)
    odd = torch.cat([buf[:1], buf[:-1]])[1:]                        # the same values, 4 bytes off a 16-byte boundary
    assert odd.data_ptr() % 16 == 4
    g_odd, loss_odd = net.gradient(odd[:16 * n].view(n, 16), odd[16 * n:20 * n].view(n, 4))
    assert loss_odd == loss_tc and np.array_equal(g_odd, g_tc)
    net.set_tensor_path(1)
    g_ms, loss_ms = net.gradient(X, T)
    assert loss_tc == loss_ms
    for (gw, gb), (rw, rb) in zip(_params_list(g_tc), _params_list(g_ms)):
        assert np.abs(gw - rw).max() <= 1e-5 * np.abs(rw).max()
        assert np.abs(gb - rb).max() <= 1e-5 * np.abs(rb).max()


@pytest.mark.parametrize("n,centre,scale", [(2, 0.0, 1.0), (127, 3.0, 0.5), (128 * 33 + 5, 1e4, 1.0), (700001, -2.0, 3.0),
                                            (1000, 1e22, 1e21), (5000, 1e-30, 1e-30)])
def test_statistics_edges(n, centre, scale):
    """The one-pass statistics against FP64 ones of the same values: tails of a
    block and of a fold, means far from zero, an odd address, and squares
    beyond or below FP32, which go to (or give the same as) the FP64 passes.
    Means and scales come back as FP32 (relative error 2^-24, bound 1e-6 of the
    deviation or of the value); the target scales as FP64 from sums of pairs of
    FP32 words (2^-45 at worst, bound 1e-12)."""
    import torch
    from paper_1801_03690_gb300 import MLP
    net = MLP(seed=1)
    rng = np.random.default_rng(n)
    buf = (centre + scale * rng.normal(size=20 * n + 1)).astype(np.float32)
    X = buf[1:16 * n + 1].reshape(n, 16)
    X[:, 13] = 0.37                                          # a constant column
    T = buf[16 * n + 1:].reshape(n, 4)
    dev = torch.tensor(buf, device="cuda")
    Xd, Td = dev[1:16 * n + 1].view(n, 16), dev[16 * n + 1:].view(n, 4)
    net.fit_input_norm(Xd)
    mean, istd = net.input_norm()
    X64, T64 = X.astype(np.float64), T.astype(np.float64)
    m, s = X64.mean(0), X64.std(0, ddof=1)
    s = np.where(s > 1e-6 * (np.abs(m) + 1.0), s, 1.0)
    np.testing.assert_allclose(mean, m, rtol=1e-6, atol=1e-6 * X64.std(0, ddof=1).max())
    np.testing.assert_allclose(istd, 1.0 / s, rtol=1e-6)
    Tn, sm, sp = net.fit_target_scales(Td)
    em, ep = max(T64[:, :3].std(ddof=1), 1e-12), max(T64[:, 3].std(ddof=1), 1e-12)
    assert abs(sm - em) <= 1e-12 * em and abs(sp - ep) <= 1e-12 * ep
    ref = T / np.array([sm, sm, sm, sp], dtype=np.float32)
    np.testing.assert_allclose(Tn.cpu().numpy(), ref, rtol=2.0 ** -22)
    Xd[n - 1, 3] = float("nan")
    with pytest.raises(Exception):
        net.fit_input_norm(Xd)


@pytest.mark.parametrize("side", [False, True])
def test_train_step_is_ordered_against_the_caller(side):
    """A step without a loss reads its batch after the work queued before the
    call (a long one and the copies that fill the batch) and before what is
    queued after it (the batch is overwritten at once), on the default stream
    and on one that does not block on it.  The pass sums in a fixed order, so
    the parameters are those of a run that waits at every point."""
    import torch
    from paper_1801_03690_gb300 import MLP
    g = torch.Generator(device="cuda").manual_seed(4)
    data = [(torch.randn((3000, 16), generator=g, device="cuda"), torch.randn((3000, 4), generator=g, device="cuda"))
            for _ in range(4)]
    want = MLP(seed=8)
    for X, T in data:
        torch.cuda.synchronize()
        want.train_step(X, T, 1e-3, want_loss=True)
    net = MLP(seed=8)
    Xb, Tb = torch.zeros((3000, 16), device="cuda"), torch.zeros((3000, 4), device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream() if side else torch.cuda.default_stream()):
        for X, T in data:
            torch.cuda._sleep(10_000_000)
            Xb.copy_(X)
            Tb.copy_(T)
            net.train_step(Xb, Tb, 1e-3)
            Xb.fill_(float("nan"))
            Tb.fill_(float("nan"))
        got = net.get_params()
    torch.cuda.synchronize()
    assert np.array_equal(got, want.get_params())


def test_a_wait_that_runs_out_leaves_the_network_as_it_was():
    """With a limit of 0 every tensor-core wait counts as run out (the kernel
    still lets its products finish).  The call that reports it is the next one
    that waits; the steps up to then change neither weights nor moments nor the
    step count, so training goes on as if they had not been asked for."""
    import torch
    from paper_1801_03690_gb300 import MLP, MMError
    g = torch.Generator(device="cuda").manual_seed(9)
    X, T = torch.randn((700, 16), generator=g, device="cuda"), torch.randn((700, 4), generator=g, device="cuda")
    net, twin = MLP(seed=8), MLP(seed=8)
    for n in (net, twin):
        n.train_step(X, T, 1e-2)
        n.train_step(X, T, 1e-2)
    before = net.get_params()
    net.set_wait_limit(0)
    net.train_step(X, T, 1e-2)
    net.set_wait_limit(2_000_000_000)
    net.train_step(X, T, 1e-2)                               # sound, but after one that was not and is not reported yet
    with pytest.raises(MMError):
        net.get_params()
    assert np.array_equal(net.get_params(), before)
    net.set_wait_limit(0)
    for call in (lambda: net.train_step(X, T, 1e-2, want_loss=True), lambda: net.gradient(X, T), lambda: net.forward(X)):
        with pytest.raises(MMError):
            call()
        assert np.array_equal(net.get_params(), before)      # reported once
    net.set_wait_limit(2_000_000_000)
    for _ in range(2):
        assert net.train_step(X, T, 1e-2, want_loss=True) == twin.train_step(X, T, 1e-2, want_loss=True)
    assert np.array_equal(net.get_params(), twin.get_params())
    with pytest.raises(MMError):
        net.set_wait_limit(-1)


@pytest.mark.parametrize("kind", ["default", "blocking", "side"])
def test_statistics_wait_for_the_data(kind):
    """The statistics of data that are still in the making on the default
    stream, on one that blocks on it and on a current stream that does not:
    the same as those of finished data (the sums have a fixed order)."""
    import ctypes
    import torch
    from paper_1801_03690_gb300 import MLP
    g = torch.Generator(device="cuda").manual_seed(2)
    X0, T0 = torch.randn((5000, 16), generator=g, device="cuda"), torch.randn((5000, 4), generator=g, device="cuda")
    torch.cuda.synchronize()
    net = MLP(seed=1)
    net.fit_input_norm(X0)
    want = (*net.input_norm(), *net.fit_target_scales(T0)[1:])
    handle = ctypes.c_void_p()
    if kind == "blocking":
        assert int(torch.cuda.cudart().cudaStreamCreate(ctypes.addressof(handle))) == 0
    stream = {"default": torch.cuda.default_stream, "side": torch.cuda.Stream,
              "blocking": lambda: torch.cuda.ExternalStream(handle.value)}[kind]()
    X, T = torch.zeros_like(X0), torch.zeros_like(T0)
    torch.cuda.synchronize()

    def make():
        torch.cuda._sleep(10_000_000)
        X.copy_(X0)
        T.copy_(T0)

    with torch.cuda.stream(stream):
        make()
        if kind == "side":
            net.fit_input_norm(X)
    if kind != "side":
        net.fit_input_norm(X)
    mean, istd = net.input_norm()
    X.zero_(), T.zero_()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        make()
        if kind == "side":
            got = net.fit_target_scales(T)
    if kind != "side":
        got = net.fit_target_scales(T)
    assert np.array_equal(mean, want[0]) and np.array_equal(istd, want[1]) and got[1:] == want[2:]
    torch.cuda.synchronize()
    if kind == "blocking":
        assert int(torch.cuda.cudart().cudaStreamDestroy(handle.value)) == 0


@pytest.mark.parametrize("rows_per_thread", [1, 8, 32])
def test_target_scales_hold_fp64_sums(rows_per_thread):
    """Equal squares, whose rounding errors all have one sign, over a full fold
    of every thread and less.  Sums in FP64 from a tree of 64 additions (fold,
    warp, block, the blocks' partials) lose 64 x 2^-53 at most, the deviation
    half of that; two more for the division and the root."""
    import torch
    from paper_1801_03690_gb300 import MLP
    n = rows_per_thread * 1024 * torch.cuda.get_device_properties(0).multi_processor_count
    a = np.float32(float.fromhex("0x1.1f95f4p+0"))
    T = torch.full((n, 4), float(a), device="cuda")
    T[n // 2:] = -float(a)
    _, sm, sp = MLP(seed=1).fit_target_scales(T)
    for got, count in ((sm, 3 * n), (sp, n)):
        want = np.longdouble(a) * np.sqrt(np.longdouble(count) / np.longdouble(count - 1))
        assert abs(np.longdouble(got) / want - 1) <= 34 * 2.0 ** -53


@pytest.mark.parametrize("n", [1, 127, 129, 20011])
def test_forward_on_odd_addresses(n):
    """Inputs and outputs off a 16-byte boundary take scalar loads and stores;
    the outputs are those of aligned arrays, bit by bit."""
    import ctypes as C
    import torch
    from paper_1801_03690_gb300 import MLP
    net = MLP(seed=4)
    g = torch.Generator(device="cuda").manual_seed(n)
    X = torch.randn((n, 16), generator=g, device="cuda")
    Y = net.forward(X)
    xb, yb = torch.zeros(16 * n + 1, device="cuda"), torch.full((4 * n + 2,), 7.0, device="cuda")
    xb[1:] = X.reshape(-1)
    torch.cuda.synchronize()
    for x, y in ((xb[1:], yb[1:-1]), (X, yb[1:-1]), (xb[1:], torch.empty(4 * n, device="cuda"))):
        rc = net._lib.mm_mlp_forward(net._h, C.c_void_p(x.data_ptr()), n, C.c_void_p(y.data_ptr()))
        assert rc == 0 and torch.equal(y.view(n, 4), Y)
    assert yb[0] == 7.0 and yb[-1] == 7.0


@pytest.mark.parametrize("path", [0, 1])
@pytest.mark.parametrize("tiles", [0, 1, "sms"])
def test_adam_steps_match_fp64(path, tiles):
    """Training steps against Adam in FP64 from the gradient that each step has
    (the same pass, without the update), at 1 row, one row more than a tile and
    one more than a tile per SM; and the BF16 copies are those of the weights.
    Per step a weight rounds once (2^-24 of itself, counted twice), and its
    change, at most 1.1 lr in these four steps, has the rounding errors of the
    moments, quotients and root (about ten of 2^-24) and that of 1 - beta2^k,
    where the difference of two numbers near one keeps 7e-6: together below
    2e-5 of 2 lr."""
    import torch
    from paper_1801_03690_gb300 import MLP
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 1 + 128 * (sms if tiles == "sms" else tiles)
    net = MLP(seed=6)
    net.set_tensor_path(path)
    g = torch.Generator(device="cuda").manual_seed(n)
    lr, b1, b2 = np.float32(2e-3), float(np.float32(0.9)), float(np.float32(0.999))
    p = net.get_params().astype(np.float64)
    m, v = np.zeros_like(p), np.zeros_like(p)
    for k in range(1, 5):
        X, T = torch.randn((n, 16), generator=g, device="cuda"), torch.randn((n, 4), generator=g, device="cuda")
        gr, loss = net.gradient(X, T)
        assert net.train_step(X, T, float(lr), want_loss=True) == loss
        gr = gr.astype(np.float64)
        m, v = b1 * m + (1 - b1) * gr, b2 * v + (1 - b2) * gr * gr
        p = p - float(lr) * (m / (1 - b1 ** k)) / (np.sqrt(v / (1 - b2 ** k)) + 1e-8)
        got = net.get_params()
        assert np.all(np.abs(got - p) <= k * (2.0 ** -23 * np.abs(p) + 2e-5 * 2 * float(lr)))
    twin = MLP(seed=1)
    twin.set_tensor_path(path)
    twin.set_params(got)
    assert torch.equal(net.forward(X), twin.forward(X))
