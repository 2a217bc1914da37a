"""The surrogate network's GPU kernels against the FP64 oracle: forward
outputs and every parameter gradient in the FP32 check mode (<= 1e-5) and
with BF16 tensor-core products (<= 2e-2), the fused inference kernel against
the training kernels, AdamW against the oracle's update, and a monotone
training loss on a fixed batch."""
import numpy as np
import pytest

from oracle import mlp_oracle as M
from paper_2408_15115_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _data(n, seed):
    rng = np.random.default_rng(seed)
    x = rng.standard_normal((n, M.N_IN)) * rng.uniform(0.5, 3.0, M.N_IN) + rng.uniform(-2, 2, M.N_IN)
    y = np.tanh(x[:, :6] * 0.7) + 0.1 * x[:, 6:12] * x[:, 12:18] + 0.3
    return x, y


def _norm(x, y):
    mx, sx = M.standardisation(x)
    my, sy = M.standardisation(y)
    return mx, sx, my, sy


def _net(precision, p, norm, cap=512):
    from paper_2408_15115_gb300 import turret as T
    net = T.MLP(p.astype(np.float32), batch_cap=cap, precision=precision)
    net.set_norm(*[v.astype(np.float32) for v in norm])
    return net


def _oracle(p, x, y, norm):
    mx, sx, my, sy = norm
    # the oracle sees the float32 values the GPU sees
    f = lambda a: np.asarray(a, dtype=np.float32).astype(np.float64)
    xs = (f(x) - f(mx)) / f(sx)
    ts = (f(y) - f(my)) / f(sy)
    out, _ = M.forward(f(p), xs)
    L, g = M.loss_and_grad(f(p), xs, ts)
    return out * f(sy) + f(my), L, g


def _per_tensor_err(g, ref):
    worst = 0.0
    for k, (o, s) in M.OFFSETS.items():
        n = int(np.prod(s))
        a, b = g[o:o + n], ref[o:o + n]
        worst = max(worst, float(np.abs(a - b).max() / max(np.abs(b).max(), 1e-30)))
    return worst


@pytest.mark.parametrize("precision,tol", [("fp32", 1e-5), ("bf16", 2e-2)])
def test_forward_and_gradients_vs_oracle(precision, tol):
    # 300 rows: several 64-row tiles and a ragged tail
    x, y = _data(300, 1)
    norm = _norm(x, y)
    p = I.mlp_init_params(3)
    net = _net(precision, p, norm)
    want_y, want_L, want_g = _oracle(p, x, y, norm)
    got_y = net.forward(x).cpu().numpy().astype(np.float64)
    assert np.abs(got_y - want_y).max() / np.abs(want_y).max() < tol
    L, g = net.loss_grad(x, y)
    assert abs(L - want_L) / want_L < tol
    assert _per_tensor_err(g.cpu().numpy().astype(np.float64), want_g) < tol
    net.close()


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_inference_kernel_matches_training_forward(precision):
    x, y = _data(37, 2)  # three blocks of 16 rows, ragged
    norm = _norm(x, y)
    net = _net(precision, I.mlp_init_params(4), norm)
    a = net.forward(x).cpu().numpy()
    b = net.infer(x).cpu().numpy()
    if precision == "bf16":
        # same BF16 operands and k order of the mma products
        assert np.array_equal(a, b)
    else:
        assert np.abs(a - b).max() <= 1e-5 * np.abs(a).max()
    net.close()


def test_adamw_step_vs_oracle():
    import torch
    x, y = _data(256, 5)
    norm = _norm(x, y)
    p = I.mlp_init_params(6).astype(np.float32).astype(np.float64)
    net = _net("fp32", p, norm)
    lr, wd = 1e-3, 0.01
    xt = torch.tensor(x, dtype=torch.float32, device="cuda:0")
    yt = torch.tensor(y, dtype=torch.float32, device="cuda:0")
    torch.cuda.synchronize()
    net.train_step(xt, yt, lr=lr, weight_decay=wd)
    got = net.params().astype(np.float64)
    _, _, g = _oracle(p, x, y, norm)
    want, _, _ = M.adamw(p, g, np.zeros_like(p), np.zeros_like(p), 1, lr, wd=wd)
    # the first step moves each parameter by lr g / (|g| + eps): compare where
    # the gradient is not vanishing (its sign is then unambiguous)
    sig = np.abs(g) > 1e-4 * np.abs(g).max()
    assert sig.mean() > 0.5
    assert np.abs(got - want)[sig].max() < 1e-6
    net.close()


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_training_loss_is_monotone_on_a_fixed_batch(precision):
    import torch
    x, y = _data(512, 7)
    norm = _norm(x, y)
    net = _net(precision, I.mlp_init_params(8), norm)
    xt = torch.tensor(x, dtype=torch.float32, device="cuda:0")
    yt = torch.tensor(y, dtype=torch.float32, device="cuda:0")
    torch.cuda.synchronize()
    losses = [net.train_step(xt, yt, lr=3e-4) for _ in range(60)]
    assert all(b < a for a, b in zip(losses, losses[1:])), losses
    assert losses[-1] < 0.5 * losses[0]
    net.close()


@pytest.mark.parametrize("n", [1, 31, 33, 257, 7000])
def test_bf16_gradients_at_block_and_slice_edges(n):
    # 32-row blocks, 256-row gradient slices, and more slices than the first
    # partial-sum buffer holds; the BF16 bar of the gradient test above
    x, y = _data(max(n, 64), 9)  # the standardisation needs some spread
    norm = _norm(x, y)
    x, y = x[:n], y[:n]
    p = I.mlp_init_params(10)
    net = _net("bf16", p, norm, cap=n)
    want_y, want_L, want_g = _oracle(p, x, y, norm)
    got_y = net.forward(x).cpu().numpy().astype(np.float64)
    assert np.abs(got_y - want_y).max() / np.abs(want_y).max() < 2e-2
    L, g = net.loss_grad(x, y)
    assert abs(L - want_L) / want_L < 2e-2
    assert _per_tensor_err(g.cpu().numpy().astype(np.float64), want_g) < 2e-2
    net.close()


@pytest.mark.parametrize("n", [9728, 9729, 9856, 9857, 19456, 19457, 39000, 78000])
def test_many_rows_give_the_bits_of_few(n):
    # above 304 x 32 rows a block may take 128 of them (an even number of rounds of
    # narrow blocks, or more than eight): at the edges of the rule, of a block and of
    # a round, and several rounds.  A row's products, sums
    # and their order are the same in every block, so its outputs are too.
    x, y = _data(n, 6)
    net = _net("bf16", I.mlp_init_params(5), _norm(x, y))
    whole = net.infer(x).cpu().numpy()
    parts = np.concatenate([net.infer(x[i:i + 4001]).cpu().numpy() for i in range(0, n, 4001)])
    assert np.array_equal(whole.view(np.uint32), parts.view(np.uint32))
    net.close()


@pytest.mark.parametrize("precision", ["bf16", "fp32"])
def test_training_step_outlives_its_inputs(precision):
    # the network's stream is busy when the steps are enqueued; their inputs are
    # dropped at once and the next allocations of that size overwritten
    import torch
    x, y = _data(256, 3)
    norm, p = _norm(x, y), I.mlp_init_params(2)
    xs = torch.tensor(x, dtype=torch.float32, device="cuda:0")
    ys = torch.tensor(y, dtype=torch.float32, device="cuda:0")
    want, got = _net(precision, p, norm), _net(precision, p, norm)
    torch.cuda.synchronize()
    for k in range(3):
        want.train_step(xs * (k + 1), ys + k)
    for _ in range(2):
        with torch.cuda.stream(got.stream):
            torch.cuda._sleep(20_000_000)  # about 10 ms
        for k in range(3):
            a, b = xs * (k + 1), ys + k
            assert got.train_step(a, b, want_loss=False) is None
            del a, b
            junk = [torch.full_like(xs, 7.0), torch.full_like(ys, -7.0)]  # noqa: F841
        torch.cuda.synchronize()
        assert np.array_equal(got.params().view(np.uint32), want.params().view(np.uint32))
        got.close()
        got = _net(precision, p, norm)
    want.close()
    got.close()


def test_training_step_beside_a_capture():
    # a capture of the caller's stream neither takes the step in nor refuses it
    import torch
    x, y = _data(64, 3)
    norm, p = _norm(x, y), I.mlp_init_params(2)
    xs = torch.tensor(x, dtype=torch.float32, device="cuda:0")
    ys = torch.tensor(y, dtype=torch.float32, device="cuda:0")
    want, got = _net("bf16", p, norm), _net("bf16", p, norm)
    torch.cuda.synchronize()
    want.train_step(xs, ys)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        z = xs + 1.0
        got.train_step(xs, ys, want_loss=False)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(z, xs + 1.0)
    assert np.array_equal(got.params().view(np.uint32), want.params().view(np.uint32))
    want.close()
    got.close()


def test_epochs_are_gathered_in_parts(monkeypatch):
    # the parts change neither the minibatches nor their order, and bound the
    # memory an epoch takes beside a large set (its own size is 671 MB here)
    import torch
    from paper_2408_15115_gb300 import surrogate as S
    x, y = (torch.tensor(a, dtype=torch.float32, device="cuda:0") for a in _data(1000, 3))
    runs = []
    for rows in (S.GATHER_ROWS, 100, 1):
        monkeypatch.setattr(S, "GATHER_ROWS", rows)
        net, hist = S.train(x, y, epochs=2, batch=64, seed=4)
        runs.append((hist, net.params()))
        net.close()
    monkeypatch.undo()
    for hist, p in runs[1:]:
        assert hist == runs[0][0]
        assert np.array_equal(p.view(np.uint32), runs[0][1].view(np.uint32))
    n = 1 << 22
    x, y = x.repeat(-(-n // 1000), 1)[:n].clone(), y.repeat(-(-n // 1000), 1)[:n].clone()
    net = _net("bf16", I.mlp_init_params(2), _norm(*(a[:1000].cpu().numpy().astype(np.float64) for a in (x, y))),
               cap=1 << 14)
    torch.cuda.synchronize()
    torch.cuda.reset_peak_memory_stats()
    before = torch.cuda.memory_allocated()
    S.train(x, y, epochs=1, batch=1 << 14, net=net)
    assert torch.cuda.max_memory_allocated() - before < 8 * n + 2 * 160 * S.GATHER_ROWS + (1 << 24)
    net.close()
