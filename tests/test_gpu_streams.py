"""Memory that passes between the caller's stream and a context's own: what the
caller's stream still reads or writes is finished before the context uses it."""
import numpy as np
import pytest

from paper_2408_15115_gb300 import inputs as I

pytestmark = pytest.mark.gpu

BUSY = 20_000_000  # cycles, about 10 ms


def _small(seed):
    from paper_2408_15115_gb300 import turret as T
    t = T.Turret(20, 20, 28, 0.05, 2.5, (0, 0, -1e-4), 0, 0, 1, 2, sponge=4)
    t.set_fields(*I.random_state((28, 20, 20), u_amp=0.01, rho_amp=0.001, kmax=2, seed=seed))
    return t


@pytest.mark.parametrize("read", ["macro", "populations"])
def test_field_reads_follow_the_readers_of_their_memory(read):
    # the first read is still being copied on the caller's stream when its memory
    # is handed to the second
    import torch
    a, b = _small(1), _small(2)
    want = [getattr(t, read)().cpu() for t in (a, b)]
    first = getattr(a, read)()
    where = first.data_ptr()
    torch.cuda._sleep(BUSY)
    copy = first.clone()
    del first
    second = getattr(b, read)()
    assert second.data_ptr() == where
    assert torch.equal(copy.cpu(), want[0])
    assert torch.equal(second.cpu(), want[1])
    a.close()
    b.close()


def test_workspaces_and_logs_follow_the_writers_of_their_memory():
    # a context, its surface and its log are made from memory that the caller's
    # stream still writes; then the log is replaced while steps write the old one
    import torch
    from paper_2408_15115_gb300 import turret as T
    V, Tr = I.sphere(3, 5.0)

    def run(busy):
        if busy:
            torch.cuda.empty_cache()
            junk = torch.empty(1 << 27, dtype=torch.uint8, device="cuda:0")
            torch.cuda._sleep(BUSY)
            junk.fill_(0x3f)
            del junk
        t = _small(3)
        t.load_surface(V, Tr, (9.6, 10.2, 16.3))
        if busy:
            torch.cuda._sleep(BUSY)
        t.set_log(8)
        t.step(9)
        first = t.log_records()
        t.set_log(16)
        junk = [torch.full((8, T.Turret.LOG_REC), 5.0, dtype=torch.float64, device="cuda:0") for _ in range(4)]
        t.step(3)
        out = [first.cpu().numpy(), t._log.cpu().numpy(), t.populations().cpu().numpy()]
        assert all(bool((j == 5.0).all()) for j in junk)
        t.close()
        return out

    want = run(False)
    for a, b in zip(run(True), want):
        assert np.array_equal(a, b, equal_nan=True)


def test_networks_in_use_are_kept():
    # a refused change of the predictor leaves the context with its network, and
    # the network keeps its memory; a replaced one outlives the steps that read it
    import torch
    from paper_2408_15115_gb300 import turret as T
    V, Tr = I.sphere(3, 5.0)

    def net(seed):
        n = T.MLP(I.mlp_init_params(seed).astype(np.float32), batch_cap=64)
        n.set_norm(np.zeros(T.MLP_IN), np.ones(T.MLP_IN), np.zeros(T.MLP_OUT), np.full(T.MLP_OUT, 1e-3))
        return n

    def run(spoil):
        t = _small(4)
        t.load_surface(V, Tr, (9.6, 10.2, 16.3))
        keep = [net(1), net(2)]
        t.set_predictor("mlp", keep[0], resid_theta=1e30)
        if spoil:
            with pytest.raises(T.TurretError):
                t.set_predictor("mlp", net(9), slip_eps=-1.0)
            assert t._net is keep[0]
            keep[0] = None
        t.step(9)
        t.set_predictor("mlp", keep[1], resid_theta=1e30)
        junk = torch.full((1 << 20,), -1, dtype=torch.int32, device="cuda:0")  # noqa: F841
        t.step(3)
        assert t.predictor_stats()["net_steps"] > 0
        out = t.populations().cpu().numpy()
        t.close()
        return out

    want = run(False)
    assert np.array_equal(run(True), want)
