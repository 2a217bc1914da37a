"""GPU parity of the standalone spreading operator (Sec. 2.2, step l = 1)
with the oracle's dense loops, on a ragged grid, plus its domain check."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2408_15115_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _case(seed=0, shape=(28, 20, 24), n=4):
    nz, ny, nx = shape
    V, T = I.icosphere(n, 5.5)
    rng = np.random.default_rng(seed)
    X = V + np.array([nx / 2 - 0.37, ny / 2 + 0.21, nz / 2 + 0.05]) + 0.1 * rng.standard_normal(3)
    h = 1e-3 * rng.standard_normal((X.shape[0], 3))
    dS = O.mesh_props(V, T)["dS"]
    return X, h, dS, shape


def _gpu_spread(X, h, dS, shape):
    import torch
    from paper_2408_15115_gb300 import turret as T
    dev = torch.device("cuda:0")
    Xt = torch.tensor(np.ascontiguousarray(X.T), dtype=torch.float32, device=dev)
    ht = torch.tensor(np.ascontiguousarray(h.T), dtype=torch.float32, device=dev)
    dt = torch.tensor(dS, dtype=torch.float32, device=dev)
    return T.ibm_spread(Xt, ht, dt, shape).cpu().numpy()


def test_spread_matches_oracle():
    X, h, dS, shape = _case()
    got = np.moveaxis(_gpu_spread(X, h, dS, shape), 0, -1).astype(np.float64)
    want = O.spread(h, X, dS, shape, (False, False, False))
    # FP32 weights and sums of at most ~30 terms per cell
    assert np.abs(got - want).max() <= 1e-5 * np.abs(want).max()
    # total force is conserved by the spreading (partition of unity)
    assert np.abs(got.reshape(-1, 3).sum(0) - (h * dS[:, None]).sum(0)).max() < 1e-5 * np.abs(h * dS[:, None]).sum()


def test_spread_is_reproducible():
    X, h, dS, shape = _case(seed=3)
    a = _gpu_spread(X, h, dS, shape)
    b = _gpu_spread(X, h, dS, shape)
    assert np.array_equal(a, b)


def test_spread_rejects_marker_outside_grid():
    from paper_2408_15115_gb300 import turret as T
    X, h, dS, shape = _case()
    X = X.copy()
    X[0] = (0.5, 5.0, 5.0)  # stencil starts at -1
    with pytest.raises(T.TurretError) as e:
        _gpu_spread(X, h, dS, shape)
    assert e.value.status == 7


@pytest.mark.parametrize("shape,n,radius,copies", [((4, 4, 4), 4, 0.0, 1), ((9, 7, 5), 4, 0.3, 1), ((40, 61, 35), 9, 8.0, 1),
                                                   ((18, 22, 20), 5, 3.0, 8)])
def test_spread_lists_at_grid_and_list_edges(shape, n, radius, copies):
    """One tile; grids no multiple of a tile; many empty tiles; lists of more
    candidates than one staged chunk (a surface repeated at the same place)."""
    nz, ny, nx = shape
    V, T = I.icosphere(n, 1.0)
    rng = np.random.default_rng(7)
    centre = np.array([nx, ny, nz]) / 2.0 - 0.5
    X = np.concatenate([radius * V + centre + 0.05 * rng.standard_normal(3) for _ in range(copies)])
    X = X.astype(np.float32).astype(np.float64)  # the positions the GPU sees
    h = 1e-3 * rng.uniform(0.2, 1.0, (X.shape[0], 3))
    dS = rng.uniform(0.5, 1.0, X.shape[0])
    got = np.moveaxis(_gpu_spread(X, h, dS, shape), 0, -1).astype(np.float64)
    want = O.spread(h, X, dS, shape, (False, False, False))
    # a cell sums at most m non-negative terms: FP32 weights (a few ulp) and m
    # additions give a relative error below (m + 16) 2^-24; the oracle's
    # stencil skips the same cells (m <= all markers, a loose bound)
    tol = (X.shape[0] + 16) * 2.0 ** -24
    assert np.abs(got - want).max() <= tol * np.abs(want).max()
    assert np.array_equal(got == 0.0, want == 0.0) or np.abs(want[got == 0.0]).max() <= tol * np.abs(want).max()


def _spread_into(X, h, dS, shape, offset, fill):
    # the C call on a field `offset` floats past a 256-byte boundary and a scratch,
    # both full of `fill` bytes
    import ctypes as C
    import torch
    from paper_2408_15115_gb300 import turret as T
    nz, ny, nx = shape
    n, L = X.shape[0], T.lib()
    dev = [torch.tensor(np.ascontiguousarray(a.T), dtype=torch.float32, device="cuda:0") for a in (X, h, dS)]
    nb = L.ibm_spread_workspace_bytes(nx, ny, nz, n)
    ws = torch.full((nb + 256,), fill, dtype=torch.uint8, device="cuda:0")
    out = torch.full((4 * (3 * nx * ny * nz + 64 + offset),), fill, dtype=torch.uint8, device="cuda:0")
    out = out[(-out.data_ptr()) % 256 + 4 * offset:][:12 * nx * ny * nz]
    rc = L.ibm_spread(*[C.c_void_p(d.data_ptr()) for d in dev], n, nx, ny, nz, C.c_void_p(out.data_ptr()),
                      C.c_void_p(ws.data_ptr() + (-ws.data_ptr()) % 256), C.c_size_t(nb),
                      C.c_void_p(torch.cuda.current_stream().cuda_stream))
    return rc, out.cpu().numpy().view(np.float32).reshape((3,) + shape)


@pytest.mark.parametrize("offset", [0, 1, 2])
@pytest.mark.parametrize("shape", [(8, 8, 8), (23, 31, 29)])
def test_spread_clears_every_cell_no_stencil_reaches(shape, offset):
    # 0xff bytes are NaN: no cell keeps what the field or the scratch held, and a
    # cell outside every stencil is zero exactly, on aligned and unaligned fields
    nz, ny, nx = shape
    rng = np.random.default_rng(1)
    X = 1.5 + np.array([nx - 4.5, ny - 4.5, nz - 4.5]) * rng.uniform(0.0, 0.3, (40, 3))
    X = X.astype(np.float32).astype(np.float64)
    h, dS = rng.uniform(0.5, 1.0, (40, 3)), rng.uniform(0.5, 1.0, 40)
    rc, got = _spread_into(X, h, dS, shape, offset, 0xff)
    assert rc == 0
    reach = np.zeros(shape, dtype=bool)
    for x, y, z in np.floor(X).astype(int):
        reach[z - 1:z + 3, y - 1:y + 3, x - 1:x + 3] = True
    assert reach.any() and not reach.all()
    assert np.isfinite(got).all() and (got[:, ~reach] == 0.0).all()
    want = O.spread(h, X, dS, shape, (False, False, False))
    tol = (40 + 16) * 2.0 ** -24  # as above: sums of at most 40 positive terms
    assert np.abs(np.moveaxis(got, 0, -1) - want).max() <= tol * np.abs(want).max()


@pytest.mark.parametrize("n", [511, 512, 513, 1024, 1025, 2048, 2049])
def test_spread_of_long_lists(n):
    # n markers in one cell: lists that are ranked (512 at most) and sorted, at the
    # edges of the padded sizes; one more than a list holds is refused.  The sum's
    # order is that of the markers, whatever order they arrive in: repeated calls
    # agree bitwise
    shape = (8, 8, 8)
    rng = np.random.default_rng(n)
    X = (4.1 + 0.8 * rng.random((n, 3))).astype(np.float32).astype(np.float64)
    h, dS = rng.uniform(0.2, 1.0, (n, 3)), rng.uniform(0.5, 1.0, n)
    rc, got = _spread_into(X, h, dS, shape, 0, 0x3f)
    if n > 2048:
        assert rc == 8
        return
    assert rc == 0
    want = O.spread(h, X, dS, shape, (False, False, False))
    tol = (n + 16) * 2.0 ** -24  # as above, n positive terms
    assert np.abs(np.moveaxis(got, 0, -1) - want).max() <= tol * np.abs(want).max()
    for _ in range(3):
        assert np.array_equal(_spread_into(X, h, dS, shape, 0, 0xff)[1], got)
