"""The forms a call is run in agree bitwise: reads of the fields on x-adjacent
pairs and one cell at a time, windows swept as flat blocks, and coupled steps
whose tile lists are built ahead (beside the far cells, or each launch beside the
one before it) against one launch after another."""
import ctypes as C

import numpy as np
import pytest

from oracle import oracle as O
from paper_2408_15115_gb300 import inputs as I

from cases import gpu_velocity, make_pair, rel_max, sphere_case

pytestmark = pytest.mark.gpu


def _fields(shape, seed=1):
    return I.random_state(shape, u_amp=0.01, rho_amp=0.001, kmax=3, seed=seed)


def _both_reads(t, name, n):
    # an 8-byte aligned array takes the pair form, one 4 bytes further on the other
    import torch
    cells = int(np.prod(t.shape))
    buf = torch.empty(2 * n * cells + 1, dtype=torch.float32, device=t.device)
    assert buf.data_ptr() % 8 == 0
    rows = [buf[:n * cells], buf[n * cells + 1:]]
    assert rows[1].data_ptr() % 8 == 4
    for r in rows:
        assert getattr(t._L, name)(t.ctx, C.c_void_p(r.data_ptr())) == 0
    return [r.cpu().numpy().view(np.uint32) for r in rows]


@pytest.mark.parametrize("storage", ["f16", "bf16"])
@pytest.mark.parametrize("shape,bc,sponge", [((4, 2, 64), (0, 0, 0, 0), 0), ((6, 4, 128), (0, 1, 1, 2), 2),
                                             ((10, 6, 64), (1, 0, 1, 1), 0)])
def test_field_reads_on_pairs(storage, shape, bc, sponge):
    nz, ny, nx = shape
    t, _ = make_pair(nx, ny, nz, 0.05, bc, sponge=sponge, storage=storage, fields=_fields(shape, 11))
    for steps in (0, 3):
        t.step(steps)
        for name, n in (("lbm_copy_macro", 4), ("lbm_copy_populations", 27)):
            a, b = _both_reads(t, name, n)
            assert np.array_equal(a, b), (name, steps)


def test_field_reads_on_pairs_of_a_sliding_window():
    # a heavy sphere falls through its anchor: the ring turns and planes enter
    V, T = sphere_case()
    t, _ = make_pair(64, 32, 48, 0.05, (0, 0, 1, 2), kappa=2.5, g=(0, 0, -1e-3), sponge=6, slide=1, anchor=0.5,
                     storage="f16", particle=(V, T, (31.5, 15.5, 24.0), (0, 0, -0.05), (0, 0, 0)))
    for _ in range(12):
        t.step(4)
        a, b = _both_reads(t, "lbm_copy_macro", 4)
        assert np.array_equal(a, b)


@pytest.mark.parametrize("nx,ny", [(31, 5), (33, 3), (127, 4), (129, 7)])
@pytest.mark.parametrize("storage,tol", [("f32", 1e-5), ("f16", 2e-3)])
def test_windows_as_flat_blocks(nx, ny, storage, tol):
    # planes that end one cell before and after a block of 128 cells and a warp;
    # the bars of the same 100 steps on the 40 x 10 x 12 window
    shape = (9, ny, nx)
    t, s = make_pair(nx, ny, 9, 0.03, (1, 1, 1, 2), sponge=3, storage=storage, fields=_fields(shape, 4))
    t.step(100)
    s.fluid_step(100)
    u, _ = gpu_velocity(t)
    assert rel_max(u, s.velocity()) < tol


@pytest.mark.parametrize("window", [(32, 32, 64), (96, 96, 96)])
@pytest.mark.parametrize("storage", ["f32", "f16"])
@pytest.mark.parametrize("steps", [1, 8, 27])
def test_lists_built_ahead(window, storage, steps):
    # 252 markers: the small window overlaps its launches, the large one (3511
    # cells per marker) builds its lists beside the far cells
    nx, ny, nz = window
    V, T = sphere_case()
    out = []
    for flags in ({}, {"no_graph": 1}):
        t, _ = make_pair(nx, ny, nz, 0.05, (0, 0, 1, 2), kappa=2.5, g=(0, 0, -1e-4), sponge=8, slide=1, anchor=0.5,
                         storage=storage, flags=flags,
                         particle=(V, T, (nx / 2 - 0.5, ny / 2 - 0.5, nz / 2.0), (0, 0, -0.02), (0, 0, 0)))
        assert {(32, 32, 64): 0, (96, 96, 96): 3000}[window] * t.state()["n_markers"] <= nx * ny * nz
        t.step(steps)
        t.step(2)
        s = t.state()
        out.append((np.concatenate([np.ravel(s[k]) for k in ("r", "v", "w", "F", "T")]),
                    t.populations().cpu().numpy()))
    assert np.array_equal(out[0][0], out[1][0])
    assert np.array_equal(out[0][1], out[1][1])


def _alone_and_batched(make, steps):
    # a batch launches every kernel after the one before it, from plain lists: no
    # launch of a step starts beside another of its stream, or is built quietly
    from paper_2408_15115_gb300 import turret as T
    out = []
    for batched in (False, True):
        t = make()
        if batched:
            b = T.Batch([t])
            b.step(steps)
            b.close()
        else:
            t.step(steps)
        s = t.state()
        out.append((np.concatenate([np.ravel(s[k]) for k in ("r", "v", "w", "F", "T")]),
                    t.populations().cpu().numpy()))
        t.close()
    assert np.array_equal(out[0][0], out[1][0])
    assert np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("window", [(32, 32, 64), (96, 96, 96)])
@pytest.mark.parametrize("warm", [False, True])
@pytest.mark.parametrize("cycles", [1, 4])
def test_overlapped_and_quiet_steps_equal_plain_ones(window, warm, cycles):
    # windows as above, also with cycles started from the previous force and with a
    # single cycle (none but the first force in the paper's form)
    nx, ny, nz = window
    V, T = sphere_case()

    def make():
        return make_pair(nx, ny, nz, 0.05, (0, 0, 1, 2), kappa=2.5, g=(0, 0, -1e-4), sponge=8, slide=1, anchor=0.5,
                         flags={"ibm_cycles": cycles}, predictor=(True, 1e-4) if warm else None,
                         particle=(V, T, (nx / 2 - 0.5, ny / 2 - 0.5, nz / 2.0), (0, 0, -0.02), (0, 0, 0)))[0]

    _alone_and_batched(make, 29)


def test_a_surface_with_one_marker_set():
    # 77,442 markers: a second set of the arrays of a time level would take more than
    # 1 GiB, so the levels share one and the particle update waits for the spreading
    from paper_2408_15115_gb300 import turret as T
    V, Tr = I.icosphere(88, 66.0)

    def make():
        t = T.Turret(160, 160, 176, 0.05, 2.5, (0, 0, -1e-5), 0, 0, 1, 2, sponge=8)
        t.load_surface(V, Tr, (79.6, 79.4, 80.3), (0.001, 0, -0.01), (0, 1e-4, 0))
        assert 1 << 30 < t._ibm_ws.numel() < 2 << 30
        return t

    _alone_and_batched(make, 19)
