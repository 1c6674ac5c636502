"""The step's kernel variants, each chosen by a rule on sizes and types, at the
sizes where it can go wrong, against the FP64 oracle: edges of tiles,
remainders, the smallest and largest of a variant's range.

Bars: those of the parity tests -- FP64 1e-10 in C on psi >= 0.01 and in u,
FP32 2e-5 in C and 1e-6 in u after a few steps.
"""
import numpy as np
import pytest
import torch

import workloads as W
from oracle import Oracle
from oracle.ddcc_oracle3d import Oracle3D

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def D():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2311_10314_gb300 import build as B
    B.build()
    import paper_2311_10314_gb300 as D
    return D


def _against_oracle(D, pb, precision, steps, **kw):
    o = Oracle(pb.params, pb.psi, pb.C0, pb.cos_theta, pb.cos_theta_field)
    o.step(steps)
    ref = {k: v.numpy() for k, v in o.macroscopic().items()}
    sim = D.Sim(pb.params, pb.psi, pb.C0, pb.cos_theta, pb.cos_theta_field, precision=precision, **kw)
    sim.step(steps)
    got = sim.fields()
    sim.close()
    fl = pb.psi >= 0.01
    tc, tu = (1e-10, 1e-10) if precision == D.DDCC_FP64 else (2e-5, 1e-6)
    assert np.abs(ref["C"] - got["C"])[:, fl].max() <= tc
    assert max(np.abs(ref[k] - got[k])[fl].max() for k in ("ux", "uy")) <= tu


@pytest.mark.parametrize("nx,ny,N,py,field", [
    (64, 11201, 4, 1, True),     # one tile wide, one row over a tile
    (191, 3751, 4, 0, False),    # a column short of three tiles, walls
    (256, 3700, 3, 1, True),
    (641, 2101, 2, 0, True),     # one column into the eleventh tile
])
def test_fp32_wide_tiles(D, nx, ny, N, py, field):
    """States beyond L2 (over 128 MB) take the 64 x 4 tiles in FP32."""
    assert nx * ny * (11 * N + 3) * 4 > 128 << 20
    pb = W.random_problem(nx, ny, N, seed=nx + N, periodic_y=py, theta_field=field, width=6.0, n_circles=12, n_drops=9)
    _against_oracle(D, pb, D.DDCC_FP32, 3)


@pytest.mark.parametrize("nx,ny,N,py,field", [
    (3, 3, 2, 1, True),          # the smallest grid
    (31, 5, 3, 0, True),         # under one block of either kernel
    (33, 4, 4, 1, False),        # one column over a block
    (64, 8, 2, 0, False),        # whole blocks
    (65, 13, 3, 1, True),        # node numbering that straddles rows
    (161, 97, 4, 0, True),
])
def test_fp64_step_and_ghost_ring(D, nx, ny, N, py, field):
    """The FP64 pair of kernels, stepped plainly and replayed (9 steps), and
    the one-node ghost ring of the lagged plane a in the saved state, which
    the reverse step reads."""
    from paper_2311_10314_gb300 import _lib
    pb = W.random_problem(nx, ny, N, seed=nx + ny, periodic_y=py, theta_field=field, width=6.0)
    _against_oracle(D, pb, D.DDCC_FP64, 9)
    sim = D.Sim(pb.params, pb.psi, pb.C0, pb.cos_theta, pb.cos_theta_field, precision=D.DDCC_FP64)
    sim.step(9)
    state = sim.save_state()
    sim.close()
    org, pitch, plane = _lib.state_layout(nx, ny, N, 8)
    a = torch.as_strided(state.view(torch.float64), (ny + 2, nx + 2), (pitch, 1),
                         org + 9 * N * plane - pitch - 1).cpu().numpy()
    wrap = np.pad(a[1:-1, 1:-1], ((0, 0), (1, 1)), mode="wrap")
    assert np.array_equal(a, np.pad(wrap, ((1, 1), (0, 0)), mode="wrap" if py else "symmetric"))


@pytest.mark.parametrize("precision,path", [(1, "fused"), (1, "split"), (0, "split"), (0, "fused")])
@pytest.mark.parametrize("nx,ny,nz,N,field", [
    (33, 9, 12, 2, True),     # copies node by node, one column and row over a block
    (31, 8, 5, 3, False),
    (64, 17, 4, 3, True),     # copies by quads, fewest planes a chunk can have
    (36, 10, 9, 4, False),    # no staged node values
])
def test_3d_paths_on_ragged_boxes(D, nx, ny, nz, N, field, precision, path):
    """The fused step with both kinds of copies and with and without staged
    values, and the three kernels, in both precisions."""
    pb = W.random_problem_3d(nx, ny, nz, N, seed=nx + N, theta_field=field, width=5.0)
    o = Oracle3D(pb.params, pb.psi, pb.C0, pb.cos_theta, pb.cos_theta_field)
    o.step(5)
    ref = {k: v.numpy() for k, v in o.macroscopic().items()}
    sim = D.Sim3D(pb.params, pb.psi, pb.C0, pb.cos_theta, pb.cos_theta_field, precision=precision, path=path)
    sim.step(5)
    got = sim.fields()
    sim.close()
    fl = pb.psi >= 0.01
    tc, tu = (1e-10, 1e-10) if precision == D.DDCC_FP64 else (2e-5, 1e-6)
    assert np.abs(ref["C"] - got["C"])[:, fl].max() <= tc
    assert max(np.abs(ref[k] - got[k])[fl].max() for k in ("ux", "uy", "uz")) <= tu


@pytest.mark.parametrize("nx,ny,N,px,py,open_x", [
    (25, 3, 2, 1, 1, False),      # narrowest fused grid; three rows keep the fill launch
    (33, 4, 3, 1, 0, False),      # one column into the second tile
    (64, 16, 2, 0, 0, False),     # whole tiles, walls all round
    (35, 9, 3, 1, 1, False),      # last tile within the ring's two columns
    (97, 33, 4, 0, 1, False),
    (48, 17, 3, 0, 0, True),      # open ends write their own copies
    (41, 22, 2, 0, 1, True),
])
def test_fp32_step_writes_its_ghost_rings(D, nx, ny, N, px, py, open_x):
    """After steps of the fused kernel (plain and replayed) the 2-node ring of
    the phase populations and the 1-node ring of the lagged plane a hold the
    copies that loading the state anew would put there, bit for bit."""
    from paper_2311_10314_gb300 import _lib
    pb = W.random_problem(nx, ny, N, seed=nx * ny, periodic_x=px, periodic_y=py, theta_field=True, width=6.0)
    y = np.arange(ny) + 0.5
    ox = (0.01 * y * (ny - y) / ny ** 2, np.full((N - 1, ny), 0.2)) if open_x else None
    sim = D.Sim(pb.params, pb.psi, pb.C0, pb.cos_theta, pb.cos_theta_field, precision=D.DDCC_FP32, open_x=ox)
    org, pitch, plane = _lib.state_layout(nx, ny, N, 4)

    def rings():
        s = sim.save_state().view(torch.float32)
        f = torch.as_strided(s, (9 * (N - 1), ny + 4, nx + 4), (plane, pitch, 1), org - 2 * pitch - 2)
        a = torch.as_strided(s, (ny + 2, nx + 2), (pitch, 1), org + 9 * N * plane - pitch - 1)
        return f.cpu().numpy().copy(), a.cpu().numpy().copy()

    for n in (1, 6):
        sim.step(n)
        got = rings()
        sim.load_state(sim.save_state())      # refills every ghost frame
        want = rings()
        assert np.isfinite(want[0]).all()
        assert np.array_equal(got[0], want[0])
        assert np.array_equal(got[1], want[1])
    sim.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("open_x", [False, True])
def test_long_replay_matches_plain_launches(D, precision, open_x):
    """Past 128 replayed steps ddcc_step uses the eight-step graph too: the
    state after calls of many lengths, from either copy, is bit for bit that
    of a handle whose launches stay plain (profiling on)."""
    from paper_2311_10314_gb300 import _lib
    pb = W.random_problem(70, 45, 3, seed=21, periodic_x=0 if open_x else 1, periodic_y=0, theta_field=True, width=5.0)
    ox = (np.full(45, 0.002), np.full((2, 45), 0.1)) if open_x else None
    sims = [D.Sim(pb.params, pb.psi, pb.C0, pb.cos_theta, pb.cos_theta_field, precision=precision, open_x=ox)
            for _ in range(2)]
    _lib.ddcc_profile(sims[0].h, True)
    for n in (127, 4, 8, 9, 15, 16, 3, 27, 10):
        for s in sims:
            s.step(n)
        _lib.ddcc_kernel_times(sims[0].h)
    assert sims[0].steps == sims[1].steps == 219
    a, b = sims[0].save_state(), sims[1].save_state()
    fa, fb = sims[0].fields(), sims[1].fields()
    assert np.isfinite(fa["C"]).all()
    for k in ("C", "ux", "uy", "P", "mu"):
        assert np.array_equal(fa[k], fb[k]), k
    org, pitch, plane = _lib.state_layout(70, 45, 3, 8 if precision == 0 else 4)
    v = [torch.as_strided(s.view(torch.float64 if precision == 0 else torch.float32), (36, 45, 70), (plane, pitch, 1), org)
         for s in (a, b)]
    assert torch.equal(*v)
    for s in sims:
        s.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nx,ny,N", [(3, 3, 2), (33, 17, 3), (130, 45, 4)])
def test_fields_in_one_call_are_the_fields_read_one_by_one(D, nx, ny, N, precision):
    """ddcc_read_fields (in groups of the staging area's planes) against
    ddcc_read, which a second handle of the same run uses."""
    pb = W.random_problem(nx, ny, N, seed=nx, theta_field=True, width=6.0)
    sims = [D.Sim(pb.params, pb.psi, pb.C0, pb.cos_theta, pb.cos_theta_field, precision=precision) for _ in range(2)]
    for s in sims:
        s.step(5)
    a = sims[0].fields()
    b = sims[1]
    assert np.array_equal(a["C"], np.stack([b.read(D.FIELD_C + i) for i in range(N)]))
    assert np.array_equal(a["mu"], np.stack([b.read(D.FIELD_MU + i) for i in range(N)]))
    for k, f in (("rho", D.FIELD_RHO), ("ux", D.FIELD_UX), ("uy", D.FIELD_UY), ("P", D.FIELD_P)):
        assert np.array_equal(a[k], b.read(f)), k
    for s in sims:
        s.close()


@pytest.mark.parametrize("N", [2, 3, 4])
@pytest.mark.parametrize("rates", [(1.0, 1.2, 1.2, 1.2, 1.2), (0.9, 1.6, 1.6, 1.6, 1.6), (1.0, 1.2, 1.1, 1.2, 1.2),
                                   (1.0, 1.2, 1.2, 1.2, 1.0)])
def test_fp64_phase_rates(D, N, rates):
    """FP64 against the oracle with one phase-LB rate above first order (its
    own collision) and with rates that differ (the transforms), and the phase
    mass, which the collision carries in its rest population."""
    pb = W.random_problem(70, 33, N, seed=5 + N, periodic_y=0, theta_field=True, width=6.0)
    pb.params["s_f"] = list(rates)
    _against_oracle(D, pb, D.DDCC_FP64, 20)
    sim = D.Sim(pb.params, pb.psi, pb.C0, pb.cos_theta, pb.cos_theta_field, precision=D.DDCC_FP64)
    m0 = sim.mass()
    sim.step(200)
    assert np.abs(sim.mass() - m0).max() <= 1e-13 * np.abs(m0).max()
    sim.close()


@pytest.mark.parametrize("off", [0, 1, 4])
def test_device_save_to_any_address(D, off):
    """A device save behind queued steps, at any byte offset, and its load."""
    pb = W.random_problem(65, 21, 3, seed=2, width=6.0)
    a, b = (D.Sim(pb.params, pb.psi, pb.C0, pb.cos_theta, pb.cos_theta_field, precision=D.DDCC_FP32) for _ in range(2))
    a.step(7)
    buf = torch.zeros(a.state_bytes() + off, dtype=torch.uint8, device="cuda")[off:]
    a.save_state(buf)
    a.step(3)
    b.load_state(buf)
    assert b.steps == 7
    b.step(3)
    assert np.array_equal(a.fields()["C"], b.fields()["C"])
    for s in (a, b):
        s.close()


@pytest.mark.parametrize("nx,N,path", [(32, 3, "fused"), (33, 2, "fused"), (33, 3, "split"), (34, 4, "split"),
                                       (31, 4, "fused"), (36, 4, "fused")])
def test_3d_default_path_in_fp32(D, nx, N, path):
    """The path taken where the caller leaves the choice, bit for bit that of
    the forced one, and both paths against the oracle."""
    pb = W.random_problem_3d(nx, 9, 7, N, seed=nx, theta_field=True, width=5.0)
    sims = [D.Sim3D(pb.params, pb.psi, pb.C0, pb.cos_theta, pb.cos_theta_field, precision=D.DDCC_FP32, path=p)
            for p in ("auto", path)]
    for s in sims:
        s.step(5)
    v = [np.stack([s.read(k) for k in (*range(D.FIELD_C, D.FIELD_C + N), D.FIELD_UX, D.FIELD_UY)]) for s in sims]
    assert np.array_equal(*v)
    o = Oracle3D(pb.params, pb.psi, pb.C0, pb.cos_theta, pb.cos_theta_field)
    o.step(5)
    ref = {k: t.numpy() for k, t in o.macroscopic().items()}
    fl = pb.psi >= 0.01
    assert np.abs(ref["C"] - v[0][:N])[:, fl].max() <= 2e-5
    assert max(np.abs(ref[k] - v[0][N + j])[fl].max() for j, k in enumerate(("ux", "uy"))) <= 1e-6
    for s in sims:
        s.close()
