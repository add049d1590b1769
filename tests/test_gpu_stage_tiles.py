"""The step kernels at the sizes where their tiling changes: 3D psi stages by small
tiles (16 x 8 x 4 and 32 x 8 x 4) against the marching ones and the oracle, both 2D
tiles (16 x 8, and 32 x 16 from 304 * 512 sites on), the depth chosen for a large box,
and the threaded read of a large field."""
import numpy as np
import pytest

import oracle as O
import paper_1104_0078_gb300 as F
from paper_1104_0078_gb300 import inputs as I

from gpu_helpers import field_error, flb_params, oracle_params, weights_column

pytestmark = pytest.mark.gpu

BASE = dict(dim=3, q=19, tau=0.8, kT=1e-4, A=-0.05, B=0.3, K=0.04, M=0.1, scheme=1, integrator=2, coupling=3, seed=5)
# one tile, one past its edges, one short of them, several ragged ones; 64 x 40 x 52 and 63 x 33 x 45
# are boxes of 32-wide tiles
SHAPES = [(4, 4, 4), (16, 8, 4), (17, 9, 5), (31, 7, 19), (64, 40, 52), (63, 33, 45)]


def _start(s, d, seed=7):
    N = d["nx"] * d["ny"] * d.get("nz", 1)
    f0 = weights_column(d["q"]) + I.random_deviations(d["q"], N, 2e-3, seed)
    psi0 = I.random_field(N, 0.05, seed + 1)
    s.set_fields(psi=psi0)
    s.set_populations(f0)
    return f0, psi0


def _run(d, steps, zc=None):
    s = F.Solver(flb_params(d))
    _start(s, d)
    if zc is not None:
        s.set_tuning(zc)
    s.step(steps)
    return (s.get_populations(), *s.get_psi_u())


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("q", [19, 15])
@pytest.mark.parametrize("extra", [{}, dict(integrator=4), dict(integrator=1, coupling=2), dict(kT=0.0),
                                   dict(integrator=4, kT=0.0, coupling=0), dict(storage=F.FLB_F16_DEV)])
def test_small_tiles_equal_marching(shape, q, extra):
    d = dict(BASE, q=q, nx=shape[0], ny=shape[1], nz=shape[2])
    d.update(extra)
    for a, b in zip(_run(d, 5), _run(d, 5, zc=8)):
        assert np.array_equal(a, b)


def test_depth_of_a_large_box_changes_no_bit():
    # above 1.3 million sites the marching stage runs with a depth taken from the box
    d = dict(BASE, nx=121, ny=120, nz=93)
    for a, b in zip(_run(d, 2), _run(d, 2, zc=64)):
        assert np.array_equal(a, b)


def _against_oracle(d, steps, tol_f, tol_psi):
    s = F.Solver(flb_params(d))
    f0, psi0 = _start(s, d)
    s.step(steps)
    op = oracle_params(d)
    st = O.State(op, f0.copy(), psi0.copy(), np.zeros((3, op.n)), 0)
    st.advance(steps)
    assert field_error(s.get_populations(), st.f, weights_column(d["q"])) < tol_f
    psi, u = s.get_psi_u()
    assert field_error(psi, st.psi) < tol_psi
    assert field_error(u[:d["dim"]], st.u[:d["dim"]]) < tol_f


# FP32: a step rounds at 6e-8 of each quantity's largest terms; 1e-5 as in the parity tests.
# FP16 deviations: a stored population is off by 2^-11 of itself, after 8 steps at most 4e-3 and with
# extremes of five times the rms 2e-2; psi is advected by u ~ 5e-3, off by as much of
# itself: 8 * 2e-2 * 5e-3 * 2 = 1.6e-3.
@pytest.mark.parametrize("shape", [(17, 9, 5), (63, 33, 45), (130, 5, 7)])
@pytest.mark.parametrize("extra", [dict(scheme=0), dict(scheme=0, integrator=4, coupling=2), dict(scheme=2),
                                   dict(scheme=0, laplacian=3), dict(laplacian=1), dict(q=15),
                                   dict(scheme=0, force_grad=3)])
def test_3d_tiles_match_oracle(shape, extra):
    d = dict(BASE, nx=shape[0], ny=shape[1], nz=shape[2])
    d.update(extra)
    _against_oracle(d, 8, 1e-5, 1e-5)


@pytest.mark.parametrize("shape", [(4, 4), (16, 8), (17, 9), (47, 31), (400, 392), (397, 395)])
@pytest.mark.parametrize("extra", [dict(scheme=0), dict(scheme=1), dict(scheme=2, integrator=1),
                                   dict(scheme=0, integrator=4, laplacian=1), dict(scheme=1, integrator=4, kT=0.0),
                                   dict(scheme=1, force_grad=3, gamma_ghost=0.3)])
def test_2d_tiles_match_oracle(shape, extra):
    d = dict(BASE, dim=2, q=9, nx=shape[0], ny=shape[1])
    d.update(extra)
    _against_oracle(d, 8, 1e-5, 1e-5)


@pytest.mark.parametrize("dim,q,shape", [(2, 9, (47, 31)), (2, 9, (397, 395)), (3, 19, (17, 9, 5)), (3, 15, (63, 33, 45))])
@pytest.mark.parametrize("scheme", [0, 1])
def test_fp16_tiles_match_oracle(dim, q, shape, scheme):
    d = dict(BASE, dim=dim, q=q, nx=shape[0], ny=shape[1], scheme=scheme, storage=F.FLB_F16_DEV)
    if dim == 3:
        d["nz"] = shape[2]
    _against_oracle(d, 8, 2e-2, 1.6e-3)


@pytest.mark.parametrize("shape", [(127, 128, 129), (128, 128, 128)])
def test_read_of_a_large_field(shape):
    # 2^21 values are where the read splits over threads: just below it and at it
    d = dict(BASE, nx=shape[0], ny=shape[1], nz=shape[2])
    N = shape[0] * shape[1] * shape[2]
    s = F.Solver(flb_params(d))
    psi = I.random_field(N, 0.05, 3)
    u = np.stack([I.random_field(N, 1e-2, 4 + a) for a in range(3)])
    s.set_fields(psi=psi, u=u)
    assert np.array_equal(s.get_psi(), psi)
    p, v = s.get_psi_u()
    assert np.array_equal(p, psi)
    assert np.array_equal(v, u)


@pytest.mark.parametrize("q", [19, 15])
@pytest.mark.parametrize("extra", [{}, dict(force_grad=3), dict(storage=F.FLB_F16_DEV), dict(coupling=2)])
def test_batched_in_two_groups_equals_plain(q, extra):
    # above 600 thousand sites a batched step runs as two chains of kernels; with boxes whose
    # padded rows end within and at a group of four x
    shapes = [(84, 84, 70), (60, 61, 37), (4, 5, 6), (17, 9, 5), (33, 7, 70)]
    ds = [{**BASE, "q": q, "nx": nx, "ny": ny, "nz": nz, "seed": 40 + r, **extra}
          for r, (nx, ny, nz) in enumerate(shapes)]
    assert sum(nx * ny * nz for nx, ny, nz in shapes) >= 600000
    runs = []
    for mode in (F.FLB_MODE_PLAIN, F.FLB_MODE_BATCHED):
        s = F.Solver([flb_params(d) for d in ds])
        for r, d in enumerate(ds):
            N = d["nx"] * d["ny"] * d["nz"]
            s.set_fields(rep=r, psi=I.random_field(N, 0.05, 8 + r))
            s.set_populations(weights_column(q) + I.random_deviations(q, N, 2e-3, 7 + r), rep=r)
        s.set_mode(mode)
        s.step(5)
        runs.append([(s.get_populations(r), *s.get_psi_u(r)) for r in range(len(ds))])
    for ra, rb in zip(*runs):
        for a, b in zip(ra, rb):
            assert np.array_equal(a, b)


# boxes whose launches are small enough for several to be in flight together
@pytest.mark.parametrize("d", [
    dict(dim=2, q=9, nx=397, ny=395, scheme=0, gamma_ghost=0.3, gamma_bulk=-0.4),
    dict(dim=2, q=9, nx=397, ny=395, scheme=1, gamma_ghost=0.3, force_grad=3),
    dict(dim=2, q=9, nx=397, ny=395, scheme=0, gamma_ghost=0.3, storage=F.FLB_F16_DEV),
    dict(dim=2, q=9, nx=420, ny=371, scheme=1, integrator=4),
    dict(dim=2, q=9, nx=130, ny=95, scheme=0, gamma_ghost=0.3), dict(dim=2, q=9, nx=64, ny=64, scheme=1),
    dict(nx=64, ny=40, nz=52, gamma_ghost=0.3), dict(nx=32, ny=32, nz=32, q=15), dict(nx=63, ny=33, nz=45, scheme=0),
    dict(nx=48, ny=48, nz=48, q=15, scheme=0, gamma_ghost=0.3), dict(nx=48, ny=40, nz=37, integrator=4, force_grad=3),
    dict(nx=48, ny=40, nz=37, laplacian=2), dict(nx=48, ny=40, nz=37, scheme=2, laplacian=1),
    dict(nx=64, ny=40, nz=52, storage=F.FLB_F16_DEV), dict(nx=121, ny=120, nz=93), dict(nx=60, ny=60, nz=60, q=15, zc=8)])
def test_overlapped_launches_give_the_same_steps(d):
    # steps enqueued one behind the other, whose launches overlap, against steps waited for one by one
    d = dict(BASE, **d)
    s = F.Solver(flb_params(d))
    _start(s, d)
    if "zc" in d:
        s.set_tuning(d["zc"])
    start = s.get_state()
    for _ in range(8):
        s.step(1)
        s.synchronize()
    ref = s.get_state()
    for k in range(30):
        s.set_state(start)
        s.step(8)
        assert s.get_state() == ref, k


@pytest.mark.parametrize("shape", [(47, 31), (397, 395)])
@pytest.mark.parametrize("extra", [{}, dict(force_grad=3, gamma_ghost=0.3), dict(kT=0.0, coupling=0)])
def test_2d_bulk_rate_matches_oracle(shape, extra):
    # the trace relaxing at its own rate, one site a thread and two
    d = dict(BASE, dim=2, q=9, nx=shape[0], ny=shape[1], scheme=0, gamma_bulk=-0.4)
    d.update(extra)
    _against_oracle(d, 8, 1e-5, 1e-5)


@pytest.mark.parametrize("shape,chunks", [((129, 130, 131), 5), ((161, 160, 163), 9)])
def test_read_reuses_its_ring(shape, chunks):
    # psi and u of more than four chunks of 2^21 values: from the fifth on a chunk takes a slot whose
    # values the threads have converted; psi ends and a component of u begins within a chunk
    N = shape[0] * shape[1] * shape[2]
    assert -(-4 * N // 2 ** 21) == chunks
    s = F.Solver(flb_params(dict(BASE, nx=shape[0], ny=shape[1], nz=shape[2])))
    psi = I.random_field(N, 0.05, 3)
    u = np.stack([I.random_field(N, 1e-2, 4 + a) for a in range(3)])
    s.set_fields(psi=psi, u=u)
    for _ in range(3):
        p, v = s.get_psi_u()
        assert np.array_equal(p, psi)
        assert np.array_equal(v, u)
