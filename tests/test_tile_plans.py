"""The library's own tile plans against other decompositions of the same
step, at the sizes where the rules that pick them change: every plan gives
the same bits in FP32 and 16-bit arithmetic (one arithmetic for both
kernels), and FP64 differs by rounding only (about 100 operations a node and
step of 2^-53 each over 40 steps: 5e-13)."""
import dataclasses

import numpy as np
import pytest

from paper_2208_13769_gb300 import lbm
from paper_2208_13769_gb300 import workloads as W
from parity_util import rel_l2

pytestmark = [pytest.mark.gpu, pytest.mark.auto_plan]

KEYS = ("u", "v", "P", "r")
Pp = W.Edge(W.PERIODIC)
MIXED = [W.Edge(W.DIRICHLET, rate=(1e-5, -2e-5)), W.Edge(W.NEUMANN, value=(0.0, 1e-5)), Pp, Pp]


def _problem(nx, ny, edges, hole=None, seed=5):
    p = W.smooth_random(nx, ny, edges, seed=seed, amp=0.01, lam=0.3, mu=0.3)
    return dataclasses.replace(p, hole=hole) if hole else p


def _run(prob, steps, storage, carry=None, scheme=1, tuning=None):
    with lbm.Body(prob, storage=storage, compensated=carry, scheme=scheme, tuning=tuning) as b:
        b.step(steps)
        return b.read(lbm.LBM_FIELD_U | lbm.LBM_FIELD_V | lbm.LBM_FIELD_P | lbm.LBM_FIELD_R)


def _same(got, ref, storage, what):
    for k in KEYS:
        if storage == "f64":
            assert rel_l2(got[k], ref[k]) <= 5e-13, (what, k)
        else:
            assert np.array_equal(got[k], ref[k]), (what, k, rel_l2(got[k], ref[k]))


# one full wave of 11 to 27 rows (4-byte storage: 4.45 tiles per SM), fewer
# rows (short tiles), 28 and more (a wave with shorter tiles after it; the
# extrapolated scheme: 20 rows), 48 and more in 16-bit storage, 64 and 100 and
# more (18 rows), with the last strip a few columns wide
@pytest.mark.parametrize("nx,ny,storage,carry,scheme", [
    (420, 400, "f32", True, 1), (640, 640, "f32", "lo16", 0), (1000, 140, "f16", None, 1), (700, 601, "f64", None, 1),
    (126, 7001, "f32", True, 1), (250, 7000, "f32", False, 1), (130, 13501, "f32", "lo16", 1), (130, 13501, "f32", True, 2),
    (130, 13501, "f16", None, 2), (131, 23003, "f16", None, 1), (129, 23003, "bf16", None, 0),
    (130, 30011, "f32", "lo16", 1), (129, 54007, "f16", None, 0)])
def test_default_interior_plans_match_fixed_rows(nx, ny, storage, carry, scheme):
    prob = _problem(nx, ny, W.clamped_free_edges())
    got = _run(prob, 18, storage, carry, scheme)
    for rows in (8, 64):
        _same(got, _run(prob, 18, storage, carry, scheme, lbm.lbm_tuning(0, rows, 0, 2)), storage, rows)
    _same(got, _run(prob, 18, storage, carry, scheme, lbm.lbm_tuning(0, 0, -1, 1)), storage, "edge tiles")


def test_reported_tuning_of_short_tiles_is_accepted():
    """The default plan of a short-tiled body, read back, sets another one's."""
    prob = _problem(420, 400, MIXED)
    with lbm.Body(prob, storage="f32") as a:
        a.step(9)
        used, ref = lbm.lbm_get_tuning(a.ctx), a.read()
    assert used.plan == 2 and used.chunk_rows >= 8
    with lbm.Body(prob, storage="f32", tuning=used) as b:
        b.step(9)
        _same(b.read(), ref, "f32", "read back")


# band tiles of interior tiles' size (seams, a hole beside short tiles), and
# the three tile shapes of bodies that run as edge tiles only
@pytest.mark.parametrize("storage", ["f64", "f32", "f16"])
@pytest.mark.parametrize("nx,ny,edges,hole", [
    (64, 64, [Pp] * 4, None), (129, 127, MIXED, None), (203, 200, MIXED, (60, 111, 50, 101)), (301, 203, MIXED, None),
    (420, 401, [Pp] * 4, None), (501, 500, MIXED, None), (700, 620, MIXED, (200, 420, 210, 430))])
def test_edge_tile_shapes_match_other_plans(nx, ny, edges, hole, storage):
    prob = _problem(nx, ny, edges, hole)
    got = _run(prob, 40, storage)
    _same(got, _run(prob, 40, storage, tuning=lbm.lbm_tuning(0, 0, -1, 1)), storage, "edge tiles")
    _same(got, _run(prob, 40, storage, tuning=lbm.lbm_tuning(0, 0, -1, 2)), storage, "interior across the seams")


@pytest.mark.parametrize("nx,ny", [(70, 60), (420, 400)])
def test_graphs_of_both_lengths_match_single_steps(nx, ny):
    """Calls around the graphs' lengths (16 and 64 steps), from both parities."""
    prob = _problem(nx, ny, MIXED)
    with lbm.Body(prob, storage="f32", scheme=1) as a, lbm.Body(prob, storage="f32", scheme=1) as b:
        for n in (17, 16, 65, 33, 1, 83, 64, 150, 2):
            a.step(n)
            for _ in range(n):
                b.step(1)
            assert lbm.lbm_get_info(a.ctx)[0] == lbm.lbm_get_info(b.ctx)[0]
            _same(a.read(), b.read(), "f32", n)


def test_steps_on_the_legacy_stream_run():
    """No capture begins on the legacy default stream (handle 1): its calls of
    up to 64 steps are launches."""
    prob = _problem(420, 400, MIXED)
    with lbm.Body(prob, storage="f32", stream=1) as a, lbm.Body(prob, storage="f32") as b:
        a.step(33)
        b.step(33)
        _same(a.read(), b.read(), "f32", "legacy stream")


def test_steps_recorded_by_a_caller_replay():
    """A call of more than a short graph's steps on a stream being captured is
    recorded as launches; its replay is those steps."""
    import torch
    prob = _problem(420, 400, MIXED)
    s = torch.cuda.Stream()
    with lbm.Body(prob, storage="f32", stream=s.cuda_stream) as a, lbm.Body(prob, storage="f32") as b:
        a.step(70)
        lbm.lbm_sync(a.ctx)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
            a.step(20)
        with torch.cuda.stream(s):
            g.replay()
        s.synchronize()
        b.step(90)
        _same(a.read(), b.read(), "f32", "replay")


@pytest.mark.parametrize("storage", ["f32", "f16", "f64"])
@pytest.mark.parametrize("sizes", [[(70, 60), (200, 130), (131, 90)],  # a few rows a wave
                                   [(1000, 1500), (260, 1900), (900, 90)]])  # long and short tiles
def test_batch_plans_match_fixed_rows(sizes, storage):
    probs = [_problem(nx, ny, [Pp] * 4 if k % 2 else W.clamped_free_edges(), seed=k) for k, (nx, ny) in enumerate(sizes)]
    res = []
    for tuning in (None, lbm.lbm_tuning(0, 16, 0, 0), lbm.lbm_tuning(0, 300, 1, 0)):
        bodies = [lbm.Body(p, storage=storage) for p in probs]
        try:
            with lbm.Batch(bodies, tuning=tuning) as batch:
                batch.step(21)
                batch.sync()
            res.append([b.read() for b in bodies])
        finally:
            for b in bodies:
                b.close()
    for other in res[1:]:
        for got, ref in zip(res[0], other):
            _same(got, ref, storage, "batch")


@pytest.mark.parametrize("given", ["u0", "v0", ""])
def test_initial_fields_left_out_are_zero(given):
    """u0 and v0 share an allocation: one, the other or neither given."""
    prob = _problem(90, 50, MIXED)
    u0, v0 = prob.initial()
    zero = np.zeros((50, 90, 2))
    u = u0 if given == "u0" else None
    v = v0 if given == "v0" else None
    a = dataclasses.replace(prob, make_initial=None, u0=u, v0=v)
    b = dataclasses.replace(prob, make_initial=None, u0=zero if u is None else u, v0=zero if v is None else v)
    _same(_run(a, 9, "f32"), _run(b, 9, "f32"), "f32", given)


def test_read_out_quotients_at_zero_and_without_inverse():
    """The stresses' quotients by J at J = 0, at a negative and a huge J and at
    zero numerators are those of the division (the formulas of the read-out,
    a few roundings of them apart: 1e-13 of the largest term)."""
    nx, ny, lam, mu = 48, 16, 0.4, 0.3
    u0 = np.zeros((ny, nx, 2))
    x, y = np.meshgrid(np.arange(nx), np.arange(ny))
    u0[:, 8:16, 0] = -x[:, 8:16]  # h11 = -1: J = 0
    u0[:, 16:24, 0] = -2.5 * x[:, 16:24]
    u0[:, 24:32, 0] = 2.0 ** 520 * x[:, 24:32]
    u0[:, 32:40, 1] = 1e-3 * x[:, 32:40]
    prob = W.Problem(nx=nx, ny=ny, lam=lam, mu=mu, rho0=1.0, omega=1.0, dX=1.0, body=(0.0, 0.0), edges=[Pp] * 4, u0=u0,
                     v0=np.zeros((ny, nx, 2)))
    with lbm.Body(prob, storage="f64") as b:
        got = b.read(allow_unstable=True)
    d = lambda a, axis: (np.roll(a, -1, axis) - np.roll(a, 1, axis)) * 0.5
    with np.errstate(all="ignore"):
        h11, h12, h21, h22 = d(u0[..., 0], 1), d(u0[..., 0], 0), d(u0[..., 1], 1), d(u0[..., 1], 0)
        jm1 = h11 + h22 + (h11 * h22 - h12 * h21)
        J = 1.0 + jm1
        F = [1.0 + h11, h12, h21, 1.0 + h22]
        G = [F[3] / J, -F[2] / J, -F[1] / J, F[0] / J]
        c = 0.5 * lam * jm1 * (2.0 + jm1)
        P = np.stack([mu * (f - g) + c * g for f, g in zip(F, G)], -1)
        S = np.stack([(P[..., 0] * F[0] + P[..., 1] * F[1]) / J, (P[..., 0] * F[2] + P[..., 1] * F[3]) / J,
                      (P[..., 2] * F[2] + P[..., 3] * F[3]) / J], -1)
        size = sum(abs(mu * f) + abs(mu * g) + abs(c * g) for f, g in zip(F, G))[..., None]
    inner = np.ones(nx, bool)  # away from the jumps of u0, where the sums cancel
    inner[[0, 7, 8, 15, 16, 23, 24, 31, 32, 39, 40, 47]] = False
    for name, ref, scale in (("P", P, size), ("sigma", S, size * (abs(F[0]) + abs(F[1]) + abs(F[2]) + abs(F[3]))[..., None]
                                                    / abs(J)[..., None])):
        a, r = np.asarray(got[name]).reshape(ny, nx, -1)[:, inner], ref[:, inner]
        z = np.broadcast_to(scale, ref.shape)[:, inner]
        assert np.array_equal(np.isnan(a), np.isnan(r)) and np.array_equal(np.isinf(a), np.isinf(r)), name
        ok = np.isfinite(r) & np.isfinite(z)
        assert ok.any() and np.all(np.abs(a[ok] - r[ok]) <= 1e-13 * z[ok]), name
