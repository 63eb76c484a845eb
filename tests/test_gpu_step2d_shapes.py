"""The tile shapes of the 2D step: 64 x 2 (FP32 states beyond 129 MB), 64 x 4
with two nodes per thread (16-bit storage, at least 1500 such tiles) and 32 x 4,
on sizes at and next to those lines, whole and ragged last tiles, every kind of
boundary, solid nodes and both collisions, against the FP64 oracle.

FP32 fields to 1e-5 (the repository's bar).  16-bit storage: a step rounds each
stored deviation once, to u = 2^-11 (FP16) or 2^-8 (BF16) of itself, so N steps
move a moment by at most N u times the sum of the deviations it is made of:
at most 2 for phi, 0.5 for U (its own reference removed, plus the change next
to the crystal), 0.1 for rho and u.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

STEPS = 5
SIZES = [(1024, 563),  # FP32: 129.1 MB, 64 x 2 tiles, an odd last row
         (1055, 571),  # the same, ragged on both sides
         (1024, 562)]  # 128.9 MB: 32 x 4 tiles
SIZES16 = [(960, 400),   # 16-bit: 15 x 100 tiles of 64 x 4, all whole
           (901, 397),   # as many, ragged on both sides
           (960, 396)]   # one row of tiles fewer: 32 x 4
BOUNDS = {
    "inflow": dict(bc=(1, 0, 0), u_in=0.01, U_in=0.4),
    "inflow_walls": dict(bc=(1, 2, 0), u_in=0.01, U_in=0.4),
    "periodic": dict(bc=(0, 0, 0), body=(1e-5, 2e-5, 0.0)),
    "walls_x": dict(bc=(2, 0, 0), body=(0.0, 1e-5, 0.0)),
}


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available(), "these tests need a CUDA GPU"
    import _pairs
    return _pairs


def problem(P, size, bounds, flow=1):
    nx, ny = size
    p = P.params(nx=nx, ny=ny, flow=flow, fold=5, eps=0.03, theta0=0.2, **BOUNDS[bounds])
    # crystals on the left and right edge columns and across the top edge too
    y, x = np.mgrid[0:ny, 0:nx].astype(float)
    rng = np.random.default_rng(5)
    r = np.minimum.reduce([np.hypot(x - cx, y - cy) for cx, cy in
                           ((0, ny / 2), (nx - 1, ny / 3), (nx / 2, 0), (65, 9))])
    phi = np.tanh((12.0 - r) / (np.sqrt(2.0) * 2.0)) + 0.01 * rng.uniform(-1, 1, r.shape)
    U = 0.4 + 0.01 * rng.uniform(-1, 1, r.shape)
    v = [0.01 * rng.uniform(-1, 1, r.shape) for _ in range(3)]
    return p, (phi, U, 1.0 + 1e-3 * rng.uniform(-1, 1, r.shape), v)


@pytest.mark.parametrize("bounds", BOUNDS)
@pytest.mark.parametrize("size", SIZES, ids=str)
def test_fp32(P, size, bounds):
    p, fields = problem(P, size, bounds)
    a, b = P.pair(p, "fp32", fields=fields)
    a.step(STEPS)
    b.step(STEPS, P.THREADS)
    errs = P.max_errors(a, b)
    assert max(errs.values()) < 1e-5, errs
    a.close()


@pytest.mark.parametrize("storage,u", [("fp16", 2.0 ** -11), ("bf16", 2.0 ** -8)])
@pytest.mark.parametrize("size", SIZES16, ids=str)
def test_16bit(P, size, storage, u):
    p, fields = problem(P, size, "inflow")
    a, b = P.pair(p, storage, fields=fields)
    a.step(STEPS)
    b.step(STEPS, P.THREADS)
    errs = P.max_errors(a, b)
    n = STEPS + 1  # the initial state is rounded too
    assert errs["phi"] < n * u * 2.0 and errs["U"] < n * u * 0.5, errs
    assert max(errs["rho"], errs["ux"], errs["uy"]) < n * u * 0.1, errs
    a.close()


@pytest.mark.parametrize("chm", [0, 1])
@pytest.mark.parametrize("size", SIZES[:2], ids=str)
def test_solids_and_collision(P, size, chm):
    import oracle
    import paper_2206_02145_gb300 as L
    p, (phi, U, rho, v) = problem(P, size, "inflow_walls")
    mask = np.zeros(phi.shape, bool)
    mask[100:300, 60:68] = True      # across a tile edge
    mask[0:3, 200:230] = True        # on the wall
    mask[-2:, -40:-37] = True        # in the last tiles
    a = L.Sim(dim=2, nx=p["nx"], ny=p["ny"], bc=p["bc"], flow=1, fold=5, eps_aniso=0.03,
              theta0=0.2, u_inlet=0.01, u0_inlet=0.4, collision=chm)
    b = oracle.Oracle(oracle.Params(dim=2, nx=p["nx"], ny=p["ny"], bc=p["bc"], flow=1, fold=5,
                                    eps=0.03, theta0=0.2, u_inlet=0.01, u0_inlet=0.4,
                                    collision=chm))
    for s in (a, b):
        s.init_fields(phi, U, rho, v[0], v[1], None)
        s.set_solid(mask)
    a.step(STEPS)
    b.step(STEPS, P.THREADS)
    errs = P.max_errors(a, b)
    assert max(errs.values()) < 1e-5, errs
    a.close()


# ---- the two-node tiles (and the 32 x 4 ones next to them) in 16-bit storage ----
UNITS = [("fp16", 2.0 ** -11), ("bf16", 2.0 ** -8)]


def within_storage_bounds(errs, u):
    n = STEPS + 1  # the initial state is rounded too
    assert errs["phi"] < n * u * 2.0 and errs["U"] < n * u * 0.5, errs
    assert max(errs.get(k, 0.0) for k in ("rho", "ux", "uy")) < n * u * 0.1, errs


def obstacles(size):
    nx, ny = size
    mask = np.zeros((ny, nx), bool)
    mask[100:300, 60:68] = True      # across a tile edge
    mask[0:3, 200:230] = True        # on the wall: rows 0 and 2 are one thread's
    mask[41, 300:303] = True         # one of a thread's two nodes
    mask[-2:, -40:-37] = True        # in the last tiles
    return mask


def solid_pair(P, size, bounds, storage, chm):
    import oracle
    import paper_2206_02145_gb300 as L
    p, (phi, U, rho, v) = problem(P, size, bounds)
    kw = dict(dim=2, nx=p["nx"], ny=p["ny"], bc=p["bc"], flow=1, fold=5, theta0=0.2,
              u_inlet=p["u_in"], u0_inlet=p["U_in"], collision=chm)
    a = L.Sim(storage=P.STORAGE[storage], eps_aniso=0.03, body_force=p["body"], **kw)
    b = oracle.Oracle(oracle.Params(eps=0.03, body=p["body"], **kw))
    for s in (a, b):
        s.init_fields(phi, U, rho, v[0], v[1], None)
        s.set_solid(obstacles(size))
    return a, b


@pytest.mark.parametrize("storage,u", UNITS)
@pytest.mark.parametrize("bounds", [k for k in BOUNDS if k != "inflow"])
@pytest.mark.parametrize("size", SIZES16, ids=str)
def test_16bit_boundaries(P, size, bounds, storage, u):
    p, fields = problem(P, size, bounds)
    a, b = P.pair(p, storage, fields=fields)
    a.step(STEPS)
    b.step(STEPS, P.THREADS)
    within_storage_bounds(P.max_errors(a, b), u)
    a.close()


@pytest.mark.parametrize("storage,u", UNITS)
@pytest.mark.parametrize("bounds", ["periodic", "walls_x"])
@pytest.mark.parametrize("size", SIZES16[:2], ids=str)
def test_16bit_without_flow(P, size, bounds, storage, u):
    p, fields = problem(P, size, bounds, flow=0)
    a, b = P.pair(p, storage, fields=fields)
    a.step(STEPS)
    b.step(STEPS, P.THREADS)
    within_storage_bounds(P.max_errors(a, b, ("phi", "U")), u)
    a.close()


@pytest.mark.parametrize("storage,u", UNITS)
@pytest.mark.parametrize("chm", [0, 1])
@pytest.mark.parametrize("bounds", ["inflow_walls", "periodic"])
@pytest.mark.parametrize("size", SIZES16, ids=str)
def test_16bit_solids_and_collision(P, size, bounds, chm, storage, u):
    a, b = solid_pair(P, size, bounds, storage, chm)
    a.step(STEPS)
    b.step(STEPS, P.THREADS)
    within_storage_bounds(P.max_errors(a, b), u)
    a.close()


@pytest.mark.parametrize("solids", [False, True])
@pytest.mark.parametrize("chm", [0, 1])
@pytest.mark.parametrize("bounds", BOUNDS)
def test_two_nodes_per_thread_round_like_one(P, bounds, chm, solids):
    # the batched step runs every one- and two-node shape in turn while it tunes; the
    # single step of this size holds two nodes per thread: the same bits
    import paper_2206_02145_gb300 as L
    size = SIZES16[1]
    p, (phi, U, rho, v) = problem(P, size, bounds)
    kw = dict(dim=2, nx=p["nx"], ny=p["ny"], bc=p["bc"], flow=1, fold=5, theta0=0.2,
              eps_aniso=0.03, u_inlet=p["u_in"], u0_inlet=p["U_in"], body_force=p["body"],
              storage=L.FP16_SHIFTED, collision=chm)
    one = L.Sim(**kw)
    batch = L.Batch([kw], [(10.0, 10.0, 0.0, 4.0, 0.4, 0.0, 1)])
    for s in (one, batch.instance(0)):
        s.init_fields(phi, U, rho, v[0], v[1], None)
        if solids:
            s.set_solid(obstacles(size))
    one.step(60)
    batch.step(60)
    assert batch.tuning()["tuned"]
    # (the header names the node of the batch's seed; the arrays follow it)
    np.testing.assert_array_equal(one.state()[P.HDR:], batch.instance(0).state()[P.HDR:])
    one.close()
    batch.close()
