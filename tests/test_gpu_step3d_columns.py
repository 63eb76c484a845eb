"""The 3D step's columns of 32 x 8 nodes and its chunks of 1 to 8 planes, on the
smallest grids, whole and ragged last columns and chunks, every kind of
boundary, solid nodes and both collisions, against the FP64 oracle.

Tolerances as for the 2D tile shapes: FP32 fields to 1e-5; N steps of 16-bit
storage move a moment by at most N u (u = 2^-11 in FP16, 2^-8 in BF16) times the
sum of the deviations it is made of, at most 2 for phi, 0.5 for U and 0.1 for
rho and u.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

STEPS = 5
SIZES = [(4, 4, 4),      # smaller than a column's halo box
         (32, 8, 8),     # one column, chunks of 1
         (33, 9, 17),    # one node beyond a column each way
         (64, 40, 61),   # whole columns, an odd last chunk
         (97, 63, 83)]   # ragged columns and chunks
BOUNDS = {
    "inflow": dict(bc=(1, 0, 0), u_in=0.01, U_in=0.4),
    "inflow_walls": dict(bc=(1, 2, 2), u_in=0.01, U_in=0.4),
    "periodic": dict(bc=(0, 0, 0), body=(1e-5, 2e-5, -1e-5)),
    "walls_x": dict(bc=(2, 0, 2), body=(0.0, 1e-5, 0.0)),
}


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available(), "these tests need a CUDA GPU"
    import _pairs
    return _pairs


def problem(P, size, bounds):
    nx, ny, nz = size
    p = P.params(dim=3, nx=nx, ny=ny, nz=nz, flow=1, fold=0, eps=0.03, **BOUNDS[bounds])
    # crystals on two faces, an edge and inside
    z, y, x = np.mgrid[0:nz, 0:ny, 0:nx].astype(float)
    rng = np.random.default_rng(7)
    r = np.minimum.reduce([np.sqrt((x - a) ** 2 + (y - b) ** 2 + (z - c) ** 2) for a, b, c in
                           ((0, ny / 2, nz / 2), (nx - 1, 0, nz / 3), (nx / 2, ny / 2, nz - 1),
                            (nx / 3, ny / 3, nz / 4))])
    phi = np.tanh((6.0 - r) / (np.sqrt(2.0) * 2.0)) + 0.01 * rng.uniform(-1, 1, r.shape)
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
    errs = P.max_errors(a, b, ("phi", "U", "rho", "ux", "uy", "uz"))
    assert max(errs.values()) < 1e-5, errs
    a.close()


@pytest.mark.parametrize("storage,u", [("fp16", 2.0 ** -11), ("bf16", 2.0 ** -8)])
@pytest.mark.parametrize("size", SIZES, ids=str)
def test_16bit(P, size, storage, u):
    p, fields = problem(P, size, "inflow_walls")
    a, b = P.pair(p, storage, fields=fields)
    a.step(STEPS)
    b.step(STEPS, P.THREADS)
    errs = P.max_errors(a, b, ("phi", "U", "rho", "ux", "uy", "uz"))
    n = STEPS + 1  # the initial state is rounded too
    assert errs["phi"] < n * u * 2.0 and errs["U"] < n * u * 0.5, errs
    assert max(errs[k] for k in ("rho", "ux", "uy", "uz")) < n * u * 0.1, errs
    a.close()


@pytest.mark.parametrize("chm", [0, 1])
@pytest.mark.parametrize("size", SIZES[2:], ids=str)
def test_solids_and_collision(P, size, chm):
    import oracle
    import paper_2206_02145_gb300 as L
    p, (phi, U, rho, v) = problem(P, size, "inflow_walls")
    mask = np.zeros(phi.shape, bool)
    mask[3:12, 2:6, 20:-1] = True    # across a column's and a chunk's edge
    mask[0:2, -3:, 4:9] = True       # on two walls
    mask[-1, 1, -5:-3] = True        # in the last chunk and column
    kw = dict(dim=3, nx=p["nx"], ny=p["ny"], nz=p["nz"], bc=p["bc"], flow=1, fold=0,
              u_inlet=0.01, u0_inlet=0.4, collision=chm)
    a = L.Sim(eps_aniso=0.03, **kw)
    b = oracle.Oracle(oracle.Params(eps=0.03, **kw))
    for s in (a, b):
        s.init_fields(phi, U, rho, *v)
        s.set_solid(mask)
    a.step(STEPS)
    b.step(STEPS, P.THREADS)
    errs = P.max_errors(a, b, ("phi", "U", "rho", "ux", "uy", "uz"))
    assert max(errs.values()) < 1e-5, errs
    a.close()


# chunks of 8 planes (the longest), ragged columns and a ragged last chunk
EIGHT = (60, 150, 62)


@pytest.mark.parametrize("storage,u", [("fp32", 0.0), ("fp16", 2.0 ** -11)])
def test_chunks_of_eight_planes(P, storage, u):
    p, fields = problem(P, EIGHT, "inflow_walls")
    a, b = P.pair(p, storage, fields=fields)
    a.step(STEPS)
    b.step(STEPS, P.THREADS)
    errs = P.max_errors(a, b, ("phi", "U", "rho", "ux", "uy", "uz"))
    n = STEPS + 1  # the initial state is rounded too
    assert errs["phi"] < 1e-5 + n * u * 2.0 and errs["U"] < 1e-5 + n * u * 0.5, errs
    assert max(errs[k] for k in ("rho", "ux", "uy", "uz")) < 1e-5 + n * u * 0.1, errs
    a.close()


@pytest.mark.parametrize("storage,u", [("fp32", 0.0), ("fp16", 2.0 ** -11), ("bf16", 2.0 ** -8)])
@pytest.mark.parametrize("bounds", ["inflow_walls", "periodic"])
@pytest.mark.parametrize("size", SIZES + [EIGHT], ids=str)
def test_without_flow(P, size, bounds, storage, u):
    nx, ny, nz = size
    p, (phi, U, rho, v) = problem(P, size, bounds)
    p = P.params(dim=3, nx=nx, ny=ny, nz=nz, flow=0, fold=0, eps=0.03,
                 **{k: w for k, w in BOUNDS[bounds].items() if k != "body"})
    a, b = P.pair(p, storage, fields=(phi, U, rho, v))
    a.step(STEPS)
    b.step(STEPS, P.THREADS)
    errs = P.max_errors(a, b, ("phi", "U"))
    n = STEPS + 1
    assert errs["phi"] < 1e-5 + n * u * 2.0 and errs["U"] < 1e-5 + n * u * 0.5, errs
    a.close()
