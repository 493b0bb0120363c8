"""The default kernel's two forms against the general two-pass kernel.

The default kind runs the two-phase step on most lattices and the pipelined
march on FP32 ones whose h populations are larger than twice the L2 cache; a
batch steps small lattices in groups and large ones by themselves.  Each form
is compared with the two-pass kernel (pinned to the oracle by the parity
tests) on the same inputs, at sizes where it can go wrong: cell counts that
are and are not multiples of the 16-byte loads, one-cell extents, the edges
of a block, no wall nodes, open boundaries, both A-A parities.

Tolerances: the rounding of a step differs between the forms (pair form
against per-direction form of the same sums), so phi, rho and P agree to the
parity bars of the oracle tests relative to the field's scale (FP64 1e-11,
FP32 1e-5); at 16-bit storage one flip of a stored population per cell and
step is allowed, 2 (1 - w_0) 2^-m with m = 9 (BF16) and 12 (FP16) bits.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

FIELDS = ("phi", "rho", "P")


def _tol(storage, n):
    flip = 2 * (2.0 / 3.0) * n
    return {"fp64": 1e-11, "fp32": 1e-5, "fp16": flip * 2.0 ** -12, "bf16": flip * 2.0 ** -9}[storage]


def _case(dims, walls, theta=70.0):
    import synth
    nx, ny, nz = dims
    shapes = []
    if walls:
        shapes.append(synth.Plane((0, 0, 0.5), (0, 0, 1)))
        if nx > 8:
            shapes.append(synth.Box((nx // 2, 0, 0), (nx // 2 + 2, max(1, ny // 3), nz)))
    g = synth.Geometry(nx, ny, nz, shapes, theta_deg=theta)
    p = dict(synth.sessile_sphere_params(theta), Fex=(1e-8, -2e-8, 0.0))
    init = dict(center=(nx / 2.0 + 0.37, ny / 2.0 - 0.21, nz / 2.0 + 0.13),
                R=max(1.5, min(dims) / 3.0))
    return g, p, init


def _lattice(case, storage, kind=3, bounds=False):
    from paper_2512_01032_gb300 import pflb
    g, p, init = case
    L = pflb.Lattice(g.nx, g.ny, g.nz, solid=g.solid, wall_normal=g.normals(),
                     theta_cells=g.theta(), solid_frac=g.solid_frac(), storage=storage, **p)
    L.set_kernel(kind)
    L.init_tanh(0, init["center"], init["R"], P0=1e-3)
    if bounds:
        L.set_x_boundaries(dict(type="velocity", u=(1e-4, 0, 0), phi=0.0),
                           dict(type="pressure", P=1e-3), ramp_steps=3)
    return L


def _close(A, B, tol):
    assert A.t == B.t
    for f in FIELDS:
        a, b = A.read(f), B.read(f)
        assert np.isfinite(a).all()
        assert np.abs(a - b).max() <= tol * max(np.abs(a).max(), 1e-3 if f != "phi" else 1.0), f


@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp16", "bf16"])
@pytest.mark.parametrize("dims,walls,bounds", [
    ((37, 23, 11), True, False), ((36, 32, 9), True, False), ((24, 10, 8), False, False),
    ((1, 6, 5), False, False), ((64, 1, 1), False, False), ((65, 3, 1), False, False),
    ((3, 8, 6), True, True), ((33, 9, 7), True, True), ((40, 8, 8), False, True)])
def test_two_phase_step_matches_two_pass(dims, walls, bounds, storage):
    c = _case(dims, walls)
    A, B = _lattice(c, storage, 3, bounds), _lattice(c, storage, 1, bounds)
    for L in (A, B):
        L.step(2)
        L.set_diag_every(1)
        L.step(3)
    _close(A, B, _tol(storage, 5))
    a, b = A.last_diag(), B.last_diag()
    for k in ("mass", "n_heavy", "n_p_heavy", "n_p_light", "region_mass", "cl_count", "nonfinite"):
        assert a[k] == pytest.approx(b[k], rel=max(2e-6, _tol(storage, 5)), abs=1e-12), k


@pytest.mark.parametrize("storage", ["fp32", "bf16"])
def test_batch_of_large_small_and_open_lattices(storage):
    """Lattices of 131072 cells and more are stepped by themselves inside a
    batch: the same bits as outside it.  Small and open ones, stepped in
    groups, agree with the two-pass kernel."""
    from paper_2512_01032_gb300 import pflb
    specs = [((100, 64, 64), True, False), ((37, 23, 11), True, False), ((33, 9, 7), True, True),
             ((40, 14, 12), False, False)]
    mixed = [_lattice(_case(d, w), storage, 3, b) for d, w, b in specs]
    ref = [_lattice(_case(d, w), storage, 3 if k == 0 else 1, b)
           for k, (d, w, b) in enumerate(specs)]
    mixed[1].step(1)
    ref[1].step(1)
    B = pflb.Batch(mixed)
    B.step(3)
    B.step(2, diag_last=True)
    for k, (A, M) in enumerate(zip(ref, mixed)):
        A.step(4)
        A.step_diag(1)
        _close(M, A, _tol(storage, 6))
        if k == 0:
            for f in ("phi", "P", "ux"):
                assert np.array_equal(A.read(f), M.read(f)), f
        assert M.last_diag()["mass"] == pytest.approx(A.last_diag()["mass"],
                                                      rel=max(2e-6, _tol(storage, 6)))
    B.close()


@pytest.mark.parametrize("storage,dims", [("fp32", (160, 151, 160)), ("fp32", (188, 142, 145)),
                                          ("bf16", (204, 185, 184))])
def test_lattices_beyond_l2(storage, dims):
    import torch
    h = dims[0] * dims[1] * dims[2] * (19 * 4 if storage == "fp32" else 20 * 2)
    assert h > 2 * torch.cuda.get_device_properties(0).L2_cache_size
    c = _case(dims, True)
    A, B = _lattice(c, storage, 3), _lattice(c, storage, 1)
    for L in (A, B):
        L.step(2)
        L.step_diag(1)
    _close(A, B, _tol(storage, 3))
    assert A.last_diag()["mass"] == pytest.approx(B.last_diag()["mass"],
                                                  rel=max(2e-6, _tol(storage, 3)))
