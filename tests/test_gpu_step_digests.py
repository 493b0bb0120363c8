"""Steps in FP32 arithmetic keep their bits: checkpoints after a few steps
against SHA-256 digests (golden/step_digests.json) taken on a GB300 from the
marching kernels, which stepped these lattices first (commit ea09c90).

The switch of the mobility correction (Eq. 4) turns one rounding into 1e-3 of
phi at an interface cell within tens of steps, so a result that is the same to
rounding is not the same result after a long run.  Covered: periodic and open
x, widths that are and are not multiples of 4, walls and none, body force and
none, FP32, BF16 and FP16 storage, steps without and with diagnostics, alone
and in batches (small lattices in groups, large ones by themselves).

The populations are compared, not the fields: FP16's rounding hides most
differences of one FP32 rounding, so the lattices are large enough for the few
that are left (about one stored value in a million).  The digests do not cover
FP64, whose collision form changed with the two-phase step.
"""
import hashlib
import json
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "step_digests.json")
STORAGES = ("fp32", "bf16", "fp16")
PARAMS = dict(sigma=0.005, W=4.0, M=0.02, rho_H=1.0, rho_L=1e-3, nu_H=0.1, nu_L=0.2,
              theta_deg=60.0, mobility_corr=1, F_mode=0, free_slip=1, blend=0.95)
# name: dims, square channel walls, body force, open x
LATTICES = {
    "drop_96x80x72": ((96, 80, 72), False, False, False),
    "drop_61x54x45": ((61, 54, 45), False, False, False),
    "channel_96x50x40": ((96, 50, 40), True, True, False),
    "channel_100x40x40": ((100, 40, 40), True, False, False),
    "channel_63x44x40": ((63, 44, 40), True, True, False),
    "open_72x34x34": ((72, 34, 34), True, False, True),
    "open_53x31x29": ((53, 31, 29), True, True, True),
    "channel_107x38x37": ((107, 38, 37), True, True, False),  # by itself in a batch
}
BATCH = ("channel_63x44x40", "open_53x31x29", "drop_61x54x45", "channel_107x38x37",
         "channel_100x40x40", "drop_96x80x72")


def _lattice(name, storage):
    from paper_2512_01032_gb300 import pflb
    (nx, ny, nz), walls, force, bounds = LATTICES[name]
    solid = np.zeros((nz, ny, nx), np.uint8)
    nrm = np.zeros((nz, ny, nx, 3))
    if walls:
        solid[(0, nz - 1), :, :] = 1
        solid[:, (0, ny - 1), :] = 1
        nrm[:, 1, :, 1], nrm[:, ny - 2, :, 1] = 1.0, -1.0
        nrm[1, :, :, 1:], nrm[nz - 2, :, :, 1:] = (0.0, 1.0), (0.0, -1.0)
    p = dict(PARAMS, Fex=(1e-7, -2e-8, 3e-8) if force else (0.0, 0.0, 0.0))
    L = pflb.Lattice(nx, ny, nz, solid=solid.reshape(-1), wall_normal=nrm.reshape(-1),
                     storage=storage, **p)
    # the tanh profile of the interface, from operations that every machine
    # rounds alike: e^u as (1 + u / 1024)^1024
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij", sparse=True)
    r = np.sqrt((x - 0.4 * nx) ** 2 + (y - 0.47 * ny) ** 2 + (z - 0.52 * nz) ** 2)
    e = 1.0 + np.clip(0.3 * min(ny, nz) - r, -30.0, 30.0) / 1024.0
    for _ in range(10):
        e = e * e
    phi = e / (1.0 + e) * (1 - solid)
    L.init_phi(phi.reshape(-1))
    if bounds:
        L.set_x_boundaries(dict(type="velocity", u=(1e-4, 0, 0), phi=0.0),
                           dict(type="pressure", P=1e-4), ramp_steps=4)
    return L


def _digest(L, tmp):
    """SHA-256 of a checkpoint: header, populations, wall populations, ghosts.
    A zero counts as a zero whatever its sign (the FP16 rest population of a
    gas cell underflows to one or the other)."""
    f = os.path.join(str(tmp), "state.bin")
    L.save(f)
    raw = np.fromfile(f, np.uint8)
    nx, ny, nz, nw, storage, _ = np.frombuffer(raw[8:56].tobytes(), np.int64)
    sha = hashlib.sha256(raw[:56].tobytes())
    n = 2 * (39 * nx * ny * nz + 18 * nw) if storage >= 2 else 0  # bytes of 16-bit values
    for part, t, minus in ((raw[56:56 + n], np.uint16, 0x8000), (raw[56 + n:], np.uint32, 1 << 31)):
        v = part.copy().view(t)
        v[v == minus] = 0
        sha.update(v.tobytes())
    return sha.hexdigest()


def single(name, storage, diag, tmp):
    L = _lattice(name, storage)
    L.set_diag_every(1 if diag else 0)
    L.step(7)
    d = _digest(L, tmp)
    assert np.abs(L.read("P")).max() < 0.1  # a run that blew up says little
    L.close()
    return d


def batch(storage, tmp, kind=3):
    from paper_2512_01032_gb300 import pflb
    lats = [_lattice(n, storage) for n in BATCH]
    lats[0].step(1)  # the other A-A parity
    for L in lats:
        L.set_kernel(kind)
    B = pflb.Batch(lats)
    out = {}
    for steps, last in ((3, False), (4, True)):
        B.step(steps, diag_last=last)
        for n, L in zip(BATCH, lats):
            out[f"batch {n} {storage} t{L.t}"] = _digest(L, tmp)
            assert np.abs(L.read("P")).max() < 0.1
    B.close()
    for L in lats:
        L.close()
    return out


def _golden():
    with open(GOLDEN) as f:
        return json.load(f)["digests"]


@pytest.mark.parametrize("diag", [0, 1])
@pytest.mark.parametrize("storage", STORAGES)
@pytest.mark.parametrize("name", sorted(LATTICES))
def test_steps_keep_their_bits(name, storage, diag, tmp_path):
    assert single(name, storage, diag, tmp_path) == _golden()[f"{name} {storage} diag{diag}"]


@pytest.mark.parametrize("storage", STORAGES)
def test_batch_steps_keep_their_bits(storage, tmp_path):
    got, want = batch(storage, tmp_path), _golden()
    assert [k for k in got if got[k] != want[k]] == []


@pytest.mark.parametrize("kind", [0, 1, 2, 4])
def test_a_lattice_s_kind_does_not_change_a_batch(kind, tmp_path):
    """Small lattices in groups and large ones by themselves alike."""
    got, want = batch("fp32", tmp_path, kind), _golden()
    assert [k for k in got if got[k] != want[k]] == []
