"""The z-marching step kernel (k_pipe) by itself.

The default kind marches only FP32 lattices whose h populations are larger
than twice the L2 cache; PFLB_KERNEL_MARCH takes the march at any size, so that
it can be held to the oracle on the parity cases (the bars of
test_gpu_parity.py) and to the bits of the two-phase step.  Each test asserts
the form that ran.
"""

import numpy as np
import pytest

from tests import _cases as CS
from tests import test_gpu_parity as PAR
from tests import test_gpu_step_digests as SD

pytestmark = pytest.mark.gpu

MARCH, PIPE = 4, 3


def _pair(case):
    G, Orc = CS.make_pair(*case, storage="fp32", kernel=MARCH)
    assert G.marches() and G.get_kernel()["kind"] == MARCH
    return G, Orc


@pytest.mark.parametrize("force", [False, True])
def test_march_matches_oracle_without_walls(force):
    """Periodic droplet, no wall lists: the force-free variant at the steps of
    test_static_droplet_400_steps, the other over its first ones (between them
    FP32 and FP64 part by up to 5e-5 of phi and come together again)."""
    g, p, init = CS.droplet_case()
    p = dict(p, Fex=(1e-8, -2e-8, 5e-9) if force else (0.0, 0.0, 0.0))
    G, Orc = _pair((g, p, init))
    PAR._compare(G, Orc, [0, 1, 2, 7] + ([] if force else [400]), "fp32", 2 * p["sigma"] / init["R"],
                 "march drop")


@pytest.mark.parametrize("diag", [0, 1])
def test_march_matches_oracle_with_walls(diag):
    """Sessile drop on a ball between plates: ghosts, bounce-back, specular
    links, per-block wall lists; without and with diagnostics."""
    g, p, init = CS.sessile_case(32, 60.0)
    G, Orc = _pair((g, p, init))
    G.set_diag_every(diag)
    PAR._compare(G, Orc, [1, 2, 25, 120], "fp32", 2 * p["sigma"] / init["R"], "march sessile")
    if diag:
        phi = Orc.macros()["phi"]
        assert G.last_diag()["nonfinite"] == 0
        # the sum is over the state before the step; mass is conserved to FP32 rounding
        assert G.last_diag()["mass"] == pytest.approx(phi.sum(), rel=1e-5)


@pytest.mark.parametrize("case", ["slit", "channel"])
def test_march_matches_oracle_on_ragged_tiles(case):
    """Extents that are not multiples of the 32 x 4 tile (96 x 16 x 4 and 40 x
    14 x 12), walls and a body force; 20 steps without the band (see
    test_slit_with_force_and_viscosity_ratio)."""
    g, p, init = CS.slit_case() if case == "slit" else CS.channel_case()
    G, Orc = _pair((g, dict(p, free_slip=0), init))
    PAR._compare(G, Orc, [3, 20], "fp32", 2 * p["sigma"] / 16.0, case)


@pytest.mark.parametrize("diag", [0, 1])
@pytest.mark.parametrize("name", [n for n in sorted(SD.LATTICES)
                                  if SD.LATTICES[n][0][0] % 4 == 0 and not SD.LATTICES[n][3]])
def test_march_keeps_its_bits(name, diag, tmp_path):
    """The checkpoint digests that the two-phase step is held to."""
    L = SD._lattice(name, "fp32")
    L.set_kernel(MARCH)
    assert L.marches()
    L.set_diag_every(diag)
    L.step(7)
    assert SD._digest(L, tmp_path) == SD._golden()[f"{name} fp32 diag{diag}"]


def test_depth_changes_keep_the_results_to_the_bit(tmp_path):
    """Every depth from set_kernel and from the autotuner, also across a switch
    to another kind and to open boundaries and back: the wall lists follow the
    depth in effect (a list of another depth would have blocks update other
    blocks' wall nodes)."""
    name = "channel_96x50x40"
    A, B = SD._lattice(name, "fp32"), SD._lattice(name, "fp32")
    A.set_kernel(MARCH)
    opened = (dict(type="velocity", u=(1e-5, 0, 0), phi=0.0), dict(type="pressure", P=0.0))
    for lz in (3, 10, -1, 16, 32, 5):
        A.set_kernel(MARCH, lz=lz)
        assert A.marches()
        A.step(2)
        A.step_diag(1)
    A.set_kernel(PIPE, lz=7)  # two phases; the lists stay those of depth 5
    assert not A.marches()
    A.step(1)
    A.set_kernel(MARCH)
    assert A.marches() and A.get_kernel()["lz"] == 7
    A.step(2)
    A.set_x_boundaries(*opened)
    assert not A.marches() and A.get_kernel()["kind"] == PIPE
    A.set_kernel(MARCH, lz=12)
    A.step(2)
    A.set_x_boundaries(None, None)
    assert A.marches() and A.get_kernel()["lz"] == 12
    A.step(2)
    t = A.t
    lz = A.tune(trial_steps=3)
    assert A.marches() and A.get_kernel() == dict(kind=MARCH, bx=32, by=4, lz=lz)
    A.step(3)
    for _ in range(6):
        B.step(2)
        B.step_diag(1)
    B.step(3)
    B.set_x_boundaries(*opened)
    B.step(2)
    B.set_x_boundaries(None, None)
    B.step(2)
    assert not B.marches() and B.t == t
    B.step(A.t - t)
    assert SD._digest(A, tmp_path) == SD._digest(B, tmp_path)


def test_which_lattices_march():
    from paper_2512_01032_gb300 import pflb
    import torch
    l2 = torch.cuda.get_device_properties(0).L2_cache_size
    n = 4 * int(np.ceil((2.4 * l2 / 76.0) ** (1.0 / 3.0) / 4.0))
    big = pflb.Lattice(n + (-n) % 32, n, n)
    assert big.marches() and big.get_kernel()["kind"] == PIPE
    big.set_kernel(0)
    assert not big.marches()
    big.close()
    for dims, storage in (((64, 32, 32), "fp64"), ((64, 32, 32), "bf16"), ((63, 32, 32), "fp32")):
        L = pflb.Lattice(*dims, storage=storage)
        L.set_kernel(MARCH)
        assert not L.marches() and L.get_kernel()["kind"] == PIPE, (dims, storage)
        L.init_tanh(0, (16, 16, 16), 8.0)
        L.step(2)
        assert np.isfinite(L.read("phi")).all()
        L.close()
    small = pflb.Lattice(64, 32, 32)
    assert not small.marches()
