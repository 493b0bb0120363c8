"""FP64 batches: a small lattice steps in a batch in about the time of its own
kernels (its fields: test_gpu_batch.py).

An FP64 block is one warp and the step is bound by the FP64 rate, so an item of
several blocks' cells adds their whole time to the step: items of 128 cells
took 98 us per step for one 16^3 lattice in a batch (the tile march before them
73), items of 32 take 34.  The bound is between the two: a batch step may take
2.2 times the lattice's own step and a tenth of a millisecond more for the
uploads and events of a call over its 64 steps.
"""
import pytest

import synth

pytestmark = pytest.mark.gpu

STEPS = 64


def _lattice(n, walls, stream):
    from paper_2512_01032_gb300 import pflb
    g, p, init = synth.sessile_sphere(n, 60.0) if walls else synth.static_droplet(n, n / 4.0)
    L = pflb.Lattice(g.nx, g.ny, g.nz, solid=g.solid, wall_normal=g.normals(),
                     theta_cells=g.theta(), stream=stream, storage="fp64", **p)
    L.init_tanh(0, init["center"], init["R"])
    return L


def _best_us(step, stream):
    import torch
    step(STEPS)
    best = float("inf")
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        with torch.cuda.stream(stream):
            a.record()
            step(STEPS)
            b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3 / STEPS)
    return best


@pytest.mark.parametrize("n,walls", [(16, False), (16, True), (24, False)])
def test_small_fp64_lattice_in_a_batch(n, walls):
    import torch
    from paper_2512_01032_gb300 import pflb
    stream = torch.cuda.Stream()
    A, M = _lattice(n, walls, stream), _lattice(n, walls, stream)
    B = pflb.Batch([M], stream=stream)
    own, batch = _best_us(A.step, stream), _best_us(B.step, stream)
    assert batch <= 2.2 * own + 100.0 / STEPS, (own, batch)
    B.close()
