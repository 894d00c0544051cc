"""GPU tests of the Newton-Schulz chain: one launch that runs every phase of
every iteration, its tiles ordered by counters in global memory (Section 2's
iteration on the tensor cores).

The sizes are the edges of its choices: matrices inside one tile and just past
one, 128- and 256-column tiles (the switch is at one 256 x 256 APPLY tile per
CTA pair, 76 of them), Gram tiles whole and split along K, more shapes than one
launch takes (eight), and the stable-rank mask, whose tile lists are compacted
on the device."""

import numpy as np
import pytest

import oracle as O
from paper_2605_19811_gb300 import synth
from tests.lm_testutil import bits, host_tensor, ns_closed_form_rows, rel_fro, stored_values, tall

pytestmark = pytest.mark.gpu

QUINTIC = O.NS_QUINTIC


def _msign(xh, precision, steps=5):
    import torch
    from paper_2605_19811_gb300 import lionmuon as L
    out = torch.empty(xh.shape, dtype=torch.float32, device="cuda")
    L.msign_ns(xh.cuda(), out, steps, *QUINTIC, eps=1e-7, precision=precision)
    return stored_values(out)


# inside one tile; one past 128, 256; 384 = 1.5 tiles; a long Gram split into
# parts; 72 and 90 APPLY tiles of 256 x 256 (narrow and full-width tiles)
@pytest.mark.parametrize("shape", [(128, 256), (129, 257), (257, 255), (384, 384), (640, 12800), (12800, 250),
                                   (2000, 2100), (2100, 2400)])
@pytest.mark.parametrize("precision,dtype,tol", [(1, "bf16", 2e-2), (2, "f32", 2e-5)])
def test_msign_at_tile_edges(shape, precision, dtype, tol):
    xh = host_tensor(synth.draw_matrix(shape, seed=shape[0]), dtype)
    got = _msign(xh, precision)
    want = ns_closed_form_rows(stored_values(xh), 5, *QUINTIC, 1e-7)
    assert rel_fro(tall(got), want) <= tol


def _steps(shapes, profile, steps=3, dtype="bf16", **cfg):
    import torch
    from paper_2605_19811_gb300 import lionmuon as L
    params = [host_tensor(w, dtype).cuda() for w in synth.init_weights(shapes, seed=1)]
    opt = L.LionMuon(params, **cfg)
    opt.profile(profile)
    for t in range(steps):
        opt.step([host_tensor(x, dtype).cuda() for x in synth.draw_grads(shapes, "student_t", seed=0, step=t)], t)
    torch.cuda.synchronize()
    assert opt.status() == 0
    out = [bits(p) for p in params] + [bits(opt.momentum(i)) for i in range(len(params))]
    opt.close()
    return out


# nine shapes: two launches; a 20000-long Gram split next to short ones; tables
# whose last iteration folds a and whose last does not; a wide set (256-column
# tiles) and a small one (128)
NINE = [(64 * k, 64 * k + 128) for k in range(1, 10)]
CASES = [(NINE, {}), ([(768, 768), (20000, 768), (768, 2304), (768,)], {}),
         ([(512, 640), (640, 512)], dict(ns_coeffs=((8.4, -25.0, 18.0), (4.1, -3.1, 0.6), (1.5, -0.5, 0.0)))),
         ([(768, 3072)] * 4, dict(ns_coeffs=((1.5, -0.5, 0.0), (3.4445, -4.775, 2.0315)))),
         ([(512, 1024), (1024, 512)] * 3, dict(schedule=1, srank_alpha=0.02))]


@pytest.mark.parametrize("shapes,cfg", CASES)
@pytest.mark.parametrize("precision,dtype", [(1, "bf16"), (2, "f32")])
def test_one_launch_equals_one_launch_per_phase(shapes, cfg, precision, dtype):
    """With profiling on every phase has a launch of its own: the same tiles
    without the overlap of phases, so a missing dependency would show."""
    cfg = dict(period=1, **cfg) if "schedule" not in cfg else cfg
    a = _steps(shapes, False, dtype=dtype, ns_precision=precision, **cfg)
    b = _steps(shapes, True, dtype=dtype, ns_precision=precision, **cfg)
    for x, y in zip(a, b):
        np.testing.assert_array_equal(x, y)
