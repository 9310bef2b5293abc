"""Launch rules picked by size: each side of a rule against the FP64 oracle.

A pixel's sums are the same terms in another order on either side, so every
case is held to the float32 bound of the repository's other comparisons.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
import paper_2104_00618_gb300 as vct  # noqa: E402
import vct_synth as vs  # noqa: E402
from gpu_cases import gpu_pyramid  # noqa: E402


# (width, height, tile or None, lanes per pixel, specular, occlusion, diffuse cones):
# None takes the default shape (8 x 4 tiles at these sizes).  1 x 1 tiles of
# 110 x 101 pixels pass four tiles per warp of a full chip, where a tile's
# cones are one item; every other case has one item per group of cones, the
# last group short when the lanes do not divide the cones.
@pytest.mark.parametrize("w,h,tile,lpp,spec,occ,nd", [
    (1, 1, None, 1, 1, 1, 6), (33, 5, None, 1, 0, 0, 1), (40, 37, None, 1, 1, 0, 6),
    (40, 37, (8, 8), 4, 1, 1, 5), (40, 37, (3, 7), 2, 0, 1, 0), (110, 101, (1, 1), 1, 1, 1, 2),
    (110, 101, (1, 1), 8, 1, 1, 6)])
@pytest.mark.parametrize("det", [False, True])
def test_adjoint_items(w, h, tile, lpp, spec, occ, nd, det):
    n = 16
    rng = np.random.default_rng(w * 100 + h)
    scene = vs.box_scene(n, 4, 5, room=True)
    view = vs.interior_view(scene, w, h, rng, with_roughness=False)
    dirs, wts = vs.cone_table_ring6()
    prm = vs.trace_params(dirs[:nd], wts[:nd], 1.0, spec_enable=spec, spec_aperture_min=0.3,
                          occ_enable=occ, light=scene["light"])
    grid = rng.uniform(0.05, 0.3, size=(n, n, n, 4)).astype(np.float32)
    g = [rng.normal(size=(w * h, 4)), rng.normal(size=(w * h, 4)), rng.normal(size=w * h)]
    ref = oracle.trace_backward(oracle.build_mips(grid), view, prm, *g)
    dev = tuple(torch.from_numpy(a.astype(np.float32)).cuda() for a in g)
    cfg = None if tile is None else vct.launch_config(tile[0], tile[1], lpp)
    got = vct.trace_backward(gpu_pyramid(grid), [vct.View.from_host(view)], [dev], prm, cfg=cfg,
                             deterministic=det).cpu().numpy().astype(np.float64)
    assert np.abs(got - ref).max() <= 1e-4 * np.abs(ref).max()
    assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)
