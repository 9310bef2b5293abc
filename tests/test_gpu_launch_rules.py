"""Launch rules picked by size: each side of a rule, bit for bit against another
launch shape or, for the adjoint's float atomics, against the FP64 oracle within
the float32 bound of the repository's other comparisons.
"""
import ctypes

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
    P, v = gpu_pyramid(grid), vct.View.from_host(view)
    got = vct.trace_backward(P, [v], [dev], prm, cfg=cfg, deterministic=det)
    if det and tile is None:
        # either default tile: 8 wide, so a round of 32 lanes is the same 8 x 4
        # pixels, and the reproducible sums the same bits on any device
        for t in ((8, 4), (8, 8)):
            assert torch.equal(got, vct.trace_backward(P, [v], [dev], prm, deterministic=True,
                                                       cfg=vct.launch_config(*t)))
    got = got.cpu().numpy().astype(np.float64)
    assert np.abs(got - ref).max() <= 1e-4 * np.abs(ref).max()
    assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)


# Brick builds read only the 16^3 blocks with an occupied brick, listed 256
# at a time per CTA: no block, one voxel, a scattered quarter, every block,
# and (n = 1024) more blocks per CTA than one list holds.
@pytest.mark.parametrize("n,fill", [(16, "none"), (16, "one"), (32, "all"), (64, "some"),
                                    (128, "one"), (256, "some"), (256, "none"), (1024, "some")])
@pytest.mark.parametrize("dtype", ["f32", "f16"])
@pytest.mark.parametrize("planned", [True, False])
def test_brick_build_lists(n, fill, dtype, planned):
    if n == 1024 and dtype == "f32":
        pytest.skip("the binary16 case covers the lists of this size")
    gen = torch.Generator(device="cuda").manual_seed(n)
    g = torch.zeros((n, n, n, 4), device="cuda")
    if fill == "one":
        g[n - 1, 0, n // 2, 3] = 0.5
    elif fill == "all":
        g.uniform_(0.1, 1.0, generator=gen)
    elif fill == "some":  # one voxel in each of a quarter of the 16^3 blocks
        m = n // 16
        pick = torch.rand((m, m, m), device="cuda", generator=gen) < 0.25
        z, y, x = pick.nonzero().mul(16).add(5).unbind(1)
        g[z, y, x] = torch.rand((len(z), 4), device="cuda", generator=gen)
    dense = vct.build_mips(g, dtype=dtype)
    if planned:
        bricks = vct.build_mips(g, dtype=dtype, layout="bricks")
    else:
        bricks = vct.Pyramid(n, dtype=dtype, layout="bricks",
                             occupied=vct.plan_bricks(g, dtype=dtype)[0])
        bricks.storage.fill_(255)  # nothing may be left from before
        vct.build_mips(g, dtype=dtype, out=bricks)
    if planned:
        vct.pyramid_status(bricks)
    for l in range(1 if n == 1024 else 0, dense.levels):
        assert torch.equal(vct.read_level(dense, l), vct.read_level(bricks, l)), l


# Pyramids cut off inside their bricked levels (n = 128 has four, n = 256 takes
# the scan of several CTAs).
@pytest.mark.parametrize("n,levels", [(16, 1), (64, 1), (64, 2), (128, 1), (128, 3), (128, 4),
                                      (256, 1), (256, 4)])
def test_brick_build_few_levels(n, levels):
    g = torch.rand((n, n, n, 4), device="cuda")
    g[: n // 2] = 0
    dense = vct.build_mips(g, levels=levels)
    bricks = vct.build_mips(g, levels=levels, layout="bricks")
    vct.pyramid_status(bricks)
    for l in range(levels):
        assert torch.equal(vct.read_level(dense, l), vct.read_level(bricks, l)), l


# A stream is anything with a cuda_stream handle, here as in every other call.
def test_brick_build_takes_a_stream_handle():
    class Handle:
        def __init__(self, stream):
            self.cuda_stream = stream.cuda_stream

    g = torch.rand((32, 32, 32, 4), device="cuda")
    want = vct.read_level(vct.build_mips(g, layout="bricks"), 1)
    torch.cuda.synchronize()
    for side in (torch.cuda.Stream(), torch.cuda.default_stream()):
        for stream in (side, Handle(side)):
            P = vct.build_mips(g, layout="bricks", stream=stream)
            side.synchronize()
            assert torch.equal(vct.read_level(P, 1), want)


def test_planned_build_checks_its_pool_and_scratch():
    lib, abi = vct.lib(), vct._abi
    g = torch.rand((64, 64, 64, 4), device="cuda")
    occ, _ = vct.plan_bricks(g)
    sb = lib.vct_pyramid_plan_scratch_bytes(64, 7, abi.VCT_F32)
    scratch = torch.zeros(sb, dtype=torch.uint8, device="cuda")
    at = ctypes.c_void_p(scratch.data_ptr())
    stream = torch.cuda.current_stream().cuda_stream
    assert lib.vct_pyramid_plan_bricks(ctypes.c_void_p(g.data_ptr()), 64, 7, abi.VCT_F32, at, sb,
                                       None, None, stream) == abi.VCT_OK
    small = vct.Pyramid(64, layout="bricks", occupied=occ - 1)
    small.storage.zero_()
    p = small.struct()
    args = (ctypes.c_void_p(g.data_ptr()), ctypes.byref(p))
    assert lib.vct_build_mips_planned(*args, at, sb - 1, stream) == abi.VCT_ERR_WORKSPACE
    assert lib.vct_build_mips_planned(*args, None, sb, stream) == abi.VCT_ERR_WORKSPACE
    assert lib.vct_build_mips_planned(*args, at, sb, stream) == abi.VCT_OK
    with pytest.raises(vct.VctError) as e:
        vct.pyramid_status(small)
    assert e.value.status == abi.VCT_ERR_WORKSPACE
    assert not vct.read_level(small, 0).any()
    assert torch.allclose(vct.read_level(small, 6), g.mean(dim=(0, 1, 2)), rtol=1e-5)
    d = vct.Pyramid(64).struct()
    assert lib.vct_build_mips_planned(args[0], ctypes.byref(d), at, sb,
                                      stream) == abi.VCT_ERR_INVALID_ARG


# What a planned build makes of a scratch that is not its plan: one of fewer
# levels, of another edge, never planned, or with slots beyond its count, must
# neither store outside the pool (the guard after it) nor go unreported.
@pytest.mark.parametrize("case", ["levels", "edge", "unplanned", "slots"])
@pytest.mark.parametrize("dtype", ["f32", "f16"])
def test_planned_build_refuses_other_plans(case, dtype):
    lib, abi = vct.lib(), vct._abi
    dt = vct.DTYPES[dtype]
    g = torch.rand((64, 64, 64, 4), device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    occ, nbytes = vct.plan_bricks(g, dtype=dtype)
    sb = lib.vct_pyramid_plan_scratch_bytes(64, 7, dt)
    scratch = torch.randint(0, 255, (sb,), dtype=torch.uint8, device="cuda")
    at = ctypes.c_void_p(scratch.data_ptr())
    if case != "unplanned":
        other = torch.rand((32, 32, 32, 4), device="cuda") if case == "edge" else g
        levels = {"levels": 1, "edge": 6, "slots": 7}[case]
        assert lib.vct_pyramid_plan_bricks(ctypes.c_void_p(other.data_ptr()), len(other), levels,
                                           dt, at, sb, None, None, stream) == abi.VCT_OK
    if case == "slots":
        tables = scratch[256:256 + 4 * 64].view(torch.int32)
        tables[:3] = torch.tensor([occ + 1, 2 ** 31 - 1, -1], device="cuda")
    P = vct.Pyramid(64, dtype=dtype, layout="bricks", occupied=occ)
    P.storage = torch.full((nbytes + 2 ** 20,), 77, dtype=torch.uint8, device="cuda")
    P.storage[:256] = 0
    p = P.struct()
    p.bytes = nbytes
    assert lib.vct_build_mips_planned(ctypes.c_void_p(g.data_ptr()), ctypes.byref(p), at, sb,
                                      stream) == abi.VCT_OK
    with pytest.raises(vct.VctError) as e:
        vct.pyramid_status(P)
    assert e.value.status == abi.VCT_ERR_WORKSPACE
    assert (P.storage[nbytes:] == 77).all()
    if case != "slots":
        assert not vct.read_level(P, 0).any()
        assert torch.allclose(vct.read_level(P, 6), g.mean(dim=(0, 1, 2)),
                              rtol=1e-5 if dtype == "f32" else 2e-3)


class _KernelNode(ctypes.Structure):  # CUDA_KERNEL_NODE_PARAMS_v1
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3),
                ("block", ctypes.c_uint * 3), ("shared", ctypes.c_uint),
                ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p)]


def _launch(P, view, prm, cfg=None):
    """(CTAs, threads per CTA, work-queue cursor afterwards) of a trace's one
    kernel.  The cursor counts the items and one last pull by every warp (or
    group of warps), so it tells tiles apart."""
    ws = torch.zeros(256, dtype=torch.uint8, device="cuda")
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        vct.trace(P, view, prm, cfg=cfg, workspace=ws)
    drv = ctypes.CDLL("libcuda.so.1")
    raw = ctypes.c_void_p(graph.raw_cuda_graph())
    count = ctypes.c_size_t()
    assert drv.cuGraphGetNodes(raw, None, ctypes.byref(count)) == 0
    nodes = (ctypes.c_void_p * count.value)()
    assert drv.cuGraphGetNodes(raw, nodes, ctypes.byref(count)) == 0
    kernels = []
    for node in nodes:
        kind = ctypes.c_int()
        assert drv.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        if kind.value == 0:  # a kernel
            k = _KernelNode()
            assert drv.cuGraphKernelNodeGetParams(ctypes.c_void_p(node), ctypes.byref(k)) == 0
            kernels.append(k)
    assert len(kernels) == 1
    graph.replay()
    queue = int(ws[:56].cpu().numpy().view(np.uint32)[12])
    return kernels[0].grid[0], kernels[0].block[0], queue


# A launch without a shape shares a tile's cones among 4 warps (up to 4 tiles of
# 8 x 4 pixels per SM, three cones and more besides the specular one), 2 (up to
# 32 per SM, two cones and more) or none; widths below 0 are multiples of the
# SM count, heights then on a limit and just above it.  Each against one warp
# per 16 x 8 tile: the cones march the same steps and D sums them in the same
# order, so every output has the same bits.
@pytest.mark.parametrize("w,h,spec,occ,nd,rough,warps", [
    (1, 1, 1, 1, 6, False, 4), (9, 5, 0, 1, 1, False, 2), (37, 21, 1, 0, 2, True, 2),
    (64, 33, 0, 0, 5, False, 4), (60, 40, 1, 1, 32, False, 4), (160, 121, 1, 1, 32, True, 2),
    (-8, 16, 1, 1, 6, True, 4), (-8, 17, 1, 1, 6, True, 2), (-8, 16, 0, 1, 6, False, 4),
    (-8, 128, 1, 1, 1, True, 2), (-8, 129, 1, 1, 1, True, 0), (-8, 128, 0, 1, 2, False, 2),
    (-8, 129, 0, 1, 2, False, 0), (300, 200, 1, 0, 0, True, 0)])
@pytest.mark.parametrize("dtype,layout,flags", [("f32", "dense", 0), ("f16", "bricks", 0),
                                                ("f32", "aniso", 0), ("f32", "dense", 15),
                                                ("f32", "dense", 32 + 24)])
def test_forward_shapes(w, h, spec, occ, nd, rough, warps, dtype, layout, flags):
    n = 16
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    w = w if w > 0 else -w * sms
    rng = np.random.default_rng(w + h)
    scene = vs.box_scene(n, 4, 5, room=True)
    view = vs.interior_view(scene, w, h, rng, with_roughness=rough)
    view["mask"] = (rng.random(w * h) >= 0.1).astype(np.uint8)
    dirs, wts = vs.cone_table_ring6()
    dirs, wts = np.tile(dirs, (6, 1)), np.tile(wts, 6) / 6
    prm = vs.trace_params(dirs[:nd], wts[:nd], 1.0, spec_enable=spec, spec_aperture_min=0.3,
                          spec_aperture_max=0.9, occ_enable=occ, light=scene["light"])
    prm = vs.variant_params(prm, flags)
    P = vct.build_mips(torch.from_numpy(scene["grid"]).cuda(), dtype=dtype, layout=layout)
    out = []
    for cfg in (None, vct.launch_config(16, 8, 1)):
        v = vct.View.from_host(view)
        if flags & vct.FLAG_SHADE:
            v.albedo = torch.full((w * h, 3), 0.7, device="cuda")
            v.alloc_outputs(radiance=True)
        if cfg is None:
            tiles = -(-w // 8) * -(-h // 4)
            shared = (min(-(-tiles * warps // 8), 2 * sms), 256) if warps else None
            own = _launch(P, v, prm)
            assert own[:2] == shared if warps else own == _launch(
                P, v, prm, vct.launch_config(8, 16 if rough and spec else 8))
        v.alloc_cone_state(prm).cone_state.zero_()
        stats = vct.read_stats(vct.trace(P, v, prm, cfg=cfg))
        out.append((v, stats))
    (a, sa), (b, sb) = out
    assert sa == sb
    assert torch.equal(a.cone_state, b.cone_state)
    for x, y in ((a.out_diffuse, b.out_diffuse), (a.out_specular, b.out_specular),
                 (a.out_visibility, b.out_visibility), (a.out_radiance, b.out_radiance)):
        assert x is None or torch.equal(x, y)


# Tiles of 192 pixels and more of dense float32 frames run in two CTAs of 256
# threads per SM, just below that in one of 512; an explicit CTA count is one
# of CTAs of 256.  The same pixels in the same warps' order: the same bits.
# Eight pyramids take the most shared memory.
@pytest.mark.parametrize("tile,views", [((8, 24), 1), ((16, 16), 1), ((8, 23), 1), ((12, 16), 8)])
def test_forward_cta_sizes(tile, views):
    w, h = 1001, 701
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(views)
    scene = vs.box_scene(16, 4, 5, room=True)
    dirs, wts = vs.cone_table_ring6()
    prm = vs.trace_params(dirs[:2], wts[:2], 1.0, spec_enable=1, spec_aperture_min=0.3,
                          spec_aperture_max=0.9, occ_enable=1, light=scene["light"])
    P = [vct.build_mips(torch.from_numpy(scene["grid"]).cuda()) for _ in range(views)]
    host = vs.interior_view(scene, w, h, rng, with_roughness=True)
    out = []
    for per_sm in (0, 1, 2):
        v = [vct.View.from_host({**host, "pyramid": i}) for i in range(views)]
        cfg = vct.launch_config(*tile, 1, per_sm)
        ctas, threads, _ = _launch(P, v, prm, cfg)
        if per_sm:
            assert (ctas, threads) == (per_sm * sms, 256)
        else:
            assert (ctas, threads) == ((2 * sms, 256) if tile[0] * tile[1] >= 192 else (sms, 512))
        for x in v:
            x.alloc_outputs()
        stats = vct.read_stats(vct.trace(P, v, prm, cfg=cfg))
        out.append((v, stats))
    (a, sa) = out[0]
    for b, sb in out[1:]:
        assert sa == sb
        for x, y in zip(a, b):
            assert torch.equal(x.out_diffuse, y.out_diffuse)
            assert torch.equal(x.out_specular, y.out_specular)
            assert torch.equal(x.out_visibility, y.out_visibility)


# The default tile where the specular aperture follows the roughness: 8 x 16
# below 400 pixels per warp of a full chip, 8 x 24 below 1000, 16 x 16 from
# there; each side of both lines, against the same launch with that shape given
# and the pixels of another.  (A view as wide as the chip has warps.)
@pytest.mark.parametrize("h,tile", [(399, (8, 16)), (400, (8, 24)), (999, (8, 24)),
                                    (1000, (16, 16))])
@pytest.mark.parametrize("dtype,layout,flags", [("f32", "dense", 0), ("f16", "dense", 0),
                                                ("f32", "bricks", 8)])
def test_default_tiles(h, tile, dtype, layout, flags):
    w = 16 * torch.cuda.get_device_properties(0).multi_processor_count
    scene = vs.box_scene(16, 4, 5, room=True)
    dirs, wts = vs.cone_table_ring6()
    prm = vs.trace_params(dirs[:2], wts[:2], 1.0, spec_enable=1, spec_aperture_min=0.3,
                          spec_aperture_max=0.9, occ_enable=1, light=scene["light"])
    prm = vs.variant_params(prm, flags)
    part = vs.interior_view(scene, w // 8, h, np.random.default_rng(h), with_roughness=True)
    host = {**part, "width": w}
    for k in ("position", "normal", "roughness", "mask"):
        a = np.asarray(part[k])
        host[k] = np.tile(a.reshape(h, w // 8, -1), (1, 8, 1)).reshape(-1)
    P = vct.build_mips(torch.from_numpy(scene["grid"]).cuda(), dtype=dtype, layout=layout)
    v = vct.View.from_host(host)
    assert _launch(P, v, prm) == _launch(P, v, prm, vct.launch_config(*tile))
    own = (v.out_diffuse.clone(), v.out_specular.clone(), v.out_visibility.clone())
    vct.trace(P, v, prm, cfg=vct.launch_config(16, 8))
    assert torch.equal(v.out_diffuse, own[0])
    assert torch.equal(v.out_specular, own[1])
    assert torch.equal(v.out_visibility, own[2])


# Four, five and all eight pyramids of a call: from five up the step tables
# pass the shared memory of a plain launch.  Each view alone gives the same
# bits, in the default shape (whose warps share tiles here) as in a given one.
@pytest.mark.parametrize("n_pyr", [4, 5, 8])
@pytest.mark.parametrize("lpp,cfg", [(1, True), (1, False), (4, True)])
@pytest.mark.parametrize("layout,flags", [("dense", 0), ("bricks", 0), ("aniso", 0), ("dense", 15)])
def test_many_pyramids(n_pyr, lpp, cfg, layout, flags):
    rng = np.random.default_rng(n_pyr)
    scene = vs.box_scene(16, 4, 5, room=True)
    view = vs.interior_view(scene, 40, 37, rng, with_roughness=True)
    dirs, wts = vs.cone_table_ring6()
    prm = vs.trace_params(dirs, wts, 1.0, spec_enable=1, spec_aperture_min=0.3,
                          spec_aperture_max=0.9, occ_enable=1, light=scene["light"])
    prm = vs.variant_params(prm, flags)
    grid = torch.from_numpy(scene["grid"]).cuda()
    P = [vct.build_mips(grid * (0.5 + 0.05 * i), layout=layout) for i in range(n_pyr)]
    shape = vct.launch_config(8, 8, lpp) if cfg else None

    def make(i):
        v = vct.View.from_host({**view, "pyramid": i})
        if flags:
            v.albedo = torch.full((40 * 37, 3), 0.7, device="cuda")
            v.alloc_outputs(radiance=True)
        return v

    got = [make(i) for i in range(n_pyr)]
    vct.trace(P, got, prm, cfg=shape)
    for i in range(n_pyr):
        one = make(0)
        vct.trace([P[i]], [one], prm, cfg=shape or vct.launch_config(8, 8, 1))
        assert torch.equal(got[i].out_specular, one.out_specular)
        assert torch.equal(got[i].out_visibility, one.out_visibility)
        assert torch.equal(got[i].out_diffuse, one.out_diffuse)


# Sizes whose level 4 passes one tail CTA's 4096 texels, whole and cut off
# inside the levels that several CTAs make: the streaming build and the
# block-wise one (a grid 16 bytes past a 32-byte boundary) give the same bits.
@pytest.mark.parametrize("levels", [5, 6, 7, 9, 10])
@pytest.mark.parametrize("dtype", ["f32", "f16"])
def test_large_build_paths_agree(levels, dtype):
    n = 512
    buf = torch.empty(4 * n ** 3 + 8, device="cuda")
    buf[4:4 + 4 * n ** 3].uniform_(generator=torch.Generator(device="cuda").manual_seed(5))
    shifted = buf[4:4 + 4 * n ** 3].view(n, n, n, 4)
    a = vct.build_mips(shifted, levels=levels, dtype=dtype)
    b = vct.build_mips(shifted.clone(), levels=levels, dtype=dtype)
    for l in range(levels):
        assert torch.equal(vct.read_level(a, l), vct.read_level(b, l)), l


# Tuning never leaves a call slower than the library's own pick: not the call
# it was run for (a shape is kept only if it beat that pick), and not a small
# call of the same kind, whose warps share tiles.
@pytest.mark.parametrize("rough", [False, True])
def test_autotune_leaves_small_calls_alone(rough):
    scene = vs.box_scene(32, 4, 5, room=True)
    dirs, wts = vs.cone_table_ring6()
    prm = vs.trace_params(dirs, wts, 1.0, spec_enable=1, spec_aperture_min=0.3,
                          spec_aperture_max=0.9, occ_enable=1, light=scene["light"])
    P = vct.build_mips(torch.from_numpy(scene["grid"]).cuda())
    rng = np.random.default_rng(3)
    small, mid, large = (vct.View.from_host(vs.interior_view(scene, w, h, rng,
                                                             with_roughness=rough))
                         for w, h in ((100, 91), (270, 200), (1024, 768)))
    own = [_launch(P, v, prm) for v in (small, mid, large)]
    for v, o in ((small, own[0]), (mid, own[1])):  # warps that share tiles
        assert o != _launch(P, v, prm, vct.launch_config(8, 8))
    best = vct.autotune(P, large, prm)
    assert _launch(P, small, prm) == own[0] and _launch(P, mid, prm) == own[1]
    assert _launch(P, large, prm) in (own[2], _launch(P, large, prm, best))
    # one warp marching a tile's cones in series takes about twice as long as
    # four sharing them, so no candidate wins here
    vct.autotune(P, small, prm)
    assert _launch(P, small, prm) == own[0]
