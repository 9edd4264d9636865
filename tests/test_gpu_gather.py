"""The gather kernel (every footprint streamed through shared memory) against
the FP64 oracle and, bit for bit, against the footprint-cache kernel: both do
the same arithmetic in the same order (GPU only)."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import paper_2102_12739_gb300 as dg  # noqa: E402
from paper_2102_12739_gb300 import synth  # noqa: E402
from tests.test_gpu_parity import (G_UV, G_W, TOL, dev, oracle_all, rel_l2,  # noqa: E402
                                   small_workload, upload)

pytestmark = pytest.mark.gpu


def bits(a):
    return np.ascontiguousarray(a).view(np.uint32)


def degrid_both(dtype, comp, sub, uvw, offs, chunk=256):
    """(footprint-cache result, gather result, their status counts)."""
    codes, scale = (sub, None) if dtype == "c64" else dg.pack_subgrids(sub, dtype)
    outs, stats = [], []
    for gather in (False, True):
        with dg.DegridPlan(dtype=dtype, device=sub.device, compensated=comp, gather=gather) as p:
            p.set_tuning(chunk, 8, 0)
            assert p.gather == gather
            outs.append(p.degrid(codes, uvw, offs, scale=scale).cpu().numpy())
            stats.append(p.status())
    return outs[0], outs[1], stats


@pytest.mark.parametrize("comp", [False, True])
@pytest.mark.parametrize("dtype", ["c64", "f16", "bf16"])
@pytest.mark.parametrize("kind", ["scatter", "mixed", "line"])
def test_gather_matches_oracle_and_the_cached_path_bitwise(kind, dtype, comp):
    d = dev()
    # ragged lists: an empty one, 513 = 16 x 32 + 1, 3 (< one stage of 4)
    w = small_workload([700, 0, 513, 64, 3], kind=kind, seed=41)
    w.uvw[9] = [np.nan, 10.0, 1.5]
    w.uvw[-1] = [600.0, 10.0, 1.5]                 # outside the subgrid
    sub_np = synth.subgrid_stack(5)
    sub, uvw, offs = upload(w, sub_np)
    cached, gathered, stats = degrid_both(dtype, comp, sub, uvw, offs)
    assert stats == [2, 2]
    np.testing.assert_array_equal(bits(cached), bits(gathered))
    assert gathered[9] == 0 and gathered[-1] == 0
    ref, bad = oracle.degrid(G_UV, G_W, sub_np.astype(np.complex128), w.uvw, w.vis_offsets)
    assert bad == 2
    assert rel_l2(gathered, ref) <= TOL[dtype]


def test_gather_chunk_sizes_give_the_same_bits():
    d = dev()
    w = small_workload([1000, 37, 0, 2049], kind="scatter", seed=43)
    sub_np = synth.subgrid_stack(4)
    sub, uvw, offs = upload(w, sub_np)
    outs = []
    with dg.DegridPlan(device=d, gather=True) as p:
        for chunk in (32, 64, 256, 1024):
            p.set_tuning(chunk, 8, 0)
            outs.append(p.degrid(sub, uvw, offs).cpu().numpy())
        assert p.status() == 0
    for o in outs[1:]:
        np.testing.assert_array_equal(bits(outs[0]), bits(o))


def test_gather_full_size_scattered_workload_every_visibility():
    # 16 subgrids x 250,000 scattered visibilities, the launch configuration
    # the benchmark times for this workload; every visibility against the
    # oracle and bitwise against the footprint-cache kernel
    d = dev()
    w = synth.workload("scatter16_250k")
    sub_np = w.subgrids()
    sub, uvw, offs = upload(w, sub_np)
    ref = oracle_all(w, lambda s: sub_np[s])
    for dtype in ("c64", "bf16"):
        cached, gathered, stats = degrid_both(dtype, False, sub, uvw, offs, chunk=256)
        assert stats == [0, 0]
        np.testing.assert_array_equal(bits(cached), bits(gathered))
        assert rel_l2(gathered, ref) <= TOL[dtype]


def test_gather_host_entry_point_and_graph_capture():
    d = dev()
    w = small_workload([300, 0, 150, 77], kind="scatter", seed=47)
    sub_np = synth.subgrid_stack(4)
    sub, uvw, offs = upload(w, sub_np)
    with dg.DegridPlan(device=d, gather=True) as p:
        ref = p.degrid(sub, uvw, offs).cpu().numpy()
        host = p.degrid_host(sub_np, w.uvw, w.vis_offsets).numpy()
        np.testing.assert_array_equal(bits(host), bits(ref))
        out = torch.empty(w.n_vis, dtype=torch.complex64, device=d)
        s = torch.cuda.Stream(d)
        with torch.cuda.stream(s):
            p.degrid(sub, uvw, offs, out=out)       # sizes the scratch before capture
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            p.degrid(sub, uvw, offs, out=out)
        out.zero_()
        g.replay()
        torch.cuda.synchronize()
        np.testing.assert_array_equal(bits(out.cpu().numpy()), bits(ref))
        assert p.status() == 0


def test_gather_is_refused_where_it_cannot_run():
    d = dev()
    with dg.DegridPlan(device=d, g_uv2=synth.default_table_2d()) as p2:
        with pytest.raises(dg.DegridError):
            p2.set_gather(True)
        assert not p2.gather
    with dg.DegridPlan(shape=(64, 64, 8), device=d) as p8:
        with pytest.raises(dg.DegridError):
            p8.set_gather(True)
        p8.set_gather(False)
    with dg.DegridPlan(device=d) as p:
        assert dg.load().degrid_plan_set_gather(p.handle, 2) == dg._native.DG_ERR_ARG
        v = ctypes.c_int(-1)
        assert dg.load().degrid_plan_get_gather(p.handle, ctypes.byref(v)) == 0 and v.value == 0


@pytest.mark.parametrize("kind", ["scatter", "mixed", "line"])
def test_scatter_gridding_matches_oracle(kind):
    # the adjoint with the plan's gather setting: one tensor reduce-add per
    # visibility; ragged lists, an empty subgrid, invalid points, accumulate
    d = dev()
    w = small_workload([1500, 0, 513, 64, 3], kind=kind, seed=61)
    w.uvw[9] = [np.nan, 10.0, 1.5]
    w.uvw[-1] = [600.0, 10.0, 1.5]
    y = synth.adjoint_vis(w.n_vis)
    uvw = torch.from_numpy(w.uvw).to(d)
    offs = torch.from_numpy(w.vis_offsets).to(d)
    yd = torch.from_numpy(y).to(d)
    ref, bad = oracle.grid(G_UV, G_W, synth.SUBGRID_SHAPE, 5, w.uvw, w.vis_offsets, y)
    assert bad == 2
    with dg.DegridPlan(device=d, gather=True) as p:
        got = p.grid(yd, uvw, offs, 5).cpu().numpy()
        assert p.status() == 2
        assert rel_l2(got, ref) <= TOL["c64"]
        assert np.all(got[1] == 0)
        base = torch.ones((5,) + synth.SUBGRID_SHAPE, dtype=torch.complex64, device=d)
        acc = p.grid(yd, uvw, offs, 5, out=base, accumulate=True).cpu().numpy()
        assert p.status() == 2
        assert rel_l2(acc - 1, ref) <= TOL["c64"]
    with dg.DegridPlan(device=d) as p0:             # the run-accumulating kernel agrees
        other = p0.grid(yd, uvw, offs, 5).cpu().numpy()
    assert rel_l2(got, other) <= 1e-6


def test_scatter_gridding_full_size_and_dot_product():
    # 16 subgrids x 250,000 scattered visibilities: the whole gridded stack
    # against the oracle, and <D s, y> = <s, G y> with both directions on the
    # gather kernels
    d = dev()
    w = synth.workload("scatter16_250k")
    sub_np = w.subgrids()
    sub, uvw, offs = upload(w, sub_np)
    y = synth.adjoint_vis(w.n_vis)
    yd = torch.from_numpy(y).to(d)
    with dg.DegridPlan(device=d, gather=True) as p:
        g = p.grid(yd, uvw, offs, w.n_subgrids)
        dvis = p.degrid(sub, uvw, offs)
        assert p.status() == 0
        lhs = torch.vdot(dvis.to(torch.complex128), yd.to(torch.complex128)).item()
        rhs = torch.vdot(sub.to(torch.complex128).flatten(), g.to(torch.complex128).flatten()).item()
        gnp = g.cpu().numpy()
    assert abs(lhs - rhs) <= 1e-5 * abs(lhs)
    ref, _ = oracle.grid(G_UV, G_W, synth.SUBGRID_SHAPE, w.n_subgrids, w.uvw, w.vis_offsets, y)
    assert rel_l2(gnp, ref) <= TOL["c64"]


TILED = [   # shape, counts, kind: enough visibilities per tile for the tile kernels
    ((48, 48, 4), [250000], "scatter"),
    ((71, 135, 4), [40000, 0, 170001, 33], "scatter"),         # tiles end inside and at the last start
    ((103, 87, 4), [220000, 1], "line"),                        # dense: whole warps in one tile
    ((512, 512, 4), [260000, 1], "mixed"),
]


@pytest.mark.parametrize("shape,counts,kind", TILED)
@pytest.mark.parametrize("dtype,comp", [("c64", False), ("f16", True), ("bf16", False)])
def test_tiled_degridding_is_bitwise_the_cached_path(shape, counts, kind, dtype, comp):
    d = dev()
    w = small_workload(counts, kind=kind, shape=shape, seed=91)
    uvw_np = w.uvw.copy()
    bad = [0, 31, 32, 1777, len(uvw_np) - 1]
    uvw_np[bad] = [[np.nan, 9, 1.5], [1e9, 9, 1.5], [9, -2, 1.5], [9, 9, 77.0], [3.4, 1e300, 1.2]]
    # the corners of the valid box: first and last start of the first and last tile
    ny, nx, _ = shape
    uvw_np[100:104] = [[3, 3, 1.0], [nx - 5 + 0.999, 3, 1.5], [3, ny - 5 + 0.999, 1.99], [nx - 5, ny - 5, 1.0]]
    sub = torch.from_numpy(synth.subgrid_stack(len(counts), shape=shape)).to(d)
    codes, scale = (sub, None) if dtype == "c64" else dg.pack_subgrids(sub, dtype)
    uvw, offs = torch.from_numpy(uvw_np).to(d), torch.from_numpy(w.vis_offsets).to(d)
    outs = []
    for gather in (False, True):
        with dg.DegridPlan(shape=shape, dtype=dtype, device=d, compensated=comp, gather=gather) as p:
            out = torch.full((w.n_vis,), float("nan"), dtype=torch.complex64, device=d)
            outs.append(p.degrid(codes, uvw, offs, scale=scale, out=out).cpu().numpy())
            assert p.status() == len(bad)
    np.testing.assert_array_equal(outs[0].view(np.uint64), outs[1].view(np.uint64))


@pytest.mark.parametrize("shape,counts,kind", TILED)
def test_tiled_gridding_matches_oracle(shape, counts, kind):
    d = dev()
    w = small_workload(counts, kind=kind, shape=shape, seed=92)
    uvw_np = w.uvw.copy()
    uvw_np[[5, 1234]] = [[np.inf, 9, 1.5], [9, 9, -1.0]]
    y = synth.adjoint_vis(w.n_vis)
    ref, bad = oracle.grid(G_UV, G_W, shape, len(counts), uvw_np, w.vis_offsets, y)
    assert bad == 2
    with dg.DegridPlan(shape=shape, device=d, gather=True) as p:
        args = (torch.from_numpy(y).to(d), torch.from_numpy(uvw_np).to(d), torch.from_numpy(w.vis_offsets).to(d),
                len(counts))
        out = p.grid(*args)
        assert p.status() == 2
        assert rel_l2(out.cpu().numpy(), ref) <= 2e-6
        p.grid(*args, out=out, accumulate=True)
        assert rel_l2(out.cpu().numpy(), 2 * ref) <= 2e-6
        assert p.status() == 2


def test_a_captured_call_larger_than_the_tiles_workspace():
    # a plan that has only seen few visibilities cannot grow its workspace
    # inside a capture: the call is captured through the gather kernel
    d = dev()
    shape = (64, 64, 4)
    w = small_workload([300000], kind="scatter", shape=shape, seed=93)
    sub = torch.from_numpy(synth.subgrid_stack(1, shape=shape)).to(d)
    uvw, offs = torch.from_numpy(w.uvw).to(d), torch.from_numpy(w.vis_offsets).to(d)
    out = torch.zeros(w.n_vis, dtype=torch.complex64, device=d)
    with dg.DegridPlan(shape=shape, device=d) as p:
        p.degrid(sub, uvw, offs)                        # the chunk table, without tiles
        p.set_gather(True)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            p.degrid(sub, uvw, offs, out=out)
        g.replay()
        torch.cuda.synchronize()
        first = out.cpu().numpy()
        second = p.degrid(sub, uvw, offs).cpu().numpy()         # by tiles
        assert p.status() == 0
    np.testing.assert_array_equal(first.view(np.uint64), second.view(np.uint64))


@pytest.mark.parametrize("dtype,comp", [("c64", False), ("c64", True), ("f16", False), ("bf16", True)])
def test_gather_and_scatter_kernels_on_many_lists(dtype, comp):
    # more lists than a call by pieces takes and too few visibilities for
    # tiles: every footprint by itself (ragged lists, empty ones, invalid
    # visibilities), bit for bit the cached path; gridding against the oracle
    d = dev()
    shape = (32, 40, 4)
    rng = np.random.default_rng(5)
    counts = [int(c) for c in rng.integers(0, 12, 300)] + [700, 0, 513]
    w = small_workload(counts, kind="scatter", shape=shape, seed=97)
    uvw_np = w.uvw.copy()
    uvw_np[::97] = [9.0, 9.0, -4.0]
    sub_np = synth.subgrid_stack(len(counts), shape=shape)
    sub = torch.from_numpy(sub_np).to(d)
    codes, scale = (sub, None) if dtype == "c64" else dg.pack_subgrids(sub, dtype)
    uvw, offs = torch.from_numpy(uvw_np).to(d), torch.from_numpy(w.vis_offsets).to(d)
    outs = []
    for gather in (False, True):
        with dg.DegridPlan(shape=shape, dtype=dtype, device=d, compensated=comp, gather=gather) as p:
            outs.append(p.degrid(codes, uvw, offs, scale=scale).cpu().numpy())
            assert p.status() == len(uvw_np[::97])
    np.testing.assert_array_equal(bits(outs[0]), bits(outs[1]))
    if dtype == "c64":
        y = synth.adjoint_vis(w.n_vis)
        ref, _ = oracle.grid(G_UV, G_W, shape, len(counts), uvw_np, w.vis_offsets, y)
        with dg.DegridPlan(shape=shape, device=d, gather=True) as p:
            out = p.grid(torch.from_numpy(y).to(d), uvw, offs, len(counts)).cpu().numpy()
            assert p.status() == len(uvw_np[::97])
        assert rel_l2(out, ref) <= 2e-6
