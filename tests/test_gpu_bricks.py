"""The quad brick form where its work splits: bricks holding every number of
particles around a warp's 32 and a block's trip, long bricks, the last bricks of an axis that hold fewer cells, positions on both
sides of the halo's edge.  Bars as in test_gpu_parity (FP32 interpolation
1e-5 of the rms velocity, a Heun step dt times that)."""
import math

import numpy as np
import pytest
import torch

import oracle
import paper_2005_13193_gb300 as ps
from paper_2005_13193_gb300 import synth

pytestmark = pytest.mark.gpu
TWO_PI = 2 * math.pi
DEV = "cuda"


def _counted_positions(n, brick, counts, seed):
    """Brick b (x fastest) holds counts[b % len(counts)] particles, the first one
    of each on the brick's low corner and the second just below its high one."""
    rng = np.random.Generator(np.random.PCG64(seed))
    nb = [-(-n[d] // brick[d]) for d in range(3)]
    cols = []
    for b in range(nb[0] * nb[1] * nb[2]):
        m = counts[b % len(counts)]
        o = (b % nb[0], b // nb[0] % nb[1], b // (nb[0] * nb[1]))
        lo = np.array([o[d] * brick[d] for d in range(3)], dtype=np.float64)[:, None]
        hi = np.array([min(n[d], (o[d] + 1) * brick[d]) for d in range(3)],
                      dtype=np.float64)[:, None]
        u = rng.random((3, m))
        if m > 0:
            u[:, 0] = 0.0
        if m > 1:
            u[:, 1] = 1.0 - 1e-9
        cols.append((lo + u * (hi - lo)) * (TWO_PI / np.array(n, dtype=np.float64)[:, None]))
    return np.concatenate(cols, axis=1)


@pytest.mark.parametrize("n,brick", [((32, 16, 24), (8, 8, 8)), ((30, 21, 18), (8, 8, 8)),
                                     ((16, 130, 8), (2, 60, 2)), ((24, 20, 16), (12, 5, 8))])
@pytest.mark.parametrize("dtype,bar", [(ps.F32X4, 1e-5), (torch.float32, 1e-5),
                                       (ps.F16X4, 4e-3)])
def test_bricks_of_every_fill(n, brick, dtype, bar):
    counts = [0, 1, 7, 8, 9, 31, 32, 33, 63, 64, 65, 71, 72, 96, 97, 127, 128, 129, 200]
    field = synth.random_field(n, ncomp=3, seed=5).astype(np.float32)
    cref = oracle.spline_coeffs(field.astype(np.float64))
    pos = _counted_positions(n, brick, counts, seed=6)
    pos = np.ascontiguousarray(
        pos[:, np.random.Generator(np.random.PCG64(7)).permutation(pos.shape[1])])
    sf = ps.SplineField.from_field(torch.from_numpy(field).to(DEV), dtype)
    pg = torch.from_numpy(pos).to(DEV)
    bins = ps.bin_particles(n, brick, pg)
    ref, gref = oracle.interp(cref, pos, grad=True)
    rms, cmax = np.sqrt((ref ** 2).mean()), np.abs(cref).max()
    st = torch.zeros(4, dtype=torch.int32, device=DEV)
    vel = sf.interp(pg, bins=bins, status=st)
    velg, grad = sf.interp(pg, grad=True, bins=bins, status=st)
    # 16-bit values: half a unit of 2^-11 of the line's scale (below 2 max|c|)
    # per coefficient, the weights (their derivatives) summing to 1 (2 per axis)
    q = 0.0 if bar < 1e-4 else 2.0 ** -11 * cmax
    for v in (vel, velg):
        assert np.abs(v.cpu().numpy() - ref).max() <= 1e-5 * rms + q
    for d in range(3):
        tol = (1e-5 * 3 * cmax + 2 * q) * n[d] / TWO_PI
        assert np.abs(grad[:, d].cpu().numpy() - gref[:, d]).max() <= tol
    dt = 0.3 * TWO_PI / max(n)
    new_ref, u1 = oracle.rk2_step(cref, pos, dt)
    tr = ps.Tracker(sf, pg.clone(), brick=brick)
    tr.step(dt)
    ids = tr.ids.cpu().numpy()
    if q == 0.0:
        assert np.abs(tr.pos.cpu().numpy() - new_ref[:, ids]).max() <= dt * 1e-5 * rms + 1e-14
    # the counts the step took are those of the positions it wrote
    x1 = tr.pos.clone()
    off = torch.empty_like(tr.offsets)
    xs = torch.empty_like(x1)
    ps.ps_rk2_sort(n, brick, x1, xs, off, tr.ws, counted=True, status=st)
    np.testing.assert_array_equal(off.cpu().numpy(),
                                  oracle.bin_particles(n, brick, x1.cpu().numpy())[1])
    assert ps.ps_status_read(st)[0] == 0


@pytest.mark.parametrize("dtype", [ps.F32X4, torch.float32, ps.BF16X4])
def test_results_by_way_of_bin_order(dtype):
    # with a workspace a permuted call stores in bin order and puts the rows in
    # place afterwards: the same bits, for every row count and a ragged last block
    n, brick = (40, 24, 17), (8, 8, 8)
    field = synth.random_field(n, ncomp=3, seed=15).astype(np.float32)
    sf = ps.SplineField.from_field(torch.from_numpy(field).to(DEV), dtype)
    for np_ in (1, 1023, 5000):
        pg = torch.from_numpy(synth.uniform_particles(np_, seed=16) * 1.3 - 0.5).to(DEV)
        bins = ps.bin_particles(n, brick, pg)
        kw = dict(scale=sf.scale, perm=bins.perm, bin_offsets=bins.offsets, brick=brick)

        def both(rows, call):
            outs = []
            for ws in (None, ps.workspace(ps._lib().ps_unsort_workspace_size(np_, rows))):
                o = torch.full((rows, np_), math.nan, device=DEV)
                call(o, ws)
                outs.append(o)
            assert not torch.isnan(outs[0]).any() and torch.equal(*outs)

        both(3, lambda o, ws: ps.ps_interp(sf.coef, n, pg, o, ws=ws, **kw))
        both(12, lambda o, ws: ps.ps_interp(sf.coef, n, pg, o[:3], grad=o[3:], ws=ws, **kw))
        both(18, lambda o, ws: ps.ps_interp_hessian(sf.coef, n, pg, o, ws=ws, **kw))
        kw["scale_n"] = kw.pop("scale")
        both(6, lambda o, ws: ps.ps_lagrangian_accel(sf.coef, n, pg, o[3:], coef_np1=sf.coef,
                                                     scale_np1=sf.scale, vel=o[:3], ws=ws, **kw))


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64, torch.int64])
@pytest.mark.parametrize("np_,rows", [(1, 1), (1023, 3), (1025, 18), (70000, 5)])
def test_permute_rows(dtype, np_, rows):
    g = torch.Generator(DEV).manual_seed(np_)
    perm = torch.randperm(np_, device=DEV, generator=g)
    src = torch.randint(-2**20, 2**20, (rows, np_), device=DEV, generator=g).to(dtype)
    dst = torch.empty_like(src)
    ps.ps_permute_rows(src, perm, dst, to_bins=True)
    assert torch.equal(dst, src[:, perm])
    back = torch.empty_like(src)
    ps.ps_permute_rows(dst, perm, back, to_bins=False)
    assert torch.equal(back, src)


@pytest.mark.parametrize("n,brick", [((24, 16, 40), (8, 8, 8)), ((9, 21, 5), (8, 8, 8)),
                                     ((3, 4, 5), (8, 8, 8)), ((20, 18, 12), (5, 7, 3)),
                                     ((40, 8, 8), (20, 4, 4)), ((32, 16, 24), (8, 8, 8))])
@pytest.mark.parametrize("crowd", [False, True])
def test_binned_adjoint(n, brick, crowd):
    # a cell holding more particles than one warp takes (512), bricks below and
    # above the staging threshold, positions outside the box, stale bins
    rng = np.random.Generator(np.random.PCG64(25))
    field = synth.random_field(n, ncomp=3, seed=26).astype(np.float32)
    cref = oracle.spline_coeffs(field.astype(np.float64))
    pos = np.ascontiguousarray(rng.random((3, 4000)) * TWO_PI * 1.5 - 1.0)
    if crowd:
        pos[:, :2500] = (rng.random((3, 2500)) + 1.0) * TWO_PI / np.array(n)[:, None]
    w = rng.standard_normal((3, pos.shape[1])).astype(np.float32)
    gp_ref, gf_ref = oracle.interp_backward(cref, pos, w.astype(np.float64))
    sf = ps.SplineField.from_field(torch.from_numpy(field).to(DEV), torch.float32)
    pg, wg = torch.from_numpy(pos).to(DEV), torch.from_numpy(w).to(DEV)
    bins = ps.bin_particles(n, brick, pg)
    stale = ps.bin_particles(n, brick, (pg + 0.7).contiguous())
    cmax, wsum = np.abs(cref).max(), np.abs(w).sum(0).max()
    direct = torch.empty_like(pg)
    ps.ps_interp_backward(sf.coef, n, pg, wg, direct, None)
    ws = ps.workspace(ps.ps_backward_workspace_size(n, brick))
    for b, w_ in ((bins, None), (bins, ws), (stale, ws)):
        g_pos = torch.empty_like(pg)
        g_field = torch.empty((3,) + tuple(reversed(n)), dtype=torch.float32, device=DEV)
        st = torch.zeros(4, dtype=torch.int32, device=DEV)
        ps.ps_interp_backward(sf.coef, n, pg, wg, g_pos, g_field, status=st, perm=b.perm,
                              bin_offsets=b.offsets, brick=brick, ws=w_)
        assert torch.equal(g_pos, direct)  # the same sums in the same order
        assert ps.ps_status_read(st)[0] == 0
        for d in range(3):
            tol = 1e-5 * 3 * (n[d] / TWO_PI) * cmax * wsum
            assert np.abs(g_pos[d].cpu().numpy() - gp_ref[d]).max() <= tol
        gf = g_field.cpu().numpy()
        assert np.abs(gf - gf_ref).max() <= 1e-5 * np.abs(gf_ref).max() + 1e-6


@pytest.mark.parametrize("least", [0, 10**6])
def test_autograd_bins_enough_particles(least, monkeypatch):
    monkeypatch.setattr(ps, "_FN_MIN_IN_L2", least)  # binned, and in the particles' order
    n = (32, 24, 16)
    field = synth.random_field(n, ncomp=3, seed=35).astype(np.float32)
    cref = oracle.spline_coeffs(field.astype(np.float64))
    pos = synth.uniform_particles(60_000, seed=36)
    w = np.random.Generator(np.random.PCG64(37)).standard_normal((3, 60_000)).astype(np.float32)
    gp_ref, gf_ref = oracle.interp_backward(cref, pos, w.astype(np.float64))
    x = torch.from_numpy(pos).to(DEV).requires_grad_()
    f = torch.from_numpy(field).to(DEV).requires_grad_()
    u = ps.interp_autograd(x, f)
    ref = oracle.interp(cref, pos)
    assert np.abs(u.detach().cpu().numpy() - ref).max() <= 1e-5 * np.sqrt((ref ** 2).mean())
    gp, gf = torch.autograd.grad(u, (x, f), torch.from_numpy(w).to(DEV))
    for d in range(3):
        tol = 1e-5 * 3 * (n[d] / TWO_PI) * np.abs(cref).max() * np.abs(w).sum(0).max()
        assert np.abs(gp[d].cpu().numpy() - gp_ref[d]).max() <= tol
    assert np.abs(gf.cpu().numpy() - gf_ref).max() <= 1e-5 * np.abs(gf_ref).max() + 1e-6


@pytest.mark.parametrize("n", [(100, 60, 300), (192, 64, 101), (250, 200, 100), (255, 200, 90),
                               (300, 64, 50), (320, 49, 75), (384, 64, 50), (510, 64, 50),
                               (640, 33, 50), (767, 50, 50), (768, 33, 50)])
def test_streamed_solve_of_any_row(n):
    # grids that take two passes, with rows that fill a warp's chunks, leave its
    # last lanes empty or a lane's chunk cut short, copied in pieces of 4, 2 and
    # 1 values; nodes and planar rows hold the same bits, the transposed solve
    # (in place) the same values
    field = synth.random_field(n, ncomp=3, seed=45).astype(np.float32)
    f = torch.from_numpy(field).to(DEV)
    ref = oracle.spline_coeffs(field.astype(np.float64))
    tol = 2e-6 * np.abs(field).max()
    p4 = ps.SplineField.from_field(f, ps.F32X4)
    p32 = ps.SplineField.from_field(f, torch.float32)
    assert np.abs(p32.padded().cpu().numpy() - ref).max() <= tol
    assert torch.equal(p4.padded(), p32.padded())
    assert torch.count_nonzero(p32.coef[..., n[0] + 3:]) == 0
    # an offset start: the field is 4-byte aligned only
    g = torch.empty(f.numel() + 1, device=DEV)[1:].view_as(f).copy_(f)
    q32 = ps.SplineField.from_field(g, torch.float32)
    assert torch.equal(q32.padded(), p32.padded())
    # the transposed solve, after a scatter
    pos = synth.uniform_particles(3000, seed=46)
    w = np.random.Generator(np.random.PCG64(47)).standard_normal((3, 3000)).astype(np.float32)
    _, gf_ref = oracle.interp_backward(ref, pos, w.astype(np.float64))
    gf = torch.empty((3,) + tuple(reversed(n)), device=DEV)
    ps.ps_interp_backward(p32.coef, n, torch.from_numpy(pos).to(DEV), torch.from_numpy(w).to(DEV),
                          None, gf)
    assert np.abs(gf.cpu().numpy() - gf_ref).max() <= 1e-5 * np.abs(gf_ref).max() + 1e-6


@pytest.mark.parametrize("n", [(4, 4, 4), (16, 16, 15), (16, 16, 16), (17, 16, 16)])
def test_offsets_of_few_and_many_bins(n):
    # one-cell bins: 64, 3840 and 4096 are scanned by one block, 4352 in three phases
    pos = synth.uniform_particles(30_000, seed=41)
    bins = ps.bin_particles(n, 1, torch.from_numpy(pos).to(DEV))
    np.testing.assert_array_equal(bins.offsets.cpu().numpy(),
                                  oracle.bin_particles(n, (1, 1, 1), pos)[1])


@pytest.mark.parametrize("n", [(8, 8, 8), (24, 16, 9), (64, 64, 128), (64, 72, 128)])
@pytest.mark.parametrize("np_", [(1 << 17) - 1, 1 << 17, 135_001])
def test_sort_of_many_particles_into_few_bins(n, np_):
    # counted in shared memory from 2^17 particles on in up to 1024 bins (1152: not)
    pos = synth.uniform_particles(np_, seed=43) * 1.4 - 0.8
    pos[:, np_ - 1] = 0.0  # where the bin of a position that is not finite is, too
    pg = torch.from_numpy(pos).to(DEV)
    pg[1, np_ - 1] = math.nan
    st = torch.zeros(4, dtype=torch.int32, device=DEV)
    bins = ps.bin_particles(n, 8, pg, status=st)
    assert ps.ps_status_read(st) == [ps._abi.PS_DEV_NONFINITE_POS, np_ - 1, 0, 1]
    ref_bin, ref_off, _ = oracle.bin_particles(n, (8, 8, 8), pos)
    np.testing.assert_array_equal(bins.bin_of.cpu().numpy(), ref_bin)
    np.testing.assert_array_equal(bins.offsets.cpu().numpy(), ref_off)
    perm = bins.perm.cpu().numpy()
    np.testing.assert_array_equal(np.sort(perm), np.arange(np_))
    np.testing.assert_array_equal(ref_bin[perm], np.sort(ref_bin))


@pytest.mark.parametrize("dtype", [torch.float32, ps.F32X4, ps.F16X4])
@pytest.mark.parametrize("brick", [(8, 8, 8), (16, 16, 8)])
def test_batch_launch_per_step_equals_one_launch(dtype, brick):
    # the default (a launch per phase and step; bricks whose halo needs more than
    # 48 KB too) against all steps in one launch, which a graph of more than 1024
    # steps takes by itself
    sizes, nps = [32, 48, 24], [3000, 9000, 700]
    assert ps.ps_tune_get("batch_persistent") == 0
    flds = [(None, ps.SplineField.from_field(
        torch.from_numpy(synth.random_field((e,) * 3, ncomp=3, seed=50 + e).astype(np.float32))
        .to(DEV), dtype)) for e in sizes]
    pos0 = torch.from_numpy(synth.uniform_particles(sum(nps), seed=51)).to(DEV)
    for nsteps, forms in ((3, ((0, False), (0, True), (1, False))), (1025, ((0, True), (1, True)))):
        out = []
        for persistent, use_graph in forms:
            ps.ps_tune_set("batch_persistent", persistent)
            try:
                plan = ps.BatchPlan([(e,) * 3 for e in sizes], nps, coef_dtype=dtype, brick=brick)
                pos, ids = pos0.clone(), torch.arange(sum(nps), device=DEV)
                st = torch.zeros(4, dtype=torch.int32, device=DEV)
                plan.run(flds, pos, nsteps, 1e-4, solve=False, ids=ids, use_graph=use_graph,
                         status=st)
                assert ps.ps_status_read(st)[0] == 0
            finally:
                ps.ps_tune_set("batch_persistent", 0)
            out.append(torch.empty_like(pos).index_copy_(1, ids, pos))
        assert all(torch.equal(o, out[0]) for o in out[1:])


def test_one_launch_barrier_wait_gives_up():
    # as wait_probe does in the staged bricks: after the first grid barrier every
    # block waits on a word that nothing sets, gives up and leaves
    sf = ps.SplineField.from_field(torch.randn((3, 24, 24, 24), device=DEV))
    pos = torch.from_numpy(synth.uniform_particles(5000, seed=53)).to(DEV)
    plan = ps.BatchPlan([(24, 24, 24)], [5000])
    st = torch.zeros(4, dtype=torch.int32, device=DEV)
    ps.ps_tune_set("batch_persistent", 1)
    ps.ps_tune_set("wait_probe", 20000)
    try:
        plan.run([(None, sf)], pos, 3, 1e-3, solve=False, use_graph=False, status=st)
        assert ps.ps_status_read(st)[0] == ps._abi.PS_DEV_TIMEOUT
    finally:
        ps.ps_tune_set("wait_probe", 0)
        ps.ps_tune_set("batch_persistent", 0)


@pytest.mark.parametrize("rows", [3, 6, 12, 18])
def test_rows_that_no_slot_names_are_left_alone(rows):
    # slots beyond the last offset, and particles whose slot names another one:
    # by way of bin order too, their rows keep what they held
    n, brick, np_ = (24, 16, 16), (8, 8, 8), 3000
    sf = ps.SplineField.from_field(torch.from_numpy(
        synth.random_field(n, ncomp=3, seed=61).astype(np.float32)).to(DEV))
    pg = torch.from_numpy(synth.uniform_particles(np_, seed=62)).to(DEV)
    bins = ps.bin_particles(n, brick, pg)
    offsets = bins.offsets.clone()
    offsets[-3:] = offsets[-4]  # the last bricks' particles are in no bin
    perm = bins.perm.clone()
    perm[100:200] = perm[:100].clone()
    covered = perm[:int(offsets[-1])]
    left = torch.ones(np_, dtype=torch.bool, device=DEV).index_fill_(0, covered, False)
    assert left.sum() > 150
    outs = []
    for ws in (None, ps.workspace(ps._lib().ps_unsort_workspace_size(np_, rows))):
        if ws is not None:
            ws.fill_(0x55)
        o = torch.full((rows, np_), 7.0, device=DEV)
        kw = dict(perm=perm, bin_offsets=offsets, brick=brick, ws=ws)
        if rows == 3:
            ps.ps_interp(sf.coef, n, pg, o, **kw)
        elif rows == 6:
            ps.ps_lagrangian_accel(sf.coef, n, pg, o[3:], vel=o[:3], **kw)
        elif rows == 12:
            ps.ps_interp(sf.coef, n, pg, o[:3], grad=o[3:], **kw)
        else:
            ps.ps_interp_hessian(sf.coef, n, pg, o, **kw)
        assert torch.all(o[:, left] == 7.0)
        outs.append(o)
    assert torch.equal(*outs)


def test_scratch_only_for_rows_that_can_use_it(monkeypatch):
    # one component, FP64 coefficients and the thread-per-particle kernel store
    # each value at its own place
    n, np_ = (24, 16, 16), 2000
    pg = torch.from_numpy(synth.uniform_particles(np_, seed=63)).to(DEV)
    bins = ps.bin_particles(n, 8, pg)
    f = torch.from_numpy(synth.random_field(n, ncomp=3, seed=64).astype(np.float32)).to(DEV)
    three = ps.SplineField.from_field(f)
    asked = []
    real = ps.workspace
    monkeypatch.setattr(ps, "_unsort_pays", lambda *a: True)
    monkeypatch.setattr(ps, "workspace", lambda *a: asked.append(a) or real(*a))
    others = [ps.SplineField.from_field(f[:1].contiguous()),
              ps.SplineField.from_field(f, torch.float64)]
    del asked[:]
    for sf in others:
        sf.interp(pg, grad=True, bins=bins)
        sf.hessian(pg, bins=bins)
    ps.ps_tune_set("brick_kernel", 2)
    try:
        three.interp(pg, grad=True, bins=bins)
    finally:
        ps.ps_tune_set("brick_kernel", -1)
    assert not asked
    three.hessian(pg, bins=bins)
    assert len(asked) == 1


@pytest.mark.parametrize("handle", [False, True])
def test_scratch_belongs_to_the_stream_of_the_call(handle, monkeypatch):
    # freed when the call returns, it must come back to that stream only
    n, np_ = (65, 40, 33), 2000
    f = torch.from_numpy(synth.random_field(n, ncomp=3, seed=65).astype(np.float32)).to(DEV)
    pg = torch.from_numpy(synth.uniform_particles(np_, seed=66)).to(DEV)
    monkeypatch.setattr(ps, "_unsort_pays", lambda *a: True)
    ref = ps.SplineField.from_field(f)
    bins = ps.bin_particles(n, 8, pg)
    grad_ref = ref.interp(pg, grad=True, bins=bins)[1]
    seen = []
    real = ps.workspace
    monkeypatch.setattr(ps, "workspace", lambda *a: (
        seen.append(torch.cuda.current_stream().cuda_stream), real(*a))[1])
    side = torch.cuda.Stream()
    for s in (side, torch.cuda.default_stream()):
        del seen[:]
        torch.cuda.synchronize()
        arg = s.cuda_stream if handle else s
        sf = ps.SplineField.from_field(f, stream=arg)
        bins = ps.bin_particles(n, 8, pg, stream=arg)
        grad = sf.interp(pg, grad=True, bins=bins, stream=arg)[1]
        sf.hessian(pg, bins=bins, stream=arg)
        sf.acceleration(pg, bins=bins, stream=arg)
        torch.cuda.synchronize()
        assert len(seen) == 5 and set(seen) == {s.cuda_stream}
        assert torch.equal(grad, grad_ref)


def test_planar_solve_without_memory_for_its_scratch(monkeypatch):
    # planar FP32 coefficients need none: they are solved in place; nodes do
    n = (65, 40, 33)
    field = synth.random_field(n, ncomp=3, seed=67).astype(np.float32)
    f = torch.from_numpy(field).to(DEV)

    def no_memory(*a):
        raise torch.cuda.OutOfMemoryError("none left")

    monkeypatch.setattr(ps, "workspace", no_memory)
    sf = ps.SplineField.from_field(f)
    ref = oracle.spline_coeffs(field.astype(np.float64))
    assert np.abs(sf.padded().cpu().numpy() - ref).max() <= 2e-6 * np.abs(field).max()
    with pytest.raises(torch.cuda.OutOfMemoryError):
        ps.SplineField.from_field(f, ps.F32X4)


@pytest.mark.parametrize("dtype", [ps.F32X4, torch.float32, torch.bfloat16, ps.BF16X4])
@pytest.mark.parametrize("brick", [(8, 8, 8), (16, 16, 16), (20, 16, 12)])
def test_acceleration_from_two_fields_in_large_bricks(dtype, brick):
    # bricks whose two halos do not fit into shared memory side by side: the later
    # field's nodes come from global memory, at each particle's own cell
    n, np_ = (48, 40, 33), 6000
    fields = [synth.random_field(n, ncomp=3, seed=s).astype(np.float32) for s in (70, 71)]
    a, b = (ps.SplineField.from_field(torch.from_numpy(f).to(DEV), dtype) for f in fields)
    pos = synth.uniform_particles(np_, seed=72)
    pg = torch.from_numpy(pos).to(DEV)
    got = a.acceleration(pg, later=b, dt_field=0.1, bins=ps.bin_particles(n, brick, pg))
    ref = a.acceleration(pg, later=b, dt_field=0.1)  # the unbinned kernel
    # both evaluate the same coefficients: velocities 1e-5 of their rms, gradients
    # 3e-5 max|c| n/L, as above (each side once)
    u, grad = a.interp(pg, grad=True)
    cmax = 3 * max(np.abs(f).max() for f in fields)
    tol = 2 * (3 * float(grad.abs().max()) * 1e-5 * cmax +
               3 * float(u.abs().max()) * 3e-5 * cmax * max(n) / TWO_PI + 2 * 1e-5 * cmax / 0.1)
    assert float((got - ref).abs().max()) <= tol
    assert float((b.interp(pg) - u).abs().max()) / 0.1 > 100 * tol  # the later field counts


@pytest.mark.parametrize("dtype", [ps.F32X4, torch.float32, ps.F16X4, torch.bfloat16])
def test_acceleration_from_one_field(dtype):
    # the convective part alone, bricks staged and not, a ragged last brick; bars as
    # above: velocities 1e-5 of their rms, gradients 3e-5 max|c| n/L, 16-bit values
    # compared with the unbinned kernel of the same coefficients
    n, brick, np_ = (40, 24, 17), (8, 8, 8), 1500
    field = synth.random_field(n, ncomp=3, seed=68).astype(np.float32)
    sf = ps.SplineField.from_field(torch.from_numpy(field).to(DEV), dtype)
    pos = synth.uniform_particles(np_, seed=69)
    pg = torch.from_numpy(pos).to(DEV)
    bins = ps.bin_particles(n, brick, pg)
    got = sf.acceleration(pg, bins=bins)
    vel, grad = (t.cpu().numpy().astype(np.float64) for t in sf.interp(pg, grad=True))
    if dtype in (ps.F32X4, torch.float32):
        vel, grad = oracle.interp(oracle.spline_coeffs(field.astype(np.float64)), pos, grad=True)
    ref = (grad * vel[None]).sum(1)
    gtol = 3e-5 * np.abs(field).max() * 3 * max(n) / TWO_PI
    tol = 3 * (np.abs(grad).max() * 1e-5 * np.sqrt((vel ** 2).mean()) + np.abs(vel).max() * gtol)
    assert np.abs(got.cpu().numpy() - ref).max() <= tol
    # the time derivative of a field that does not change adds nothing
    assert torch.equal(sf.acceleration(pg, later=sf, dt_field=0.5, bins=bins), got)


def _staged_and_not(n, brick, per, dtype, seed):
    """Every brick call's results with halos staged as the dispatch has it, and with
    every stencil from global memory."""
    nbins = math.prod(-(-n[d] // brick[d]) for d in range(3))
    pos = torch.from_numpy(synth.uniform_particles(per * nbins, seed=seed)).to(DEV)
    a, b = (ps.SplineField.from_field(torch.from_numpy(
        synth.random_field(n, ncomp=3, seed=seed + i).astype(np.float32)).to(DEV), dtype)
        for i in (1, 2))
    bins, xs = ps.bin_particles(n, brick, pos, want_sorted=True)
    bins.perm = None
    dt = 0.4 * TWO_PI / max(n)
    out = []
    try:
        for least in (8, 1 << 20):
            ps.ps_tune_set("brick_min_stage", least)
            st = torch.zeros(4, dtype=torch.int32, device=DEV)
            r = [*a.interp(xs, grad=True, bins=bins, status=st), a.interp(xs, bins=bins),
                 a.hessian(xs, bins=bins), a.acceleration(xs, bins=bins),
                 a.acceleration(xs, later=b, dt_field=0.1, bins=bins)]
            for later in (None, b):
                x, v = xs.clone(), torch.empty((3, xs.shape[1]), device=DEV)
                ps.ps_rk2_step(a.coef, n, x, dt, coef_np1=later.coef if later else None,
                               scale_n=a.scale, scale_np1=later.scale if later else None,
                               vel_out=v, brick=brick, rebin=0, bin_offsets=bins.offsets,
                               status=st)
                r += [x, v]
            assert ps.ps_status_read(st)[0] == 0
            out.append(r)
    finally:
        ps.ps_tune_set("brick_min_stage", 8)
    return out


@pytest.mark.parametrize("dtype", [ps.F32X4, torch.float32, ps.BF16X4, torch.float16])
@pytest.mark.parametrize("per", [9, 13, 15, 21, 63, 65, 130])
def test_halos_staged_or_not(per, dtype):
    # around the densities from which a second field's halo is staged
    staged, plain = _staged_and_not((32, 24, 16), (8, 8, 8), per, dtype, 80)
    assert all(torch.equal(s, p) for s, p in zip(staged, plain))


@pytest.mark.parametrize("dtype", [ps.F32X4, torch.float32, ps.F16X4, torch.float16])
@pytest.mark.parametrize("brick", [(8, 5, 8), (8, 1, 4), (4, 9, 4), (12, 5, 3), (7, 13, 2)])
def test_halo_planes_with_further_rows(brick, dtype):
    # halos of a multiple of 4 rows per plane lie with rows that no stencil uses
    staged, plain = _staged_and_not((24, 26, 16), brick, 40, dtype, 90)
    assert all(torch.equal(s, p) for s, p in zip(staged, plain))


@pytest.mark.parametrize("dtype", [ps.F32X4, torch.float32, torch.float16])
@pytest.mark.parametrize("brick,per", [((8, 1, 8), 4), ((8, 5, 8), 20), ((8, 5, 8), 60)])
def test_sparse_bricks_of_unfavourable_height(brick, per, dtype):
    # with few particles second derivatives and accelerations take the unbinned
    # kernels, with more the staged ones: both within the bars of the FP32 sums
    n = (24, 25, 16)
    np_ = per * math.prod(-(-n[d] // brick[d]) for d in range(3))
    sf = ps.SplineField.from_field(torch.from_numpy(
        synth.random_field(n, ncomp=3, seed=95).astype(np.float32)).to(DEV), dtype)
    pg = torch.from_numpy(synth.uniform_particles(np_, seed=96)).to(DEV)
    bins = ps.bin_particles(n, brick, pg)
    for call, unit in ((sf.hessian, 6 * (max(n) / TWO_PI) ** 2),
                       (sf.acceleration, 9 * max(n) / TWO_PI)):
        got, ref = call(pg, bins=bins), call(pg)
        assert torch.equal(got, ref) == (per < 30)
        cmax = float(sf.padded().abs().max())
        scale = cmax if call == sf.hessian else cmax ** 2
        assert float((got - ref).abs().max()) <= 1e-5 * 8 * unit * scale
    with pytest.raises(RuntimeError):  # a brick that the staged form refuses
        sf.hessian(pg, bins=ps.Bins((30, 5, 8), bins.offsets, None, bins.perm))


@pytest.mark.parametrize("per", [30, 110])
def test_planar_16_bit_halos_in_ragged_boxes(per):
    # below and above the density from which both fields' halos are staged there
    staged, plain = _staged_and_not((30, 21, 17), (8, 8, 8), per, torch.bfloat16, 100)
    assert all(torch.equal(s, p) for s, p in zip(staged, plain))


def test_differentiable_call_bins_what_its_gradients_need(monkeypatch):
    # the tensors kept for the backward pass are saved tensors: hooks see them and they
    # are freed with the graph
    n, np_ = (32, 24, 16), 60_000
    f = torch.from_numpy(synth.random_field(n, ncomp=3, seed=97).astype(np.float32)).to(DEV)
    x = torch.from_numpy(synth.uniform_particles(np_, seed=98)).to(DEV)
    monkeypatch.setattr(ps, "_FN_MIN_IN_L2", 0)
    sorts = []
    real = ps.bin_particles
    monkeypatch.setattr(ps, "bin_particles", lambda *a, **k: sorts.append(a) or real(*a, **k))
    saved = []

    def pack(t):
        saved.append(t)
        return t

    xr, fr = x.clone().requires_grad_(), f.clone().requires_grad_()
    with torch.autograd.graph.saved_tensors_hooks(pack, lambda t: t):
        u = ps.interp_autograd(xr, fr)
    assert len(sorts) == 1 and len(saved) == 4  # pos; permutation, offsets, sorted positions
    assert {t.dtype for t in saved} == {torch.float64, torch.int64, torch.int32}
    torch.autograd.grad(u, (xr, fr), torch.ones_like(u))
    with pytest.raises(RuntimeError):  # freed
        torch.autograd.grad(u, (xr, fr), torch.ones_like(u))
    # what is asked of the limits: the gradients that the call will need
    asked = []
    monkeypatch.setattr(ps, "_fn_binned", lambda n, m, *want: asked.append(want) or False)
    for a, b, want in ((x, f, (False, False)), (xr, f, (True, False)), (x, fr, (False, True)),
                       (xr, fr, (True, True))):
        v = ps.interp_autograd(a, b)
        assert asked.pop() == want and v.requires_grad == any(want)
        assert float((v - u).detach().abs().max()) <= 2e-5 * float(u.detach().abs().max())
        with torch.no_grad():
            v = ps.interp_autograd(a, b)
        assert asked.pop() == (False, False) and not v.requires_grad
    assert len(sorts) == 1


@pytest.mark.parametrize("n", [(168, 33, 200), (236, 100, 150), (226, 200, 150), (225, 200, 150),
                               (484, 150, 50), (612, 50, 50), (518, 100, 50), (519, 100, 50),
                               (528, 33, 50), (88, 49, 393)])
def test_streamed_solve_of_larger_boxes(n):
    # two passes by the rule for whole chunks, chunks cut short, and odd rows
    test_streamed_solve_of_any_row(n)


@pytest.mark.parametrize("dtype", [ps.F32X4, torch.float32])
def test_bricks_scale_as_the_unbinned_kernels(dtype):
    # the constant factor of the sums, from a fit against 64 bits of the same
    # coefficients (rounding noise 1e-7 / sqrt(600,000) = 2e-10): that of 1/6 rounded to
    # FP32 on each axis, 8.94e-8, in bricks and out of them
    n, np_ = (32, 24, 40), 200_000
    field = synth.random_field(n, ncomp=3, seed=110).astype(np.float32)
    f = torch.from_numpy(field).to(DEV)
    sf = ps.SplineField.from_field(f, dtype)
    pos = synth.uniform_particles(np_, seed=111)
    pg = torch.from_numpy(pos).to(DEV)
    bins = ps.bin_particles(n, 8, pg)
    ref = torch.from_numpy(oracle.interp(sf.padded().cpu().numpy().astype(np.float64), pos)).to(DEV)

    def factor(a, b):
        return float((a.double() * b).sum() / (b * b).sum() - 1)

    direct, binned = factor(sf.interp(pg), ref), factor(sf.interp(pg, bins=bins), ref)
    assert abs(direct - 8.94e-8) <= 5e-9 and abs(binned - 8.94e-8) <= 5e-9


def test_slots_next_to_2_31():
    # the last particles of the largest set: the trip after them begins beyond 2^31
    np_, m, n = 2**31 - 1, 77, (16, 16, 16)
    if torch.cuda.mem_get_info()[0] < 100e9:
        pytest.skip("needs 100 GB")
    f = torch.from_numpy(synth.random_field(n, ncomp=3, seed=120).astype(np.float32)).to(DEV)
    last = (torch.from_numpy(synth.uniform_particles(m, seed=121)).to(DEV) + TWO_PI) / 2
    pos = torch.empty((3, np_), dtype=torch.float64, device=DEV)
    pos[:, np_ - m:] = last
    offsets = torch.full((9,), np_ - m, dtype=torch.int32, device=DEV)
    offsets[8] = np_  # all in the last brick
    small = torch.zeros(9, dtype=torch.int32, device=DEV)
    small[8] = m
    buf = torch.empty((3, np_), dtype=torch.float32, device=DEV)
    for field, dtype, kernel in ((f, torch.float32, -1), (f, ps.F16X4, -1), (f, torch.float32, 2),
                                 (f[:1].contiguous(), torch.float32, -1)):
        sf = ps.SplineField.from_field(field, dtype)
        ref = torch.empty((sf.ncomp, m), device=DEV)
        ps.ps_tune_set("brick_kernel", kernel)
        try:
            ps.ps_interp(sf.coef, n, last, ref, scale=sf.scale, bin_offsets=small, brick=8)
            ps.ps_interp(sf.coef, n, pos, buf[:sf.ncomp], scale=sf.scale, bin_offsets=offsets,
                         brick=8)
        finally:
            ps.ps_tune_set("brick_kernel", -1)
        assert torch.equal(buf[:sf.ncomp, np_ - m:], ref)
    sf = ps.SplineField.from_field(f)
    out = []
    for p, o, w in ((last, small, ref := torch.randn((3, m), device=DEV)), (pos, offsets, buf)):
        buf[:, np_ - m:] = ref
        g = torch.empty_like(f)
        ps.ps_interp_backward(sf.coef, n, p, w, None, g, bin_offsets=o, brick=8,
                              ws=ps.workspace(ps.ps_backward_workspace_size(n, 8)))
        out.append(g)
    assert torch.equal(*out)
    del pos, buf, w
    torch.cuda.empty_cache()


@pytest.mark.parametrize("brick,per", [((8, 5, 8), 20), ((8, 5, 8), 24), ((4, 4, 4), 11),
                                       ((4, 4, 4), 14), ((20, 3, 3), 17), ((20, 3, 3), 20)])
def test_planar_16_bit_halos_from_a_particle_per_four_rows(brick, per):
    staged, plain = _staged_and_not((26, 22, 18), brick, per, torch.float16, 130)
    assert all(torch.equal(s, p) for s, p in zip(staged, plain))


@pytest.mark.parametrize("dtype", [ps.F32X4, torch.float32, torch.bfloat16, ps.F16X4])
@pytest.mark.parametrize("n,brick", [((32, 40, 34), (16, 16, 32)), ((32, 20, 34), (29, 17, 17))])
def test_largest_halos(n, brick, dtype):
    # nearly all of the shared memory: staged without padding where that alone fits
    staged, plain = _staged_and_not(n, brick, 300, dtype, 140)
    assert all(torch.equal(s, p) for s, p in zip(staged, plain))
