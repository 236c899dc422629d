"""Sizes at which the tiles, strips and chunks of the kernels end: one row or column past a tile, fewer
rows than CTAs, frames narrower than a warp, series of a few frames, against the oracle.

Bounds as for the same steps at ordinary sizes: levels and registered frames a few FP32 roundings of
values of order 1, energies 1e-6 relative, gradients 2e-4 of their largest entry.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2010_12478_gb300 import binding as B
from paper_2010_12478_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2010_12478_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"


@pytest.mark.parametrize("shape", [(8, 512), (9, 513), (7, 511), (17, 1025), (3, 3), (600, 31)])
@pytest.mark.parametrize("storage", ["f32", "bf16", "f16"])
def test_pyramid_levels_at_tile_edges(shape, storage):
    H, W = shape
    img = np.random.default_rng(2).uniform(0, 1, size=(H, W)).astype(np.float32)
    h2, w2 = (H + 1) // 2, (W + 1) // 2
    dt = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}[storage]
    out = torch.full((H * W + h2 * w2,), -7.0, dtype=dt, device="cuda")
    B.Context(B.Config()).pyramid(torch.from_numpy(img).cuda(), 2, storage, out)
    got = out.float().cpu().numpy().astype(np.float64)
    l0, l1 = got[:H * W].reshape(H, W), got[H * W:].reshape(h2, w2)
    assert np.array_equal(l0, torch.from_numpy(img).to(dt).double().numpy())
    tol = {"f32": 3e-7, "bf16": 8e-3, "f16": 1e-3}[storage]
    np.testing.assert_allclose(l1, O.downsample(l0), rtol=tol, atol=tol)


@pytest.mark.parametrize("shape", [(17, 33), (65, 513), (240, 37), (3, 129), (129, 3)])
@pytest.mark.parametrize("far", [0.0, 40.0])
def test_energy_and_gradient_at_strip_edges(shape, far):
    # far: every sample beyond the template's border on one side of the frame, so the mean that stands
    # there (the border of a level, its model at the pixel centres) carries the energy
    H, W = shape
    rng = np.random.default_rng(11)
    R, T = (rng.uniform(0, 1, size=(H, W)).astype(np.float32) for _ in range(2))
    g = O.grid_for(W, H)
    c = rng.uniform(-0.5, 0.5, size=(2, g.ny, g.nx))
    c[0] += far * np.linspace(0.0, 1.0, g.nx)[None, :]
    cd = torch.from_numpy(np.ascontiguousarray(c.transpose(1, 2, 0)).astype(np.float32)).cuda()
    gd = torch.zeros((g.ny, g.nx, 2), device="cuda")
    dR, dT = torch.from_numpy(R).cuda(), torch.from_numpy(T).cuda()
    E = B.Context(B.Config(mode="nonrigid")).energy_grid(dR, dT, cd, gd)
    Eo, go = O.grid_energy(R, T, 0, g, cd.cpu().numpy().transpose(2, 0, 1).astype(np.float64), 2.0)
    assert abs(E - Eo) <= 1e-6 * abs(Eo)
    np.testing.assert_allclose(gd.cpu().numpy().transpose(2, 0, 1), go, atol=2e-4 * np.abs(go).max())
    th = [0.01, 0.3 + 0.2 * far, -0.2]
    E, gr = B.Context(B.Config()).energy_rigid(dR, dT, th)
    Eo, gro = O.rigid_energy(R, T, th)
    assert abs(E - Eo) <= 1e-6 * abs(Eo)
    assert np.abs(gr - gro).max() <= 1e-4 * max(1.0, np.abs(gro).max())


@pytest.mark.parametrize("N", [1, 2, 5, 65, 131])
def test_registered_mean_over_any_number_of_frames(N):
    # the frames of a chunk, and so the number of chunks, follow from the sizes
    F = synth.make_series(synth.SeriesSpec(N, 70, 133, step=2.0, snr=(10.0, 10.0), seed=4)).frames
    rng = np.random.default_rng(N)
    els = [(0, k + 1, *(float(v) for v in rng.uniform(-1, 1, 3) * (0.02, 6.0, 6.0))) for k in range(N - 1)]
    mean = torch.empty((70, 133), device="cuda")
    out = torch.empty((N, 70, 133), device="cuda")
    B.Context(B.Config()).warp(F.cuda(), elems=els, out=out, mean=mean)
    want, wmean = O.register_series(F.numpy().astype(np.float64), "rigid",
                                    [np.array(e[2:], np.float32).astype(np.float64) for e in els])
    assert np.abs(out.cpu().numpy() - want).max() <= 1e-5
    assert np.abs(mean.cpu().numpy() - wmean).max() <= 1e-5


@pytest.mark.parametrize("shape", [(65, 129), (100, 97), (33, 160)])
@pytest.mark.parametrize("grid", [1, 2, 4, 20, 32, 40, 64])
def test_gradient_for_every_kind_of_cell_width(shape, grid):
    # strips of many cells, of one cell, of a part of one; widths that divide a warp and that do not; the
    # column and row past the last cell (129 = 2^7 + 1)
    H, W = shape
    if grid <= 2:
        H, W = 33, 41   # as many points as shared memory holds
    rng = np.random.default_rng(21)
    R, T = (rng.uniform(0, 1, size=(H, W)).astype(np.float32) for _ in range(2))
    g = O.grid_for(W, H, grid)
    c = rng.uniform(-0.9, 0.9, size=(g.ny, g.nx, 2)).astype(np.float32)
    gd = torch.zeros((g.ny, g.nx, 2), device="cuda")
    E = B.Context(B.Config(mode="nonrigid", grid=grid)).energy_grid(
        torch.from_numpy(R).cuda(), torch.from_numpy(T).cuda(), torch.from_numpy(c).cuda(), gd)
    Eo, go = O.grid_energy(R, T, 0, g, c.transpose(2, 0, 1).astype(np.float64), 2.0)
    assert abs(E - Eo) <= 1e-6 * abs(Eo)
    np.testing.assert_allclose(gd.cpu().numpy().transpose(2, 0, 1), go, atol=2e-4 * np.abs(go).max())


@pytest.mark.parametrize("shape,grid", [((64, 60000), 64), ((65, 60001), 96)])
def test_gradient_of_thousands_of_strips(shape, grid):
    # more 32-column strips than shared memory has slots for: a warp walks a cell's chunks (two of them; three,
    # with a column past the last cell), and there is a single band of cell rows
    H, W = shape
    rng = np.random.default_rng(22)
    R, T = (rng.uniform(0, 1, size=(H, W)).astype(np.float32) for _ in range(2))
    g = O.grid_for(W, H, grid)
    c = rng.uniform(-0.9, 0.9, size=(g.ny, g.nx, 2)).astype(np.float32)
    gd = torch.zeros((g.ny, g.nx, 2), device="cuda")
    E = B.Context(B.Config(mode="nonrigid", grid=grid)).energy_grid(
        torch.from_numpy(R).cuda(), torch.from_numpy(T).cuda(), torch.from_numpy(c).cuda(), gd)
    Eo, go = O.grid_energy(R, T, 0, g, c.transpose(2, 0, 1).astype(np.float64), 2.0)
    assert abs(E - Eo) <= 1e-6 * abs(Eo)
    np.testing.assert_allclose(gd.cpu().numpy().transpose(2, 0, 1), go, atol=2e-4 * np.abs(go).max())


@pytest.mark.parametrize("cluster", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("levels,grid,metric", [(1, 16, 1), (3, 16, 1), (2, 24, 0), (2, 16, 2)])
def test_pair_for_every_band_split(cluster, levels, grid, metric):
    # bands of many, one and no cell rows per CTA, cell widths down to 4, each scalar product: three steps
    # per level take both sides through the same trials, so only rounding separates their end points
    # (a gradient off by 1e-6 of itself, steps of at most half a pixel: far below 1e-3 px)
    spec = synth.SeriesSpec(2, 107, 140, step=1.0, field_amp=1.0, snr=(10.0, 10.0), seed=8)
    F = synth.make_series(spec).frames
    cfg = B.Config(mode="nonrigid", cluster=cluster, levels=levels, grid=grid, metric=metric, max_iter=3)
    out = torch.empty((2, 107, 140), device="cuda")
    _, st = B.Context(cfg).pairwise(F[0].cuda(), F[1].cuda(), field_out=out)
    oc = O.Config(levels=levels, max_iter=3, max_rejects=cfg.max_rejects, tol_grad=cfg.tol_grad,
                  tol_rel_e=cfg.tol_rel_e, armijo_c=cfg.armijo_c, tau0=cfg.tau0, step_cap=cfg.step_cap, lam=cfg.lam,
                  mode="nonrigid", grid=grid, metric=metric, sigma=cfg.sigma, tol_coarse=cfg.tol_coarse)
    F = F.numpy()
    c_o, st_o = O.register_nonrigid(O.pyramid(F[0], levels), O.pyramid(F[1], levels), None, oc)
    assert O.max_px_error(out.cpu().numpy(), c_o, 107, 140, "nonrigid", grid) <= 1e-3
    assert st["iters"] == list(st_o.iters) and st["evals"] == list(st_o.evals)
    assert abs(st["energy"] - st_o.energy) <= 1e-6 * abs(st_o.energy)


def test_a_grid_too_large_for_one_cta_takes_more():
    # 65 x 65 points: one CTA cannot hold the control state and its slots; the results are those of a
    # cluster that can
    F = synth.make_series(synth.SeriesSpec(2, 513, 513, step=1.0, field_amp=1.0, snr=(10.0, 10.0), seed=9),
                          device="cuda").frames
    outs = []
    for cluster in (1, 16):
        ctx = B.Context(B.Config(mode="nonrigid", grid=8, cluster=cluster, max_iter=2))
        outs.append(torch.empty((2, 513, 513), device="cuda"))
        ctx.pairwise(F[0], F[1], field_out=outs[-1])
        assert ctx.last_timing()["cluster"] >= cluster
    assert float((outs[0] - outs[1]).abs().max()) <= 1e-4


@pytest.mark.parametrize("mode", ["rigid", "nonrigid"])
def test_pair_takes_frames_and_fields_from_anywhere(mode):
    # device frames and fields are used where they are, anything else is staged: the same result, bit for bit
    F = synth.make_series(synth.SeriesSpec(2, 90, 101, step=1.5, field_amp=1.0, snr=(10.0, 10.0), seed=3)).frames
    ctx = B.Context(B.Config(mode=mode))
    dev = F.cuda()
    rev = torch.stack([F[1], F[0]]).cuda()   # the template in front of the reference
    init = torch.full((2, 90, 101), 0.25)
    runs = []
    for R, T in ((dev[0], dev[1]), (F[0], F[1]), (F[0].pin_memory(), dev[1]), (rev[1], rev[0])):
        if mode == "rigid":
            runs.append(torch.tensor(ctx.pairwise(R, T, init=(0.001, 0.25, 0.25))[1]["theta"], dtype=torch.float64))
            continue
        for where in ("cuda", "cpu"):
            out = torch.empty((2, 90, 101), device=where)
            ctx.pairwise(R, T, field_in=init.to(where), field_out=out)
            same = init.to(where).clone()   # the result over the initial guess
            ctx.pairwise(R, T, field_in=same, field_out=same)
            runs += [out.cpu(), same.cpu()]
    assert all(torch.equal(r, runs[0]) for r in runs)
    if mode == "nonrigid":
        g = O.grid_for(101, 90)
        c = torch.zeros((g.ny, g.nx, 2), device="cuda") + 0.3
        E = [B.Context(B.Config(mode=mode)).energy_grid(R, T, c) for R, T in ((dev[0], dev[1]), (F[0], dev[1]), (rev[1], rev[0]))]
        assert E[0] == E[1] == E[2]


@pytest.mark.parametrize("mode", ["rigid", "nonrigid"])
def test_level_means_of_levels_with_fewer_rows_than_ctas(mode):
    # most CTAs that sum a level's mean have no row of it and reach the exchange at once: many frames side by
    # side, the coarsest level 2 x 2 pixels.  A frame's means, and with them a pair's result, do not depend on
    # the launch they are in: identical frames give identical operators, at the energy of a pair on its own
    pair = synth.make_series(synth.SeriesSpec(2, 8, 7, step=0.5, snr=(10.0, 10.0), seed=5)).frames
    F = torch.cat([pair] * 256).contiguous().cuda()
    cfg = B.Config(mode=mode, levels=3, max_iter=3)
    ctx = B.Context(cfg)
    out = torch.empty((2, 8, 7), device="cuda")
    _, one = ctx.pairwise(F[0], F[1], field_out=out if mode == "nonrigid" else None)
    for _ in range(4):
        _, st = ctx.scan(F, exec="level")
        assert {s["energy"] for s in st[:len(F) - 1:2]} == {st[0]["energy"]}
        assert {s["energy"] for s in st[1:len(F) - 1:2]} == {st[1]["energy"]}
    # another cluster size, another order of the sums: the relative energy bar of the parity tests
    assert abs(one["energy"] - st[0]["energy"]) <= 1e-5 * max(abs(one["energy"]), 1e-2)


class _At:
    """Floats at any byte of a device buffer, as a caller's packed record may hold them."""

    def __init__(self, a, off):
        self.shape = a.shape
        raw = a.contiguous().view(torch.uint8).reshape(-1)
        self.buf = torch.zeros(raw.numel() + 16, dtype=torch.uint8, device="cuda")
        self.at = self.buf[off:off + raw.numel()]
        self.at.copy_(raw)

    def data_ptr(self):
        return self.at.data_ptr()

    def is_contiguous(self):
        return True

    def floats(self):
        return self.at.clone().view(torch.float32).reshape(self.shape).cpu()


@pytest.mark.parametrize("off", [1, 2, 6, 4])
def test_frames_and_fields_off_a_floats_alignment_are_staged(off):
    # the kernels load floats: device memory off their alignment goes through the staging copy, as host memory
    # does; frames a fraction of a float apart do too
    F = synth.make_series(synth.SeriesSpec(2, 40, 37, step=1.0, field_amp=0.5, snr=(10.0, 10.0), seed=6)).frames.cuda()
    init = torch.full((2, 40, 37), 0.25, device="cuda")
    for R, T in ((_At(F[0], off), _At(F[1], off)), (F[0], _At(F[1], off)), (_At(F[0], off), F[1])):
        ctx = B.Context(B.Config(mode="rigid"))
        assert ctx.pairwise(R, T)[1] == ctx.pairwise(F[0], F[1])[1]
        assert ctx.energy_rigid(R, T, [0.01, 0.2, 0.1])[0] == ctx.energy_rigid(F[0], F[1], [0.01, 0.2, 0.1])[0]
        ctx = B.Context(B.Config(mode="nonrigid"))
        want, got = torch.empty((2, 40, 37), device="cuda"), _At(torch.zeros((2, 40, 37), device="cuda"), off)
        ctx.pairwise(F[0], F[1], field_in=init, field_out=want)
        ctx.pairwise(R, T, field_in=_At(init, off), field_out=got)
        assert torch.equal(got.floats(), want.cpu())


@pytest.mark.parametrize("grid,past,metric", [(32, 0, 1), (32, 1, 1), (32, 1, 2), (17, 1, 1), (40, 1, 0)])
def test_the_largest_accepted_grid_of_three_rows(grid, past, metric):
    # 892 x 3 control points, the most that reg_grid_dims takes at three rows, with and without a column past the
    # last cell, cells of a strip each and of two chunks: two bands of one cell row in 16 CTAs
    W, H = 891 * grid + past, 2 * grid + past
    assert B.grid_dims(W, H, grid, 1)[:2] == (892, 3)
    rng = np.random.default_rng(31)
    R = rng.uniform(0, 1, size=(H, W)).astype(np.float32)
    T = (0.5 * (R + np.roll(R, 1, axis=1))).astype(np.float32)
    dR, dT = torch.from_numpy(R).cuda(), torch.from_numpy(T).cuda()
    g = O.grid_for(W, H, grid)
    c = rng.uniform(-0.9, 0.9, size=(g.ny, g.nx, 2)).astype(np.float32)
    gd = torch.zeros((g.ny, g.nx, 2), device="cuda")
    E = B.Context(B.Config(mode="nonrigid", levels=1, grid=grid)).energy_grid(dR, dT, torch.from_numpy(c).cuda(), gd)
    Eo, go = O.grid_energy(R, T, 0, g, c.transpose(2, 0, 1).astype(np.float64), 2.0)
    assert abs(E - Eo) <= 1e-6 * abs(Eo)
    np.testing.assert_allclose(gd.cpu().numpy().transpose(2, 0, 1), go, atol=2e-4 * np.abs(go).max())
    # one accepted step from the identity, as in test_pair_for_every_band_split
    cfg = B.Config(mode="nonrigid", levels=1, grid=grid, metric=metric, max_iter=1)
    out = torch.empty((2, H, W), device="cuda")
    _, st = B.Context(cfg).pairwise(dR, dT, field_out=out)
    oc = O.Config(levels=1, max_iter=1, max_rejects=cfg.max_rejects, tol_grad=cfg.tol_grad, tol_rel_e=cfg.tol_rel_e,
                  armijo_c=cfg.armijo_c, tau0=cfg.tau0, step_cap=cfg.step_cap, lam=cfg.lam, mode="nonrigid", grid=grid,
                  metric=metric, sigma=cfg.sigma, tol_coarse=cfg.tol_coarse)
    c_o, st_o = O.register_nonrigid(O.pyramid(R, 1), O.pyramid(T, 1), None, oc)
    assert O.max_px_error(out.cpu().numpy(), c_o, H, W, "nonrigid", grid) <= 1e-3
    assert st["iters"] == list(st_o.iters) and abs(st["energy"] - st_o.energy) <= 1e-6 * abs(st_o.energy)


@pytest.mark.parametrize("cap", [1e-3, 3.7e-4])
def test_a_capped_step_has_the_caps_length_in_64_bits(cap):
    # the step controller works in FP64: a first step that the cap shortens has exactly its length in the flow's
    # metric, a few roundings of 1.1e-16 (a length held in FP32 is off by up to 6e-8)
    F = synth.make_series(synth.SeriesSpec(2, 96, 110, step=1.0, snr=(10.0, 10.0), seed=15)).frames.cuda()
    _, st = B.Context(B.Config(levels=1, max_iter=1, step_cap=cap)).pairwise(F[0], F[1])
    a, x, y = st["theta"]
    assert st["iters"] == [1] and st["rejects"] == 0
    assert abs(np.sqrt((0.25 * (96 + 110) * a) ** 2 + x * x + y * y) / cap - 1.0) <= 1e-13


def _lattice(shift, period=13.3, n=512):
    y, x = np.mgrid[0:n, 0:n].astype(np.float64)
    return 0.5 + 0.2 * np.cos(2 * np.pi * (x + shift) / period) + 0.2 * np.cos(2 * np.pi * (y + 0.5 * shift) / period)


def _ncc_energy(R, T):
    # 1 - NCC of two images pixel by pixel, in extended precision (sums of FP64 products in FP64, as the oracle's,
    # are off by 1e-5 of an energy of 7e-6 at an offset of 25 times the contrast)
    r, t = (v.astype(np.longdouble) - v.astype(np.longdouble).mean() for v in (R, T))
    return float(1 - (r * t).sum() / np.sqrt((r * r).sum() * (t * t).sum()))


@pytest.mark.parametrize("shift", [0.01, 0.1])
@pytest.mark.parametrize("gain,offset", [(1.0, 0.0), (1.3, 0.0), (3.0, 0.0), (0.2, 0.0), (1.0, 5.0), (-1.0, 0.0), (1.3, -5.0)])
def test_small_energies_at_any_gain_and_offset(shift, gain, offset):
    # 1 - NCC does not see gain and offset, and its rounding must not either.  At the identity the rigid model's
    # samples are the pixels, so only the sums round: relative to the energy, as the difference that is summed is as
    # small as the energy (the bar of the energies, 1e-6).  The nonrigid model's samples round to 6e-8 of their own
    # value, 1e-4 of the difference at E = 7e-6, at random over the pixels: a few 1e-6 of the energy
    R = _lattice(0.0).astype(np.float32)
    T = (gain * _lattice(shift) + offset).astype(np.float32)
    dR, dT = torch.from_numpy(R).cuda(), torch.from_numpy(T).cuda()
    E, _ = B.Context(B.Config()).energy_rigid(dR, dT, [0.0, 0.0, 0.0])
    Ex = _ncc_energy(R, T)
    assert abs(E - Ex) <= 1e-6 * Ex
    if abs(offset) > 1.0:
        return
    g = O.grid_for(512, 512)
    c = np.zeros((g.ny, g.nx, 2), np.float32)
    gd = torch.zeros((g.ny, g.nx, 2), device="cuda")
    E = B.Context(B.Config(mode="nonrigid")).energy_grid(dR, dT, torch.from_numpy(c).cuda(), gd)
    Eo, go = O.grid_energy(R, T, 0, g, c.transpose(2, 0, 1).astype(np.float64), 2.0)
    assert abs(E - Eo) <= 1e-5 * abs(Eo)
    np.testing.assert_allclose(gd.cpu().numpy().transpose(2, 0, 1), go, atol=2e-4 * np.abs(go).max())


@pytest.mark.parametrize("mode", ["rigid", "nonrigid"])
@pytest.mark.parametrize("gain,offset", [(3.0, 0.0), (0.25, 2.0)])
def test_pairs_of_different_gain_and_offset_match_the_oracle(mode, gain, offset):
    F = synth.make_series(synth.SeriesSpec(2, 120, 131, step=1.0, field_amp=1.0, snr=(10.0, 10.0), seed=8)).frames.numpy()
    R, T = F[0], (gain * F[1] + offset).astype(np.float32)
    cfg = B.Config(mode=mode)
    out = torch.empty((2, 120, 131), device="cuda") if mode == "nonrigid" else None
    _, st = B.Context(cfg).pairwise(torch.from_numpy(R).cuda(), torch.from_numpy(T).cuda(), field_out=out)
    oc = O.Config(levels=cfg.levels, max_iter=cfg.max_iter, max_rejects=cfg.max_rejects, tol_grad=cfg.tol_grad,
                  tol_rel_e=cfg.tol_rel_e, armijo_c=cfg.armijo_c, tau0=cfg.tau0, step_cap=cfg.step_cap, lam=cfg.lam,
                  mode=mode, metric=cfg.metric, sigma=cfg.sigma, tol_coarse=cfg.tol_coarse)
    Rp, Tp = O.pyramid(R, cfg.levels), O.pyramid(T, cfg.levels)
    p_o, st_o = O.register_nonrigid(Rp, Tp, None, oc) if mode == "nonrigid" else O.register_rigid(Rp, Tp, np.zeros(3), oc)
    got = out.cpu().numpy() if mode == "nonrigid" else np.array(st["theta"])
    assert O.max_px_error(got, p_o, 120, 131, mode) <= 0.02
    assert abs(st["energy"] - st_o.energy) <= 1e-5 * abs(st_o.energy)


@pytest.mark.parametrize("value", [0.0, 0.5, 0.3, -7.1, 1000.3])
@pytest.mark.parametrize("which", ["template", "reference", "both"])
def test_a_constant_image_has_energy_one_and_no_gradient(value, which):
    rng = np.random.default_rng(3)
    img = torch.from_numpy(rng.uniform(0, 1, size=(128, 117)).astype(np.float32)).cuda()
    const = torch.full_like(img, value)
    R = const if which != "template" else img
    T = const if which != "reference" else img
    E, g = B.Context(B.Config()).energy_rigid(R, T, [0.01, 0.37, -2.21])
    assert E == 1.0 and not g.any()
    nx, ny, _ = B.grid_dims(117, 128)
    c = torch.zeros((ny, nx, 2), device="cuda") + 0.37   # a translation: no regulariser
    gd = torch.ones_like(c)
    E = B.Context(B.Config(mode="nonrigid")).energy_grid(R, T, c, gd)
    assert E == 1.0 and not gd.any()


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf"), "f16"])
@pytest.mark.parametrize("which", ["template", "reference", "both"])
@pytest.mark.parametrize("mode", ["rigid", "nonrigid"])
def test_samples_that_are_not_finite_are_no_constant_image(mode, which, bad):
    # one pixel that is not finite, or that FP16 storage cannot hold: the energy is NaN (not that of a constant
    # image), and no step is taken
    F = synth.make_series(synth.SeriesSpec(2, 64, 70, step=1.0, snr=(10.0, 10.0), seed=2)).frames.cuda()
    R, T = F[0].clone(), F[1].clone()
    for img in ([R] if which == "reference" else [T] if which == "template" else [R, T]):
        img[30, 33] = 1e6 if bad == "f16" else bad
    nx, ny, _ = B.grid_dims(70, 64)
    if bad != "f16":
        ctx = B.Context(B.Config(mode=mode))
        E = ctx.energy_rigid(R, T, [0.0, 0.3, 0.2])[0] if mode == "rigid" else ctx.energy_grid(
            R, T, torch.full((ny, nx, 2), 0.3, device="cuda"))
        assert np.isnan(E)
    for cluster in (1, 16):
        out = torch.empty((2, 64, 70), device="cuda") if mode == "nonrigid" else None
        _, st = B.Context(B.Config(mode=mode, cluster=cluster, storage="f16" if bad == "f16" else "f32")).pairwise(R, T, field_out=out)
        assert np.isnan(st["energy"]) and st["iters"] == [0, 0]


def test_registered_mean_of_the_longest_series():
    # 64 frames for each of the 65,535 chunks that a launch's grid holds: a shorter chunk would make more of them
    N = 64 * 65535
    g = torch.Generator(device="cuda").manual_seed(3)
    F = torch.rand((N, 2, 2), device="cuda", generator=g)
    mean = torch.empty((2, 2), device="cuda")
    B.Context(B.Config(mode="nonrigid", levels=1)).warp(F, grids=torch.zeros((N - 1, 2, 2, 2), device="cuda"), mean=mean)
    assert float((mean.double() - F.double().mean(dim=0)).abs().max()) <= 1e-5


@pytest.mark.parametrize("H,grid", [(38545, 16), (38577, 16), (9637, 4)])
def test_pair_of_a_tall_frame_in_two_bands(H, grid):
    # 2,410 control rows of 2 points: two CTAs hold bands of 1,205 cell rows in one segment, the longest there is;
    # 2,412 rows take four CTAs
    W = grid + 1
    assert B.grid_dims(W, H, grid, 1)[0] == 2 and 2410 <= B.grid_dims(W, H, grid, 1)[1] <= 2412
    rng = np.random.default_rng(17)
    R = rng.uniform(0, 1, size=(H, W)).astype(np.float32)
    T = (0.5 * (R + np.roll(R, 1, axis=0))).astype(np.float32)
    outs = []
    for cluster in (2, 16):
        ctx = B.Context(B.Config(mode="nonrigid", levels=1, grid=grid, max_iter=1, cluster=cluster))
        outs.append(torch.empty((2, H, W), device="cuda"))
        _, st = ctx.pairwise(torch.from_numpy(R).cuda(), torch.from_numpy(T).cuda(), field_out=outs[-1])
        assert ctx.last_timing()["cluster"] == (4 if H == 38577 and cluster == 2 else cluster)
    cfg = B.Config()
    oc = O.Config(levels=1, max_iter=1, max_rejects=cfg.max_rejects, tol_grad=cfg.tol_grad, tol_rel_e=cfg.tol_rel_e,
                  armijo_c=cfg.armijo_c, tau0=cfg.tau0, step_cap=cfg.step_cap, lam=cfg.lam, mode="nonrigid", grid=grid,
                  metric=cfg.metric, sigma=cfg.sigma, tol_coarse=cfg.tol_coarse)
    c_o, st_o = O.register_nonrigid(O.pyramid(R, 1), O.pyramid(T, 1), None, oc)
    for out in outs:   # one accepted step, as in test_pair_for_every_band_split
        assert O.max_px_error(out.cpu().numpy(), c_o, H, W, "nonrigid", grid) <= 1e-3


@pytest.mark.parametrize("exec", ["level", "plain", "graph", "persistent"])
def test_scans_and_streams_of_a_grid_too_large_for_one_cta_take_two(exec):
    # 65 x 65 points need 292 KB in one CTA and 178 KB in each of two: asked for one, every executor and a stream
    # take two, with the results of two
    F = synth.make_series(synth.SeriesSpec(3, 513, 513, step=1.0, field_amp=1.0, snr=(10.0, 10.0), seed=9), device="cuda").frames
    els = {}
    for cluster in (1, 2):
        ctx = B.Context(B.Config(mode="nonrigid", grid=8, cluster=cluster, max_iter=2))
        els[cluster] = ctx.scan(F, schedule="sequential", exec=exec)[0]
        assert ctx.last_timing()["cluster"] == 2
    assert els[1] == els[2]
    if exec == "plain":
        s = B.Stream(B.Context(B.Config(mode="nonrigid", grid=8, cluster=1, max_iter=2)), 513, 513)
        for k in range(3):
            assert s.submit(F[k], k) == B.REG_OK
        got = []
        for _ in range(100):
            got += s.poll(timeout_us=100000)
            if len(got) == 3:
                break
        s.close()
        assert [r["elem"] for r in got[1:]] == els[2] and all(r["status"] == 0 for r in got)
