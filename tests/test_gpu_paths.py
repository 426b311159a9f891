"""GPU tests of the launch rules: every kernel a call can be routed to, at the
edges where the rule or the kernel's tiling changes, against the other route
or the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2603_09668_gb300 import binding as B
from paper_2603_09668_gb300 import inputs

from gpu_util import rel_l2, to_dev

pytestmark = pytest.mark.gpu


# HOME-LBM: a call of several steps on populations against the same steps one
# call at a time. Above 2^20 cells one step runs the tile kernel, below it the
# population kernels too, so both routes and both parities of the last step
# meet. The two round alike except for contraction: 5e-7 of the largest moment
# per step (a few float32 roundings of sums of order one).
@pytest.mark.parametrize("shape,bc_x", [((131, 103, 79), 1), ((130, 97, 85), 0), ((33, 7, 5), 1),
                                        ((2, 2, 2), 0)])
@pytest.mark.parametrize("steps", [1, 2, 3, 4, 5])
def test_home_steps_on_populations(shape, bc_x, steps):
    nx, ny, nz = shape
    g = torch.Generator(device="cuda").manual_seed(5)
    lbm = B.LBM(shape, 0.6, u_inlet=(0.05, 0.01, -0.02), force=(1e-5, 0.0, -2e-5), bc_x=bc_x)
    a = lbm.moments()
    lbm.home_init(a, 1.0, (0.04, 0.0, 0.01))
    a[:4] += 5e-3 * torch.randn(a[:4].shape, generator=g, device="cuda")
    solid = (torch.rand((nz, ny, nx), generator=g, device="cuda") < 0.1).to(torch.uint8)
    b, start = a.clone(), a.clone()
    lbm.home_step(a, solid, steps)
    for _ in range(steps):
        lbm.home_step(b, solid, 1)
    assert torch.isfinite(a).all()
    assert (a - b).abs().max().item() <= 5e-7 * steps
    keep = solid.bool().expand(10, nz, ny, nx)
    assert torch.equal(a[keep], start[keep])
    lbm.close()


def _mpm_case(n, n_grid, material, seed=0):
    """A deformed block of n particles in lattice order with 5% pinned."""
    g = np.random.default_rng(seed)
    sub = max(2, int(np.ceil((n / 3.0) ** (1 / 3))))
    x = inputs.block_particles(lo=(0.3, 0.3, 0.3), size=0.3, sub=sub, per_sub=3, seed=seed)[:, :n]
    st = inputs.perturbed_state(np.ascontiguousarray(x), v_scale=0.2, c_scale=1.0, f_scale=0.02, seed=seed)
    pin = (g.random(n) < 0.05).astype(np.uint8)
    st[1][:, pin != 0] = 0.0
    st[2][:, pin != 0] = 0.0
    vol = 0.3 ** 3 / n
    pr = dict(n_grid=n_grid, dt=5e-5, gravity=(0.0, -9.8, 0.0), bc_band=3, material=material, E=2e4,
              nu=0.3, p_mass=1000.0 * vol, p_vol=vol)
    return pr, st, pin


def _dev(st):
    return B.MpmState(*(to_dev(np.ascontiguousarray(a)) for a in st))


# The layer-split kernels (P2G and G2P up to 2^17 particles, the fused kernel up
# to 38,912) and the paired kernel above them, with and without vector loads,
# against the one-particle-per-thread kernels, around the CTA's 32 particles and
# the rules' edges. The same formulas summed in another order:
# the bounds of the paired kernels' test (x, F 1e-5; v, C 1e-3 of the largest).
@pytest.mark.parametrize("n", [1, 31, 32, 33, 95, 1000, 32768, 32772, 65535, 65537, 131072, 131073])
@pytest.mark.parametrize("material,sort_every", [(0, 0), (1, 3)])
def test_layer_split_forward(n, material, sort_every):
    pr, st, pin = _mpm_case(n, 64 if n > 5000 else 24, material)
    wind = B.WindField(to_dev(inputs.fourier_wind(9, 3, seed=4)), 7 * pr["dt"])
    got = []
    for mode in (B.P2G_AUTO, B.P2G_WARP):
        mpm = B.MPM.from_params(pr, max_particles=n, p2g_mode=mode)
        s, p = _dev(st), to_dev(pin)
        ids = torch.arange(n, dtype=torch.int32, device="cuda")
        out = B.MpmState.empty_like(s)
        mpm.substep(s, out, p, wind, 0.0)
        mpm.rollout(out, p, ids, wind, pr["dt"], 6, sort_every)
        mpm.device_status()
        assert torch.equal(torch.sort(ids.long()).values, torch.arange(n, device="cuda"))
        back = [torch.empty_like(a) for a in out]
        for b, a in zip(back, out):
            b[:, ids.long()] = a
        assert torch.equal(p.cpu(), torch.from_numpy(pin)[ids.cpu().long()])
        got.append(back)
        mpm.close()
    for k, tol in ((0, 1e-5), (3, 1e-5)):
        assert (got[0][k] - got[1][k]).abs().max().item() <= tol
    for k in (1, 2):
        assert (got[0][k] - got[1][k]).abs().max() <= 1e-3 * got[1][k].abs().max()


@pytest.mark.parametrize("n", [38912, 38913, 38916])
def test_fused_layer_split_at_the_rule(n):
    test_layer_split_forward(n, 0, 3)


def test_layer_split_reports_a_particle_off_the_grid():
    pr, st, pin = _mpm_case(70, 24, 0)
    st[0][0, 40] = 0.999
    mpm = B.MPM.from_params(pr, max_particles=70)
    s = _dev(st)
    wind = B.WindField(to_dev(inputs.constant_wind(2, 1, (1.0, 0.0, 0.0))), 1.0)
    mpm.rollout(s, to_dev(pin), None, wind, 0.0, 3, 0)
    with pytest.raises(B.DiffWindError):
        mpm.device_status()
    assert s.x[0, 40].item() == st[0][0, 40] and s.v[:, 40].abs().max().item() == 0.0
    assert torch.isfinite(s.x).all()
    mpm.close()


# The fused reverse pass (two launches per substep) against the four-launch one
# of p2g_mode WARP: the same sums in another order, relative L2 1e-4 per block,
# as between the batched and the single-scene adjoints.
@pytest.mark.parametrize("n", [1, 33, 1000, 40001])
@pytest.mark.parametrize("material,steps", [(0, 2), (1, 3), (0, 5)])
def test_fused_reverse_segment(n, material, steps):
    pr, st, pin = _mpm_case(n, 64 if n > 5000 else 24, material, seed=1)
    wind = B.WindField(to_dev(inputs.fourier_wind(9, 3, seed=4)), 7 * pr["dt"])
    g = torch.Generator(device="cuda").manual_seed(2)
    g0 = [torch.randn(a.shape, generator=g, device="cuda") for a in st]
    got = []
    for mode in (B.P2G_AUTO, B.P2G_WARP):
        mpm = B.MPM.from_params(pr, max_particles=n + 5, p2g_mode=mode)
        gs = B.MpmState(*(a.clone() for a in g0))
        gw, gE = torch.ones_like(wind.values), torch.ones(1, device="cuda")
        tape = torch.empty((steps - 1) * 24 * n, device="cuda")
        for _ in range(2):  # the second call starts from the first one's gradient
            mpm.segment_adjoint(_dev(st), tape, gs, to_dev(pin), wind, pr["dt"], steps, gw, gE)
        mpm.device_status()
        got.append([a.cpu().numpy().astype(np.float64) for a in (*gs, gw, gE)])
        mpm.close()
    for k, (a, b) in enumerate(zip(*got)):
        # dL/dx of an isolated particle is a difference of equal terms: both
        # passes are 2e-4 off the float64 value there (the other blocks 1e-5)
        if n > 1 or k > 0:
            assert rel_l2(a, b) <= 1e-4, k


# The wind gradient's scatter, per axis within a 4^3 block of grid nodes or tap
# by tap where the wind grid is as fine as the MPM grid, against the oracle's
# reverse substep: relative L2 1e-4, the adjoint's stated target.
@pytest.mark.parametrize("nf,frames", [(1, 1), (2, 3), (5, 1), (9, 2), (12, 3), (17, 2), (40, 2)])
def test_wind_gradient_scatter(nf, frames):
    pr, st, pin = _mpm_case(400, 18, 0, seed=3)
    wind = inputs.fourier_wind(nf, frames, seed=6)
    t = 0.3
    g = [np.random.default_rng(k).standard_normal(a.shape).astype(np.float32) for k, a in enumerate(st)]
    gw = torch.zeros(wind.shape, device="cuda")
    mpm = B.MPM.from_params(pr, max_particles=400)
    gi = B.MpmState.empty_like(_dev(st))
    mpm.substep_adjoint(_dev(st), _dev(g), gi, to_dev(pin), B.WindField(to_dev(wind), 1.0), t, gw)
    mpm.device_status()
    ref = oracle.mpm_substep_adjoint(pr, tuple(a.astype(np.float64) for a in st),
                                     (wind.astype(np.float64), nf, frames, 1.0), t,
                                     tuple(a.astype(np.float64) for a in g), pinned=pin)[1]
    assert rel_l2(gw.cpu().numpy().ravel(), np.asarray(ref).ravel()) <= 1e-4
    mpm.close()


def _gaussians(n, sigma, seed, opacity):
    """Gaussians in a unit slab seen from 2 units away, with distinct depths."""
    g = np.random.default_rng(seed)
    x = g.uniform(-0.4, 0.4, (3, n)).astype(np.float32)
    x[2] = (g.permutation(n) / n - 0.5).astype(np.float32) * 0.8
    F = np.tile(np.eye(3).reshape(9, 1), (1, n)) + g.uniform(-0.1, 0.1, (9, n))
    s0 = np.zeros((6, n))
    s0[:3] = np.asarray(sigma) ** 2
    col = g.uniform(0.0, 1.0, (3, n))
    op = g.uniform(*opacity, n)
    return [np.ascontiguousarray(a.astype(np.float32)) for a in (x, F, s0, col, op)]


# Tile lists: up to 4,096 Gaussians of a tile by the sort in shared memory, more
# by the radix sorts; a Gaussian meeting more than 16 tiles is listed by its
# whole warp. Every Gaussian covers the whole image (q < 9 everywhere), so no
# pixel depends on the cut-off. Image: n float32 roundings of a convex sum,
# 1e-5; gradients relative L2 1e-4 as in the renderer's parity test.
@pytest.mark.parametrize("n,size,opacity", [(1, (9, 8), (0.5, 0.9)), (40, (161, 97), (0.1, 0.5)),
                                            (33, (8, 200), (0.1, 0.5)), (4096, (12, 9), (0.01, 0.1)),
                                            (4097, (12, 9), (0.01, 0.1))])
def test_gaussian_tile_lists(n, size, opacity):
    from oracle import gsplat as G
    W, H = size
    arrs = _gaussians(n, 1.5, 7, opacity)
    f = 0.4 * max(W, H)
    kw = (np.eye(3), (0.0, 0.0, 2.0), f, f, W / 2, H / 2, W, H)
    dcam, ocam = B.camera(*kw), G.camera(*kw)
    r = B.GaussianRenderer(n, W, H)
    d = [to_dev(a) for a in arrs]
    img = r.render(dcam, *d)
    ref = G.render(*arrs, ocam)
    assert np.abs(img.cpu().numpy() - ref).max() <= 1e-5
    if n <= 64:
        g_img = np.random.default_rng(1).standard_normal((3, H, W)).astype(np.float32)
        gs = [torch.zeros_like(d[k]) for k in (0, 1, 3, 4)]
        r.backward(dcam, *d, to_dev(g_img), *gs)
        grad = G.render_grad(*arrs, ocam, g_img)
        for name, got in zip(("x", "F", "color", "opacity"), gs):
            assert rel_l2(got.cpu().numpy(), grad[name]) <= 1e-4, name
    r.close()


# The sorted lists do not depend on the path: small Gaussians, one tile crowded
# past the limit, drawn with and without the crowd's last members (which lie
# behind everything, at zero opacity, so that the image must not change).
def test_gaussian_list_paths_agree():
    n = 6000
    x, F, s0, col, op = _gaussians(n, 0.004, 8, (0.1, 0.9))
    x[:2, :4095] = np.random.default_rng(2).uniform(0.0, 0.02, (2, 4095))
    k = 5000
    op[k:] = 0.0
    x[:2, k:] = 0.01
    x[2, k:] = 0.9 + 0.001 * np.arange(n - k) / n
    cam = B.camera(np.eye(3), (0.0, 0.0, 2.0), 90.0, 90.0, 50.0, 40.0, 100, 80)
    r = B.GaussianRenderer(n, 100, 80)
    imgs = [r.render(cam, *(to_dev(np.ascontiguousarray(a[..., :m])) for a in (x, F, s0, col, op)))
            for m in (k, n)]
    assert torch.equal(imgs[0], imgs[1]) and imgs[0].max() > 0.3
    r.close()


# D-SSIM on 32 x 16 tiles: images smaller than the window, exactly one tile, and
# one pixel more; the oracle's tolerances (test_gpu_gsplat.py).
@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 4, 3), (3, 16, 32), (1, 17, 33), (5, 31, 65)])
def test_dssim_tiles(shape):
    from oracle import gsplat as G
    g = np.random.default_rng(11)
    a = g.random(shape).astype(np.float32)
    b = np.clip(a + 0.1 * g.standard_normal(shape), 0, 1).astype(np.float32)
    ref_loss, ref_g = G.dssim_loss(a, b)
    loss, grad = torch.zeros(1, device="cuda"), torch.zeros(shape, device="cuda")
    B.image_dssim_loss(to_dev(a), to_dev(b), loss, 2.0, grad)
    assert loss.item() == pytest.approx(2.0 * ref_loss, rel=1e-4)
    assert rel_l2(grad.cpu().numpy(), 2.0 * ref_g) <= 1e-4
    l2 = torch.zeros(1, device="cuda")
    B.image_dssim_loss(to_dev(a), to_dev(b), l2, 2.0)
    assert abs(l2.item() - loss.item()) <= 1e-6  # the block sums' order: 4 ulp of the weight


# Weight gradients of a g with a few single nonzero voxels (corners, faces, tile
# and slice edges): each tap's entry is a sum of few products of small whole
# numbers, exact in any order.
@pytest.mark.parametrize("shape", [(16, 32), (32, 32), (32, 16)])
@pytest.mark.parametrize("n", [16, 48])
def test_weight_gradient_of_single_voxels(n, shape):
    cin, cout = shape
    rng = np.random.default_rng(3)
    X = rng.integers(-8, 9, (cin, n, n, n)).astype(np.float64)
    G = np.zeros((cout, n, n, n))
    e = n - 1
    for v in ((0, 0, 0), (e, e, e), (0, e, 8), (7, 8, 15), (8, 7, 16 % n), (e, 0, 0), (5, 15, e), (1, 2, 3)):
        G[(slice(None), *v)] = rng.integers(-8, 9, cout)
    Xp = np.pad(X, ((0, 0), (1, 1), (1, 1), (1, 1)))
    ref = np.stack([np.einsum("ozyx,izyx->oi", G, Xp[:, dz:dz + n, dy:dy + n, dx:dx + n], optimize=True)
                    for dz in range(3) for dy in range(3) for dx in range(3)])

    def planar(a):
        p = np.moveaxis(a.reshape(-1, 8, n, n, n), 1, 4).reshape(-1, n ** 3, 8)
        return torch.tensor(np.ascontiguousarray(p)).to(torch.bfloat16).cuda()

    s = B.Surrogate(n)
    gw, gb = torch.zeros(27 * cout * cin, device="cuda"), torch.zeros(cout, device="cuda")
    s.weight_grad(cin, cout, planar(X), planar(G), gw, gb)
    s.device_status()
    assert np.array_equal(gw.cpu().numpy().reshape(27, cout, cin), ref)
    assert np.array_equal(gb.cpu().numpy(), G.sum(axis=(1, 2, 3)))
    s.close()


# The features kernel with paired and with scalar loads (a lattice or a mask
# that starts off its alignment) does the same operations in the same order.
@pytest.mark.parametrize("n", [16, 48])
def test_surrogate_features_alignment(n):
    rng = np.random.default_rng(5)
    N = 2 * n
    f = torch.tensor(0.02 * rng.standard_normal((19, N, N, N)).astype(np.float32), device="cuda")
    solid = torch.tensor((rng.random((N, N, N)) < 0.3).astype(np.uint8), device="cuda")
    fo = torch.empty(f.numel() + 1, device="cuda")[1:].view(f.shape)
    so = torch.empty(solid.numel() + 1, dtype=torch.uint8, device="cuda")[1:].view(solid.shape)
    fo.copy_(f)
    so.copy_(solid)
    s = B.Surrogate(n)
    got = [s.features(a, b, 20.0, torch.empty((n ** 3, 16), device="cuda"))
           for a, b in ((f, solid), (fo, solid), (f, so), (f, None), (fo, None))]
    assert torch.equal(got[0], got[1]) and torch.equal(got[0], got[2]) and torch.equal(got[3], got[4])
    rho = 1.0 + f.double().sum(0)
    cells = torch.where(solid == 0, rho - 1.0, 0.0).view(n, 2, n, 2, n, 2).sum((1, 3, 5))
    count = (solid == 0).double().view(n, 2, n, 2, n, 2).sum((1, 3, 5))
    ref = torch.where(count > 0, 20.0 * cells / count.clamp(min=1), 0.0).reshape(-1)
    # 19 populations and 8 cells summed in float32 around rho = 1: 27 half ulp of 1, scaled
    assert (got[0][:, 0].double() - ref).abs().max() <= 27 * 6e-8 * 20
    s.close()


# The one-launch inference pass where the grid has more CTAs than the volume
# has output slices (16^3: 32 slices), launch after launch, against the
# per-layer kernels: the same operations on the same operands (the tolerance of
# that comparison at 64^3).
def test_inference_with_idle_ctas():
    n = 16
    g = torch.Generator(device="cuda").manual_seed(9)
    s = B.Surrogate(n)
    s.set_params(0.1 * torch.randn(s.nparams, generator=g, device="cuda"))
    outs = []
    for keep in (True, False):
        for k in range(40):
            feats = torch.randn((n ** 3, 16), generator=torch.Generator(device="cuda").manual_seed(k),
                                device="cuda")
            s.set_features(feats)
            out = torch.empty((n ** 3, 16), device="cuda")
            s.forward(out, keep_activations=keep)
            outs.append(out)
    s.device_status()
    for a, b in zip(outs[:40], outs[40:]):
        assert a.abs().max() > 0 and (a - b).abs().max() <= 1e-6 * a.abs().max()
    s.close()


# The loss of a target that starts off a 16-byte boundary (scalar loads): the
# same gradients bit for bit; the loss up to the order of its 432 block sums, one
# rounding each.
@pytest.mark.parametrize("offset", [1, 2, 3])
def test_surrogate_loss_alignment(offset):
    n = 48
    g = torch.Generator(device="cuda").manual_seed(4)
    s = B.Surrogate(n)
    s.set_params(0.1 * torch.randn(s.nparams, generator=g, device="cuda"))
    feats = torch.randn((n ** 3, 16), generator=g, device="cuda")
    feats[:, 4] = (torch.rand(n ** 3, generator=g, device="cuda") < 0.3).float()
    s.set_features(feats)
    target = torch.randn((n ** 3, 16), generator=g, device="cuda")
    off = torch.empty(target.numel() + 4, device="cuda")[offset:offset + target.numel()].view(target.shape)
    off.copy_(target)
    assert target.data_ptr() % 16 == 0 and off.data_ptr() % 16 == 4 * offset and off.is_contiguous()
    got = []
    for t in (target, off):
        loss = torch.zeros(1, device="cuda")
        s.forward()
        s.loss(t, loss)
        s.zero_grads()
        s.backward()
        got.append((loss.item(), s.grads()))
    s.device_status()
    assert got[0][0] > 0 and abs(got[0][0] - got[1][0]) <= 432 * 1.2e-7 * got[0][0]
    assert got[0][1].abs().max() > 0 and torch.equal(got[0][1], got[1][1])
    s.close()


# Two handles that differentiate on two streams into one g_E and one wind
# gradient: every segment's part arrives. 80 parts of one sign in any order:
# 80 roundings, and the segments' own sums in any order, 1e-4.
def test_segments_of_two_streams_share_a_gradient():
    n, steps, calls = 64, 2, 40
    pr, st, pin = _mpm_case(n, 24, 0, seed=2)
    wind = B.WindField(to_dev(inputs.fourier_wind(5, 1, seed=4)), 1.0)
    g0 = [0.1 * torch.randn(a.shape, generator=torch.Generator(device="cuda").manual_seed(6), device="cuda")
          for a in st]

    def work(mpm, gw, gE, tape, stream, calls):
        with torch.cuda.stream(stream):
            for _ in range(calls):
                gs = B.MpmState(*(a.clone() for a in g0))
                mpm.segment_adjoint(state, tape, gs, pin_d, wind, 0.0, steps, gw, gE)

    state, pin_d = _dev(st), to_dev(pin)
    mpms = [B.MPM.from_params(pr, max_particles=n) for _ in range(2)]
    tapes = [torch.empty((steps - 1) * 24 * n, device="cuda") for _ in range(2)]
    streams = [torch.cuda.Stream() for _ in range(2)]
    sums = []
    for rounds in ((1,), (calls, calls)):  # one segment alone, then both streams at once
        gw, gE = torch.zeros_like(wind.values), torch.zeros(1, device="cuda")
        torch.cuda.synchronize()
        for k, c in enumerate(rounds):
            work(mpms[k], gw, gE, tapes[k], streams[k], c)
        torch.cuda.synchronize()
        sums.append((gw.cpu().numpy(), gE.item()))
    for m in mpms:
        m.device_status()
        m.close()
    (gw1, gE1), (gw2, gE2) = sums
    assert gE1 != 0 and abs(gE2 - 2 * calls * gE1) <= 1e-4 * abs(2 * calls * gE1)
    assert rel_l2(gw2, 2 * calls * gw1.astype(np.float64)) <= 1e-4


# As many Gaussians that meet more than 16 tiles as a 32-bit count of their
# warps' work items (16 each) no longer holds: the call is refused, and the
# handle still renders.
def test_gaussian_queue_of_2_28():
    n, W, H = 1 << 28, 64, 64
    if torch.cuda.mem_get_info()[0] < 90 << 30:
        pytest.skip("needs 90 GB of device memory")
    r = B.GaussianRenderer(n, W, H)
    x, F, s0 = (torch.zeros((k, n), device="cuda") for k in (3, 9, 6))
    F[::4] = 1.0
    s0[:3] = 4.0
    col, op = torch.full((3, n), 0.5, device="cuda"), torch.full((n,), 0.25, device="cuda")
    cam = B.camera(np.eye(3), (0.0, 0.0, 2.0), 40.0, 40.0, W / 2, H / 2, W, H)
    with pytest.raises(B.DiffWindError, match="too long"):
        r.render(cam, x, F, s0, col, op)
    few = [a[..., :3].contiguous() for a in (x, F, s0, col, op)]
    # three layers, each covers the image: at the centre C = 0.5 (1 - (1 - 0.25)^3)
    img = r.render(cam, *few)
    assert abs(img[0, H // 2, W // 2].item() - 0.5 * (1 - 0.75 ** 3)) <= 1e-3
    r.close()
    del x, F, s0, col, op
    torch.cuda.empty_cache()


# A list whose length no 32-bit (nor 36-bit) count holds, 2^18 Gaussians on all
# 2^18 tiles of an image, is refused; the handle still renders.
def test_gaussian_list_of_2_36_entries():
    n, W = 1 << 18, 4096
    r = B.GaussianRenderer(n, W, W)
    x, F, s0 = (torch.zeros((k, n), device="cuda") for k in (3, 9, 6))
    F[::4] = 1.0
    s0[:3] = 4.0
    col, op = torch.full((3, n), 0.5, device="cuda"), torch.full((n,), 0.25, device="cuda")
    cam = B.camera(np.eye(3), (0.0, 0.0, 2.0), 2560.0, 2560.0, W / 2, W / 2, W, W)
    with pytest.raises(B.DiffWindError, match="too long"):
        r.render(cam, x, F, s0, col, op)
    img = r.render(cam, *[a[..., :3].contiguous() for a in (x, F, s0, col, op)])
    assert abs(img[0, W // 2, W // 2].item() - 0.5 * (1 - 0.75 ** 3)) <= 1e-3
    r.close()


# Lists too long for 8 x 8 tiles (the second by the indices' step past the end: 2^31
# - 2 entries), made on 16 x 16: Gaussians about the optical
# axis that cover the image (q < 9 everywhere), at a few pixels against the
# float64 composite, with the gradients of those pixels. A pixel is a product of
# n factors, each rounded twice: n^0.5 x 1.2e-7 = 2 to 3e-5 of the image if the
# roundings are independent, allowed 1e-4. dL/dopacity is a difference of two
# such terms, allowed 1e-3 relative L2.
@pytest.mark.parametrize("size,n", [((2048, 2048), 32769), ((1736, 1208), 65538)])
def test_gaussian_list_on_coarse_tiles(size, n):
    (W, H), g = size, np.random.default_rng(3)
    if torch.cuda.mem_get_info()[0] < 120 << 30:
        pytest.skip("needs 120 GB of device memory")
    assert n * ((W + 7) // 8) * ((H + 7) // 8) > 2 ** 31 - 4096
    f, s = 0.4 * W, 1.5
    x, F, s0 = np.zeros((3, n), np.float32), np.zeros((9, n), np.float32), np.zeros((6, n), np.float32)
    x[2] = (g.permutation(n) / n - 0.5) * 0.8
    F[::4] = 1.0
    s0[:3] = s * s
    col = g.uniform(0.0, 1.0, (3, n)).astype(np.float32)
    op = (g.uniform(0.5, 1.5, n) * 3.0 / n).astype(np.float32)
    cam = B.camera(np.eye(3), (0.0, 0.0, 2.0), f, f, W / 2, H / 2, W, H)
    d = [to_dev(a) for a in (x, F, s0, col, op)]
    r = B.GaussianRenderer(n, W, H)
    img = r.render(cam, *d)
    pix = [(0, 0), (W - 1, H - 1), (W // 2, H // 2 - 1), (W - 16, H - 1), (17, 15)]
    g_img = torch.zeros((3, H, W), device="cuda")
    for k, (px, py) in enumerate(pix):
        g_img[:, py, px] = torch.tensor([1.0, -0.5, 0.25]) * (k + 1)
    gs = [torch.zeros_like(d[k]) for k in (0, 1, 3, 4)]
    r.backward(cam, *d, g_img, *gs)
    tz = 2.0 + x[2].astype(np.float64)
    order = np.argsort(tz)
    gc, go = np.zeros((3, n)), np.zeros(n)
    for k, (px, py) in enumerate(pix):
        e = np.exp(-0.5 * ((px + 0.5 - W / 2) ** 2 + (py + 0.5 - H / 2) ** 2) / (f * s / tz) ** 2)[order]
        a, c = op.astype(np.float64)[order] * e, col.astype(np.float64)[:, order]
        T = np.concatenate([[1.0], np.cumprod(1.0 - a)[:-1]])
        part = np.cumsum(T * a * c, axis=1)
        C = part[:, -1:]
        assert np.abs(img[:, py, px].cpu().numpy() - C[:, 0]).max() <= 1e-4
        w = np.array([1.0, -0.5, 0.25])[:, None] * (k + 1)
        gc[:, order] += w * T * a
        go[order] += (w * (T * c - (C - part) / (1.0 - a))).sum(0) * e
    assert rel_l2(gs[2].cpu().numpy(), gc) <= 1e-4 and rel_l2(gs[3].cpu().numpy(), go) <= 1e-3
    r.close()


# Little free memory: room for the list but not for the colours in front of its
# batches, so the backward walks the tiles; room only for the list on 16 x 16
# tiles. The same pixels composited in the same order: the same
# image, gradients up to the order of their sums over pixels, relative L2 1e-5.
@pytest.mark.parametrize("n", [2000, 4500])  # tiles sorted in shared memory; radix sorts (more per entry)
def test_gaussian_lists_in_little_memory(n):
    W = 1024 if n < 4096 else 640
    f = 0.4 * W
    cam = B.camera(np.eye(3), (0.0, 0.0, 2.0), f, f, W / 2, W / 2, W, W)
    d = [to_dev(a) for a in _gaussians(n, 3.0, 7, (0.0005, 0.001))]
    g_img = torch.randn((3, W, W), generator=torch.Generator(device="cuda").manual_seed(1), device="cuda")
    fine = n * (W // 8) ** 2
    lists, before = fine * (12 if n < 4096 else 16), ((n + 63) // 64) * 1024 * (W // 8) ** 2
    got, used = [], []
    for room in (None, lists + before // 2, int(0.75 * lists)):
        r = B.GaussianRenderer(n, W, W)
        img, gs = torch.empty_like(g_img), [torch.zeros_like(d[k]) for k in (0, 1, 3, 4)]
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        hog = []
        while room is not None and torch.cuda.mem_get_info()[0] - room > 32 << 20:
            left = torch.cuda.mem_get_info()[0] - room
            hog.append(torch.empty(min(left, 8 << 30) // (2 << 20) * (2 << 20), dtype=torch.uint8, device="cuda"))
        free = torch.cuda.mem_get_info()[0]
        r.render(cam, *d, image=img)
        r.backward(cam, *d, g_img, *gs)
        torch.cuda.synchronize()
        used.append(free - torch.cuda.mem_get_info()[0])
        got.append((img.cpu(), [a.cpu().numpy() for a in gs]))
        r.close()
        hog.clear()
        torch.cuda.empty_cache()
    assert used[0] >= lists + before and lists <= used[1] < lists + before and used[2] < lists, (used, lists, before)
    assert got[0][0].max() > 0.3
    for img, gs in got[1:]:
        assert torch.equal(img, got[0][0])
        for a, b in zip(gs, got[0][1]):
            assert rel_l2(a, b) <= 1e-5


def _kernels(call, path):
    """The kernel names of a call, from its capture (the call has run before)."""
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    g.enable_debug_mode()
    with torch.cuda.graph(g, stream=torch.cuda.Stream()):
        call()
    g.debug_dump(str(path))
    return path.read_text()


# What each p2g_mode runs, from the kernel names of a captured call: PAIR the
# paired fused kernel at every size, AUTO the layer kernels up to their counts.
@pytest.mark.parametrize("mode,n,fused", [("PAIR", 500, "k_g2p2g_pair"), ("PAIR", 38913, "k_g2p2g_pair"),
                                          ("AUTO", 500, "k_layer_g2p"), ("AUTO", 38913, "k_g2p2g_pair"),
                                          ("WARP", 500, "k_g2p2g")])
@pytest.mark.filterwarnings("ignore:DEBUG")
def test_kernels_of_a_mode(mode, n, fused, tmp_path):
    pr, st, pin = _mpm_case(n, 24, 0)
    mpm = B.MPM.from_params(pr, max_particles=n, p2g_mode=getattr(B, "P2G_" + mode))
    s, pin_d = _dev(st), to_dev(pin)
    wind = B.WindField(to_dev(inputs.constant_wind(2, 1, (1.0, 0.0, 0.0))), 1.0)
    mpm.rollout(s, pin_d, None, wind, 0.0, 3, 0)
    text = _kernels(lambda: mpm.rollout(s, pin_d, None, wind, 0.0, 3, 0), tmp_path / "g.dot")
    layers = ["k_layer_p2g", "k_layer_g2p"] if mode == "AUTO" else []  # the first P2G, the last G2P
    for name in ("k_g2p2g_pair", "k_layer_g2p", "k_layer_p2g", "k_grid_update_active"):
        assert (name in text) == (name in (fused, "k_grid_update_active", *layers)), name
    assert fused in text
    mpm.close()


# A segment whose recompute runs the paired kernel (P2G_PAIR) on few particles,
# odd counts and a partly filled last warp, against the one-particle kernels of
# P2G_WARP: states and gradients, relative L2 1e-4 per block, as the fused reverse
# pass above. (dL/dE is left out: one number, the sum of n terms of both signs that
# cancel to 2e-6 here, while every mode is 3e-10 off its float64 value.)
@pytest.mark.parametrize("n", [33, 130, 1000])
@pytest.mark.parametrize("material,steps", [(0, 2), (1, 4)])
def test_paired_recompute_of_a_segment(n, material, steps):
    pr, st, pin = _mpm_case(n, 24, material, seed=1)
    wind = B.WindField(to_dev(inputs.fourier_wind(9, 3, seed=4)), 7 * pr["dt"])
    g = torch.Generator(device="cuda").manual_seed(2)
    g0 = [torch.randn(a.shape, generator=g, device="cuda") for a in st]
    got = []
    for mode in (B.P2G_PAIR, B.P2G_WARP):
        mpm = B.MPM.from_params(pr, max_particles=n, p2g_mode=mode)
        gs = B.MpmState(*(a.clone() for a in g0))
        gw = torch.zeros_like(wind.values)
        tape = torch.empty((steps - 1) * 24 * n, device="cuda")
        mpm.segment_adjoint(_dev(st), tape, gs, to_dev(pin), wind, pr["dt"], steps, gw)
        mpm.device_status()
        got.append([a.cpu().numpy().astype(np.float64) for a in (tape, *gs, gw)])
        mpm.close()
    for k, (a, b) in enumerate(zip(*got)):
        assert rel_l2(a, b) <= 1e-4, k


# A particle whose F is not a number (or has det F = -inf) has no stress: its mass and
# momentum reach the grid, and the particles around it stay finite; the call
# reports it. (The paired kernel's Neo-Hookean form never did so.) Against the
# same call with an inverted F in its place, which adds the same: x, v and F within
# 1e-6, atomics' order (which C's factor 4 / dx carries beyond that).
@pytest.mark.parametrize("bad", [float("nan"), float("-inf")])
@pytest.mark.parametrize("mode,material,steps", [(m, k, s) for m in ("AUTO", "WARP", "ATOMIC", "TILE")
                                                 for k in (0, 1) for s in (1, 3)]
                         + [("PAIR", 0, 1), ("PAIR", 1, 3)])
def test_a_particle_without_a_stress(mode, material, steps, bad):
    n, p = 200, 70
    pr, st, pin = _mpm_case(n, 24, material, seed=5)
    wind = B.WindField(to_dev(inputs.constant_wind(2, 1, (1.0, 0.0, 0.0))), 1.0)
    out = []
    for F in (bad, -1.0):
        st[3][:, p] = np.eye(3).reshape(9) * -1.0
        st[3][0, p] = F
        mpm = B.MPM.from_params(pr, max_particles=n, p2g_mode=getattr(B, "P2G_" + mode))
        s = _dev(st)
        if steps == 1:
            mpm.substep(s, s, to_dev(pin), wind, 0.0)
        else:
            mpm.rollout(s, to_dev(pin), None, wind, 0.0, steps, 0)
        with pytest.raises(B.DiffWindError):
            mpm.device_status()
        out.append([a.cpu().numpy() for a in s])
        mpm.close()
    for k, (a, b) in enumerate(zip(*out)):
        if k == 3:
            a, b = np.delete(a, p, 1), np.delete(b, p, 1)
        assert np.isfinite(a).all(), k
        if k != 2:
            assert np.abs(a - b).max() <= 1e-6 * max(1.0, np.abs(b).max()), k


# Wind cotangents that are not finite reach the wind nodes that their grid nodes
# sample and no others: the same ones as in the oracle's reverse substep (of a
# particle whose grid nodes lie between wind nodes, so that no weight is zero).
@pytest.mark.parametrize("nf,frames", [(6, 2), (5, 3), (9, 2)])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_wind_gradient_of_a_bad_cotangent(nf, frames, bad):
    pr, st, pin = _mpm_case(400, 18, 0, seed=3)
    wind, t = inputs.fourier_wind(nf, frames, seed=6), 0.3
    g = [np.random.default_rng(k).standard_normal(a.shape).astype(np.float32) for k, a in enumerate(st)]
    p = int(np.flatnonzero((pin == 0) & (st[0] * 18 < 7.4).all(0))[3])
    g[1][0, p] = bad
    gw = torch.zeros(wind.shape, device="cuda")
    mpm = B.MPM.from_params(pr, max_particles=400)
    mpm.substep_adjoint(_dev(st), _dev(g), B.MpmState.empty_like(_dev(st)), to_dev(pin),
                        B.WindField(to_dev(wind), 1.0), t, gw)
    ref = oracle.mpm_substep_adjoint(pr, tuple(a.astype(np.float64) for a in st),
                                     (wind.astype(np.float64), nf, frames, 1.0), t,
                                     tuple(a.astype(np.float64) for a in g), pinned=pin)[1]
    got, ref = gw.cpu().numpy().reshape(-1, 3), np.asarray(ref).reshape(-1, 3)
    assert 0 < np.isfinite(ref).sum() and np.array_equal(np.isfinite(got), np.isfinite(ref))
    ok = np.isfinite(ref)
    assert rel_l2(got[ok], ref[ok]) <= 1e-4
    mpm.close()


# The counts up to which a substep of AUTO runs the layer kernels.
@pytest.mark.parametrize("n,layers", [(38912, ("p2g", "g2p")), (38913, ("g2p",)), (65536, ("g2p",)), (65537, ())])
@pytest.mark.filterwarnings("ignore:DEBUG")
def test_kernels_of_a_substep(n, layers, tmp_path):
    pr, st, pin = _mpm_case(n, 24, 0)
    mpm = B.MPM.from_params(pr, max_particles=n)
    s, pin_d = _dev(st), to_dev(pin)
    wind = B.WindField(to_dev(inputs.constant_wind(2, 1, (1.0, 0.0, 0.0))), 1.0)
    mpm.substep(s, s, pin_d, wind, 0.0)
    text = _kernels(lambda: mpm.substep(s, s, pin_d, wind, 0.0), tmp_path / "g.dot")
    for k in ("p2g", "g2p"):
        assert ("k_layer_" + k in text) == (k in layers)
    mpm.close()


# The count up to which a segment's reverse pass runs in two launches a substep,
# and the gradients on both sides of it against P2G_WARP's: relative L2 1e-4 per
# block (dL/dE left out, as in the paired recompute's test).
@pytest.mark.parametrize("n,chain", [(196608, True), (196609, False)])
@pytest.mark.filterwarnings("ignore:DEBUG")
def test_kernels_of_a_segment(n, chain, tmp_path):
    pr, st, pin = _mpm_case(n, 64, 0)
    s, pin_d, steps = _dev(st), to_dev(pin), 3
    wind = B.WindField(to_dev(inputs.fourier_wind(9, 3, seed=4)), 7 * pr["dt"])
    gen = torch.Generator(device="cuda").manual_seed(2)
    g0 = [torch.randn(a.shape, generator=gen, device="cuda") for a in st]
    got = []
    for mode in (B.P2G_AUTO, B.P2G_WARP):
        mpm = B.MPM.from_params(pr, max_particles=n, p2g_mode=mode)
        gs = B.MpmState(*(a.clone() for a in g0))
        gw, tape = torch.zeros_like(wind.values), torch.empty((steps - 1) * 24 * n, device="cuda")
        call = lambda: mpm.segment_adjoint(s, tape, gs, pin_d, wind, 0.0, steps, gw)
        call()
        mpm.device_status()
        got.append([a.cpu().numpy().astype(np.float64) for a in (*gs, gw)])
        if mode == B.P2G_AUTO:
            text = _kernels(call, tmp_path / "g.dot")
            assert ("k_layer_rev" in text) == chain and ("k_rev_g2p" in text) == (not chain)
        mpm.close()
    for k, (a, b) in enumerate(zip(*got)):
        assert rel_l2(a, b) <= 1e-4, k


# HOME-LBM steps on populations or by tiles, by the lattice's cells, the steps of
# the call and whether there is a mask.
@pytest.mark.parametrize("shape,steps,masked,chain", [
    ((128, 128, 64), 1, 0, True), ((128, 128, 65), 1, 0, False), ((128, 128, 65), 3, 0, True),
    ((128, 128, 128), 4, 0, True), ((128, 128, 129), 8, 1, False), ((128, 128, 129), 10, 0, True),
    ((256, 128, 129), 10, 0, False), ((256, 128, 129), 10, 1, True), ((256, 128, 224), 3, 0, True),
    ((256, 128, 225), 3, 0, False), ((256, 128, 225), 30, 1, False)])
@pytest.mark.filterwarnings("ignore:DEBUG")
def test_kernels_of_home_steps(shape, steps, masked, chain, tmp_path):
    lbm = B.LBM(shape, 0.6, u_inlet=(0.05, 0.0, 0.0), bc_x=1)
    m = lbm.moments()
    lbm.home_init(m, 1.0, (0.04, 0.0, 0.01))
    solid = torch.zeros(shape[::-1], dtype=torch.uint8, device="cuda") if masked else None
    lbm.home_step(m, solid, steps)
    text = _kernels(lambda: lbm.home_step(m, solid, steps), tmp_path / "g.dot")
    assert ("k_home_open" in text) == chain and ("k_home_step" in text) == (not chain)
    lbm.close()


# Queued Gaussians (more than 16 tiles each) in numbers around the queue's warps
# (4,864: one each, several each, a part each): all are listed in all tiles, each
# once. Against the image drawn in nine parts of nine tiles each, which queue
# none: Gaussians on the optical axis, whose pixel offsets are the same floats in
# the parts, so the same bits.
@pytest.mark.parametrize("n", [1, 2, 303, 305, 1621, 2433, 4863, 4864, 4865, 9000])
def test_gaussian_queue_shares(n):
    W, p = 72, 24
    g = torch.Generator(device="cuda").manual_seed(n)
    x, F, s0 = (torch.zeros((k, n), device="cuda") for k in (3, 9, 6))
    x[2] = torch.linspace(-0.4, 0.4, n, device="cuda")
    F[::4] = 1.0
    s0[:3] = 4.0
    d = (x, F, s0, torch.rand((3, n), generator=g, device="cuda"), torch.full((n,), 0.5 / n ** 0.5, device="cuda"))
    whole, part = B.GaussianRenderer(n, W, W), B.GaussianRenderer(n, p, p)
    img = whole.render(B.camera(np.eye(3), (0.0, 0.0, 2.0), 400.0, 400.0, W / 2, W / 2, W, W), *d)
    assert img.max() > 0.1
    for y in range(0, W, p):
        for x0 in range(0, W, p):
            cam = B.camera(np.eye(3), (0.0, 0.0, 2.0), 400.0, 400.0, W / 2 - x0, W / 2 - y, p, p)
            assert torch.equal(part.render(cam, *d), img[:, y:y + p, x0:x0 + p]), (x0, y)
    whole.close()
    part.close()


# The weight gradient's partial sums are held once per CTA that can run: a
# 27 x 32 x 32 block of floats each (the mma.sync kernel has fewer chunks at 16^3).
def test_surrogate_partial_sums_memory():
    B.Surrogate(16).close()  # the library's own first allocations
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    s = B.Surrogate(16)
    used = free - torch.cuda.mem_get_info()[0]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert used <= sms * 27 * 32 * 32 * 4 + (10 << 20)
    s.close()
