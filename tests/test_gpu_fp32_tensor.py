"""The FP32 tier on the tensor cores and the paired contraction: edges of the row pairs, the
column tiles and the accumulation groups, strengths at the ends of FP32's range, and the
CUDA-core sum where the workspace bound holds no more.

Bar of the FP32 tier, 1e-6: the sines and cosines of A and B are each off by at most 2^-21.4
(3.6e-7), together 5.1e-7 in the mean square; an accumulation of two 32-pixel chunks rounds
toward zero 16 times at its full size, about 16 x 2^-25 x 2/3 = 3.2e-7; the 16-bit pairs hold
22 bits and the FP32 sums add less."""
import numpy as np
import pytest

import oracle
from paper_2307_09226_gb300 import synth
from paper_2307_09226_gb300.synth import Radar

pytestmark = pytest.mark.gpu
FP32_BAR = 1e-6


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2307_09226_gb300 import _abi, device
    ctx = device.Context(0)
    yield torch, _abi, device, ctx
    ctx.close()


@pytest.mark.parametrize("tier,bar", [("fp32", FP32_BAR), ("split_fp16", 2e-5), ("split_bf16", 2e-5)])
@pytest.mark.parametrize("V,Ns,L,n_az,n_el", [
    (1, 128, 16, 16, 8),     # one row tile of the pair, the fewest pixels the rule takes
    (1, 129, 17, 43, 3),     # one row in the second tile; a chunk with one pixel
    (1, 255, 15, 40, 25),
    (3, 171, 129, 33, 31),   # 513 rows: an odd number of tiles; two column tiles
    (2, 256, 136, 64, 16),
    (17, 13, 40, 30, 20),    # a tile over more channels than the phase ring holds
    (1, 40, 8, 300, 100),    # 30,000 pixels: groups of two chunks
])
def test_pair_edges(env, tier, bar, V, Ns, L, n_az, n_el):
    torch, _abi, device, ctx = env
    f = synth.Frame(Radar(M=V, N=1, Ns=Ns, L=L), synth.random_frame(Radar(M=V, N=1, Ns=Ns, L=L), n_az, n_el, seed=Ns,
                                                                   mask_frac=0.0 if n_az * n_el < 200 else 0.2))
    got = ctx.synth(f.radar, device.upload(f), tier).cpu().numpy()
    assert ctx.sync_status() == _abi.OK
    assert oracle.rel_l2(got, oracle.cube_separable(f.radar, f.pixels)) <= bar


@pytest.mark.parametrize("tier,bar", [("fp32", FP32_BAR), ("split_fp16", 2e-5), ("fp16", 1e-2)])
@pytest.mark.parametrize("top", [1e-40, 1e-30, 1e30, 1e37])
def test_strengths_at_the_ends_of_the_range(env, tier, bar, top):
    """The power-of-two scale of sigma neither overflows nor underflows: the cube is that of
    ordinary strengths, scaled (normal results: 1e-30 and above)."""
    torch, _abi, device, ctx = env
    f = synth.parity_frame(seed=91, M=2, N=2, Ns=64, L=24, n_az=40, n_el=20)
    m = float(np.max(np.abs(np.stack([f.pixels.sigma_re, f.pixels.sigma_im]))))
    if top > 1:  # a cube of a few strong pixels stays below FP32's largest number
        f.pixels.sigma_re[8:] = 0.0
        f.pixels.sigma_im[8:] = 0.0
    f.pixels.sigma_re[:] = (f.pixels.sigma_re / m * top).astype(np.float32)
    f.pixels.sigma_im[:] = (f.pixels.sigma_im / m * top).astype(np.float32)
    got = ctx.synth(f.radar, device.upload(f), tier, out_dtype="complex128").cpu().numpy()
    assert ctx.sync_status() == _abi.OK and np.all(np.isfinite(got))
    # subnormal strengths and sums have an absolute resolution of 1.4e-45
    err = np.linalg.norm(got - oracle.cube_separable(f.radar, f.pixels))
    ref = np.linalg.norm(oracle.cube_separable(f.radar, f.pixels))
    assert err <= bar * ref + 1.5e-45 * np.sqrt(got.size) * (1 if top < 1e-37 else 0)


def test_weak_pixels_keep_their_bits(env):
    """One pixel 1e4 times stronger than the 8,000 others: the others' cube alone, recovered by
    linearity, keeps the accuracy that FP32 sums at the strong pixel's size leave."""
    torch, _abi, device, ctx = env
    f = synth.parity_frame(seed=92, M=1, N=2, Ns=96, L=32, n_az=100, n_el=80, mask_frac=0.0)
    f.pixels.sigma_re[4000] = 1e4 * np.max(np.abs(f.pixels.sigma_re))
    ref = oracle.cube_separable(f.radar, f.pixels)
    got = ctx.synth(f.radar, device.upload(f), "fp32").cpu().numpy()
    assert oracle.rel_l2(got, ref) <= FP32_BAR


def test_a_workspace_bound_leaves_the_cuda_core_sum(env):
    """Contexts whose budget holds the CUDA-core sum's workspace but not the tensor cores' keep
    taking the call; a batch beyond the budget gives the same bits as its frames alone."""
    torch, _abi, device, ctx = env
    radar = Radar(M=2, N=4, Ns=64, L=64)
    frames = [synth.random_frame(radar, 80, 60, seed=s, mask_frac=0.3) for s in range(5)]
    pxs = [device.upload(f) for f in frames]
    P = frames[0].P
    pinned = device.Context(0)
    _abi.rsim_set_plan(pinned.h, radar, P, _abi.TIER_FP32, splits=2)
    direct = _abi.rsim_workspace_size(pinned.h, radar, P, _abi.TIER_FP32)
    tensor = _abi.rsim_workspace_size(ctx.h, radar, P, _abi.TIER_FP32)
    assert direct < tensor
    small = device.Context(0, hbm_budget_bytes=tensor - 256)
    got = small.synth(radar, pxs[0], "fp32").cpu().numpy()
    assert small.sync_status() == _abi.OK
    assert oracle.rel_l2(got, oracle.cube_separable(radar, frames[0])) <= 2e-5
    alone = [ctx.synth(radar, px, "fp32").cpu().numpy() for px in pxs]
    two = device.Context(0, hbm_budget_bytes=2 * tensor + 4096)
    cubes = two.synth_batch(radar, pxs, "fp32")
    assert two.sync_status() == _abi.OK
    for a, c in zip(alone, cubes):
        assert np.array_equal(a, c.cpu().numpy())
    for c in (pinned, small, two):
        c.close()


def test_tuning_keeps_the_engine_and_its_accuracy(env):
    torch, _abi, device, _ = env
    c = device.Context(0)
    f = synth.parity_frame(seed=93, M=2, N=4, Ns=128, L=64, n_az=64, n_el=64)
    before = c.synth(f.radar, device.upload(f), "fp32").cpu().numpy()
    plan = _abi.rsim_autotune(c.h, f.radar, f.pixels.P, _abi.TIER_FP32)
    assert plan.tuned == 1 and plan.as_dict() == _abi.rsim_get_plan(c.h, f.radar, f.pixels.P, _abi.TIER_FP32).as_dict()
    ref = oracle.cube_separable(f.radar, f.pixels)
    after = c.synth(f.radar, device.upload(f), "fp32").cpu().numpy()
    assert oracle.rel_l2(before, ref) <= FP32_BAR and oracle.rel_l2(after, ref) <= FP32_BAR
    c.close()


@pytest.mark.parametrize("tier,bar", [("fp32", FP32_BAR), ("split_fp16", 2e-5)])
def test_odd_column_tiles_take_no_padding(env, tier, bar):
    """40 columns of l: 640 bytes of operand images and 28 of phases a pixel, so that 96,000
    pixels fit the static workspace of 64 MiB, which images padded to 48 columns (768) pass."""
    torch, _abi, device, ctx = env
    radar = Radar(M=1, N=1, Ns=64, L=40)
    px = synth.random_frame(radar, 300, 320, seed=11)
    d = device.upload(px)
    cube = torch.empty((1, 64, 40), dtype=torch.complex64, device="cuda")
    assert _abi.rsim_synth_static(radar, d, _abi.TIERS[tier], cube) == _abi.OK, _abi.last_error()
    torch.cuda.synchronize()
    got = cube.cpu().numpy()
    assert np.array_equal(got, ctx.synth(radar, d, tier).cpu().numpy())
    assert oracle.rel_l2(got, oracle.cube_separable(radar, px)) <= bar


@pytest.mark.parametrize("tier", ["fp32", "bf16", "fp16", "split_fp16", "split_bf16"])
@pytest.mark.parametrize("V,Ns,L", [(1, 64, 16), (1, 128, 128), (2, 96, 40), (3, 128, 64)])
def test_frames_of_few_tiles_are_split(env, tier, V, Ns, L):
    """One to three tiles of 65,536 pixels: enough splits to give most SMs a unit."""
    torch, _abi, device, ctx = env
    plan = _abi.rsim_get_plan(ctx.h, Radar(M=V, N=1, Ns=Ns, L=L), 65536, _abi.TIERS[tier])
    assert plan.splits >= 32


@pytest.mark.parametrize("tier", ["split_fp16", "fp16"])
def test_complex128_cubes_beyond_the_range_of_fp32(env, tier):
    """Eight pixels of 1.5e38 at one place: their sum passes FP32's largest number, but a
    complex128 cube holds it when the tile is written directly (one split, one accumulation
    group)."""
    torch, _abi, device, ctx = env
    f = synth.parity_frame(seed=94, M=1, N=2, Ns=64, L=24, n_az=8, n_el=1, mask_frac=0.0)
    px = f.pixels
    for a in (px.range, px.az, px.el, px.vel):
        a[:] = a[0]
    px.sigma_re[:], px.sigma_im[:] = np.float32(1.5e38), 0.0
    assert _abi.rsim_get_plan(ctx.h, f.radar, px.P, _abi.TIERS[tier]).splits == 1
    ref = oracle.cube_separable(f.radar, px)
    assert np.abs(ref.real).max() > 3.5e38
    got = ctx.synth(f.radar, device.upload(f), tier, out_dtype="complex128").cpu().numpy()
    assert ctx.sync_status() == _abi.OK and np.all(np.isfinite(got))
    assert oracle.rel_l2(got / 1e38, ref / 1e38) <= (2e-5 if tier == "split_fp16" else 1e-2)


@pytest.mark.parametrize("one_phase", [True, False])
def test_no_systematic_loss_beside_the_cuda_core_sum(env, one_phase):
    """The tensor cores' accumulator rounds toward zero, which shortens every sum, most visibly
    where strengths share a phase (rendered scenes: rho |n.d| / R^2).  Both forms have the same
    phasors, so their projections on the exact cube differ by the accumulation, and in single
    frames by the roundings of the strongest pixels' operands: over the frames by less than
    2^-23 in the mean, one unit in the last place.  And no frame's error is larger than the
    CUDA-core sum's, up to 10% for its own roundings."""
    torch, _abi, device, ctx = env
    lengths = []
    for V, Ns, L in [(2, 64, 17), (1, 128, 64), (2, 40, 8)]:
        for n_az, n_el in [(64, 32), (140, 130), (200, 200), (256, 256)]:
            radar = Radar(M=V, N=1, Ns=Ns, L=L)
            px = synth.random_frame(radar, n_az, n_el, seed=n_az + V, mask_frac=0.3)
            g = np.random.default_rng(n_el)
            hit = (px.sigma_re != 0) | (px.sigma_im != 0)
            amp = np.where(hit, g.uniform(0.1, 1.0, px.P) / np.where(hit, px.range, 1.0) ** 2, 0.0)
            phase = np.zeros(px.P) if one_phase else g.uniform(0, 2 * np.pi, px.P)
            px.sigma_re[:], px.sigma_im[:] = amp * np.cos(phase), amp * np.sin(phase)
            ref = oracle.cube_separable(radar, px)
            d = device.upload(px)
            tensor = ctx.synth(radar, d, "fp32").cpu().numpy().astype(np.complex128)
            bound = _abi.rsim_workspace_size(ctx.h, radar, px.P, _abi.TIER_FP32) - 256
            small = device.Context(0, hbm_budget_bytes=bound)
            direct = small.synth(radar, d, "fp32").cpu().numpy().astype(np.complex128)
            small.close()
            lengths.append([np.vdot(ref, x).real / np.vdot(ref, ref).real - 1.0 for x in (tensor, direct)])
            errs = [oracle.rel_l2(x, ref) for x in (tensor, direct)]
            print(f"length {lengths[-1][0]:+.2e} {lengths[-1][1]:+.2e}, error {errs[0]:.2e} {errs[1]:.2e}")
            assert errs[0] <= 1.1 * errs[1]
    mean = np.mean(lengths, axis=0)
    assert abs(mean[0] - mean[1]) < 2.0 ** -23
