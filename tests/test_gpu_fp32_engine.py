"""The FP32 tier's two forms, the tensor-core form and the CUDA-core sum: which one a call
takes (plans, saved plans, workspace bounds, captures) and the CUDA-core sum's own results."""
import json

import numpy as np
import pytest

import oracle
from paper_2307_09226_gb300 import synth
from paper_2307_09226_gb300.synth import Radar

pytestmark = pytest.mark.gpu
FP32_BAR = 1e-6    # the tensor-core form (derived in test_gpu_fp32_tensor.py)
DIRECT_BAR = 2e-5  # the tier


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


def sizes(env, radar, P):
    """Workspace of the tensor-core form and of the CUDA-core sum under their default plans."""
    torch, _abi, device, ctx = env
    tensor = _abi.rsim_workspace_size(ctx.h, radar, P, _abi.TIER_FP32)
    small = device.Context(0, hbm_budget_bytes=tensor - 256)
    direct = _abi.rsim_workspace_size(small.h, radar, P, _abi.TIER_FP32)
    small.close()
    assert direct < tensor
    return tensor, direct


def split(plan):
    d = plan.as_dict()
    d.pop("tuned")
    return d


@pytest.mark.parametrize("Ns,L,n_az,n_el", [(128, 64, 64, 64), (96, 40, 60, 50), (64, 256, 90, 40), (64, 32, 10, 9)])
@pytest.mark.parametrize("tune", [False, True])
def test_a_plan_read_and_set_again_changes_nothing(env, Ns, L, n_az, n_el, tune):
    """What rsim_get_plan or rsim_autotune returns, pinned in a new context: the same form
    (its workspace), the same plan, the same bits."""
    torch, _abi, device, _ = env
    f = synth.parity_frame(seed=Ns + L, M=2, N=3, Ns=Ns, L=L, n_az=n_az, n_el=n_el)
    d, P = device.upload(f), f.pixels.P
    a, b = device.Context(0), device.Context(0)
    plan = _abi.rsim_autotune(a.h, f.radar, P, _abi.TIER_FP32) if tune else _abi.rsim_get_plan(a.h, f.radar, P, _abi.TIER_FP32)
    _abi.rsim_set_plan(b.h, f.radar, P, _abi.TIER_FP32, **split(plan))
    assert split(_abi.rsim_get_plan(b.h, f.radar, P, _abi.TIER_FP32)) == split(plan)
    assert _abi.rsim_workspace_size(a.h, f.radar, P, _abi.TIER_FP32) == _abi.rsim_workspace_size(b.h, f.radar, P, _abi.TIER_FP32)
    want, got = (c.synth(f.radar, d, "fp32").cpu().numpy() for c in (a, b))
    assert a.sync_status() == _abi.OK and b.sync_status() == _abi.OK
    assert np.array_equal(want, got)
    assert oracle.rel_l2(got, oracle.cube_separable(f.radar, f.pixels)) <= FP32_BAR
    a.close(), b.close()


def test_a_plan_of_the_cuda_core_sum_and_back(env):
    """grid 0 pins the CUDA-core sum, a CTA count the tensor-core form again; a plan read while
    the CUDA-core sum runs pins the CUDA-core sum."""
    torch, _abi, device, _ = env
    radar, P = Radar(M=2, N=4, Ns=64, L=64), 4800
    tensor, direct = sizes(env, radar, P)
    c = device.Context(0)
    _abi.rsim_set_plan(c.h, radar, P, _abi.TIER_FP32, splits=2)
    pinned = _abi.rsim_workspace_size(c.h, radar, P, _abi.TIER_FP32)
    plan = _abi.rsim_get_plan(c.h, radar, P, _abi.TIER_FP32)
    assert plan.grid == 0 and plan.splits == 2
    _abi.rsim_set_plan(c.h, radar, P, _abi.TIER_FP32, **split(plan))
    assert _abi.rsim_workspace_size(c.h, radar, P, _abi.TIER_FP32) == pinned < tensor
    free = device.Context(0)
    _abi.rsim_set_plan(c.h, radar, P, _abi.TIER_FP32, **split(_abi.rsim_get_plan(free.h, radar, P, _abi.TIER_FP32)))
    assert _abi.rsim_workspace_size(c.h, radar, P, _abi.TIER_FP32) == tensor
    free.close(), c.close()


def test_a_tuned_entry_of_the_cuda_core_sum_does_not_choose_the_form(env, tmp_path, monkeypatch):
    """A tuning file may hold an entry of the CUDA-core sum for a shape (tuned where the
    workspace bound left nothing else, or by a version of the library that had nothing else):
    it is the plan of that sum, not a choice of it, and tuning again times the form that runs."""
    torch, _abi, device, _ = env
    radar, P = Radar(M=2, N=4, Ns=128, L=64), 4000
    tensor, direct = sizes(env, radar, P)
    cache = tmp_path / "tune.json"
    cache.write_text(json.dumps({"t0_V8_Ns128_L64_b12": [2, 0, 64, 0]}))
    monkeypatch.setenv("RSIM_TUNE_CACHE", str(cache))
    c = device.Context(0)
    assert not _abi.rsim_get_plan(c.h, radar, P, _abi.TIER_FP32).tuned
    assert _abi.rsim_workspace_size(c.h, radar, P, _abi.TIER_FP32) == tensor
    small = device.Context(0, hbm_budget_bytes=tensor - 256)
    plan = _abi.rsim_get_plan(small.h, radar, P, _abi.TIER_FP32)
    assert plan.tuned == 1 and plan.splits == 2 and plan.tile_n == 64
    assert _abi.rsim_autotune(c.h, radar, P, _abi.TIER_FP32).tuned == 1
    assert any(key.startswith("t6_V8_Ns128_L64") for key in json.loads(cache.read_text()))
    assert _abi.rsim_get_plan(c.h, radar, P, _abi.TIER_FP32).grid > 0  # the tensor-core form
    small.close(), c.close()


def test_tuning_within_a_bound(env):
    """A budget that holds the default plan of the tensor-core form, but not the candidates with
    more splits: tuning takes the candidates that fit."""
    torch, _abi, device, _ = env
    radar, P = Radar(M=2, N=4, Ns=128, L=64), 4000
    tensor, direct = sizes(env, radar, P)
    c = device.Context(0, hbm_budget_bytes=tensor + 4096)
    plan = _abi.rsim_autotune(c.h, radar, P, _abi.TIER_FP32)
    assert plan.tuned == 1 and plan.as_dict() == _abi.rsim_get_plan(c.h, radar, P, _abi.TIER_FP32).as_dict()
    assert direct < _abi.rsim_workspace_size(c.h, radar, P, _abi.TIER_FP32) <= tensor + 4096
    c.close()


def test_capture_in_a_workspace_of_the_cuda_core_sum(env):
    """A call captured in a workspace that holds the CUDA-core sum but not the tensor-core form:
    it cannot grow during the capture, and the call takes the CUDA-core sum."""
    torch, _abi, device, ctx = env
    radar = Radar(M=1, N=1, Ns=64, L=64)
    px = synth.random_frame(radar, 100, 96, seed=21, mask_frac=0.2)
    tensor, direct = sizes(env, radar, px.P)
    d, cube = device.upload(px), torch.zeros((1, 64, 64), dtype=torch.complex64, device="cuda")
    ctx.synth(radar, device.upload(synth.random_frame(radar, 10, 10, seed=22)), "fp32")  # loads the kernels
    c = device.Context(0)
    # 2 MiB of row transforms: a workspace of 3 MiB
    big = Radar(M=1, N=1, Ns=512, L=512)
    assert direct < 2 << 20 and tensor > 4 << 20
    _abi.rsim_range_doppler(c.h, big, [torch.zeros((1, 512, 512), dtype=torch.complex64, device="cuda")],
                            torch.empty((1, 512, 512), device="cuda"), torch.empty(1, device="cuda"))
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        c.synth(radar, d, "fp32", cube=cube, stream=s)
    g.replay()
    torch.cuda.synchronize()
    assert c.sync_status() == _abi.OK
    assert oracle.rel_l2(cube.cpu().numpy(), oracle.cube_separable(radar, px)) <= DIRECT_BAR
    # outside a capture the workspace grows and the tensor-core form runs
    got = c.synth(radar, d, "fp32").cpu().numpy()
    assert np.array_equal(got, ctx.synth(radar, d, "fp32").cpu().numpy())
    c.close()


def test_host_call_after_the_tensor_core_form_filled_the_budget(env):
    """The staging buffer of rsim_synth_host counts against the budget with the workspace.  A
    workspace that an FP32 call on the tensor cores grew beyond the CUDA-core sum's is given
    back where the staging would otherwise be refused."""
    torch, _abi, device, ctx = env
    radar = Radar(M=2, N=4, Ns=64, L=64)
    px = synth.random_frame(radar, 80, 60, seed=31, mask_frac=0.3)
    tensor, direct = sizes(env, radar, px.P)
    cube_bytes = 8 * 64 * 64 * 8
    assert direct + direct // 8 + (1 << 20) + cube_bytes < tensor
    c = device.Context(0, hbm_budget_bytes=tensor + 4096)
    d = device.upload(px)
    want = c.synth(radar, d, "fp32").cpu().numpy()
    host = {k: torch.from_numpy(np.ascontiguousarray(a)).pin_memory() for k, a in zip(device.FIELDS, px.arrays())}
    for tier, bar in (("nufft", 2e-5), ("fp32", FP32_BAR)):
        got = c.synth_host(radar, host, tier)
        assert c.sync_status() == _abi.OK
        assert oracle.rel_l2(got.numpy(), oracle.cube_separable(radar, px)) <= bar
    assert np.array_equal(got.numpy(), want)
    c.close()


def test_staging_beyond_the_budget_stays_refused(env):
    """A staging buffer that does not fit beside the workspace other calls need is refused."""
    torch, _abi, device, ctx = env
    radar = Radar(M=2, N=4, Ns=64, L=64)
    px = synth.random_frame(radar, 80, 60, seed=32, mask_frac=0.3)
    need = _abi.rsim_workspace_size(ctx.h, radar, px.P, _abi.TIER_SPLIT_FP16)
    c = device.Context(0, hbm_budget_bytes=need + 4096)
    c.synth(radar, device.upload(px), "split_fp16")
    c.synth(radar, device.upload(px), "fp32")
    host = {k: torch.from_numpy(np.ascontiguousarray(a)).pin_memory() for k, a in zip(device.FIELDS, px.arrays())}
    with pytest.raises(_abi.RsimError) as e:
        c.synth_host(radar, host, "split_fp16")
    assert e.value.status == _abi.ERR_BUDGET
    c.close()


def test_served_requests_without_memory_for_the_operand_images(env):
    """A request whose operand images cannot be allocated runs as the CUDA-core sum; one of a
    tier that has nothing else fails with OOM, and the server goes on."""
    torch, _abi, device, _ = env
    radar = Radar(M=2, N=4, Ns=64, L=64)
    px = synth.random_frame(radar, 80, 60, seed=71, mask_frac=0.3)
    tensor, direct = sizes(env, radar, px.P)
    d = device.upload(px)
    cubes = [torch.zeros((8, 64, 64), dtype=torch.complex64, device="cuda") for _ in range(3)]
    c = device.Context(0)
    srv = _abi.rsim_server_create(c.h, slots=2, hbm_budget_bytes=2 * tensor)
    _abi.rsim_selftest_alloc_limit(c.h, tensor - 256)
    tickets = [_abi.rsim_server_submit(srv, _abi.make_request(radar, d, tier, cube))
               for tier, cube in zip((_abi.TIER_FP32, _abi.TIER_SPLIT_FP16, _abi.TIER_FP32), cubes)]
    status = [_abi.rsim_server_wait(srv, t, -1) for t in tickets]
    stats = _abi.rsim_server_stats_get(srv)
    _abi.rsim_server_destroy(srv)
    split = _abi.rsim_workspace_size(c.h, radar, px.P, _abi.TIER_SPLIT_FP16)
    assert status == [_abi.OK, _abi.ERR_OOM if split > tensor - 256 else _abi.OK, _abi.OK]
    assert stats.failed == (1 if split > tensor - 256 else 0)
    assert stats.peak_reserved_bytes < 2 * tensor
    ref = oracle.cube_separable(radar, px)
    for cube in (cubes[0], cubes[2]):
        assert oracle.rel_l2(cube.cpu().numpy(), ref) <= DIRECT_BAR
    small = device.Context(0, hbm_budget_bytes=tensor - 256)
    assert np.array_equal(cubes[0].cpu().numpy(), small.synth(radar, d, "fp32").cpu().numpy())
    small.close(), c.close()


def test_a_batch_in_parts_without_memory_for_the_largest(env):
    """A batch that goes in parts, the second of which cannot have its workspace: the whole batch
    runs as the CUDA-core sum, instead of failing after the first part."""
    torch, _abi, device, _ = env
    radar = Radar(M=2, N=4, Ns=64, L=64)
    frames = [synth.random_frame(radar, a, e, seed=81 + a, mask_frac=0.2) for a, e in ((25, 20), (80, 60))]
    tensor, direct = sizes(env, radar, 4800)
    c = device.Context(0, hbm_budget_bytes=tensor + 4096)
    _abi.rsim_selftest_alloc_limit(c.h, tensor - 256)
    pxs = [device.upload(f) for f in frames]
    cubes = c.synth_batch(radar, pxs, "fp32")
    assert c.sync_status() == _abi.OK
    for f, cube in zip(frames, cubes):
        assert oracle.rel_l2(cube.cpu().numpy(), oracle.cube_separable(radar, f)) <= DIRECT_BAR
    _abi.rsim_selftest_alloc_limit(c.h, 0)
    for f, px, cube in zip(frames, pxs, c.synth_batch(radar, pxs, "fp32")):
        assert oracle.rel_l2(cube.cpu().numpy(), oracle.cube_separable(radar, f)) <= FP32_BAR
    _abi.rsim_selftest_alloc_limit(c.h, 1)
    with pytest.raises(_abi.RsimError) as e:  # a batch that nothing holds
        c.synth_batch(radar, [device.upload(synth.random_frame(radar, 80, 60, seed=s)) for s in range(9)], "split_fp16")
    assert e.value.status in (_abi.ERR_OOM, _abi.ERR_BUDGET)
    c.close()


def test_tuning_without_memory_for_the_operand_images(env):
    """Where the tensor-core form's workspace cannot be had, tuning tunes the CUDA-core sum that
    calls then run; where only the larger candidates' cannot, it passes them over."""
    torch, _abi, device, _ = env
    radar, P = Radar(M=2, N=4, Ns=128, L=64), 4000
    tensor, direct = sizes(env, radar, P)
    for limit, form in ((tensor - 256, "direct"), (tensor + tensor // 8 + (1 << 20), "tensor")):
        c = device.Context(0)
        _abi.rsim_selftest_alloc_limit(c.h, limit)
        plan = _abi.rsim_autotune(c.h, radar, P, _abi.TIER_FP32)
        assert plan.tuned == 1 and (plan.grid > 0) == (form == "tensor")
        px = synth.random_frame(radar, 80, 50, seed=91, mask_frac=0.2)
        got = c.synth(radar, device.upload(px), "fp32").cpu().numpy()
        assert c.sync_status() == _abi.OK
        assert oracle.rel_l2(got, oracle.cube_separable(radar, px)) <= (FP32_BAR if form == "tensor" else DIRECT_BAR)
        c.close()


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("V,Ns,L,n_az,n_el,splits,tile_n", [
    (1, 128, 64, 256, 256, 8, 128),   # 65,536 pixels, whole tiles
    (3, 70, 33, 251, 130, 4, 128),    # ragged rows, columns and pixels
    (2, 200, 96, 120, 100, 7, 64),    # the narrower tile
    (1, 64, 64, 90, 60, 1, 0),        # one split: written directly
])
def test_the_cuda_core_sum(env, dtype, V, Ns, L, n_az, n_el, splits, tile_n):
    """The CUDA-core sum, pinned, at sizes that the tensor cores take by default: alone, written
    as complex128, and as a batch of uneven valid counts with the same bits."""
    torch, _abi, device, _ = env
    radar = Radar(M=V, N=1, Ns=Ns, L=L)
    frames = [synth.random_frame(radar, n_az, n_el, seed=41 + i, mask_frac=m, dtype=dtype) for i, m in enumerate((0.3, 0.0))]
    c = device.Context(0)
    _abi.rsim_set_plan(c.h, radar, frames[0].P, _abi.TIER_FP32, splits=splits, tile_n=tile_n)
    pxs = [device.upload(f) for f in frames]
    refs = [oracle.cube_separable(radar, f) for f in frames]
    alone = [c.synth(radar, px, "fp32").cpu().numpy() for px in pxs]
    for got, ref in zip(alone, refs):
        assert oracle.rel_l2(got, ref) <= DIRECT_BAR
    wide = c.synth(radar, pxs[0], "fp32", out_dtype="complex128").cpu().numpy()
    assert np.array_equal(wide.astype(np.complex64), alone[0])
    for got, want in zip(c.synth_batch(radar, pxs, "fp32"), alone):
        assert np.array_equal(got.cpu().numpy(), want)
    assert c.sync_status() == _abi.OK
    c.close()


def test_static_entry_falls_back_to_the_cuda_core_sum(env):
    """80,000 pixels and 64 columns: 82 MB of operand images pass the static workspace, the
    CUDA-core sum's scratch does not.  The result is that of a context whose budget leaves the
    same sum, bit for bit."""
    torch, _abi, device, _ = env
    radar = Radar(M=1, N=1, Ns=64, L=64)
    px = synth.random_frame(radar, 400, 200, seed=51, mask_frac=0.1)
    tensor, direct = sizes(env, radar, px.P)
    assert direct < 64 << 20 < tensor
    d = device.upload(px)
    cube = torch.empty((1, 64, 64), dtype=torch.complex64, device="cuda")
    assert _abi.rsim_synth_static(radar, d, _abi.TIER_FP32, cube) == _abi.OK, _abi.last_error()
    torch.cuda.synchronize()
    small = device.Context(0, hbm_budget_bytes=tensor - 256)
    assert np.array_equal(cube.cpu().numpy(), small.synth(radar, d, "fp32").cpu().numpy())
    assert oracle.rel_l2(cube.cpu().numpy(), oracle.cube_separable(radar, px)) <= DIRECT_BAR
    small.close()


def test_uneven_batch_across_the_pixel_limit(env):
    """A batch takes the form and the plan of its largest frame: frames of fewer than 128 pixels
    run on the tensor cores there, on the CUDA cores alone.  Each within the tier's bar, and the
    largest with the bits it has alone."""
    torch, _abi, device, ctx = env
    radar = Radar(M=2, N=2, Ns=64, L=24)
    frames = [synth.random_frame(radar, a, e, seed=60 + i, mask_frac=0.0)
              for i, (a, e) in enumerate([(5, 3), (16, 8), (1, 1), (127, 1), (60, 50), (43, 3)])]
    pxs = [device.upload(f) for f in frames]
    cubes = [x.cpu().numpy() for x in ctx.synth_batch(radar, pxs, "fp32")]
    assert ctx.sync_status() == _abi.OK
    for f, got in zip(frames, cubes):
        assert oracle.rel_l2(got, oracle.cube_separable(radar, f)) <= DIRECT_BAR
    assert np.array_equal(cubes[4], ctx.synth(radar, pxs[4], "fp32").cpu().numpy())
