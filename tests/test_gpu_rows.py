"""The batched gather (4 to 32 frames per unit): every frame of a batch has the
bits of the same frame alone (the single-frame kernels, which the parity tests
hold to the oracle), at the edges of its groupings -- frame counts around each
unit size, ragged last segments, groups cut down to one or two sensors by long
windows, odd record lengths, whole-tile units -- and a frame that holds
infinities and NaN does not touch the others."""
import numpy as np
import pytest

from paper_1501_03869_gb300 import BP, _lib, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _handle(shape, ns, nt, tile, mode):
    rng = np.random.default_rng([len(shape), ns, nt])
    dx = 0.2e-3
    origin = np.zeros(3)
    speed = (1500.0 + 900.0 * synth.smooth_field(shape, 4.0, rng)).astype(np.float32)
    hi = (np.array(shape[::-1], dtype=float) - 1) * dx
    sensors = np.zeros((ns, 3))
    sensors[:, :len(shape)] = rng.uniform(0.0, 1.0, (ns, len(shape))) * hi
    sensors[:, 0] = np.where(np.arange(ns) % 2, hi[0], 0.0)  # on two faces
    dt = 1.2 * float(np.linalg.norm(hi)) / 1500.0 / nt
    mask = None if len(shape) == 3 else (rng.uniform(size=shape) < 0.9).astype(np.uint8)
    flags = _lib.PAT_FLAG_TILE_256 if tile == 256 else _lib.PAT_FLAG_TILE_128
    if mode == "constant":
        return BP.constant(1560.0, shape, dx, origin, sensors, dt, nt, mask=mask, flags=flags)
    bp = BP(speed, dx, origin, sensors, dt, nt, mask=mask, flags=flags | _lib.PAT_FLAG_GPU_TABLE)
    if mode == "solid":
        normals = np.zeros((ns, 3))
        normals[:, 0] = np.where(np.arange(ns) % 2, -1.0, 1.0)
        # off the nodes, so that no pixel sits on a sensor
        bp.close()
        sensors[:, 1] = np.clip(sensors[:, 1], 0.3 * dx, hi[1] - 0.3 * dx)
        sensors[:, 1] = (np.floor(sensors[:, 1] / dx) + 0.37) * dx
        sensors[:, 1] = np.minimum(sensors[:, 1], hi[1] - 0.63 * dx)
        bp = BP(speed, dx, origin, sensors, dt, nt, mask=mask, flags=flags | _lib.PAT_FLAG_GPU_TABLE)
        bp.set_solid_angle(normals, np.full(ns, dx), 2 * np.pi)
    return bp


def _signals(frames, ns, nt, dtype, seed=1):
    g = torch.Generator("cuda").manual_seed(seed)
    x = torch.randn(frames, ns, nt, generator=g, device="cuda")
    if dtype == "f32":
        return x, None
    sc = x.abs().amax(dim=2).contiguous()
    return (x / sc[..., None]).to(torch.bfloat16 if dtype == "bf16" else torch.float16).contiguous(), sc


def _check(bp, sig, sc, frames):
    got = bp.reconstruct(sig, scales=sc).cpu().numpy()
    for f in frames:
        one = bp.reconstruct(sig[f:f + 1], scales=None if sc is None else sc[f:f + 1]).cpu().numpy()
        assert np.array_equal(got[f], one[0], equal_nan=True), f"frame {f}"
    bp.sync()


@pytest.mark.parametrize("mode", ["table", "constant", "solid"])
@pytest.mark.parametrize("tile", [128, 256])
@pytest.mark.parametrize("dtype", ["f32", "bf16", "f16"])
def test_frame_counts(dtype, tile, mode):
    """Every unit size (4, 8, 16, 32 frames), full and padded, three segments
    of which the last holds 22 sensors, odd record length."""
    bp = _handle((72, 80), 150, 301, tile, mode)
    with bp:
        for n in (4, 5, 8, 9, 16, 17, 25, 32, 33, 48, 57):
            sig, sc = _signals(n, 150, 301, dtype, n)
            _check(bp, sig, sc, sorted({0, 1, n // 2, n - 2, n - 1}))


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("tile", [128, 256])
def test_long_windows(tile, dtype):
    """Windows of several hundred samples: few sensors fit the ring together."""
    bp = _handle((72, 80), 67, 4001, tile, "table")
    with bp:
        assert bp.info["window"] > 500
        for n in (6, 8, 16, 32):
            sig, sc = _signals(n, 67, 4001, dtype, n)
            _check(bp, sig, sc, (0, n // 2, n - 1))


@pytest.mark.parametrize("frames", [8, 16])
@pytest.mark.parametrize("dtype", ["f32", "f16"])
def test_whole_tile_units(dtype, frames):
    """Enough tiles that a unit takes all segments and keeps the running sum."""
    bp = _handle((72, 96, 96), 131, 200, 128, "table")
    with bp:
        assert bp.info["n_tiles"] >= 8 * 4 * 152 and bp.info["split"] == 3
        sig, sc = _signals(frames, 131, 200, dtype)
        _check(bp, sig, sc, (0, 5, frames - 1))


def test_non_finite_frame_stays_alone():
    bp = _handle((72, 80), 150, 301, 128, "table")
    with bp:
        sig, _ = _signals(32, 150, 301, "f32")
        sig[3, 10, 40:60] = float("inf")
        sig[3, 11, 100] = float("nan")
        _check(bp, sig, None, (2, 3, 4, 31))


@pytest.mark.parametrize("reserved,frames", [(64, 64), (32, 32), (16, 16), (40, 32), (64, 17), (24, 8)])
def test_reserved_handle_allocates_nothing_for_shorter_rows(reserved, frames):
    """A small launch takes shorter rows than its frame count allows; what
    reserve() set aside for the longest ones holds it, so that its first call
    can already be under capture."""
    with _handle((72, 80), 64, 301, 128, "table") as bp, _handle((72, 80), 64, 301, 128, "table") as ref:
        sig, _ = _signals(frames, 64, 301, "f32")
        want = ref.reconstruct(sig)
        bp.reserve(reserved)
        out = torch.empty_like(want)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            bp.reconstruct(sig, out=out)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out.view(torch.int32), want.view(torch.int32))
        bp.sync()
        ref.sync()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("tile", [128, 256])
def test_page_locked_signals(tile, dtype):
    """Signals read over the host link, for which rows of 4 hold the gather's
    start back: the bits of device signals, call after call."""
    with _handle((72, 80), 150, 301, tile, "table") as bp:
        for n in (4, 6, 8, 12, 4):
            sig, sc = _signals(n, 150, 301, dtype, n)
            want = bp.reconstruct(sig, scales=sc).cpu()
            bp.sync()
            host = (sig if sc is None else sig.view(torch.int16)).cpu().pin_memory().numpy()
            out = torch.full_like(want, 7.0).pin_memory()
            bp.reconstruct_host(host if sc is None else host.view(np.uint16), dtype=dtype,
                                scales=None if sc is None else sc.cpu().pin_memory().numpy(), out=out.numpy())
            assert torch.equal(out.view(torch.int32), want.view(torch.int32))
