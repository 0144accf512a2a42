"""One frame through the windowed gather and through the kernel that reads the
integrand from L2 (PAT_FLAG_NO_WINDOW): the same bits for every kind of delay
and weight, tile size and format, with windows on both sides of each slot size
(128, 192, 288 and 384 rows, and longer ones that take the other kernel), one
ragged segment of sensors (the gather writes the image) and two."""
import numpy as np
import pytest

from paper_1501_03869_gb300 import BP, _lib, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _handle(mode, tile, ns, nt, extra, shape=(64, 70)):
    rng = np.random.default_rng(5)
    dx = 0.2e-3
    speed = (1500.0 + 900.0 * synth.smooth_field(shape, 4.0, rng)).astype(np.float32)
    hi = (np.array(shape[::-1], dtype=float) - 1) * dx
    sensors = np.zeros((ns, 3))
    sensors[:, 0] = np.where(np.arange(ns) % 2, hi[0], 0.0)
    sensors[:, 1] = (np.floor(rng.uniform(0.0, 1.0, ns) * (shape[0] - 2)) + 0.37) * dx  # off the nodes
    dt = 1.2 * float(np.linalg.norm(hi)) / 1500.0 / nt
    flags = extra | (_lib.PAT_FLAG_TILE_256 if tile == 256 else _lib.PAT_FLAG_TILE_128)
    if mode.startswith("constant"):
        bp = BP.constant(1560.0, shape, dx, np.zeros(3), sensors, dt, nt, flags=flags)
    else:
        bp = BP(speed, dx, np.zeros(3), sensors, dt, nt, flags=flags)
    if mode.endswith("solid"):
        normals = np.zeros((ns, 3))
        normals[:, 0] = np.where(np.arange(ns) % 2, -1.0, 1.0)
        bp.set_solid_angle(normals, np.full(ns, dx), 2 * np.pi)
    return bp


@pytest.mark.parametrize("nt", [600, 1000, 1199, 1600, 2000, 2400])
@pytest.mark.parametrize("tile", [128, 256])
@pytest.mark.parametrize("mode", ["table", "constant", "table_solid", "constant_solid"])
def test_windowed_equals_unwindowed(mode, tile, nt):
    for ns in (37, 70):
        g = torch.Generator("cuda").manual_seed(nt + ns)
        x = torch.randn(1, ns, nt, generator=g, device="cuda")
        sc = x.abs().amax(dim=2).contiguous()
        with _handle(mode, tile, ns, nt, 0) as a, _handle(mode, tile, ns, nt, _lib.PAT_FLAG_NO_WINDOW) as b:
            for dtype in (torch.float32, torch.bfloat16, torch.float16):
                s = None if dtype == torch.float32 else sc
                sig = x if s is None else (x / sc[..., None]).to(dtype).contiguous()
                ia, ib = a.reconstruct(sig, scales=s), b.reconstruct(sig, scales=s)
                assert torch.isfinite(ia).all() and bool((ia != 0).any())
                assert torch.equal(ia.view(torch.int32), ib.view(torch.int32)), (ns, dtype, a.info["window"])
            a.sync()
            b.sync()


@pytest.mark.parametrize("imaged", ["few", "scattered", "none but one"])
@pytest.mark.parametrize("ns", [40, 130])
def test_image_outside_the_mask_is_cleared(ns, imaged):
    """One segment (the gather clears) and three (the reduction does), with many
    more runs outside the mask than warps, and with a few long ones."""
    shape, dx, nt = (180, 200), 0.2e-3, 500
    mask = np.zeros(shape, dtype=np.uint8)
    if imaged == "few":
        mask[85:95, 90:110] = 1
    elif imaged == "scattered":
        mask[::2, ::3] = 1
    else:
        mask[-1, -1] = 1
    rng = np.random.default_rng(3)
    sensors = np.zeros((ns, 3))
    sensors[:, 1] = rng.uniform(0.0, 1.0, ns) * (shape[0] - 1) * dx
    with BP.constant(1500.0, shape, dx, np.zeros(3), sensors, 1.2 * 0.054 / 1500.0 / nt, nt, mask=mask) as bp:
        x = torch.randn(2, ns, nt, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
        out = torch.full(bp.out_shape(2), 7.0, device="cuda")
        bp.reconstruct(x, out=out)
        bp.sync()
        outside = torch.from_numpy(mask == 0).cuda()
        assert bool((out[:, outside] == 0).all()) and bool((out[:, ~outside] != 7.0).all())
        for f in range(2):
            one = bp.reconstruct(x[f:f + 1], out=torch.full(bp.out_shape(1), 7.0, device="cuda"))
            assert torch.equal(one[0].view(torch.int32), out[f].view(torch.int32))


@pytest.mark.parametrize("nt", [2000, 4500, 6000, 8500])
@pytest.mark.parametrize("tile", [128, 256])
@pytest.mark.parametrize("mode", ["table", "constant", "table_solid", "constant_solid"])
def test_windowed_equals_unwindowed_in_full_waves(mode, tile, nt):
    """Three segments of enough tiles that the windowed kernel takes every form
    that has a slot (the smaller launches above leave some to the other kernel)."""
    ns, shape = 130, (256, 256)
    x = torch.randn(1, ns, nt, generator=torch.Generator("cuda").manual_seed(nt), device="cuda")
    gpu = 0 if mode.startswith("constant") else _lib.PAT_FLAG_GPU_TABLE
    with _handle(mode, tile, ns, nt, gpu, shape) as a, \
            _handle(mode, tile, ns, nt, gpu | _lib.PAT_FLAG_NO_WINDOW, shape) as b:
        assert a.info["n_tiles"] * a.info["split"] == (1536 if tile == 128 else 768)
        sc = x.abs().amax(dim=2).contiguous()
        for dtype in (torch.float32, torch.float16):
            s = None if dtype == torch.float32 else sc
            sig = x if s is None else (x / sc[..., None]).to(dtype).contiguous()
            ia, ib = a.reconstruct(sig, scales=s), b.reconstruct(sig, scales=s)
            assert torch.isfinite(ia).all() and bool((ia != 0).any())
            assert torch.equal(ia.view(torch.int32), ib.view(torch.int32)), (dtype, a.info["window"])
        a.sync()
        b.sync()
