"""Plans and handles whose batches take rows of 8 to 32 frames.  Every image has
the bits of the same frames through the handle's own reconstruct() (which the
parity tests hold to the oracle)."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_1501_03869_gb300 import BP, Plan, _lib, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _handle(shape, ns, nt, tile=128, mode="table", weights=None):
    rng = np.random.default_rng([shape[0], shape[1], ns, nt])
    dx = 0.2e-3
    speed = (1500.0 + 900.0 * synth.smooth_field(shape, 4.0, rng)).astype(np.float32)
    hi = (np.array(shape[::-1], dtype=float) - 1) * dx
    sensors = np.zeros((ns, 3))
    sensors[:, 0] = np.where(np.arange(ns) % 2, hi[0], 0.0)
    sensors[:, 1] = (np.floor(rng.uniform(0.0, 1.0, ns) * (shape[0] - 2)) + 0.37) * dx  # off the nodes
    dt = 1.2 * float(np.linalg.norm(hi)) / 1500.0 / nt
    flags = _lib.PAT_FLAG_TILE_256 if tile == 256 else _lib.PAT_FLAG_TILE_128
    if mode == "constant":
        return BP.constant(1560.0, shape, dx, np.zeros(3), sensors, dt, nt, weights=weights, flags=flags)
    return BP(speed, dx, np.zeros(3), sensors, dt, nt, weights=weights, flags=flags | _lib.PAT_FLAG_GPU_TABLE)


def _set_weights(bp, ns):
    normals = np.zeros((ns, 3))
    normals[:, 0] = np.where(np.arange(ns) % 2, -1.0, 1.0)
    bp.set_solid_angle(normals, np.full(ns, 0.2e-3), 2 * np.pi)


def _signals(frames, ns, nt, dtype="f32", seed=1):
    g = torch.Generator("cuda").manual_seed(seed)
    x = torch.randn(frames, ns, nt, generator=g, device="cuda")
    if dtype == "f32":
        return x, None
    sc = x.abs().amax(dim=2).contiguous()
    return (x / sc[..., None]).to(torch.bfloat16 if dtype == "bf16" else torch.float16).contiguous(), sc


def _same(a, b):
    return torch.equal(a.view(torch.int32), b.view(torch.int32))


def _check_plan(bps, frames, dtype="f32", **kw):
    """Executes twice (the second replays the graph where there is one); returns the plan's facts."""
    sig, sc = zip(*[_signals(f, b.n_sensors, b.n_samples, dtype, i) for i, (b, f) in enumerate(zip(bps, frames))])
    sc = None if dtype == "f32" else list(sc)
    want = [b.reconstruct(s, scales=None if sc is None else sc[i]) for i, (b, s) in enumerate(zip(bps, sig))]
    plan = Plan(bps, frames, dtype=dtype, **kw)
    for _ in range(2):
        outs = [torch.full_like(w, 7.0) for w in want]
        plan.execute(list(sig), outs, scales=sc)
        plan.sync()
        assert all(_same(o, w) for o, w in zip(outs, want))
    info = plan.info
    plan.close()
    return info


@pytest.mark.parametrize("kw", [{}, dict(graph=True), dict(autotune=True, graph=True)], ids=["plain", "graph", "tuned"])
@pytest.mark.parametrize("tile,nt", [(128, 17000), (128, 20000), (256, 12000)])
def test_long_windows_of_many_frames(tile, nt, kw):
    """Windows of 1 800 to 2 900 rows: a 32-frame row of them fits no CTA."""
    with _handle((72, 80), 12, nt, tile) as a, _handle((64, 64), 9, 901, tile) as b:
        assert 1800 <= a.info["window"] <= 2900, a.info["window"]
        info = _check_plan([a, b], [32, 48], **kw)
        assert info["fb_mask"] & 32 == 0


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_autotune_where_reconstruct_falls_back(dtype):
    """The tuner takes the frames per unit that reconstruct() settles on."""
    with _handle((128, 136), 260, 30000) as bp:
        # enough units for rows of 32 frames, of which no window fits a CTA
        assert bp.info["n_tiles"] * bp.info["split"] >= 4 * 152 and bp.info["window"] > 1752
        sig, sc = _signals(32, 260, 30000, dtype)
        want = bp.reconstruct(sig, scales=sc)
        bp.autotune(sig, scales=sc)
        assert _same(bp.reconstruct(sig, scales=sc), want)
        bp.sync()


@pytest.mark.parametrize("kw", [{}, dict(graph=True), dict(autotune=True, graph=True)], ids=["plain", "graph", "tuned"])
@pytest.mark.parametrize("dtype", ["f32", "f16"])
def test_rows_follow_the_units_of_a_class(dtype, kw):
    """32-frame rows only where their units fill the chip: a small instance
    takes 8-frame rows alone, and the long ones beside enough others."""
    with _handle((72, 80), 64, 301) as small, _handle((160, 160), 256, 401) as big, \
            _handle((152, 160), 250, 399) as other:
        assert small.info["n_tiles"] < 152
        assert _check_plan([small], [32], dtype, **kw)["fb_mask"] == 8
        assert _check_plan([small, big], [8, 32], dtype, **kw)["fb_mask"] == 8 | 32
        assert _check_plan([small, big, other], [32, 32, 48], dtype, **kw)["fb_mask"] == 16 | 32


_TUNED = """
import sys
sys.path.insert(0, {root!r})
sys.path.insert(0, {root!r} + "/tests")
import test_gpu_plan_rows as t
with t._handle((72, 80), 12, 9001) as a:
    info = t._check_plan([a], [32], autotune=True, graph=True)
    assert info["tuned"] == 1
    print("ok", info["sensors_per_stage"], info["smem_budget_kb"], a.info["window"])
"""


def test_stored_shapes_that_do_not_fit(tmp_path):
    """A stored launch shape of another kernel or one that holds no group is
    tuned again, and a stored shape that fits is used."""
    path = tmp_path / "shapes"

    def run():
        r = subprocess.run([sys.executable, "-c", _TUNED.format(root=ROOT)], capture_output=True, text=True,
                           env=dict(os.environ, PAT_TUNE_CACHE=str(path)), timeout=300)
        assert r.returncode == 0 and "ok" in r.stdout, r.stderr[-2000:]
        return path.read_text().splitlines()

    first = run()
    assert len(first) == 1
    key, s, b = first[0].split()
    assert run() == first  # used, not tuned again
    for bad in ("8 1", "24 200", "-4 100", "8 -5", "0 55", "64 200"):
        path.write_text(f"{key} {bad}\n")
        assert len(run()) == 2, bad
    # as the staged kernel's shapes were stored
    assert key.startswith("rows1.")
    path.write_text(f"{key[len('rows1.'):]} 8 55\n")
    assert len(run()) == 2


@pytest.mark.parametrize("frames", [12, 48])
def test_weights_set_between_preprocess_and_gather(frames):
    """The gather takes the rows that preprocess() laid out, whatever rows the
    handle's new mode would choose.  Sensor weights of one: preprocess() puts
    the weights of its time into the multipliers."""
    ones = np.ones(70, dtype=np.float32)
    with _handle((256, 256), 70, 401, mode="constant", weights=ones) as bp, \
            _handle((256, 256), 70, 401, mode="constant") as ref:
        sig, _ = _signals(frames, 70, 401)
        _set_weights(ref, 70)
        want = ref.reconstruct(sig)
        bp.preprocess(sig)
        _set_weights(bp, 70)
        out = torch.empty_like(want)
        bp.gather(frames, out)
        bp.sync()
        assert _same(out, want)


def test_noalloc_at_the_scratch_limit():
    """32 frames that need exactly the 16 MiB in rows of 8: 36 tiles, 50 sensors,
    2 528 padded samples.  The launch takes rows of 4 (36 tiles fill no chip),
    which must not need more."""
    with _handle((64, 72), 50, 2527) as bp:
        assert bp.info["n_tiles"] == 36 and bp.info["n_samples_pad"] == 2528 and bp.info["tile_pix"] == 128
        sig, _ = _signals(32, 50, 2527)
        want = bp.reconstruct(sig)
        out = torch.full_like(want, 7.0)
        bp.reconstruct_noalloc(sig, out)
        bp.sync()
        assert _same(out, want)
        more, _ = _signals(33, 50, 2527)
        with pytest.raises(Exception, match="scratch"):
            bp.reconstruct_noalloc(more, torch.empty(bp.out_shape(33), device="cuda"))


@pytest.mark.parametrize("frames,nt,budget", [(8, 2001, 72), (8, 6001, 110), (8, 14000, 200), (5, 6001, 110)])
def test_plans_widen_the_ring_for_long_windows(frames, nt, budget):
    """Windows of 240, 728 and 1 672 rows of 8 frames, 728 of 4: the budget
    grows before a ring gets down to one group."""
    with _handle((72, 80), 12, nt) as bp:
        info = _check_plan([bp], [frames])
        kb = info["smem_budget_kb"]
        assert kb == budget if budget < 200 else kb >= budget, (kb, bp.info["window"])


@pytest.mark.parametrize("frames", [4, 16, 23, 32])
@pytest.mark.parametrize("nt", [9001, 17000, 26000, 32000])
def test_reserved_handle_allocates_nothing_for_long_windows(frames, nt):
    """1 072 to 3 912 rows per window: rows of 16 down to single frames, whose
    partial sums take the most; every frame as through the kernels for one
    frame, first under capture, then through the no-allocation path."""
    with _handle((72, 80), 12, nt) as bp, _handle((72, 80), 12, nt) as ref:
        sig, _ = _signals(frames, 12, nt)
        want = torch.cat([ref.reconstruct(sig[f:f + 1]) for f in range(frames)])
        bp.reserve(32)
        out = torch.empty_like(want)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            bp.reconstruct(sig, out=out)
        graph.replay()
        torch.cuda.synchronize()
        assert _same(out, want)
        few = sig[:4]
        out = torch.full_like(want[:4], 7.0)
        bp.reconstruct_noalloc(few, out)
        bp.sync()
        assert _same(out, want[:4])


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("tile", [128, 256])
def test_shapes_of_computed_delays(tile, dtype):
    """Constant speed: 16-bit frames take rows of 8 where FP32 takes 16, and
    8-frame rows get the shared memory of two CTAs per SM, whose registers hold
    what three would spill; stored delays keep three."""
    with _handle((160, 160), 256, 401, tile, "constant") as bp, _handle((160, 160), 256, 401, tile) as table:
        assert _check_plan([bp], [48], dtype)["fb_mask"] == (16 if dtype == "f32" else 8)
        info = _check_plan([bp], [8], dtype)
        assert info["smem_budget_kb"] == 110 and info["sensors_per_stage"] == (8 if tile == 128 else 4)
        info = _check_plan([table], [8], dtype)
        assert info["smem_budget_kb"] == 72
        _set_weights(bp, 256)
        assert _check_plan([bp], [48], dtype)["fb_mask"] == (16 if dtype == "f32" else 8)
        assert _check_plan([bp], [24], dtype)["smem_budget_kb"] == 110


def test_one_long_record_leaves_a_class_its_ctas():
    """The budget of a class follows its instances' units, not its longest window."""
    with _handle((160, 160), 130, 401) as many, _handle((24, 24), 8, 6001) as long:
        assert long.info["window"] > 512
        info = _check_plan([many, long], [8, 8])
        assert info["n_classes"] == 1 and info["smem_budget_kb"] == 72


@pytest.mark.parametrize("mode", ["table", "constant"])
@pytest.mark.parametrize("frames", [5, 8, 40])
def test_one_long_record_leaves_the_groups_of_the_others(mode, frames):
    """Groups of sensors follow the windows of each tile: an instance whose
    windows fill a third of the ring or more does not cut those of the others."""
    with _handle((96, 100), 130, 401, 128, mode) as many, _handle((24, 24), 9, 6001, 128, mode) as long:
        one = _check_plan([many], [frames])
        both = _check_plan([many, long], [frames, frames])
        assert both["fb_mask"] == one["fb_mask"] and both["sensors_per_stage"] == one["sensors_per_stage"]
