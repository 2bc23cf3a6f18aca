"""Edges of the steps that work on units of 32 x 8 pixels, against the oracle at the parity
tolerances: units with more coarse cells than they have numbers, cells outside a unit's key
window, grids of no more than 1024 cells an axis (where points leave the grid), float32 depths
beyond the range of the grid evaluation of the consistency step, one cell raised by every point,
image sizes one pixel to each side of the units' and tiles' edges, and the static entry's tables
after frames of the other variant."""
import numpy as np
import pytest

from paper_2602_01035_gb300 import scenes as S
from parity import compare, run_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _check(oracle_mod, rig, fr, **params):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_01035_gb300 import fuseflow
    ff = fuseflow.FuseFlow(rig, **params)
    try:
        gpu = run_gpu(ff, fr, torch)
        again = run_gpu(ff, fr, torch, with_trace=False)
    finally:
        ff.close()
    assert gpu["status"] == fuseflow.FUSEFLOW_OK, gpu["stats"]
    for k, v in gpu["cells"].items():                      # reproducible, traced or not
        assert np.array_equal(v, again["cells"][k], equal_nan=v.dtype.kind == "f"), k
    orc = oracle_mod.fuse_frame(rig, fr, {k: v for k, v in params.items() if k != "max_cells"})
    return compare(gpu, orc, oracle_mod), gpu


def _scattered(rig, seed, lo, hi, dtype=np.uint16):
    rng = np.random.default_rng(seed)
    shape = [(c.height, c.width) for c in rig.cameras]
    z = [rng.uniform(lo, hi, size=s).astype(dtype) for s in shape]
    return S.Frame(z, [rng.uniform(0.55, 1.0, size=s).astype(np.float32) for s in shape],
                   [rng.integers(0, 256, size=s + (3,), dtype=np.uint8) for s in shape])


@pytest.mark.parametrize("coarse,level", [
    (0.32, 2),      # more than 64 coarse cells in a unit, all in one window
    (0.015, 1),     # points more than 512 cells apart in a unit
    (0.32, 10),     # 1024 cells an axis: every cell in the window
    (0.32, 14),     # 64 cells an axis: points leave the grid
])
def test_scattered_units(oracle_mod, coarse, level):
    rig = S.tiny_rig(n=3, width=71, height=35, fx=60.0, fy=60.0)
    rep, gpu = _check(oracle_mod, rig, _scattered(rig, 5, 500, 40000), coarse_cell_m=coarse, max_level=level, n_min=2)
    assert rep["n_points_compared"] > 0.3 * gpu["stats"]["n_gated"] or level == 14
    assert (gpu["stats"]["n_out_of_range"] > 0) == (level == 14)


@pytest.mark.parametrize("coarse", [0.32, 8.0])
def test_float_depths_beyond_the_grid_range(oracle_mod, coarse):
    rig = S.tiny_rig(n=4, width=64, height=40, depth_format="f32", depth_scale=1.0, fx=60.0, fy=60.0)
    rep, gpu = _check(oracle_mod, rig, _scattered(rig, 6, 1.0, 100.0, np.float32), coarse_cell_m=coarse, max_level=1)
    assert rep["n_points_compared"] > 0.5 * gpu["stats"]["n_gated"]


@pytest.mark.parametrize("w,h", [(31, 7), (32, 8), (33, 9), (65, 17), (1, 16), (64, 33)])
def test_sizes_around_units(oracle_mod, w, h):
    rig = S.tiny_rig(n=3, width=w, height=h, fx=40.0, fy=40.0)
    _check(oracle_mod, rig, S.random_frame(rig, seed=7), n_min=2)


@pytest.mark.parametrize("equal", [False, True])
def test_representative_of_one_crowded_cell(oracle_mod, equal):
    """One cell holds every point, in one image after another of rising confidence (or all of
    one): each of tens of thousands of points raises the cell's record."""
    rig = S.tiny_rig(n=4, width=160, height=120, spread_deg=90.0)
    fr = S.random_frame(rig, seed=9)
    for c in rig.cameras:                                  # the scene to the middle of a cell
        c.t = c.t - c.R @ np.full(3, 50.0)
    rise = np.arange(rig.n_pixels, dtype=np.float32).reshape(4, 120, 160) / np.float32(4 * rig.n_pixels)
    fr = S.Frame(fr.depth, [np.full_like(c, 0.9) if equal else np.float32(0.7) + rise[i] for i, c in enumerate(fr.conf)],
                 fr.rgb)
    rep, gpu = _check(oracle_mod, rig, fr, coarse_cell_m=100.0, max_level=0)
    assert rep["n_cells_oracle"] == rep["n_cells_matched"] == 1
    order = np.concatenate([c.reshape(-1) for c in fr.conf]) * np.concatenate([d.reshape(-1) > 0 for d in fr.depth])
    assert gpu["cells"]["rep"][0] == np.argmax(order)


def test_static_calls_alternate_between_variants(oracle_mod):
    """The allocation-free entry keeps its tables between calls: a top-k frame leaves nothing in
    them that a frame of all members would read, nor the other way round."""
    import test_zz_no_alloc as Z
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_01035_gb300 import fuseflow as F
    dev, stream = torch.device("cuda"), torch.cuda.current_stream().cuda_stream
    rig = S.tiny_rig(n=3, width=160, height=120, spread_deg=30.0)
    for k, seed in ((3, 51), (0, 51), (3, 52), (0, 53)):
        fr = S.random_frame(rig, seed=seed, flying_frac=0.01)
        ff = F.FuseFlow(rig, max_cells=8192, top_k=k)
        try:
            ref = run_gpu(ff, fr, torch, with_trace=False)
        finally:
            ff.close()
        st, stats, out = Z._static_call(F, rig, fr, 8192, dev, stream, top_k=k)
        assert st == F.FUSEFLOW_OK and stats.error == 0
        Z._check_same(ref["cells"], ref["stats"], out, int(stats.n_cells))


def test_static_call_after_top_k_ran_out_of_records():
    """A top-k frame with more (tile, cell) records than the static entry holds leaves cells that
    were never listed; nothing of them may pass for a member of a later frame, not even where its
    members' confidences are negative (they do not gate without the confidence term)."""
    import test_zz_no_alloc as Z
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_01035_gb300 import fuseflow as F
    dev, stream = torch.device("cuda"), torch.cuda.current_stream().cuda_stream
    big = S.tiny_rig(n=2, width=512, height=512)
    rig = S.tiny_rig(n=3, width=160, height=120, spread_deg=30.0)
    fr = S.random_frame(rig, seed=54, flying_frac=0.01)
    low = S.Frame(fr.depth, [c - np.float32(1.5) for c in fr.conf], fr.rgb)
    for frame, params in ((low, {"use_conf": 0}), (fr, {})):
        st, stats, _ = Z._static_call(F, big, _scattered(big, 55, 500, 8000), 32768, dev, stream, top_k=3,
                                      coarse_cell_m=2.0, max_level=4, n_min=1)
        assert st == F.FUSEFLOW_OK and stats.error & 16       # more records than the buffer holds
        for _ in range(2):
            ff = F.FuseFlow(rig, max_cells=8192, **params)
            try:
                ref = run_gpu(ff, frame, torch, with_trace=False)
            finally:
                ff.close()
            st, stats, out = Z._static_call(F, rig, frame, 8192, dev, stream, **params)
            assert st == F.FUSEFLOW_OK and stats.error == 0
            Z._check_same(ref["cells"], ref["stats"], out, int(stats.n_cells))


def test_crowded_units_in_few_and_many_blocks():
    """Units of nearly 256 coarse cells: one frame alone takes the count step of few units, eight
    in a batch that of many.  The clouds are the same to the bit (no result depends on the order
    in which cells are found)."""
    from test_gpu_batch import _batch_vs_plain
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_01035_gb300 import fuseflow
    rig = S.tiny_rig(n=2, width=640, height=512, fx=600.0, fy=600.0)
    frames = [(rig, _scattered(rig, 20 + i, 500, 40000)) for i in range(8)]
    _batch_vs_plain(fuseflow, frames, coarse_cell_m=0.32, max_level=2, n_min=2, max_cells=700000)
