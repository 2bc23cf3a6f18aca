"""Values at the ends of the accepted ranges, against the oracle at the parity tolerances:
depth samples so far away that a residual leaves float32, confidences above one, and residual
sums of 2^48 grid units squared and more."""
import numpy as np
import pytest

from paper_2602_01035_gb300 import scenes as S
from parity import compare, run_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def F():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_01035_gb300 import fuseflow
    fuseflow.load()
    return fuseflow


def _fuse(F, rig, fr, with_trace=False, **params):
    ff = F.FuseFlow(rig, **params)
    try:
        gpu = run_gpu(ff, fr, torch, with_trace=with_trace)
    finally:
        ff.close()
    assert gpu["status"] == F.FUSEFLOW_OK, gpu["stats"]
    return gpu


def _with_sentinels(seed):
    """A rendered float32 frame in which 2 % of the samples are the largest finite float32, as
    sensors mark "no return"; they are not confident, so that only other cameras' points see them."""
    rig = S.tiny_rig(n=4, width=96, height=64, depth_format="f32", depth_scale=1.0, spread_deg=25.0)
    fr = S.random_frame(rig, seed=seed, zero_frac=0.02)
    rng = np.random.default_rng(seed)
    for d, c in zip(fr.depth, fr.conf):
        far = rng.random(d.shape) < 0.02
        d[far] = np.finfo(np.float32).max
        c[far] = 0.0
    return rig, fr


@pytest.mark.parametrize("top_k", [0, 7])
def test_infinite_residual_weighs_nothing(F, oracle_mod, top_k):
    rig, fr = _with_sentinels(81)
    params = {"coarse_cell_m": 0.4, "max_level": 0, "n_min": 2, "top_k": top_k}
    orc = oracle_mod.fuse_frame(rig, fr, params)
    hit = (orc["gated"] != 0) & (orc["e"] > 1e30)
    assert hit.sum() > 100
    assert np.all(np.isin(orc["key"][hit], orc["key"][(orc["gated"] != 0) & (orc["e"] < 1e3)]))
    gpu = _fuse(F, rig, fr, **params)
    rep = compare(gpu, orc)
    assert rep["n_cells_valued"] > 20


def test_infinite_residual_of_a_point(F, oracle_mod):
    from test_gpu_points import _points
    rig, fr = _with_sentinels(82)
    orc = oracle_mod.fuse_frame(rig, fr, {})
    hit = (orc["gated"] != 0) & (orc["e"] > 1e30)
    assert hit.sum() > 100
    _, _, _, w, _ = _points(F, rig, fr)
    assert np.all(w[hit] == 0.0)


@pytest.mark.parametrize("scale", [255.0, 1000.0, 65535.0, 1e30])
@pytest.mark.parametrize("top_k", [0, 3])
def test_confidences_above_one(F, oracle_mod, scale, top_k):
    """Confidence images on another scale than [0, 1] fuse to the same cloud at that scale."""
    rig, _, fr = S.config1()
    fr = S.Frame(fr.depth, [(c * np.float32(scale)).astype(np.float32) for c in fr.conf], fr.rgb)
    params = {"tau": float(np.float32(0.6) * np.float32(scale)), "top_k": top_k}
    gpu = _fuse(F, rig, fr, with_trace=True, **params)
    rep = compare(gpu, oracle_mod.fuse_frame(rig, fr, params))
    assert rep["n_cells_valued"] > 100


def test_residual_sums_past_48_bits(F, oracle_mod):
    """Cameras of one pose and 126 degrees: eight whose corner samples lie at the end of the grid's
    range, and eight more whose corners hold near points 1 mm apart, each of which differs from all
    of the first eight by nearly the whole range.  One cell a corner, exponents of 16,000 that differ
    by a half from point to point: an error of 2^-24 of a residual moves its weight by 0.1 %."""
    n, size = 16, 40
    f = (size - 1) / 2 / 1.94
    cams = [S.Camera(f, f, (size - 1) / 2, (size - 1) / 2, size, size, np.eye(3), np.zeros(3)) for _ in range(n)]
    rig = S.Rig(cams, "f32", 1.0)
    rng = np.random.default_rng(83)
    depth, conf, rgb = [], [], []
    for k in range(n):
        d, c = np.zeros((size, size), np.float32), np.zeros((size, size), np.float32)
        for y in (0, size - 1):
            for x in (0, size - 1):
                d[y, x] = 65.5 if k < 8 else 1.2 + 1e-3 * (k - 8)
                c[y, x] = 0.0 if k < 8 else 1.0
        depth.append(d)
        conf.append(c)
        rgb.append(rng.choice(np.array([0, 255], np.uint8), size=(size, size, 3)))
    fr = S.Frame(depth, conf, rgb)
    params = {"k_views": 9, "sigma_m": 1.47, "coarse_cell_m": 1.0, "max_level": 0}
    orc = oracle_mod.fuse_frame(rig, fr, params)
    e = orc["e"][orc["gated"] != 0]
    assert len(e) == 32 and e.min() > 1.6e4 and orc["stats"]["n_cells"] == 4
    rep = compare(_fuse(F, rig, fr, **params), orc)
    assert rep["n_cells_valued"] == 4
