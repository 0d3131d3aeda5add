"""The autotuner's cache: geometries of one shape that want other plans."""
import pytest

from paper_2410_14900_gb300 import api, synth, tune

pytestmark = pytest.mark.gpu


def _geometry(voxel=1.0, shift=0.0, pitch=1.0, n=64):
    V, H, W = 60, 400, 400
    o = synth.circle_orbit(V)
    P = synth.projection_matrices(o, H, W, pitch)
    for i in range(V):   # every view its own principal point
        P[i, 0] += shift * (i + 1) * P[i, 2]
    desc = dict(n_views=V, det_rows=H, det_cols=W, n_mu=500, n_s=500, pitch=pitch, ds=pitch,
                vol_x=2 * n, vol_y=2 * n, vol_z=n, voxel=(voxel,) * 3, closed_orbit=1)
    return api.Geometry(desc, P, o.vdl)


def test_a_plan_is_not_taken_for_another_geometry_of_the_shape(tmp_path, monkeypatch):
    monkeypatch.setenv("DC_TUNE_CACHE", str(tmp_path / "tune.json"))
    first = _geometry()
    assert not tune.autotune(first, chunks=(256,))["cached"]
    for other in (_geometry(shift=0.1), _geometry(voxel=2.2), _geometry(pitch=0.5)):
        r = tune.autotune(other, chunks=(256,))
        assert not r["cached"]
        t = api.dc_geometry_get_tuning(other)
        assert t["chunk_images"] == r["chunk_images"] <= t["chunk_capacity"]
    again = tune.autotune(_geometry(), chunks=(256,))
    assert again["cached"]


def test_a_cached_chunk_is_held_to_the_work_area(tmp_path, monkeypatch):
    monkeypatch.setenv("DC_TUNE_CACHE", str(tmp_path / "tune.json"))
    geom = _geometry()
    cap = api.dc_geometry_get_tuning(geom)["chunk_capacity"]
    tune._store({tune.shape_key(geom): {"chunk_images": cap + 100, "bp_nz": 16}})
    r = tune.autotune(geom)
    assert r["cached"] and r["chunk_images"] == cap
    assert api.dc_geometry_get_tuning(geom)["chunk_images"] == cap
