"""Handles of different geometries used at the same time, each from a host
thread and a stream of its own, and batches that outlive the creation of
others: the shared-memory limit of a kernel belongs to the process."""
import threading

import pytest
import torch

from paper_2410_14900_gb300 import api, synth

pytestmark = pytest.mark.gpu


def _geometry(V, H, W, n_s, vol=16):
    o = synth.sinusoid_orbit(V)
    desc = dict(n_views=V, det_rows=H, det_cols=W, n_mu=4, n_s=n_s, pitch=1.0, ds=1.0, vol_x=vol,
                vol_y=vol, vol_z=vol, voxel=(1.0, 1.0, 1.0), closed_orbit=1)
    return api.Geometry(desc, synth.projection_matrices(o, H, W, 1.0), o.vdl)


def test_two_threads_with_their_own_handles():
    # tiles of these detectors stage windows of different sizes; 64 launches a call
    geoms = [_geometry(256, 200, 256, 300), _geometry(256, 256, 256, 300),
             _geometry(256, 40, 512, 300)]
    for g in geoms:
        api.dc_geometry_set_tuning(g, 4, 0)
    sinos = [torch.randn((1, g.V) + g.sino_shape, device="cuda") for g in geoms]
    refs = [api.dc_radon2d_adjoint(g, s) for g, s in zip(geoms, sinos)]
    torch.cuda.synchronize()
    errors, start = [], threading.Barrier(len(geoms))

    def work(i):
        try:
            st = torch.cuda.Stream()
            start.wait()
            with torch.cuda.stream(st):
                for _ in range(100):
                    out = api.dc_radon2d_adjoint(geoms[i], sinos[i])
            st.synchronize()
            if not torch.equal(out, refs[i]):
                errors.append(f"geometry {i}: another result")
        except Exception as e:  # reported by the main thread
            errors.append(f"geometry {i}: {e}")

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(geoms))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def test_a_batch_runs_after_a_smaller_one_was_created():
    big, small = _geometry(5, 120, 700, 900), _geometry(5, 16, 16, 16)
    g = torch.rand((5, 120, 700), device="cuda")
    vol, ref = torch.empty(big.vol_shape, device="cuda"), torch.empty(big.vol_shape, device="cuda")
    first = api.Batch([big], persistent_filter=True)
    first.run([g], [ref])
    second = api.Batch([small], persistent_filter=True)
    first.run([g], [vol])
    torch.cuda.synchronize()
    assert torch.equal(vol, ref)
    second.close()
    first.close()
