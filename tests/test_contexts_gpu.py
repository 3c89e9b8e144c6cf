"""The C ABI in one CUDA context after another on the same device, and after a
reset of the device's primary context."""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def render_in_new_context(cu, device, primary):
    """(rgb, gradient w.r.t. the grid) of a small scene, in a context of its own or
    in the primary context, which ends with it."""
    import paper_2412_10084_gb300 as ps
    import synth
    sc = synth.make_scene("sphere64", dims=(24, 24, 24), probe_dims=(6, 6, 6))
    rays = synth.make_rays("sphere64", n_rays=64)
    params = ps.render_params(64.0, 32, 0, sc.n_fresnel)
    lib, P, n = ps.library(), ctypes.c_void_p, rays.o.shape[0]

    def ok(err):
        assert err == 0, (err, lib.psdf_last_cuda_error())

    ctx = P()
    if primary:
        ok(cu.cuDevicePrimaryCtxRetain(ctypes.byref(ctx), device))
        ok(cu.cuCtxSetCurrent(ctx))
    else:
        ok(cu.cuCtxCreate_v2(ctypes.byref(ctx), 0, device))
    try:
        def dev(a=None, floats=0):
            a = np.zeros(floats, np.float32) if a is None else np.ascontiguousarray(a, np.float32)
            p = ctypes.c_uint64()
            ok(cu.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(a.nbytes)))
            ok(cu.cuMemcpyHtoD_v2(p, a.ctypes.data_as(P), ctypes.c_size_t(a.nbytes)))
            return P(p.value)

        def host(p, floats):
            a = np.empty(floats, np.float32)
            ok(cu.cuMemcpyDtoH_v2(a.ctypes.data_as(P), ctypes.c_uint64(p.value),
                                  ctypes.c_size_t(a.nbytes)))
            return a

        gd = ps.grid_desc(sc.dims, sc.box_min, sc.box_max)
        pd = ps.ProbeDesc()
        pd.dims[:] = sc.probe_dims
        pd.sh_l, pd.n_ang, pd.dtype = sc.sh_l, sc.probes.shape[-1], ps.F32
        md = ps.MlpDesc(3 + sc.probes.shape[-1] + sc.n_fresnel, sc.width, ps.F32)
        records = np.concatenate([sc.sdf[..., None], sc.feat], -1)
        g, p, m = P(), P(), P()
        ok(lib.psdf_grid_create(ctypes.byref(gd), dev(records), ctypes.byref(g)))
        ok(lib.psdf_probes_create(ctypes.byref(pd), dev(sc.probes), ctypes.byref(p)))
        ok(lib.psdf_mlp_create(ctypes.byref(md), dev(sc.mlp), ctypes.byref(m)))
        o, d = dev(rays.o), dev(rays.d)
        rgb, depth, wsum, logT = (dev(floats=k * n) for k in (3, 1, 1, 1))
        gg, gp, gm = (dev(floats=a.size) for a in (records, sc.probes, sc.mlp))
        ok(lib.psdf_render_forward(g, p, m, ctypes.byref(params), o, d, None, n, rgb, depth, wsum,
                                   logT, None, None))
        ok(lib.psdf_render_backward(g, p, m, ctypes.byref(params), o, d, None, n,
                                    dev(np.ones((n, 3))), None, None, logT, None, gg, gp, gm,
                                    None))
        flags = ctypes.c_int32(-1)
        ok(lib.psdf_device_status(None, ctypes.byref(flags)))
        assert flags.value == 0
        out = host(rgb, 3 * n), host(gg, records.size)
        lib.psdf_grid_destroy(g)
        lib.psdf_probes_destroy(p)
        lib.psdf_mlp_destroy(m)
        return out
    finally:
        if primary:
            ok(cu.cuDevicePrimaryCtxReset_v2(device))
            ok(cu.cuCtxSetCurrent(None))
        else:
            ok(cu.cuCtxDestroy_v2(ctx))


def child(primary):
    cu = ctypes.CDLL("libcuda.so.1")
    device = ctypes.c_int()
    assert cu.cuInit(0) == 0 and cu.cuDeviceGet(ctypes.byref(device), 0) == 0
    first = render_in_new_context(cu, device, primary)
    second = render_in_new_context(cu, device, primary)
    assert np.array_equal(first[0], second[0]) and first[0].max() > 0.1
    # reductions in any order
    assert np.max(np.abs(first[1] - second[1])) <= 1e-5 * np.max(np.abs(first[1]))


@pytest.mark.parametrize("which", ["own", "primary"])
def test_one_context_after_another(which):
    run = subprocess.run([sys.executable, os.path.abspath(__file__), which], cwd=ROOT,
                         timeout=300, capture_output=True, text=True,
                         env={**os.environ, "PYTHONPATH": ROOT})
    assert run.returncode == 0, run.stderr[-2000:]


if __name__ == "__main__":
    child(sys.argv[1] == "primary")
