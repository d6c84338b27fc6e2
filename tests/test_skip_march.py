"""The plain method's skipping march (nedf_device.cuh: march_crossing_skip), compiled for the host, against the
march that evaluates every sample: the same hit and the same depth, bit for bit, for every SDF kind, bound
radii of 0.5 to 1000, twists up to 200, origins up to 1000 units away, and rays along the twist's axis at the
bound's rim, where the SDF changes at its Lipschitz bound."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_2308_04669_gb300 import scenegen as sg

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2308_04669_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")
F32 = C.POINTER(C.c_float)

SOURCE = r"""
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
using std::max;
using std::min;
static inline float __int_as_float(int i) { float f; std::memcpy(&f, &i, 4); return f; }
#include "nedf_device.cuh"
using namespace nedf;

static float uniform_march(const DevType &t, V3 ol, V3 dl, float te, float tx, int steps, int bisect, bool &hit)
{
    const float step = (tx - te) / (float)steps;
    bool prev = inside_solid(t, madd(ol, te, dl));
    for (int k = 1; k <= steps; ++k) {
        const bool in = inside_solid(t, madd(ol, std::fmaf((float)k, step, te), dl));
        if (in && !prev) {
            float lo = std::fmaf((float)(k - 1), step, te), hi = std::fmaf((float)k, step, te);
            for (int it = 0; it < bisect; ++it) {
                const float mid = 0.5f * (lo + hi);
                if (inside_solid(t, madd(ol, mid, dl))) hi = mid; else lo = mid;
            }
            hit = true;
            return 0.5f * (lo + hi);
        }
        prev = in;
    }
    hit = false;
    return INFINITY;
}

// rays with another answer than the uniform march's; *hits: rays that hit
extern "C" long long differ(int kind, const float *p, float rb, const float *o, const float *d, long long n, int steps,
                            int bisect, long long *hits)
{
    DevType t{};
    t.kind = kind;
    for (int i = 0; i < 8; ++i) t.p[i] = p[i];
    t.rb = rb;
    long long bad = 0;
    *hits = 0;
    for (long long i = 0; i < n; ++i) {
        const V3 ol = v3(o[3 * i], o[3 * i + 1], o[3 * i + 2]);
        const V3 dl = normalized(v3(d[3 * i], d[3 * i + 1], d[3 * i + 2]));
        Chord c;
        if (!bound_chord(ol, dl, rb, c)) continue;
        bool h0, h1;
        const float a = uniform_march(t, ol, dl, c.te, c.tx, steps, bisect, h0);
        const float b = march_crossing_skip(t, ol, dl, c.te, c.tx, steps, bisect, h1);
        bad += h0 != h1 || a != b;
        *hits += h0;
    }
    return bad;
}
"""


@pytest.fixture(scope="module")
def differ(tmp_path_factory):
    d = tmp_path_factory.mktemp("skip_march")
    (d / "m.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", "-w", f"-I{CUDA}/include", f"-I{CSRC}", str(d / "m.cpp"), "-o",
                    str(d / "m.so")], check=True)
    lib = C.CDLL(str(d / "m.so"))
    lib.differ.restype = C.c_longlong

    def run(kind, params, rb, o, d, steps, bisect):
        p = np.zeros(8, np.float32)
        p[:len(params)] = params
        o, d = np.ascontiguousarray(o, np.float32), np.ascontiguousarray(d, np.float32)
        hits = C.c_longlong()
        bad = lib.differ(C.c_int(kind), p.ctypes.data_as(F32), C.c_float(rb), o.ctypes.data_as(F32), d.ctypes.data_as(F32),
                         C.c_longlong(len(o)), C.c_int(steps), C.c_int(bisect), C.byref(hits))
        return bad, hits.value
    return run


def _rays(n, rb, dist, seed):
    """From a sphere of radius dist towards points of the bound sphere."""
    g = np.random.default_rng(seed)
    o, q = g.normal(size=(n, 3)), g.normal(size=(n, 3))
    o *= dist / np.linalg.norm(o, axis=1, keepdims=True)
    q *= rb * g.uniform(size=(n, 1)) ** (1 / 3) / np.linalg.norm(q, axis=1, keepdims=True)
    return o, q - o


def _params(kind, scale):
    p = [v * scale for v in sg.DEFAULT_PARAMS[kind]]
    if kind == sg.SDF_TWISTTORUS:
        p[2] = sg.DEFAULT_PARAMS[kind][2] / scale
    return p


@pytest.mark.parametrize("scale", [0.5, 1.0, 63.9, 100.0, 1000.0])
@pytest.mark.parametrize("kind", sorted(sg.DEFAULT_PARAMS))
def test_every_kind(differ, kind, scale):
    for dist, steps, bisect, n in ((1.0, 1, 0, 2000), (1.0, 97, 6, 20000), (7.0, 256, 8, 20000), (1000.0, 256, 8, 20000),
                                   (1.0, 4096, 4, 1000)):
        o, d = _rays(n, scale, dist * scale, 3)
        bad, hits = differ(kind, _params(kind, scale), scale, o, d, steps, bisect)
        assert bad == 0, (dist, steps, bad)
        assert hits > 0 or steps == 1


@pytest.mark.parametrize("rb", [1.0, 20.0, 63.9, 200.0, 1000.0])
@pytest.mark.parametrize("twist", [1.0, 30.0, 200.0])
def test_twist_at_the_bounds_rim(differ, rb, twist):
    for steps, n in ((1024, 20000), (4096, 4000), (16384, 4000)):
        for rim in (0.9, 0.99, 0.999, 0.9999):
            g = np.random.default_rng(5)
            phi, rho = g.uniform(0, 2 * np.pi, n), rb * (rim + (1 - rim) * g.uniform(0, 1, n))
            o = np.stack([rho * np.cos(phi), np.full(n, -2 * rb), rho * np.sin(phi)], 1)
            bad, _ = differ(sg.SDF_TWISTTORUS, [0.9 * rb, 0.3 * rb, twist], rb, o, np.tile([0, 1.0, 0], (n, 1)), steps, 8)
            assert bad == 0, (steps, rim, bad)


@pytest.mark.gpu
@pytest.mark.parametrize("size,many", [(40, False), (448, True)])
def test_deferred_pairs_of_large_bounds(size, many):
    """Bound radii of 60 to 500, an unscaled twist, seen from thousands of local units away: pairs deferred to a
    warp or a thread each (every pair, at a confidence bound of 1) get the depths, ids and shadows of the
    plain method's frame."""
    import dataclasses

    import torch
    from paper_2308_04669_gb300 import native
    base = sg.stress_scene(size, size - 8, nerf=False, n_inst=64)
    rbs = [60.0, 100.0, 500.0]
    types = [sg.make_type(sg.SDF_TWISTTORUS, 1, 0, 2, 64, rb=rbs[0], params=[0.55 * rbs[0], 0.2 * rbs[0], 0.5]),
             sg.make_type(sg.SDF_TORUS, 1, 1, 2, 64, rb=rbs[1], params=_params(sg.SDF_TORUS, rbs[1])),
             sg.make_type(sg.SDF_BOX, 1, 2, 2, 64, rb=rbs[2], params=_params(sg.SDF_BOX, rbs[2]))]
    for t in types:                # confidence 1/2 everywhere (inputs of hundreds saturate an untrained network)
        t.nedf_w[:] = 0.0
    it = (base.inst_type % 3).astype(np.uint32)
    sc = dataclasses.replace(base, types=types, inst_type=it, inst_s=sg.f32(base.inst_s / sg.f32(rbs)[it]))
    r = native.renderer_for(sc, precision=native.PREC_BF16)
    cam, lights = r.camera(sc.eye, sc.target, sc.fov_deg), r.lights(sc.lights[:2])
    got = []
    for source in (native.DEPTH_NEDF, native.DEPTH_MARCH):
        o = r.get_options()
        o.depth_source, o.fallback_conf, o.march_steps, o.march_bisect = source, 1.0, 256, 8
        r.set_options(o)
        n = sc.W * sc.H
        b = [torch.empty(n, device="cuda"), torch.empty(n, dtype=torch.int32, device="cuda"), torch.empty(n, device="cuda")]
        st = r.render(cam, lights, b[0], b[1], None, b[2], None, stats=True)
        torch.cuda.synchronize()
        got.append([x.cpu().numpy() for x in b] + [st])
    r.close()
    st = got[0][-1]
    assert st.fallback_pairs == st.primary_pairs + st.shadow_pairs and st.status == 0
    assert (st.primary_pairs > 32768) == many and (got[0][1] != -1).any()
    for a, b in zip(got[0][:3], got[1][:3]):
        assert np.array_equal(a, b)
