"""The frame's launch sequence on a fake CUDA runtime (host memory, no kernels; a preloaded library that logs
launches, event records and waits): a frame whose launch fails part-way leaves nothing on the light grids'
stream that the frame's stream does not wait for, whichever launch fails, captured into a graph or not."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
struct dim3 { unsigned x, y, z; };
static FILE *log_file() { static FILE *f = fopen(getenv("FAKE_LOG"), "w"); return f; }
#define LOG(...) do { fprintf(log_file(), __VA_ARGS__); fflush(log_file()); } while (0)
static dim3 cg, cb; static size_t csm; static void *cst;
static long checks = 0, next_id = 16;
static bool armed = false;
extern "C" {
void fake_arm() { armed = true; checks = 0; LOG("frame 0 0\n"); }
long fake_checks() { return checks; }
void **__cudaRegisterFatBinary(void *) { static void *h; return &h; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, void *, void *, void *, void *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
int __cudaGetKernel(void **k, const void *f) { *k = (void *)f; return 0; }
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, void *st) { cg = g; cb = b; csm = s; cst = st; return 0; }
int __cudaPopCallConfiguration(dim3 *g, dim3 *b, size_t *s, void *st) { *g = cg; *b = cb; *s = csm; *(void **)st = cst; return 0; }
int __cudaLaunchKernel(void *, dim3, dim3, void **, size_t, void *st) { LOG("launch %p 0\n", st); return 0; }
int cudaLaunchKernelExC(const void *, const void *, void **) { return 0; }
int cudaGetLastError() { const char *f = getenv("FAKE_FAIL"); return armed && f && ++checks == atol(f) ? 719 : 0; }
const char *cudaGetErrorString(int) { return "fake"; }
int cudaDeviceGetAttribute(int *v, int, int) { *v = 152; return 0; }
int cudaGetDevice(int *d) { *d = 0; return 0; }
int cudaMalloc(void **p, size_t n) { *p = calloc(n ? n : 1, 1); return *p ? 0 : 2; }
int cudaMallocHost(void **p, size_t n) { return cudaMalloc(p, n); }
int cudaFree(void *p) { free(p); return 0; }
int cudaFreeHost(void *p) { free(p); return 0; }
int cudaMemcpy(void *d, const void *s, size_t n, int) { memcpy(d, s, n); return 0; }
int cudaMemcpyAsync(void *d, const void *s, size_t n, int, void *) { memcpy(d, s, n); return 0; }
int cudaMemset(void *d, int v, size_t n) { memset(d, v, n); return 0; }
int cudaMemsetAsync(void *d, int v, size_t n, void *) { memset(d, v, n); return 0; }
int cudaStreamCreateWithFlags(void **s, unsigned) { *s = (void *)(next_id += 16); LOG("stream %p 0\n", *s); return 0; }
int cudaStreamDestroy(void *) { return 0; }
int cudaStreamSynchronize(void *) { return 0; }
int cudaStreamIsCapturing(void *, int *s) { *s = 0; return 0; }
int cudaStreamBeginCapture(void *, int) { return 0; }
int cudaStreamEndCapture(void *st, void **g) { *g = (void *)16; LOG("end %p 0\n", st); return 0; }
int cudaStreamWaitEvent(void *st, void *e, unsigned) { LOG("wait %p %p\n", st, e); return 0; }
int cudaEventCreate(void **e) { *e = (void *)(next_id += 16); return 0; }
int cudaEventCreateWithFlags(void **e, unsigned) { return cudaEventCreate(e); }
int cudaEventDestroy(void *) { return 0; }
int cudaEventRecord(void *e, void *st) { LOG("record %p %p\n", st, e); return 0; }
int cudaEventRecordWithFlags(void *e, void *st, unsigned) { return cudaEventRecord(e, st); }
int cudaEventElapsedTime(float *t, void *, void *) { *t = 1.0f; return 0; }
int cudaFuncSetAttribute(const void *, int, int) { return 0; }
int cudaGetSymbolAddress(void **p, const void *s) { *p = (void *)s; return 0; }
int cudaGraphDestroy(void *) { return 0; }
int cudaGraphExecDestroy(void *) { return 0; }
int cudaGraphInstantiate(void **g, void *, unsigned long long) { *g = (void *)16; return 0; }
int cudaGraphLaunch(void *, void *) { return 0; }
int cudaOccupancyMaxActiveClusters(int *n, const void *, const void *) { *n = 0; return 0; }
}
"""

DRIVER = """
import ctypes as C, sys
from paper_2308_04669_gb300 import native, scenegen as sg
fake = C.CDLL(None)
stream, deep, profile = (int(a) for a in sys.argv[1:])
sc = sg.three_types_scene(16, 16, nerf=False)
if deep:                # an E4M3 NeDF of more layers than its engine's shared memory holds: refused at the launch
    sc.types = [sg.make_type(t.kind, 3, i, 12, 128) for i, t in enumerate(sc.types)]
r = native.renderer_for(sc, precision=native.PREC_FP8 if deep else native.PREC_FP32, stream=stream)
r.set_profiling(profile)
fake.fake_arm()
try:
    r.render(r.camera(sc.eye, sc.target, sc.fov_deg), r.lights(sc.lights))
    print("ok", fake.fake_checks())
except native.NedfError as e:
    print("failed", fake.fake_checks())
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    from paper_2308_04669_gb300 import build
    build.build()
    d = tmp_path_factory.mktemp("fake_cuda")
    (d / "fake.cpp").write_text(FAKE)
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-w", str(d / "fake.cpp"), "-o", str(d / "fake.so")], check=True)

    def run(stream, deep, fail, profile=0):
        env = dict(os.environ, LD_PRELOAD=str(d / "fake.so"), FAKE_LOG=str(d / "log"), FAKE_FAIL=str(fail), PYTHONPATH=ROOT)
        p = subprocess.run([sys.executable, "-c", DRIVER, str(stream), str(deep), str(profile)], env=env, capture_output=True,
                           text=True, timeout=300)
        assert p.returncode == 0, p.stderr
        lines = [x.split() for x in (d / "log").read_text().splitlines()]
        at = next(i for i, x in enumerate(lines) if x[0] == "frame")
        side = [x[1] for x in lines[:at] if x[0] == "stream"]
        assert len(side) == 1
        return p.stdout.split()[0], side[0], lines[at + 1:]
    return run


def _unjoined(side, ops):
    """Launches on the side stream that no wait of another stream covers (in a captured frame, before its end)."""
    open_, recorded = 0, {}
    for op, st, ev in ops:
        if op == "launch" and st == side:
            open_ += 1
        elif op == "record":
            recorded[ev] = open_ if st == side else None
        elif op == "wait" and st != side and recorded.get(ev) == open_:
            open_ = 0
        elif op == "end":
            break
    return open_


@pytest.mark.parametrize("stream", [0, 4096])
def test_whichever_launch_fails(fake, stream):
    """Launch checks of a frame one after another, until a frame passes them all."""
    failed = 0
    for k in range(1, 40):
        out, side, ops = fake(stream, 0, k)
        assert any(op == "launch" and st == side for op, st, _ in ops)
        assert _unjoined(side, ops) == 0, k
        if out == "ok":
            break
        failed += 1
    assert 3 <= failed < 39


@pytest.mark.parametrize("stream", [0, 4096])
def test_a_shape_the_engine_refuses(fake, stream):
    out, side, ops = fake(stream, 1, 0)
    assert out == "failed" and any(op == "launch" and st == side for op, st, _ in ops)
    assert _unjoined(side, ops) == 0


@pytest.mark.parametrize("stream", [0, 4096])
def test_profiled_stages(fake, stream):
    """A profiled frame runs on the frame's stream alone; its Step-3 binning stage (the sixth) holds the six
    light-grid kernels and the two of the shadow rays."""
    out, side, ops = fake(stream, 0, 0, profile=1)
    assert out == "ok" and not any(st == side for _, st, _ in ops)
    launches = []
    for op, _, _ in ops:
        if op == "record":
            launches.append(0)
        elif op == "launch":
            launches[-1] += 1
    assert len(launches) == 9 and launches[5] == 8
