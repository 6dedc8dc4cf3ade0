"""Devices that hold fewer or smaller clusters than a B200 (a partition of one, say): the kernels in clusters give way to those
without.  Host only: a stand-in for the CUDA runtime's launch and occupancy calls refuses clusters above a limit and
launches nothing."""
import ctypes
import os
import shutil
import subprocess
import sys
import textwrap

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#include <cuda_runtime_api.h>
#include <stdlib.h>
static int limit(void) { return atoi(getenv("FAKE_CLUSTER")); }     /* CTAs of the largest cluster */
static int resident(void) { return atoi(getenv("FAKE_RESIDENT")); }   /* clusters at a time */
static int cluster_of(const cudaLaunchConfig_t* c) {
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) return (int)c->attrs[i].val.clusterDim.x;
    return 1;
}
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int d) { *v = 148; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v) {
    return a == cudaFuncAttributeNonPortableClusterSizeAllowed && limit() < 16 ? cudaErrorInvalidValue : cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* f, const cudaLaunchConfig_t* c) {
    *n = cluster_of(c) > limit() ? 0 : resident();
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
    return cluster_of(c) > limit() ? cudaErrorInvalidConfiguration : cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void* f, dim3 g, dim3 b, void** args, size_t s, cudaStream_t st) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t st) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t st, enum cudaStreamCaptureStatus* s) {
    *s = getenv("FAKE_CAPTURE") ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaPeekAtLastError(void) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
"""

PROBE = textwrap.dedent("""
    import ctypes, sys
    class Shape(ctypes.Structure):
        _fields_ = [(n, ctypes.c_int32) for n in ("B", "T", "H", "P", "io", "reserved")]
    lib = ctypes.CDLL(sys.argv[1])
    lib.ssm_launch_count.restype = ctypes.c_longlong
    op, *dims = sys.argv[2], *map(int, sys.argv[3:8])
    s = ctypes.byref(Shape(*dims, 0))
    ptr, size, null = ctypes.c_void_p(4096), ctypes.c_size_t(1 << 40), ctypes.c_void_p(0)
    calls = {"step": [lambda: lib.ssm_step(s, *[ptr] * 7, size, null)],
             "layer": [lambda: lib.ssm_layer_fwd(s, *[ptr] * 11, size, null), lambda: lib.ssm_layer_bwd(s, *[ptr] * 11, size, *[ptr] * 7, null, null)]}
    for call in calls[op]:
        n = lib.ssm_launch_count()
        print(call(), lib.ssm_launch_count() - n)
""")


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    from paper_2502_20168_b200 import build
    build.build()
    d = tmp_path_factory.mktemp("fake")
    (d / "fake.c").write_text(FAKE)
    include = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())), "include")
    subprocess.run([shutil.which("gcc") or "gcc", "-shared", "-fPIC", "-w", "-I" + include, "-o", str(d / "fake.so"), str(d / "fake.c")],
                   check=True)

    def calls(cluster, resident, *args, **more):
        """[(status, launches)] of each call where clusters above `cluster` CTAs are refused."""
        env = dict(os.environ, **more, LD_PRELOAD=str(d / "fake.so"), FAKE_CLUSTER=str(cluster), FAKE_RESIDENT=str(resident))
        r = subprocess.run([sys.executable, "-c", PROBE, build.LIB_PATH, *map(str, args)], env=env, capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr
        return [tuple(map(int, line.split())) for line in r.stdout.splitlines()]
    return calls


@pytest.mark.parametrize("B,H,P,io,size", [(16, 512, 256, 0, 16), (1, 384, 64, 0, 16), (16, 256, 128, 0, 8), (16, 256, 128, 1, 8), (3, 128, 64, 1, 4)])
def test_steps_without_clusters_take_the_two_halves(fake, B, H, P, io, size):
    assert fake(16, 14, "step", B, 1, H, P, io) == [(0, 1)]
    assert fake(size // 2, 14, "step", B, 1, H, P, io) == [(0, 2)]   # no such cluster
    groups = (B + 7) // 8
    assert fake(16, groups, "step", B, 1, H, P, io) == [(0, 1)]
    assert fake(16, groups - 1, "step", B, 1, H, P, io) == [(0, 2)]   # not all in one round


@pytest.mark.parametrize("B,H,P,io,eager,graph", [(1, 512, 256, 0, 2, 2), (3, 512, 256, 0, 2, 2), (4, 512, 256, 0, 1, 1), (4, 384, 192, 0, 1, 2),
                                                  (16, 384, 64, 0, 1, 2), (17, 384, 64, 0, 1, 1), (1, 256, 128, 0, 1, 1), (2, 256, 64, 0, 1, 2), (3, 256, 64, 1, 1, 1),
                                                  (112, 128, 64, 0, 1, 2), (113, 128, 64, 0, 1, 1)])
def test_steps_in_a_graph_take_the_two_halves_where_those_are_shorter(fake, B, H, P, io, eager, graph):
    """Launched one by one, two kernels cost their host time; in a graph only what they take on the device."""
    assert fake(16, 40, "step", B, 1, H, P, io) == [(0, eager)]
    assert fake(16, 40, "step", B, 1, H, P, io, FAKE_CAPTURE="1") == [(0, graph)]


@pytest.mark.parametrize("B,T,H,P,io,size", [(1, 64, 32, 16, 0, 8), (14, 64, 32, 16, 1, 8), (32, 64, 32, 16, 0, 4)])
def test_small_layers_without_clusters_take_separate_kernels(fake, B, T, H, P, io, size):
    (rc_f, fwd), (rc_b, bwd) = fake(16, B, "layer", B, T, H, P, io)
    assert (rc_f, rc_b, fwd) == (0, 0, 1) and bwd == (1 if B == 1 else 3)
    for cluster, resident in ((size // 2, B), (16, B - 1)):
        (rc_f, fwd), (rc_b, bwd) = fake(cluster, resident, "layer", B, T, H, P, io)
        assert (rc_f, rc_b) == (0, 0) and fwd >= 4 and bwd >= 5
