"""Host code of the library against a CUDA runtime whose calls fail, refuse or take long: small programs compiled from the library's
own sources, with the calls in question defined by the program.  No GPU."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _run(tmp_path, source, body):
    from paper_2405_17991_b200 import build
    src, exe = tmp_path / "fake.cu", tmp_path / "fake"
    src.write_text('#include "%s"\n#include <cstdio>\n#include <cstdlib>\n%s' % (os.path.join(build.CSRC, source), body))
    r = subprocess.run([build._nvcc(), "-std=c++17", "-O1", "-gencode", "arch=compute_100a,code=compute_100a", "-cudart", "shared", "-I", build.INCLUDE,
                        "-I", build.CSRC, "-Xcompiler", "-fPIC", "-o", str(exe), str(src), "-lpthread"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    lib = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "lib64")
    env = dict(os.environ, LD_LIBRARY_PATH=lib + ":" + os.environ.get("LD_LIBRARY_PATH", ""))
    return subprocess.run([str(exe)], capture_output=True, text=True, timeout=60, env=env)


def test_two_threads_may_make_their_first_tensor_map_at_once(tmp_path):
    r = _run(tmp_path, "tensor_maps.cu", r"""
#include <thread>
#include <unistd.h>
static CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                       CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill) { return CUDA_SUCCESS; }
extern "C" cudaError_t cudaGetDriverEntryPoint(const char*, void** p, unsigned long long, cudaDriverEntryPointQueryResult* q)
{
    usleep(200000);
    *p = reinterpret_cast<void*>(&encode);
    if (q) *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
int main()
{
    int rc[4];
    std::thread t[4];
    for (int i = 0; i < 4; ++i)
        t[i] = std::thread([&rc, i] { CUtensorMap m; usleep(20000 * i); rc[i] = velora::make_tmap_bf16_2d(&m, &m, 64, 64, 64, 64, 64); });
    for (auto& x : t) x.join();
    std::printf("%d %d %d %d\n", rc[0], rc[1], rc[2], rc[3]);
}
""")
    assert r.stdout.split() == ["0"] * 4, r.stdout + r.stderr


def test_a_refused_cluster_launch_falls_back_to_single_ctas(tmp_path):
    r = _run(tmp_path, "gemm_simt.cu", r"""
namespace velora {
int device_info(DeviceInfo* d) { *d = DeviceInfo{148, 227 * 1024}; return VELORA_OK; }
int after_launch() { return VELORA_OK; }
}
extern "C" cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void*, void** args)
{
    unsigned cluster = 1;
    for (unsigned i = 0; i < c->numAttrs; ++i)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) cluster = c->attrs[i].val.clusterDim.z;
    std::printf("cluster %u grid %u %u %u slice %lld\n", cluster, c->gridDim.x, c->gridDim.y, c->gridDim.z, (long long)*static_cast<int64_t*>(args[15]));
    return cluster > 1 ? cudaErrorInvalidConfiguration : cudaSuccess;
}
int main()
{
    float x[4];
    const int rc = velora::launch_gemm_simt(x, VELORA_F32, 1280, 1, x, VELORA_F32, 1280, 1, x, VELORA_F32, 288, 0, 171, 288, 1280, nullptr);
    std::printf("status %d\n", rc);
}
""")
    lines = r.stdout.splitlines()
    assert lines[-1] == "status 0", r.stdout + r.stderr
    assert lines[0].startswith("cluster 8 grid 5 3 8") and lines[1] == "cluster 1 grid 5 3 1 slice 1280", r.stdout
