"""Which arrays of a caller a kernel may touch in place of a staging copy
(csrc/sph_place.cuh), against a stand-in for the CUDA runtime that knows a few
allocations: device memory of another address than the element's alignment is
staged, as host, managed and peer memory are (a copy takes any address, a kernel's
access of it would fault), and so is an array that reaches past its allocation
(which a copy refuses)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1210_1017_gb300", "csrc")

RUNTIME = r"""
#include "sph_place.cuh"
#include <cstdio>
#include <initializer_list>
// device 0 is current; 1 MB each at 0x10000000 (its memory), 0x20000000 (of
// device 1), 0x30000000 (managed), 0x40000000 (pinned host)
static const uintptr_t MB = 1u << 20;
extern "C" cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
extern "C" cudaError_t cudaGetLastError() { return cudaSuccess; }
extern "C" cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
    const uintptr_t v = (uintptr_t)p;
    *a = cudaPointerAttributes{};
    a->device = v / 0x10000000u == 2 ? 1 : 0;
    a->type = v % 0x10000000u >= MB ? cudaMemoryTypeUnregistered
              : v / 0x10000000u <= 2 ? cudaMemoryTypeDevice
              : v / 0x10000000u == 3 ? cudaMemoryTypeManaged : cudaMemoryTypeHost;
    return cudaSuccess;
}
static CUresult range(CUdeviceptr* b, size_t* n, CUdeviceptr p) {
    *b = p / 0x10000000u * 0x10000000u;
    *n = MB;
    return p - *b < MB ? CUDA_SUCCESS : CUDA_ERROR_NOT_FOUND;
}
extern "C" cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned,
                                                        unsigned long long,
                                                        cudaDriverEntryPointQueryResult* q) {
    *f = (void*)range;
    *q = cudaDriverEntryPointSuccess;
    return cudaSuccess;
}
"""


def _run(tmp_path, body):
    src = tmp_path / "place.cpp"
    src.write_text(RUNTIME + "int main() {\n" + body + "\nreturn 0; }\n")
    exe = tmp_path / "place"
    subprocess.check_call(["g++", "-std=c++17", "-I", CSRC, "-I", "/usr/local/cuda/include",
                           str(src), "-o", str(exe)])
    return subprocess.check_output([str(exe)], text=True).split()


def test_only_aligned_memory_of_this_device_is_used_in_place(tmp_path):
    got = _run(tmp_path, r"""
    for (uintptr_t base : {0x10000000u, 0x20000000u, 0x30000000u, 0x40000000u, 0x50000000u})
        printf("%d ", sph::on_this_device((const double*)base, 3));
    printf("%d ", sph::on_this_device((const double*)nullptr, 3));
    for (uintptr_t o = 1; o <= 8; ++o)
        printf("%d%d%d ", sph::on_this_device((const double*)(0x10000000u + o), 3),
               sph::on_this_device((float*)(0x10000000u + o), 3),
               sph::on_this_device((const uint32_t*)(0x10000000u + o), 3));
    """)
    assert got[:6] == ["1", "0", "0", "0", "0", "0"]
    assert got[6:] == ["000", "000", "000", "011", "000", "000", "000", "111"]


def test_an_array_past_its_allocation_is_not_used_in_place(tmp_path):
    got = _run(tmp_path, r"""
    const size_t n = MB / 8;
    const double* p = (const double*)0x10000000u;
    printf("%d %d %d ", sph::on_this_device(p, n), sph::on_this_device(p, n + 1),
           sph::on_this_device(p + 1, n));
    printf("%d %d %d", sph::on_this_device(p + 1, n - 1), sph::on_this_device(p + n - 1, 1),
           sph::on_this_device(p, SIZE_MAX / 8));
    """)
    assert got == ["1", "0", "0", "1", "1", "0"]
