"""The mean IoU that a block of a kernel works out (csrc/miou.cuh), run on the CPU: the header is compiled for the host with a
thread per CUDA thread, barriers for __syncthreads and the warp exchanges.  Every block size that a kernel may have must give
the mean IoU of the matrix and write nothing outside the arrays it was given."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2003_10735_b200", "csrc")

CUDA_FOR_HOST = r"""
#pragma once
#include <barrier>
#include <cstdint>
#include <memory>
#include <thread>
#include <vector>
#define __device__
#define __host__
#define __forceinline__ inline
#define __shared__ static
struct Dim { unsigned x, y, z; };
inline thread_local Dim threadIdx{0, 0, 0};
inline Dim blockDim{1, 1, 1};
inline std::unique_ptr<std::barrier<>> block_barrier;
inline std::vector<std::unique_ptr<std::barrier<>>> warp_barrier;
inline std::vector<unsigned long long> lane_value;
template <class T> inline T __ldcg(const T* p) { return *p; }
inline void __syncthreads() { block_barrier->arrive_and_wait(); }
inline unsigned long long __shfl_xor_sync(unsigned, unsigned long long v, int o)
{
    lane_value[threadIdx.x] = v;
    warp_barrier[threadIdx.x / 32]->arrive_and_wait();
    const unsigned long long r = lane_value[threadIdx.x ^ o];
    warp_barrier[threadIdx.x / 32]->arrive_and_wait();
    return r;
}
"""

HARNESS = r"""
#include "miou.cuh"
#include <cstring>
// returns the number of bytes written outside the two arrays
extern "C" int run(const unsigned long long* conf, int C, int threads, int prefetched, double* out)
{
    static struct { unsigned char before[1024]; double iou[256]; unsigned char between[4096]; int present[256]; unsigned char after[4096]; } m;
    std::memset(&m, 0x5a, sizeof m);
    blockDim = {(unsigned)threads, 1, 1};
    block_barrier = std::make_unique<std::barrier<>>(threads);
    warp_barrier.clear();
    for (int k = 0; k < threads / 32; ++k) warp_barrier.push_back(std::make_unique<std::barrier<>>(32));
    lane_value.assign(threads, 0);
    std::vector<std::thread> block;
    for (int t = 0; t < threads; ++t)
        block.emplace_back([=] {
            threadIdx = {(unsigned)t, 0, 0};
            st::MiouFetch f{};
            if (prefetched) f = st::miou_fetch(conf, C);
            const double v = st::block_miou(conf, C, m.iou, m.present, prefetched ? &f : nullptr);
            if (t == 0) *out = v;
        });
    for (auto& t : block) t.join();
    int stray = 0;
    for (unsigned char b : m.before) stray += b != 0x5a;
    for (unsigned char b : m.between) stray += b != 0x5a;
    for (unsigned char b : m.after) stray += b != 0x5a;
    return stray;
}
// the same for a kernel's last block of 256 threads, which delivers the matrix as well
extern "C" double deliver(unsigned long long* conf, int C, unsigned long long* result, unsigned int* stage)
{
    static double iou[256];
    static int present[256];
    double mean = 0;
    blockDim = {256, 1, 1};
    block_barrier = std::make_unique<std::barrier<>>(256);
    warp_barrier.clear();
    for (int k = 0; k < 8; ++k) warp_barrier.push_back(std::make_unique<std::barrier<>>(32));
    lane_value.assign(256, 0);
    std::vector<std::thread> block;
    for (int t = 0; t < 256; ++t)
        block.emplace_back([=, &mean] {
            threadIdx = {(unsigned)t, 0, 0};
            const double v = st::deliver_matrix<256>(conf, C, result, stage, iou, present);
            if (t == 0) mean = v;
        });
    for (auto& t : block) t.join();
    return mean;
}
"""


@pytest.fixture(scope="module")
def block_miou(tmp_path_factory):
    d = tmp_path_factory.mktemp("miou")
    (d / "cuda_runtime.h").write_text(CUDA_FOR_HOST)
    (d / "harness.cpp").write_text(HARNESS)
    lib = d / "harness.so"
    subprocess.run(["g++", "-std=c++20", "-O1", "-shared", "-fPIC", "-pthread", "-w", f"-I{d}", f"-I{CSRC}", str(d / "harness.cpp"), "-o", str(lib)],
                   check=True)
    run = ctypes.CDLL(str(lib)).run

    def call(conf, threads, prefetched=False):
        out = ctypes.c_double()
        flat = np.ascontiguousarray(conf, np.uint64)
        stray = run(flat.ctypes.data_as(ctypes.c_void_p), conf.shape[0], threads, int(prefetched), ctypes.byref(out))
        return out.value, stray

    call.deliver = ctypes.CDLL(str(lib)).deliver
    call.deliver.restype = ctypes.c_double
    return call


def expected(conf):
    """mean over the classes with pixels of diag / (row + column - diag), added in class order"""
    total, n = 0.0, 0
    for c in range(conf.shape[0]):
        row, col, inter = int(conf[c].sum()), int(conf[:, c].sum()), int(conf[c, c])
        if row > 0:
            total += inter / (row + col - inter)
            n += 1
    return total / n if n else 0.0


def matrix(C, seed):
    rng = np.random.default_rng(seed)
    conf = rng.integers(0, 1000, (C, C)) + np.diag(rng.integers(0, 100000, C))
    conf[rng.integers(0, C)] = 0                               # a class without pixels
    return conf


# 320 threads: the backward kernel of a head with a hidden layer; 128: that of a one-layer head; 256: everything else
@pytest.mark.parametrize("threads", [64, 128, 256, 320, 512])
@pytest.mark.parametrize("C", [2, 21, 31, 32, 33, 255])        # around the size up to which the matrix is staged
def test_block_miou_stays_in_its_arrays(block_miou, C, threads):
    conf = matrix(C, 7 * C + threads)
    value, stray = block_miou(conf, threads)
    assert stray == 0
    assert value == expected(conf)                             # integer counts, the same double arithmetic in the same order


@pytest.mark.parametrize("C", [2, 19, 32])
def test_block_miou_with_prefetched_counts(block_miou, C):
    conf = matrix(C, C)
    assert block_miou(conf, 256, prefetched=True) == (expected(conf), 0)


def test_block_miou_of_an_empty_matrix(block_miou):
    assert block_miou(np.zeros((5, 5), np.int64), 320) == (0.0, 0)


@pytest.mark.parametrize("C", [2, 21, 32, 33, 45, 46, 81, 255])    # 2025, 2116: a pass of eight counts per thread ends at 2048
def test_last_block_delivers_the_matrix(block_miou, C):
    conf = matrix(C, C).astype(np.uint64)
    left, result, stage = np.append(conf, np.uint64(7)), np.full(C * C + 1, 5, np.uint64), np.full(C * C + 1, 3, np.uint32)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    assert block_miou.deliver(p(left), C, p(result), p(stage)) == expected(conf.astype(np.int64))
    assert (result[:-1] == conf.ravel()).all() and not left[:-1].any()
    assert (left[-1], result[-1], stage[-1]) == (7, 5, 3)
    assert block_miou.deliver(p(result), C, None, p(stage)) == expected(conf.astype(np.int64)) and (result[:-1] == conf.ravel()).all()
