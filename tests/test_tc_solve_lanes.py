"""The triangular solve of the tensor-core prefill (tc_solve of csrc/prefill_tc.cuh) under every
lane order that its barriers allow: U = L^-1 Y in place, heads in one, two or four value blocks.

The device function's own text is compiled for the host with the few intrinsics it uses.  Every
thread of the CTA is a fiber that runs, without being interrupted, up to its next barrier; the
fibers are taken up in a given order, so an access that only lockstep execution would order
comes out wrong.  The reference is the forward substitution, each element subtracting its
products in ascending row order with one rounding each: equal bit for bit."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_27513_gb300", "csrc")

HOST = r"""
#include <ucontext.h>
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <random>
#include <vector>
#define __device__
#define __forceinline__ inline
struct float2 { float x, y; };
struct uint4 { uint32_t x, y, z, w; };
static float2 make_float2(float x, float y) { return {x, y}; }
static uint4 make_uint4(uint32_t x, uint32_t y, uint32_t z, uint32_t w) { return {x, y, z, w}; }
static float __uint_as_float(uint32_t u) { float f; memcpy(&f, &u, 4); return f; }
static uint32_t __float_as_uint(float f) { uint32_t u; memcpy(&u, &f, 4); return u; }
static float2 splat2(float a) { return {a, a}; }
static float2 fma2(float2 a, float2 b, float2 c) { return {std::fma(a.x, b.x, c.x), std::fma(a.y, b.y, c.y)}; }
constexpr int kTcC = 64;
@CONSTANTS@
static std::vector<uint8_t> smem(64 * (kTcRowY + kTcRowL) * 4);
static void in_range(uint32_t a) { if (a % 16 || a + 16 > smem.size()) { puts("out of range"); exit(3); } }
static uint4 lds128(uint32_t a) { in_range(a); uint4 v; memcpy(&v, &smem[a], 16); return v; }
static void sts128(uint32_t a, uint4 v) { in_range(a); memcpy(&smem[a], &v, 16); }

// fibers and barriers: id 1, 2 count the threads given; 100 + warp is the warp's own
struct Barrier { int arrived = 0, phase = 0; };
static std::map<int, Barrier> bars;
struct Fiber { ucontext_t ctx; std::vector<char> stack; bool done = false; int bar = -1, phase = 0; };
static std::vector<Fiber> fibers;
static ucontext_t scheduler;
static int self;
static void arrive(int id, int threads) {
    Barrier &b = bars[id];
    if (++b.arrived == threads) { b.arrived = 0; ++b.phase; }
}
static void bar_arrive(int id, int threads) { arrive(id, threads); }
static void bar_sync(int id, int threads) {
    Fiber &f = fibers[self];
    f.bar = id;
    f.phase = bars[id].phase;
    arrive(id, threads);
    if (bars[id].phase == f.phase) swapcontext(&f.ctx, &scheduler);
    f.bar = -1;
}
static void __syncwarp() { bar_sync(100 + self / 32, 32); }

@SOLVE@

template <int NW, int NV> static void thread_main() {
    const int tid = self;
    tc_solve<NW, NV>(0u, (uint32_t)(64 * kTcRowY * 4), tid / 32, tid % 32);
    fibers[tid].done = true;
}

template <int NW, int NV> static bool check(int order) {
    std::mt19937 rng(7 * NW + NV);
    std::uniform_real_distribution<float> d(-1.f, 1.f);
    auto at = [](int off, int r, int c, int ld) { return (float *)&smem[off + 4 * (r * ld + c)]; };
    std::vector<float> L(64 * 64, 0.f), U(64 * 32 * NV);
    std::fill(smem.begin(), smem.end(), (uint8_t)0);
    for (int t = 0; t < 64; ++t)
        for (int s = 0; s < t; ++s) *at(64 * kTcRowY * 4, s, t, kTcRowL) = L[64 * t + s] = 0.2f * d(rng);
    for (int r = 0; r < 64; ++r)
        for (int c = 0; c < 32 * NV; ++c) *at(0, r, c, kTcRowY) = U[32 * NV * r + c] = d(rng);
    for (int c = 0; c < 32 * NV; ++c)
        for (int t = 0; t < 64; ++t)
            for (int s = 0; s < t; ++s)
                U[32 * NV * t + c] = std::fma(L[64 * t + s], -U[32 * NV * s + c], U[32 * NV * t + c]);
    bars.clear();
    fibers.assign(32 * NW, Fiber());
    std::vector<int> seq(32 * NW);
    for (int i = 0; i < 32 * NW; ++i) {
        seq[i] = order == 1 ? 32 * NW - 1 - i : i;
        Fiber &f = fibers[i];
        f.stack.resize(64 << 10);
        getcontext(&f.ctx);
        f.ctx.uc_stack.ss_sp = f.stack.data();
        f.ctx.uc_stack.ss_size = f.stack.size();
        f.ctx.uc_link = &scheduler;
        makecontext(&f.ctx, (void (*)())thread_main<NW, NV>, 0);
    }
    for (int left = 32 * NW; left > 0;) {
        if (order > 1) std::shuffle(seq.begin(), seq.end(), rng);
        bool ran = false;
        for (int i : seq) {
            Fiber &f = fibers[i];
            if (f.done || (f.bar >= 0 && bars[f.bar].phase == f.phase)) continue;
            self = i;
            swapcontext(&scheduler, &f.ctx);
            ran = true;
            left -= f.done;
        }
        if (!ran) { puts("no thread can run"); return false; }
    }
    for (int r = 0; r < 64; ++r)
        for (int c = 0; c < 32 * NV; ++c)
            if (memcmp(at(0, r, c, kTcRowY), &U[32 * NV * r + c], 4) != 0) {
                printf("order %d: row %d column %d is %g, expected %g\n", order, r, c, *at(0, r, c, kTcRowY), U[32 * NV * r + c]);
                return false;
            }
    return true;
}

int main() {
    for (int order = 0; order < 4; ++order)
        if (!check<@NW@, @NV@>(order)) return 1;
    return 0;
}
"""


@pytest.mark.parametrize("nv", [1, 2, 4])
@pytest.mark.parametrize("nw", [8, 16])
def test_solve_holds_in_every_lane_order(nw, nv, tmp_path):
    text = open(os.path.join(CSRC, "prefill_tc.cuh")).read()
    solve = re.search(r"^template <int NW, int NV>\n__device__ __forceinline__ void tc_solve\(.*?^}\n", text, re.S | re.M)
    consts = re.findall(r"^constexpr int (?:kTcRowL|kTcRowY) = \d+;", text, re.M)
    assert solve and len(consts) == 2
    src = tmp_path / "solve.cpp"
    src.write_text(HOST.replace("@CONSTANTS@", "\n".join(consts)).replace("@SOLVE@", solve.group(0))
                   .replace("@NW@", str(nw)).replace("@NV@", str(nv)))
    cxx = shutil.which("g++")
    assert cxx, "the test compiles the solve for the host"
    exe = str(tmp_path / "solve")
    subprocess.run([cxx, "-std=c++17", "-O1", "-ffp-contract=off", "-w", str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
