// decode_fp32.cu -- the FP32-state step (the deployment baseline of Sec. 6.1: FP32
// recurrent-state storage) and the FP32 trajectories of a calibration run, GDN and KDA.
//
// The pipelined kernel (fp32_tokens_kernel): a unit is up to four value blocks of one (slot,
// head); a CTA of four warps walks units (persistent), warp w holding a tile of d_k rows x 32
// columns in registers over the launch's tokens (one token for a decode step).  Lane (pc, cg) = (lane / 8, lane % 8) holds
// columns 4 cg .. 4 cg + 3 of the rows u = pc mod 4:
//   * a row is 128 bytes of 16-byte accesses (whole lines in memory, no bank conflicts);
//   * the sums over the rows run as four chains (rows 0, 4, 8, ..; 1, 5, 9, ..; ...), one
//     per lane quarter, which meet by two shuffles as (c0 + c1) + (c2 + c3);
//   * a lane reads the operands of its own d_k / 4 rows only and uses each for four
//     columns: 24 (KDA) 16-byte shared loads per token and tile instead of 96 with one
//     column per lane, which were the limit of a multi-token launch.
// The next unit's state lands in shared memory by bulk copies while the current one is
// computed from registers and stored; the per-channel operands (k, q, decay, beta k) are
// staged once per unit and NT tokens from copies made in the same way.
//
// Measured (B = 64, H = 32, d = 128, GDN, 268 MB of state per step, more than L2): 45.0 us, 6.0
// TB/s, bound by HBM; 47.8 us with one column per lane and each tile loaded, computed and
// stored in turn (fp32_tile_kernel, which stays for shapes that leave these CTAs part empty).  A
// calibration run over 32 documents (KDA): 16 us for one token (the 134 MB that the states move
// through L2) and 2.1 us for each further one up to eight (31 us), 2.5 us in longer runs, whose
// operands come eight tokens at a time -- FP32 arithmetic (1.3 us at the FMA rate) and the operand
// loads, with two warps per scheduler.  With one launch per token eight tokens took 127 us.
#include "damp_common.cuh"
#include "damp_internal.h"

#include <algorithm>

namespace damp {

static __device__ uint32_t g_status_fp32;

struct Fp32Params {
    float *state;
    int64_t num_slots;
    const int32_t *slot_idx;
    const void *q, *k, *v;
    const float *g, *beta;
    float *o;
    int32_t batch, H, Hqk, dv, V, VG;  // VG: groups of four value blocks per (slot, head)
    int32_t n_tokens;                  // token t's operands lie t * batch rows further on
    int64_t units;                     // of four value blocks each (pipelined kernel), or tiles
    uint32_t *status;
};

constexpr int kFp32Warps = 4;
constexpr int kFp32Ctas = 2;    // CTAs per SM: a third (168 registers a thread) spills, step 47 -> 54 us (below)
constexpr int kFp32Tokens = 8;  // tokens staged at a time by a calibration run
constexpr int kFp32TileWarps = 8;
constexpr int64_t kFp32L2Bytes = 129000000;

// A staged operand vector.  A run's loads keep their place in the program (one group of four rows
// ahead of their use): left to the compiler, they are all moved to the front of the token, over the
// registers that hold the state (170 bytes of spills; a 32 x 256 run 1805 us, so 1680).
template <bool RUN>
__device__ __forceinline__ float4 staged4(const float *p) {
    if (!RUN) return *reinterpret_cast<const float4 *>(p);
    const uint4 w = lds128(smem_u32(p));
    return make_float4(__uint_as_float(w.x), __uint_as_float(w.y), __uint_as_float(w.z), __uint_as_float(w.w));
}

// RUN: a calibration run of p.n_tokens tokens without outputs; otherwise one decode step.
// DV > 0 fixes d_v (row addresses become immediate offsets).
template <int DK, int DV, bool KDA, bool BF16, bool RUN>
__global__ void __launch_bounds__(32 * kFp32Warps, kFp32Ctas) fp32_tokens_kernel(const Fp32Params p) {
    constexpr int NT = RUN ? kFp32Tokens : 1;
    constexpr int RP = DK / 4;  // rows per lane
    constexpr int ESZ = BF16 ? 2 : 4;
    extern __shared__ __align__(128) uint8_t state_buf[];  // the next unit's state, row after row
    // staged operands: channel u = 4 i + c at [c][i], so that a lane's rows are contiguous
    __shared__ __align__(16) float sk[NT][DK], sb[NT][DK], sa[KDA ? NT : 1][DK], sq[RUN ? 1 : NT][DK];
    __shared__ __align__(16) float sv[NT][32 * kFp32Warps];
    __shared__ float salpha[NT];
    // the operands as they lie in memory (cp.async)
    __shared__ __align__(16) uint8_t rk[NT][DK * ESZ], rq[RUN ? 1 : NT][RUN ? 16 : DK * ESZ], rv[NT][kFp32Warps * 32 * ESZ];
    __shared__ __align__(16) float rg[NT][KDA ? DK : 4], rbeta[NT];
    __shared__ __align__(8) uint64_t bar_mem;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nthr = DV == 128 ? 128 : blockDim.x;
    const int pc = lane >> 3, cg = lane & 7;
    const uint32_t bar = smem_u32(&bar_mem), sbuf = smem_u32(state_buf);
    const int64_t ld = DV > 0 ? DV : p.dv;
    const int H = p.H, VG = p.VG;
    if (tid == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
    }
    __syncthreads();

    struct Unit {
        int64_t slot;
        int b, h, c0, ncol;  // batch row, head, first value block, value columns
        bool ok;             // false past the last unit
    };
    bool bad_slot = false;
    int64_t at = blockIdx.x;  // the next unit to look at
    // the next unit whose slot is in the pool
    auto next_unit = [&]() {
        Unit n{0, 0, 0, 0, 0, false};
        for (; at < p.units && !n.ok; at += gridDim.x) {
            const int64_t bh = at / VG;
            n.c0 = (int)(at - bh * VG) * kFp32Warps;
            n.b = (int)(bh / H);
            n.h = (int)(bh - (int64_t)n.b * H);
            n.ncol = DV == 128 ? 128 : min(kFp32Warps, p.V - n.c0) * kG;
            n.slot = p.slot_idx ? (int64_t)p.slot_idx[n.b] : (int64_t)n.b;
            n.ok = n.slot >= 0 && n.slot < p.num_slots;
            bad_slot |= !n.ok;
        }
        return n;
    };
    auto unit_base = [&](const Unit &n) { return p.state + (n.slot * H + n.h) * DK * ld + (int64_t)n.c0 * kG; };
    auto fetch_state = [&](const Unit &n) {  // thread 0: one copy of a whole (slot, head), or one per row
        if (tid != 0) return;
        fence_proxy_async_smem();  // the CTA's reads of the buffer before the copies' writes
        mbar_arrive_expect_tx(bar, (uint32_t)(DK * n.ncol * 4));
        const float *src = unit_base(n);
        if (VG == 1) {
            bulk_g2s(sbuf, src, (uint32_t)(DK * n.ncol * 4), bar);
        } else {
            for (int u = 0; u < DK; ++u) bulk_g2s(sbuf + (uint32_t)(u * n.ncol * 4), src + u * ld, (uint32_t)(n.ncol * 4), bar);
        }
    };
    auto fetch_operands = [&](const Unit &n, int t0, int nt) {  // of the tokens t0 .. t0 + nt - 1
        constexpr int nk = DK * ESZ / 16, nq = RUN ? 0 : nk, ng = KDA ? DK / 4 : 0;
        const int per = nk + nq + ng + n.ncol * ESZ / 16;
        const int hq = (n.h * p.Hqk) / H;
        for (int i = tid; i < nt * per; i += nthr) {
            const int s = RUN ? i / per : 0;
            int j = i - s * per;
            const int64_t row = (int64_t)(t0 + s) * p.batch + n.b;
            if (j < nk) {
                cp_async16(smem_u32(rk[s]) + 16 * j, static_cast<const uint8_t *>(p.k) + (row * p.Hqk + hq) * (DK * ESZ) + 16 * j);
            } else if ((j -= nk) < nq) {
                cp_async16(smem_u32(rq[s]) + 16 * j, static_cast<const uint8_t *>(p.q) + (row * p.Hqk + hq) * (DK * ESZ) + 16 * j);
            } else if ((j -= nq) < ng) {
                cp_async16(smem_u32(rg[s]) + 16 * j, p.g + (row * H + n.h) * DK + 4 * j);
            } else {
                j -= ng;
                cp_async16(smem_u32(rv[s]) + 16 * j,
                           static_cast<const uint8_t *>(p.v) + ((row * H + n.h) * p.dv + n.c0 * kG) * ESZ + 16 * j);
            }
        }
        if (tid < nt) {
            const int64_t row = ((int64_t)(t0 + tid) * p.batch + n.b) * H + n.h;
            cp_async4(smem_u32(&rbeta[tid]), p.beta + row);
            if (!KDA) cp_async4(smem_u32(&rg[tid][0]), p.g + row);
        }
        cp_async_commit();
    };

    const int n_tokens = RUN ? p.n_tokens : 1;
    auto ld4 = [](const float *at) { return staged4<RUN>(at); };
    Unit cur = next_unit();
    if (cur.ok) {
        fetch_state(cur);
        fetch_operands(cur, 0, min(NT, n_tokens));
    }
    uint32_t parity = 0;
    bool timed_out = false;
    while (cur.ok) {
        const Unit nxt = next_unit();
        cp_async_wait_all();
        if (!__syncthreads_and(mbar_wait_bounded(bar, parity))) {  // the state and the first tokens' operands
            timed_out = true;
            break;
        }
        parity ^= 1u;
        const bool live = warp * kG < cur.ncol;  // the last group of a d_v that is no multiple of 128 has idle warps
        float2 x[RP][2];
        if (live) {
            const uint32_t src = sbuf + (uint32_t)((pc * cur.ncol + warp * kG + 4 * cg) * 4);
#pragma unroll
            for (int i = 0; i < RP; ++i) {
                const uint4 w = lds128(src + (uint32_t)(16 * i * (DV > 0 ? DV : cur.ncol)));
                x[i][0] = make_float2(__uint_as_float(w.x), __uint_as_float(w.y));
                x[i][1] = make_float2(__uint_as_float(w.z), __uint_as_float(w.w));
            }
        }
#pragma unroll 1
        for (int t0 = 0; t0 < n_tokens; t0 += NT) {
            const int nt = min(NT, n_tokens - t0);
            if (RUN && t0 > 0) {
                cp_async_wait_all();
                __syncthreads();  // these tokens' operands are here, the last ones' staged form is read
            }
            for (int u = tid; u < DK; u += nthr) {
                const int to = (u & 3) * RP + (u >> 2);
#pragma unroll 2
                for (int s = 0; s < nt; ++s) {
                    const float kv = load_in(rk[s], u, BF16);
                    sk[s][to] = kv;
                    sb[s][to] = rbeta[s] * kv;
                    if (!RUN) sq[s][to] = load_in(rq[s], u, BF16);
                    if (KDA) sa[s][to] = expf(rg[s][u]);
                }
            }
            if (!KDA && tid < nt) salpha[tid] = expf(rg[tid][0]);
            for (int j = tid; j < cur.ncol; j += nthr) {
                for (int s = 0; s < nt; ++s) sv[s][j] = load_in(rv[s], j, BF16);
            }
            __syncthreads();
            const bool last = t0 + NT >= n_tokens;
            if (!last) {
                fetch_operands(cur, t0 + NT, min(NT, n_tokens - t0 - NT));
            } else if (nxt.ok) {
                fetch_operands(nxt, 0, min(NT, n_tokens));
            }
            if (t0 == 0 && nxt.ok) fetch_state(nxt);  // every warp has its tile in registers
            if (!live) continue;
#pragma unroll 1
            for (int s = 0; s < nt; ++s) {
                const float *ka = sk[s] + pc * RP, *ba = sb[s] + pc * RP, *aa = sa[KDA ? s : 0] + pc * RP;
                const float *qa = sq[RUN ? 0 : s] + pc * RP;
                const float alpha = KDA ? 0.f : salpha[s];
                // S_bar = Lambda S ; r = S_bar^T k
                float2 rp[2] = {splat2(0.f), splat2(0.f)};
                float4 kn = ld4(ka), an = KDA ? ld4(aa) : make_float4(alpha, alpha, alpha, alpha);
#pragma unroll
                for (int i4 = 0; i4 < RP / 4; ++i4) {
                    const float4 k4 = kn, a4 = an;
                    if (i4 + 1 < RP / 4) {
                        kn = ld4(ka + 4 * i4 + 4);
                        if (KDA) an = ld4(aa + 4 * i4 + 4);
                    }
                    const float kk[4] = {k4.x, k4.y, k4.z, k4.w}, av[4] = {a4.x, a4.y, a4.z, a4.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
#pragma unroll
                        for (int m = 0; m < 2; ++m) {
                            float2 &w = x[4 * i4 + e][m];
                            w = mul2(w, splat2(av[e]));
                            rp[m] = fma2(w, splat2(kk[e]), rp[m]);
                        }
                    }
                }
                const float4 v4 = ld4(sv[s] + warp * kG + 4 * cg);
                float4 bn = ld4(ba), qn = RUN ? bn : ld4(qa);
                float r[4] = {rp[0].x, rp[0].y, rp[1].x, rp[1].y};
#pragma unroll
                for (int m = 8; m <= 16; m <<= 1) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) r[e] += __shfl_xor_sync(kFull, r[e], m);
                }
                const float2 d[2] = {make_float2(v4.x - r[0], v4.y - r[1]), make_float2(v4.z - r[2], v4.w - r[3])};
                // S = S_bar + beta k d^T ; o = S^T q
                float2 op[2] = {splat2(0.f), splat2(0.f)};
#pragma unroll
                for (int i4 = 0; i4 < RP / 4; ++i4) {
                    const float4 b4 = bn, q4 = qn;
                    if (i4 + 1 < RP / 4) {
                        bn = ld4(ba + 4 * i4 + 4);
                        qn = RUN ? bn : ld4(qa + 4 * i4 + 4);
                    }
                    const float bb[4] = {b4.x, b4.y, b4.z, b4.w}, qv[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
#pragma unroll
                        for (int m = 0; m < 2; ++m) {
                            float2 &w = x[4 * i4 + e][m];
                            w = fma2(splat2(bb[e]), d[m], w);
                            if (!RUN) op[m] = fma2(w, splat2(qv[e]), op[m]);
                        }
                    }
                }
                if (!RUN) {
                    float o[4] = {op[0].x, op[0].y, op[1].x, op[1].y};
#pragma unroll
                    for (int m = 8; m <= 16; m <<= 1) {
#pragma unroll
                        for (int e = 0; e < 4; ++e) o[e] += __shfl_xor_sync(kFull, o[e], m);
                    }
                    // every lane of a column group holds the sums: lane (pc, cg) writes column 4 cg + pc
                    p.o[((int64_t)cur.b * H + cur.h) * ld + (cur.c0 + warp) * kG + 4 * cg + pc] =
                        pc == 0 ? o[0] : pc == 1 ? o[1] : pc == 2 ? o[2] : o[3];
                }
            }
        }
        if (live) {
            float *dst = unit_base(cur) + pc * ld + warp * kG + 4 * cg;
#pragma unroll
            for (int i = 0; i < RP; ++i) {
                const float4 w = make_float4(x[i][0].x, x[i][0].y, x[i][1].x, x[i][1].y);
                if (RUN) *reinterpret_cast<float4 *>(dst + 4 * i * ld) = w;
                else __stcs(reinterpret_cast<float4 *>(dst + 4 * i * ld), w);
            }
        }
        cur = nxt;
    }
    if (timed_out) mbar_wait_bounded(bar, parity);  // one more bounded wait before the buffer goes away
    cp_async_wait_all();
    if (tid == 0) {
        const uint32_t bits = (timed_out ? kDevWaitTimeout : 0u) | (bad_slot ? kDevBadSlot : 0u);
        if (bits) atomicOr(p.status, bits);
    }
}

// The step of the shapes whose CTAs the pipelined kernel cannot fill (launch_fp32_step): one warp
// per tile of d_k rows x 32 columns, lane j owns column j for all rows, so both sums over the rows
// are its own (as four chains, in the same order as above: same bits) and every load or store of a
// row is one 128-byte line.  d_k independent loads in flight per warp, eight warps per SM whatever
// d_v; bound by HBM latency times what those keep in flight.  Also the single tokens of a
// calibration run (no outputs: o is null).
template <int DK, int DV, bool KDA, bool BF16>
__global__ void __launch_bounds__(32 * kFp32TileWarps, 1) fp32_tile_kernel(const Fp32Params p) {
    __shared__ __align__(16) float ops[kFp32TileWarps][4][DK];  // k, q, a, beta*k per channel
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int nw = blockDim.x >> 5;
    float *sk = ops[warp][0];
    float *sq = ops[warp][1];
    float *sa = ops[warp][2];
    float *sb = ops[warp][3];

    const int64_t gw = (int64_t)blockIdx.x * nw + warp;
    const int64_t nwt = (int64_t)gridDim.x * nw;
    const int64_t t0 = p.units * gw / nwt;
    const int64_t t1 = p.units * (gw + 1) / nwt;
    bool bad_slot = false;

    for (int64_t t = t0; t < t1; ++t) {
        const int c = (int)(t % p.V);
        const int64_t bh = t / p.V;
        const int h = (int)(bh % p.H);
        const int b = (int)(bh / p.H);
        if (t == t0 || c == 0) {
            __syncwarp();
            const int hq = (h * p.Hqk) / p.H;
            const int64_t qoff = ((int64_t)b * p.Hqk + hq) * DK;
            const float beta = p.beta[(int64_t)b * p.H + h];
            const float alpha = KDA ? 0.f : expf(p.g[(int64_t)b * p.H + h]);
#pragma unroll
            for (int u = lane; u < DK; u += 32) {
                const float kv = load_in(p.k, qoff + u, BF16);
                sk[u] = kv;
                sq[u] = load_in(p.q, qoff + u, BF16);
                sa[u] = KDA ? expf(p.g[((int64_t)b * p.H + h) * DK + u]) : alpha;
                sb[u] = beta * kv;
            }
            __syncwarp();
        }
        const int64_t slot = p.slot_idx ? (int64_t)p.slot_idx[b] : (int64_t)b;
        if (slot < 0 || slot >= p.num_slots) {
            bad_slot = true;
            continue;
        }
        float *base = p.state + ((slot * p.H + h) * DK) * (int64_t)p.dv + c * kG + lane;
        // a compile-time row stride (DV > 0) turns every row address into an
        // immediate offset from one base register
        const int64_t ld = DV > 0 ? DV : p.dv;
        float x[DK];
#pragma unroll
        for (int u = 0; u < DK; ++u) x[u] = __ldcs(base + u * ld);
        const float vj = load_in(p.v, ((int64_t)b * p.H + h) * p.dv + c * kG + lane, BF16);

        // S_bar = Lambda S ; r = S_bar^T k
        float r0 = 0.f, r1 = 0.f, r2 = 0.f, r3 = 0.f;
#pragma unroll
        for (int u = 0; u < DK; u += 4) {
            const float4 a4 = *reinterpret_cast<const float4 *>(sa + u);
            const float4 k4 = *reinterpret_cast<const float4 *>(sk + u);
            x[u] *= a4.x;
            x[u + 1] *= a4.y;
            x[u + 2] *= a4.z;
            x[u + 3] *= a4.w;
            r0 = fmaf(x[u], k4.x, r0);
            r1 = fmaf(x[u + 1], k4.y, r1);
            r2 = fmaf(x[u + 2], k4.z, r2);
            r3 = fmaf(x[u + 3], k4.w, r3);
        }
        const float d = vj - ((r0 + r1) + (r2 + r3));
        // S = S_bar + beta k d^T ; o = S^T q
        float o0 = 0.f, o1 = 0.f, o2 = 0.f, o3 = 0.f;
#pragma unroll
        for (int u = 0; u < DK; u += 4) {
            const float4 b4 = *reinterpret_cast<const float4 *>(sb + u);
            const float4 q4 = *reinterpret_cast<const float4 *>(sq + u);
            x[u] = fmaf(b4.x, d, x[u]);
            x[u + 1] = fmaf(b4.y, d, x[u + 1]);
            x[u + 2] = fmaf(b4.z, d, x[u + 2]);
            x[u + 3] = fmaf(b4.w, d, x[u + 3]);
            o0 = fmaf(x[u], q4.x, o0);
            o1 = fmaf(x[u + 1], q4.y, o1);
            o2 = fmaf(x[u + 2], q4.z, o2);
            o3 = fmaf(x[u + 3], q4.w, o3);
        }
        // a fresh copy of the row pointer keeps the compiler from holding all
        // d_k load addresses live until the stores
#pragma unroll
        for (int u = 0; u < DK; ++u) __stcs(base + u * ld, x[u]);
        if (p.o) p.o[((int64_t)b * p.H + h) * p.dv + c * kG + lane] = (o0 + o1) + (o2 + o3);  // no o: calibration runs
    }
    if (bad_slot && lane == 0) atomicOr(p.status, (uint32_t)kDevBadSlot);
}


static cudaError_t fp32_params(const StepArgs &a, Fp32Params &p) {
    static std::atomic<uint32_t *> cache[64];
    const cudaError_t e = symbol_address_cached(&g_status_fp32, cache, &p.status);
    if (e != cudaSuccess) return e;
    p.state = static_cast<float *>(a.state);
    p.num_slots = a.num_slots;
    p.slot_idx = a.slot_idx;
    p.q = a.q;
    p.k = a.k;
    p.v = a.v;
    p.g = a.g;
    p.beta = a.beta;
    p.o = a.o;
    p.batch = a.batch;
    p.H = a.H;
    p.Hqk = a.Hqk;
    p.dv = a.dv;
    p.V = a.dv / kG;
    p.VG = (p.V + kFp32Warps - 1) / kFp32Warps;
    return cudaSuccess;
}

#define DAMP_PICK4(KERN_, DK_, DV_, ...)                                                           \
    if (a.kda) kern = a.in_bf16 ? KERN_<DK_, DV_, true, true __VA_ARGS__> : KERN_<DK_, DV_, true, false __VA_ARGS__>; \
    else kern = a.in_bf16 ? KERN_<DK_, DV_, false, true __VA_ARGS__> : KERN_<DK_, DV_, false, false __VA_ARGS__>;

template <bool RUN>
static cudaError_t launch_fp32(const StepArgs &a, int32_t n_tokens, cudaStream_t stream) {
    Fp32Params p{};
    cudaError_t e = fp32_params(a, p);
    if (e != cudaSuccess) return e;
    p.n_tokens = n_tokens;
    p.units = (int64_t)a.batch * a.H * p.VG;
    if (p.units == 0 || n_tokens == 0) return cudaSuccess;
    void (*kern)(Fp32Params) = nullptr;
#define DAMP_COMMA_RUN , RUN
#define DAMP_PICK(DK_)                                                                             \
    if (a.dk == DK_) {                                                                             \
        if (a.dv == 128) { DAMP_PICK4(fp32_tokens_kernel, DK_, 128, DAMP_COMMA_RUN) }              \
        else { DAMP_PICK4(fp32_tokens_kernel, DK_, 0, DAMP_COMMA_RUN) }                            \
    }
    if constexpr (RUN) { DAMP_PICK(32) }  // (a step of d_k = 32 never comes here)
    DAMP_PICK(64)
    DAMP_PICK(128)
#undef DAMP_PICK
#undef DAMP_COMMA_RUN
    if (!kern) return cudaErrorInvalidValue;
    const int warps = std::min(p.V, kFp32Warps), smem = a.dk * warps * kG * 4;
    if ((e = ensure_smem_limit(reinterpret_cast<const void *>(kern), smem)) != cudaSuccess) return e;
    const int grid = (int)std::min<int64_t>(p.units, (int64_t)sm_count() * kFp32Ctas);
    kern<<<grid, 32 * warps, smem, stream>>>(p);
    return cudaGetLastError();
}

static cudaError_t launch_fp32_tile(const StepArgs &a, cudaStream_t stream) {
    Fp32Params p{};
    const cudaError_t e = fp32_params(a, p);
    if (e != cudaSuccess) return e;
    p.n_tokens = 1;
    p.units = (int64_t)a.batch * a.H * p.V;  // tiles
    if (p.units == 0) return cudaSuccess;
    void (*kern)(Fp32Params) = nullptr;
#define DAMP_PICK(DK_)                                                                             \
    if (a.dk == DK_) {                                                                             \
        if (a.dv == 64) { DAMP_PICK4(fp32_tile_kernel, DK_, 64) }                                  \
        else if (a.dv == 128) { DAMP_PICK4(fp32_tile_kernel, DK_, 128) }                           \
        else { DAMP_PICK4(fp32_tile_kernel, DK_, 0) }                                              \
    }
    DAMP_PICK(32)
    DAMP_PICK(64)
    DAMP_PICK(128)
#undef DAMP_PICK
    if (!kern) return cudaErrorInvalidValue;
    const int64_t want = (p.units + kFp32TileWarps - 1) / kFp32TileWarps;
    kern<<<(int)std::min<int64_t>(want, (int64_t)sm_count()), 32 * kFp32TileWarps, 0, stream>>>(p);
    return cudaGetLastError();
}
#undef DAMP_PICK4

// The pipelined kernel where its CTAs are full: two CTAs of up to four warps per SM move a 32 KB
// (64 x 128) to 64 KB state each, so it needs tall tiles and whole groups of four value blocks
// (or one of three).  Measured, pipelined / tile kernel, H = 32, states from memory:
//   d_k = 128: d_v = 96, B = 64: 38 / 57 us; 128: 45 / 48; 256: 117 / 145; 1024: 488 / 578;
//     a group with idle warps: d_v = 32: 23 / 20, 64: 29 / 27, 160: 116 / 90, 288: 165 / 163;
//   d_k = 64: d_v = 128, B = 256: 84 / 98, but from L2 (B = 64) 17 / 15; 64, B = 256: 55 / 52; 160: 214 / 131;
//   d_k = 32: 32 x 32, B = 256: 40 / 17; 32 x 128: even, from L2 13 / 9.
// A call of few units gives each its own CTA, where the tile kernel packs eight tiles into one:
//   128 x 32, B = 8: 5 / 11; 64 x 64, B = 8: 3.6 / 4.3; 128 x 160, B = 2: 9.3 / 11.
// At d_k = 128 from L2 a wave of CTAs that is part full costs the pipelined kernel as much as a full
// one, where the tile kernel gives every SM a smaller share (fp32_uneven; 152 SMs, a wave is 304 units):
//   d_v = 128: 400 units 7.7 / 8.3 us, 432: 9.1 / 8.5, 528: 9.35 / 9.2, 560: 9.4 / 9.5, 784: 12.8 / 12.4,
//     1024: 14.1 / 15.8;
//   d_v = 256 (rows copied one by one), GDN: 144 units 9.1 / 10.1, 208: 10.7 / 10.2, 336: 16.9 / 13.7,
//     496: 18.4 / 16.1, 624: 24.7 / 22.2, 784: 26.0 / 25.7, 816: 26.1 / 27.2; KDA: 304 10.6 / 10.8, 336:
//     15.9 / 13.8, 528: 17.6 / 17.1, 560: 17.6 / 17.7, 624: 23.2 / 22.3, 720: 23.2 / 24.3.
static bool fp32_uneven(int64_t V, int64_t units, bool kda) {
    const int64_t sms = sm_count(), last = units % (2 * sms);
    if (V == 3) return false;
    if (V == 4) return units > 2 * sms && units < 6 * sms && 5 * last > 4 * sms && 2 * last <= 3 * sms;
    return kda ? units > 2 * sms && 5 * units <= 22 * sms && 2 * last <= 3 * sms : units > sms && 4 * units <= 21 * sms;
}

static bool fp32_pipelined(const StepArgs &a) {
    const int64_t V = a.dv / kG, VG = (V + kFp32Warps - 1) / kFp32Warps, units = (int64_t)a.batch * a.H * VG;
    const bool full = V % kFp32Warps == 0 || V == 3;
    if (a.dk == 128) return units <= sm_count() || (full && !fp32_uneven(V, units, a.kda));
    if (a.dk < 64 || VG > 1) return false;
    return units <= 2 * sm_count() || (full && (int64_t)a.batch * a.H * a.dk * a.dv * 4 > kFp32L2Bytes);
}

cudaError_t launch_fp32_step(const StepArgs &a, cudaStream_t stream) {
    return fp32_pipelined(a) ? launch_fp32<false>(a, 1, stream) : launch_fp32_tile(a, stream);
}
// A run of a few tokens has too little to gain from the states staying in registers: single steps
// on the tile kernel.  Per 12 tokens of 32 documents with the samples' error passes, run / steps:
// one token a run: GDN 128 x 128 398 / 359 us, 64 x 64 222 / 174, 32 x 32 158 / 102, KDA 128 x 64 256
// / 223, but KDA 128 x 128 366 / 386; two: GDN 128 x 128 212 / 282, 64 x 64 119 / 125, 32 x 32 86 /
// 73; three: GDN 32 x 32 even; four: GDN 32 x 32 51 / 58, 32 x 128 78 / 119.
static bool fp32_run_pays(const StepArgs &a, int32_t n_tokens) {
    const int64_t V = a.dv / kG, rows = (int64_t)n_tokens * a.dk;
    if (n_tokens == 1) return a.kda && a.dk == 128 && (V % kFp32Warps == 0 || V == 3);
    return rows >= 128;
}

cudaError_t launch_fp32_run(const StepArgs &a, int32_t n_tokens, cudaStream_t stream) {
    if (fp32_run_pays(a, n_tokens)) return launch_fp32<true>(a, n_tokens, stream);
    const int64_t B = a.batch, esz = a.in_bf16 ? 2 : 4;
    const int64_t sq = B * a.Hqk * a.dk * esz, sv = B * a.H * a.dv * esz, sg = B * a.H * (a.kda ? a.dk : 1);
    StepArgs t = a;
    for (int32_t i = 0; i < n_tokens; ++i) {
        t.q = static_cast<const uint8_t *>(a.q) + i * sq;
        t.k = static_cast<const uint8_t *>(a.k) + i * sq;
        t.v = static_cast<const uint8_t *>(a.v) + i * sv;
        t.g = a.g + i * sg;
        t.beta = a.beta + i * B * a.H;
        const cudaError_t e = launch_fp32_tile(t, stream);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t take_status_fp32(uint32_t *bits) {
    uint32_t zero = 0;
    cudaError_t e = cudaMemcpyFromSymbol(bits, g_status_fp32, sizeof(uint32_t));
    if (e != cudaSuccess) return e;
    return cudaMemcpyToSymbol(g_status_fp32, &zero, sizeof(uint32_t));
}

}  // namespace damp
