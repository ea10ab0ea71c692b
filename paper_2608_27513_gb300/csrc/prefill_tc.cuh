// prefill_tc.cuh -- the GDN prefill chunk on the tensor cores (App. A.5 prefill path),
// in the chunkwise closed form of the delta rule (Sec. 3.1, Eq. delta_update).
//
// Within a piece of C = 64 tokens, with a_t = exp(g_t), the decay from token s to token
// t f_ts = a_{s+1} ... a_t (f_tt = 1), gamma_t = a_0 ... a_t and u_t the update column
// of token t (S_t = a_t S_{t-1} + k_t u_t^T), the per-token recurrence unrolls to
//     u_t + beta_t sum_{s<t} f_ts (k_t . k_s) u_s = beta_t (v_t - gamma_t S_0^T k_t)
//     o_t = gamma_t S_0^T q_t + sum_{s<=t} f_ts (q_t . k_s) u_s
//     S_C = gamma_C S_0 + sum_s f_Cs k_s u_s^T .
// With L = I + (beta_t f_ts k_t.k_s)_{s<t} (unit lower triangular),
// M = (f_ts q_t.k_s)_{s<=t} and Y = diag(beta) (V - diag(gamma) K S_0):
//     U = L^-1 Y,  O = diag(gamma) Q S_0 + M U,  S_C = gamma_C S_0 + K^T diag(f_C.) U.
// One CTA of eight warps owns a unit for the whole chunk: a (slot, head), or one or two of
// its four value blocks where few heads run (tc_nv).  Its state stays in tensor memory
// (FP32, lane = record row) from the reconstruction of the packed records to the
// requantization.  Per piece, four tcgen05.mma products (bf16 operands, FP32
// accumulation in tensor memory, M = 128):
//     [K; Q] S_0         -> W = K S_0 (lanes 0-63), P = Q S_0 (lanes 64-127)
//     [K; Q] K^T         -> K K^T, Q K^T
//     [.; M] U           -> accumulated onto gamma P: O (lanes 64-127; rows 0-63 of the
//                           operand are whatever their bytes hold, lanes 0-63 are not read)
//     K^T (f_C. U)       -> accumulated onto gamma_C S_0
// k and q are bf16 inputs (exact operands); the FP32 operands (S_0, M, U, f_C. U) enter
// as three bf16 parts x = hi + mid + lo (24 significant bits), and a product of two split
// operands takes the six partial products down to 2^-16 relative, so the products keep
// FP32 accuracy.  U = L^-1 Y is solved by forward substitution on the CUDA cores (tc_solve:
// each warp a few rows of all columns, in register tiles), where the decay factors
// (running products and shuffle scans: no cancellation of cumulative log sums) and the
// requantization run too.  With the H_32 formats the whole chunk runs in the transformed domain
// (S~ = S H, v~ = v H, o = o~ H per value block of 32), as the other prefill kernels do.
#pragma once

#include <cuda_bf16.h>

#include "prefill.cuh"

namespace damp {

constexpr int kTcC = 64;          // tokens per piece
constexpr int kTcThreads = 256;   // two threads per tensor-memory lane (warps w and w + 4)
constexpr uint32_t kTcCols = 512; // tensor-memory columns of the CTA (one CTA per SM)
// tensor-memory columns of the accumulators: W | P then O (lanes 64-127), S, K K^T | Q K^T
constexpr uint32_t kColWP = 0, kColS = 128, kColG = 256;
// Shared memory (bytes from the base of the dynamic shared memory).  Each area is live
// from the step that writes it to the step that last reads it; areas that share bytes
// are never live together:
//   staging:        A1 [0, 32K)  B1 [32K, 128K)  records (unit start) [128K, 160K)  V [160K, 177K)
//   after [K;Q]S_0: A3 [16K, 32K)  AO [32K, 80K)  LP [80K, 97K)  YU [97K, 130K)
//   after the solve: BU [80K, 128K)  B4 [128K, 176K)
constexpr int kSmA1 = 0;        // [K; Q] bf16, K-major: 128 rows x 128 channels (K rows stay for A3)
constexpr int kSmB1 = 32768;    // S_0 as three bf16 parts, MN-major (value columns x channels)
constexpr int kSmRec = 131072;  // the four value-block records of the (slot, head)
constexpr int kSmV = 163840;    // v of the piece, bf16, 64 rows of 272 bytes
constexpr int kSmA3 = 16384;    // K^T in record-row order, bf16, MN-major (16 KB)
constexpr int kSmAO = 32768;    // [.; M] three bf16 parts, K-major (128 rows x 64 tokens, 3 x 16 KB)
constexpr int kSmLP = 81920;    // L'^T (L' = L - I strictly lower), 64 rows of 68 FP32
constexpr int kSmYU = 99328;    // Y, then U in place: 64 rows of 132 FP32
constexpr int kSmBU = 81920;    // U as three bf16 parts, K-major (value columns x tokens, 3 x 16 KB)
constexpr int kSmB4 = 131072;   // f_C. U as three bf16 parts, K-major (3 x 16 KB)
constexpr int kSmScal = 181248; // a, beta, gamma, f_C. (64 floats each), pi, g, two mbarriers, tensor-memory address
constexpr int kTcRowL = 68;     // floats per row of L'^T
constexpr int kTcRowY = 132;    // floats per row of Y / U
constexpr int kTcRowV = 272;    // bytes per row of v
constexpr int kTcMaxSort = 256;  // batch rows up to which a ragged chunk's units are ordered by length
constexpr int kSmOrder = kSmScal + 1472;
constexpr int kTcSmem = kSmOrder + 2 * kTcMaxSort + 16;
constexpr int kTcMaxRec = 8192; // largest record (d_k = 128): four fit in [kSmRec, kSmV)
__host__ __device__ constexpr int tc_rec_stride(int rec_bytes) { return (rec_bytes + 127) & ~127; }

// ---- tcgen05 / tensor-memory primitives (inline PTX) ----
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
    // shared-memory matrix descriptor: start >> 4, leading (K-direction) and stride
    // (M/N-direction) byte offsets >> 4, version 1, no swizzle
    return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}
// instruction descriptor: bf16 x bf16 -> FP32, M = 128, N, A/B MN-major when set
__host__ __device__ constexpr uint32_t tc_idesc(int n, bool a_mn, bool b_mn) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (a_mn ? 1u << 15 : 0u) | (b_mn ? 1u << 16 : 0u) |
           ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %4, 0;\n"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
                 "l"(a), "l"(b), "r"(idesc), "r"(acc)
                 : "memory");
}
__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// 32 consecutive columns of this thread's lane (warp w reaches lanes 32 (w % 4) .. + 31)
__device__ __forceinline__ void tc_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
                 "tcgen05.wait::ld.sync.aligned;"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                   "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
                   "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
                   "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr)
                 : "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tc_st32(uint32_t taddr, const float (&v)[32]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};\n"
                 "tcgen05.wait::st.sync.aligned;" ::"r"(taddr),
                 "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
                 "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])),
                 "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])), "r"(__float_as_uint(v[8])),
                 "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])),
                 "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])),
                 "r"(__float_as_uint(v[15])), "r"(__float_as_uint(v[16])), "r"(__float_as_uint(v[17])),
                 "r"(__float_as_uint(v[18])), "r"(__float_as_uint(v[19])), "r"(__float_as_uint(v[20])),
                 "r"(__float_as_uint(v[21])), "r"(__float_as_uint(v[22])), "r"(__float_as_uint(v[23])),
                 "r"(__float_as_uint(v[24])), "r"(__float_as_uint(v[25])), "r"(__float_as_uint(v[26])),
                 "r"(__float_as_uint(v[27])), "r"(__float_as_uint(v[28])), "r"(__float_as_uint(v[29])),
                 "r"(__float_as_uint(v[30])), "r"(__float_as_uint(v[31]))
                 : "memory");
}

// N = 8, 16 or 32 consecutive columns
template <int N>
__device__ __forceinline__ void tc_ldn(uint32_t taddr, float (&v)[N]) {
    static_assert(N == 8 || N == 16 || N == 32, "columns per access");
    if constexpr (N == 32) {
        tc_ld32(taddr, v);
    } else {
        uint32_t r[N];
        if constexpr (N == 16)
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
                         "tcgen05.wait::ld.sync.aligned;"
                         : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                           "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
                         : "r"(taddr)
                         : "memory");
        else
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                         "tcgen05.wait::ld.sync.aligned;"
                         : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                         : "r"(taddr)
                         : "memory");
#pragma unroll
        for (int i = 0; i < N; ++i) v[i] = __uint_as_float(r[i]);
    }
}
template <int N>
__device__ __forceinline__ void tc_stn(uint32_t taddr, const float (&v)[N]) {
    static_assert(N == 8 || N == 16 || N == 32, "columns per access");
    if constexpr (N == 32) {
        tc_st32(taddr, v);
    } else if constexpr (N == 16) {
        asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};\n"
                     "tcgen05.wait::st.sync.aligned;" ::"r"(taddr),
                     "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])),
                     "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])),
                     "r"(__float_as_uint(v[8])), "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])),
                     "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])), "r"(__float_as_uint(v[15]))
                     : "memory");
    } else {
        asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n"
                     "tcgen05.wait::st.sync.aligned;" ::"r"(taddr),
                     "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])),
                     "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7]))
                     : "memory");
    }
}

// x = hi + mid + lo as bf16 parts (each the round-to-nearest of what is left), two
// values per 32-bit word (a in the low half)
__device__ __forceinline__ void split3_pair(float a, float b, uint32_t &h, uint32_t &m, uint32_t &l) {
    const __nv_bfloat162 h2 = __floats2bfloat162_rn(a, b);
    const float2 hf = __bfloat1622float2(h2);
    const float ra = a - hf.x, rb = b - hf.y;  // exact
    const __nv_bfloat162 m2 = __floats2bfloat162_rn(ra, rb);
    const float2 mf = __bfloat1622float2(m2);
    const __nv_bfloat162 l2 = __floats2bfloat162_rn(ra - mf.x, rb - mf.y);
    memcpy(&h, &h2, 4);
    memcpy(&m, &m2, 4);
    memcpy(&l, &l2, 4);
}
// eight consecutive MN-elements of an operand as three 16-byte parts, off_m and off_l bytes
// after the first (the second form: part_bytes apart)
__device__ __forceinline__ void split3_store8(uint32_t dst, uint32_t off_m, uint32_t off_l, const float *x) {
    uint32_t h[4], m[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) split3_pair(x[2 * i], x[2 * i + 1], h[i], m[i], l[i]);
    sts128(dst, make_uint4(h[0], h[1], h[2], h[3]));
    sts128(dst + off_m, make_uint4(m[0], m[1], m[2], m[3]));
    sts128(dst + off_l, make_uint4(l[0], l[1], l[2], l[3]));
}
__device__ __forceinline__ void split3_store8(uint32_t dst, uint32_t part_bytes, const float *x) {
    split3_store8(dst, part_bytes, 2 * part_bytes, x);
}
// byte offset of element (mn, k) in an MN-major bf16 operand whose 8-element groups
// along MN are 128 B apart and whose 8-row groups along K are kstride apart
__device__ __forceinline__ uint32_t tc_mn_off(int mn, int k, uint32_t kstride) {
    return (uint32_t)(mn >> 3) * 128u + (uint32_t)(k >> 3) * kstride + (uint32_t)(k & 7) * 16u + (uint32_t)(mn & 7) * 2u;
}

__device__ __forceinline__ uint32_t lds_u16(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
// all threads of the CTA wait for the phase (bounded) and agree on the outcome
__device__ __forceinline__ bool tc_wait_all(uint32_t bar, uint32_t parity) {
    return __syncthreads_and(mbar_wait_bounded(bar, parity)) != 0;
}
// the 32 values of v as 16 pairs
__device__ __forceinline__ void tc_pairs(const float (&v)[32], float2 (&y)[16]) {
#pragma unroll
    for (int i = 0; i < 16; ++i) y[i] = make_float2(v[2 * i], v[2 * i + 1]);
}

constexpr uint32_t kIdG = tc_idesc(64, false, false);  // [K; Q] and K (KDA: X and Z), both K-major
// byte offset of element (row, k) in a K-major bf16 operand of 8-row groups 1024 B apart
// (64 columns of K: eight 16-byte core matrices per group)
__device__ __forceinline__ uint32_t tc_k64_off(int row, int k) {
    return (uint32_t)(row >> 3) * 1024u + (uint32_t)(k >> 3) * 128u + (uint32_t)(row & 7) * 16u + (uint32_t)(k & 7) * 2u;
}

// The record rows of a (slot, head) (value-block records at `recs`, `rstride` apart in shared
// memory) reconstructed into tensor-memory lane u = record row, blocks ca .. cb - 1: FP32 at the
// natural scale, FP16 rows taken into the H_32 domain with the H_32 formats (where the low
// tier's codes already are).
template <int FMT>
__device__ __forceinline__ void tc_reconstruct(const PrefillParams &p, uint32_t recs, int rstride, int u, int ca, int cb,
                                               uint32_t tS) {
    constexpr bool HAD = fmt_had(FMT);
    const int K = p.K, lo = 128 - K;
#pragma unroll 1
    for (int c = ca; c < cb; ++c) {
        const uint32_t rec = recs + (uint32_t)(c * rstride);
        float2 y[16];
        if (u < K) {
            load_hi_row(rec, u, y);
            if (HAD) hadamard_pairs(y);
        } else {
            const int r = u - K;
            const uint4 c0 = lds128(rec + (uint32_t)(p.codes_off + lo_chunk_off(r, 0, lo)));
            const uint32_t sz = lds32(rec + (uint32_t)(p.meta_off + 4 * r));
            if constexpr (fmt_u4(FMT)) {
                const uint32_t w[4] = {c0.x, c0.y, c0.z, c0.w};
                dequantize_group_u4(w, sz, 1.0f, y);
            } else {
                const uint4 c1 = lds128(rec + (uint32_t)(p.codes_off + lo_chunk_off(r, 1, lo)));
                const uint32_t w[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
                if constexpr (FMT == kFmtE4M3) dequantize_group_e4m3(w, __uint_as_float(sz), 1.0f, y);
                else dequantize_group(w, sz, 1.0f, y);
            }
        }
        float v[32];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            v[2 * i] = y[i].x;
            v[2 * i + 1] = y[i].y;
        }
        tc_st32(tS + 32 * c, v);
    }
}

__device__ __forceinline__ void bar_arrive(int id, int threads) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// U = L^-1 Y by forward substitution, in place: yu addresses row 0 of Y (rows kTcRowY floats
// apart), lt the rows of L'^T (L' = L - I, kTcRowL floats apart).  Warp w of NW owns the rows
// RW w .. RW w + RW - 1 (RW = 64 / NW) of all 32 NV columns, lane l the columns 4 l .. 4 l + 3
// (l mod 8 NV: with fewer than 128 columns lanes repeat one another's work, their loads merge),
// in registers.  Step j: warp j solves its rows among themselves and stores them; the warps
// after it take them out of their own rows, each value of L' and of U loaded once per RW x 4
// tile.  Every element subtracts its products in ascending row order.  Every thread of the CTA
// calls it; the caller synchronizes after it.  Bound by the shared loads of L' and U (3840
// cycles with 16 warps at 128 bytes a cycle): a 64-token KDA piece 8400 -> 6000 cycles against
// a thread per column and quarter of the rows, whose every 16-byte load of L' fed four products
// (on 8 of the 16 warps: 8000); the GDN chunk of B = 256 x 64 tokens 934 -> 878 us.
template <int NW, int NV>
__device__ __forceinline__ void tc_solve(uint32_t yu, uint32_t lt, int warp, int lane) {
    constexpr int RW = kTcC / NW;  // 4 or 8
    static_assert(RW % 4 == 0, "a warp's rows of L'^T are read in 16-byte vectors");
    const int r0 = RW * warp;
    const uint32_t col = yu + (uint32_t)(16 * (lane & (8 * NV - 1))), lrow = lt + (uint32_t)(4 * r0);
    float2 acc[RW][2];
    auto row = [&](int r, float2 (&v)[2]) {
        const uint4 w = lds128(col + (uint32_t)(r * kTcRowY * 4));
        v[0] = make_float2(__uint_as_float(w.x), __uint_as_float(w.y));
        v[1] = make_float2(__uint_as_float(w.z), __uint_as_float(w.w));
    };
    auto ltr = [&](int s, float (&l)[RW]) {  // L' of this warp's rows at column s
#pragma unroll
        for (int i = 0; i < RW / 4; ++i) {
            const uint4 w = lds128(lrow + (uint32_t)(s * kTcRowL * 4 + 16 * i));
            l[4 * i] = __uint_as_float(w.x);
            l[4 * i + 1] = __uint_as_float(w.y);
            l[4 * i + 2] = __uint_as_float(w.z);
            l[4 * i + 3] = __uint_as_float(w.w);
        }
    };
#pragma unroll
    for (int i = 0; i < RW; ++i) row(r0 + i, acc[i]);
    if constexpr (NV < 4) __syncwarp();  // every lane has read Y before a lane of the same columns stores U (warp 0: no barrier between)
    float own[RW][RW];  // L' of this warp's rows among themselves
#pragma unroll
    for (int a = 0; a < RW - 1; ++a) ltr(r0 + a, own[a]);
#pragma unroll 1
    for (int j = 0; j < warp; ++j) {
        bar_sync(1 + (j & 1), 32 * (NW - j));  // rows RW j .. are solved
#pragma unroll
        for (int a = 0; a < RW; ++a) {
            const int s = RW * j + a;
            float2 u[2];
            float l[RW];
            row(s, u);
            ltr(s, l);
            u[0] = make_float2(-u[0].x, -u[0].y);
            u[1] = make_float2(-u[1].x, -u[1].y);
#pragma unroll
            for (int i = 0; i < RW; ++i) {
                acc[i][0] = fma2(splat2(l[i]), u[0], acc[i][0]);
                acc[i][1] = fma2(splat2(l[i]), u[1], acc[i][1]);
            }
        }
    }
#pragma unroll
    for (int a = 0; a < RW - 1; ++a) {
        const float2 u0 = make_float2(-acc[a][0].x, -acc[a][0].y), u1 = make_float2(-acc[a][1].x, -acc[a][1].y);
#pragma unroll
        for (int i = a + 1; i < RW; ++i) {
            acc[i][0] = fma2(splat2(own[a][i]), u0, acc[i][0]);
            acc[i][1] = fma2(splat2(own[a][i]), u1, acc[i][1]);
        }
    }
#pragma unroll
    for (int i = 0; i < RW; ++i)
        sts128(col + (uint32_t)((r0 + i) * kTcRowY * 4),
               make_uint4(__float_as_uint(acc[i][0].x), __float_as_uint(acc[i][0].y), __float_as_uint(acc[i][1].x),
                          __float_as_uint(acc[i][1].y)));
    if (warp < NW - 1) bar_arrive(1 + (warp & 1), 32 * (NW - warp));
}

// The chunk-final state (tensor-memory lane u = record row u, blocks ca .. cb - 1) into the
// records at grec0 in place: FP16 rows back to the natural domain
// and rounded once, low-tier rows requantized (the affine formats at the working scale
// 2^-39, FP8 in the natural domain).  Warps holding FP16 rows store them warp-collectively.
template <int FMT>
__device__ __forceinline__ void tc_requantize(const PrefillParams &p, uint8_t *grec0, int u, int ca, int cb, int lane,
                                              uint32_t tS) {
    constexpr bool HAD = fmt_had(FMT);
    const int K = p.K, lo = 128 - K;
#pragma unroll 1
    for (int c = ca; c < cb; ++c) {
        float v[32];
        tc_ld32(tS + 32 * c, v);
        uint8_t *const grec = grec0 + (int64_t)c * p.rec_bytes;
        float2 y[16];
        tc_pairs(v, y);
        if ((u & ~31) < K) {  // the warp holds FP16 rows: the row-pair store is warp-collective
            float2 z[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) z[i] = y[i];
            if (HAD) hadamard_pairs(z);
            uint32_t own[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) own[i] = f2_to_h2(z[i].x, z[i].y);
            store_hi_row(grec, u, K, lane, own);
        }
        if (u >= K) {
            const int r = u - K;
            if constexpr (FMT == kFmtE4M3) {  // natural domain, one FP32 scale per group
                uint32_t w[8];
                const float sc = quantize_group_e4m3(y, w);
                stg128(grec + p.codes_off + lo_chunk_off(r, 0, lo), make_uint4(w[0], w[1], w[2], w[3]));
                stg128(grec + p.codes_off + lo_chunk_off(r, 1, lo), make_uint4(w[4], w[5], w[6], w[7]));
                stg32(grec + p.meta_off + 4 * r, __float_as_uint(sc));
            } else {
#pragma unroll
                for (int i = 0; i < 16; ++i) y[i] = mul2(y[i], splat2(kDown));  // exact
                if constexpr (fmt_u4(FMT)) {
                    uint32_t w[4];
                    const uint32_t szw = quantize_group_u4(y, w);
                    stg128(grec + p.codes_off + lo_chunk_off(r, 0, lo), make_uint4(w[0], w[1], w[2], w[3]));
                    stg32(grec + p.meta_off + 4 * r, szw);
                } else {
                    float mn, mx, inv, zq;
                    minmax32(y, mn, mx);
                    const float sc = scale_of(mn, mx);
                    const uint32_t szw =
                        sc == 0.0f ? affine_params_scaled(mn, mx, inv, zq) : affine_finish(sc, mn, inv, zq);
                    const float2 inv2 = splat2(inv * 0x1p-110f), zc2 = splat2(zq * 0x1p-149f);
                    uint32_t w[8];
#pragma unroll
                    for (int m = 0; m < 8; ++m) w[m] = encode4(y[2 * m], y[2 * m + 1], inv2, zc2);
                    stg128(grec + p.codes_off + lo_chunk_off(r, 0, lo), make_uint4(w[0], w[1], w[2], w[3]));
                    stg128(grec + p.codes_off + lo_chunk_off(r, 1, lo), make_uint4(w[4], w[5], w[6], w[7]));
                    stg32(grec + p.meta_off + 4 * r, szw);
                }
            }
        }
    }
}

// Which units a CTA of the persistent grid takes: in round r the units at position r * grid +
// blk of the order, in odd rounds from the other end (r * grid + grid - 1 - blk).  The order is
// head by head through the batch rows, and for a ragged chunk through the rows by falling length
// (up to kTcMaxSort rows: `order`, uint16 in shared memory, filled by tc_sort_rows), so that the
// CTAs with the longest units get the shortest ones next.  KDA, 13 rows of up to 133 tokens x 32
// heads (416 units on 152 SMs): 176 us in batch order, 134 us so.  A last round after two, four, .. of
// them that has not a unit for every CTA starts at the end whose CTAs have fewer 64-token pieces so
// far (10 rows x 32 heads, one row of 65 tokens, the others within a piece: KDA 94 us where the CTAs
// with the longest units take those as well, 72 so).  Units that all run at once keep batch order.
// The order's cost grows with the square of the rows, in every CTA: 1.7 us for 256 rows (from shared
// memory, one comparison per pair; 3.4 us before), 15 us for 512 from global memory (GDN, 512 rows of
// 64 tokens x 2 heads: 114.5 us in batch order, 129 us so), where each CTA has enough units that
// their order matters little.
// After the rows: 1 if that last round starts at the other end, else 0.
__device__ __forceinline__ void tc_sort_rows(const PrefillParams &p, uint32_t order, uint32_t scratch) {
    // (length, up to 2^22; the earlier of equal rows) as one number, larger first and distinct
    static_assert(kTcMaxSort <= 512, "a row's number takes nine bits of its key");
    const int units = p.batch * p.H, grid = (int)gridDim.x, full = units / grid;  // (fits: at most kTcMaxSort rows)
    if (units <= grid) {  // (also wherever NV < 4)
        for (int b = threadIdx.x; b < p.batch; b += blockDim.x)
            asm volatile("st.shared.u16 [%0], %1;" ::"r"(order + 2 * b), "h"((unsigned short)b) : "memory");
        if (threadIdx.x == 0) asm volatile("st.shared.u16 [%0], %1;" ::"r"(order + 2 * kTcMaxSort), "h"((unsigned short)0) : "memory");
        return;
    }
    const int n4 = (p.batch + 3) & ~3;
    for (int b = threadIdx.x; b < n4; b += blockDim.x)  // keys past the batch: 0, below every row's
        sts32(scratch + 4 * b, b < p.batch ? (uint32_t)min(min(max(p.lengths[b], 0), p.T), (1 << 22) - 1) * 512u + 512u - (uint32_t)b : 0u);
    __syncthreads();
    for (int b = threadIdx.x; b < p.batch; b += blockDim.x) {
        const uint32_t key = lds32(scratch + 4 * b);
        int rank = 0;
#pragma unroll 4
        for (int c = 0; c < n4; c += 4) {
            const uint4 w = lds128(scratch + 4 * c);
            rank += (w.x > key) + (w.y > key) + (w.z > key) + (w.w > key);
        }
        asm volatile("st.shared.u16 [%0], %1;" ::"r"(order + 2 * rank), "h"((unsigned short)b) : "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int first = 0, last = 0;  // pieces of the first and the last CTA in the full rounds
        if (full >= 2 && full <= 8 && !(full & 1)) {
            for (int i = 0; i < full; ++i) {
                auto pieces = [&](int blk) {
                    const uint32_t row = lds_u16(order + 2u * (uint32_t)((i * grid + blk) / p.H));
                    return (int)(((lds32(scratch + 4 * row) - 1u) / 512u + kTcC - 1) / kTcC);
                };
                first += pieces((i & 1) ? grid - 1 : 0);
                last += pieces((i & 1) ? 0 : grid - 1);
            }
        }
        asm volatile("st.shared.u16 [%0], %1;" ::"r"(order + 2 * kTcMaxSort), "h"((unsigned short)(first > last)) : "memory");
    }
}
struct TcUnit {
    int64_t slot;
    int b, h, mh, hq, Tb;  // batch row, held, model and q/k head, tokens
    int c0;                // first value block
    bool ok;               // false past the CTA's last unit
};
// A unit is NV of a (slot, head)'s four value blocks (the closed form's value columns are
// independent).  The fewer, the more of the work that does not depend on the values is repeated,
// but with few (slot, head) pairs the SMs would be idle: NV = 1 or 2 where all the units then still
// run at once (KDA, 32 heads: one prompt of 2048 tokens 737 us with NV = 4, 643 with 1; two of 500
// tokens 190 / 168 with 2; GDN, one prompt of 1000: 213 / 192).
__host__ __device__ constexpr int tc_nv(int64_t pairs, int sms) { return 4 * pairs <= sms ? 1 : 2 * pairs <= sms ? 2 : 4; }
// The CTA's next unit with work at or after round `round` (left after it); units without work are
// skipped, their status bits collected.
template <int NV>
__device__ __forceinline__ TcUnit tc_next_unit(const PrefillParams &p, int64_t &round, bool sorted, uint32_t order,
                                               bool &bad_slot, bool &bad_head) {
    TcUnit n{0, 0, 0, 0, 0, 0, 0, false};
    constexpr int S = 4 / NV;
    const int HS = p.H * S;
    const int64_t units = (int64_t)p.batch * HS, grid = gridDim.x;
    for (; round * grid < units && !n.ok; ++round) {
        const bool turned = (round & 1) || (sorted && (round + 1) * grid > units && lds_u16(order + 2 * kTcMaxSort));
        const int64_t at = round * grid + (turned ? grid - 1 - blockIdx.x : blockIdx.x);
        if (at >= units) continue;
        const int r = (int)(at / HS), hs = (int)(at - (int64_t)r * HS);
        n.h = hs / S;
        n.c0 = NV * (hs - n.h * S);
        n.b = sorted ? (int)lds_u16(order + 2 * r) : r;
        n.mh = p.head_map ? p.head_map[n.h] : n.h;
        n.slot = p.slot_idx ? (int64_t)p.slot_idx[n.b] : (int64_t)n.b;
        n.Tb = p.lengths ? min(max(p.lengths[n.b], 0), p.T) : p.T;
        const bool slot_ok = n.slot >= 0 && n.slot < p.num_slots, head_ok = n.mh >= 0 && n.mh < p.Hm;
        bad_slot |= !slot_ok;
        bad_head |= !head_ok;
        n.ok = slot_ok && head_ok && n.Tb > 0;
        n.hq = (int)(((int64_t)n.mh * p.Hqk) / p.Hm);
    }
    return n;
}

// One CTA of kTcThreads threads per unit of NV value blocks at a time (persistent over units);
// d_k = d_v = 128, bf16 q/k/v, low tier FMT (UINT8 or UINT4 affine, with or without H_32;
// the launchers instantiate no FP8 or row-absmax kernel).  Thread (row, half):
// row = tensor-memory lane (warps w and w + 4 reach the same lanes), half = 0 / 1 splits
// a row's value blocks (the unit's first and second half of them; with NV = 1 half 0 has the one) or a
// phase's tasks between the two.
template <int FMT, int NV>
__global__ void __launch_bounds__(kTcThreads, 1) prefill_tc_gdn_kernel(const PrefillParams p) {
    static_assert(FMT != kFmtS8Row, "the row-absmax format shares a row scale over the value blocks");
    constexpr bool HAD = fmt_had(FMT);
    constexpr int NC = 32 * NV;  // value columns of a unit
    constexpr uint32_t kIdWP = tc_idesc(NC, false, true);   // [K; Q] K-major, S_0 MN-major
    constexpr uint32_t kIdO = tc_idesc(NC, false, false);   // [.; M] and U, both K-major
    constexpr uint32_t kIdS = tc_idesc(NC, true, false);    // K^T MN-major, f_C. U K-major
    extern __shared__ __align__(128) uint8_t smem[];  // descriptors need 16-byte alignment (no swizzle)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int row = tid & 127, half = tid >> 7;
    const int ca = (half * NV + 1) / 2, cb = ((half + 1) * NV + 1) / 2;  // this half's value blocks of the unit
    const uint32_t sb = smem_u32(smem);
    const int T = p.T, Hm = p.Hm;
    const int rec_bytes = p.rec_bytes, rstride = tc_rec_stride(rec_bytes);
    const uint32_t scal = sb + (uint32_t)kSmScal;
    const uint32_t s_a = scal, s_beta = scal + 256, s_gam = scal + 512, s_rev = scal + 768, s_perm = scal + 1024;
    const uint32_t s_g = scal + 1152, bar_rec = scal + 1408, bar_mma = scal + 1416, s_taddr = scal + 1424;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s_taddr), "r"(kTcCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        mbar_init(bar_rec, 1);
        mbar_init(bar_mma, 1);
        fence_mbar_init();
    }
    if (p.lengths && p.batch <= kTcMaxSort) tc_sort_rows(p, sb + (uint32_t)kSmOrder, sb + (uint32_t)kSmB1);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = lds32(s_taddr);
    const uint32_t tl = tmem + ((uint32_t)(32 * (warp & 3)) << 16);  // this warp's lanes
    const uint32_t tWP = tl + kColWP, tS = tl + kColS, tG = tl + kColG;

    uint32_t ph_rec = 0, ph_mma = 0;
    bool bad_slot = false, bad_head = false, timed_out = false;
    bool rec_pending = false, mma_pending = false;  // a copy / a product in flight
    int64_t round = 0;
    const bool sorted = p.lengths && p.batch <= kTcMaxSort;
    auto next_unit = [&]() { return tc_next_unit<NV>(p, round, sorted, sb + (uint32_t)kSmOrder, bad_slot, bad_head); };
    auto rec_of = [&](const TcUnit &n) { return p.state + n.slot * p.slot_bytes + (int64_t)(n.h * 4 + n.c0) * rec_bytes; };
    // [K; Q] (bf16, natural channel order, K-major), v, g and beta of unit n's piece at p0
    // (cp.async; a masked token is zero, neither decays nor updates)
    auto load_piece = [&](const TcUnit &n, int p0) {
        const int nt = min(kTcC, n.Tb - p0);
#pragma unroll 1
        for (int i = tid; i < 2048; i += kTcThreads) {
            const int m = i >> 4, j = i & 15, t = m & 63;
            const uint32_t dst = sb + (uint32_t)(kSmA1 + (m >> 3) * 2048 + j * 128 + (m & 7) * 16);
            if (t < nt) {
                const uint8_t *src = static_cast<const uint8_t *>(m < 64 ? p.k : p.q) +
                                     (((int64_t)n.b * T + p0 + t) * p.Hqk + n.hq) * 256 + 16 * j;
                cp_async16(dst, src);
            } else {
                sts128(dst, make_uint4(0u, 0u, 0u, 0u));
            }
        }
#pragma unroll 1
        for (int i = tid; i < 1024; i += kTcThreads) {
            const int t = i >> 4, j = i & 15;
            const uint32_t dst = sb + (uint32_t)(kSmV + t * kTcRowV + 16 * j);
            if (t < nt)
                cp_async16(dst, static_cast<const uint8_t *>(p.v) + (((int64_t)n.b * T + p0 + t) * Hm + n.mh) * 256 + 16 * j);
            else
                sts128(dst, make_uint4(0u, 0u, 0u, 0u));
        }
        if (tid < kTcC) {  // log-decay and beta (a masked token: g = 0, beta = 0)
            const int t = tid;
            if (t < nt) {
                const int64_t gi = ((int64_t)n.b * T + p0 + t) * Hm + n.mh;
                cp_async4(s_g + 4 * t, p.g + gi);
                cp_async4(s_beta + 4 * t, p.beta + gi);
            } else {
                sts32(s_g + 4 * t, 0u);
                sts32(s_beta + 4 * t, 0u);
            }
        }
        cp_async_commit();
    };
    // unit n's four records (bulk copies), pi and first piece: issued one unit ahead, so
    // that they land while the previous unit finishes (every area they write is free then)
    auto prefetch = [&](const TcUnit &n) {
        if (tid == 0) {
            fence_proxy_async_smem();
            mbar_arrive_expect_tx(bar_rec, (uint32_t)(NV * rec_bytes));
            uint8_t *const g0 = rec_of(n);
#pragma unroll
            for (int c = 0; c < NV; ++c)
                bulk_g2s(sb + (uint32_t)(kSmRec + c * rstride), g0 + (int64_t)c * rec_bytes, (uint32_t)rec_bytes, bar_rec);
        }
        if (tid < 8) cp_async16(s_perm + 16 * tid, p.perm + (int64_t)n.h * 128 + 16 * tid);
        load_piece(n, 0);  // commits the perm copies with the piece's
        rec_pending = true;
    };

    TcUnit cur = next_unit();
    if (cur.ok) prefetch(cur);
    while (cur.ok) {
        const int b = cur.b, Tb = cur.Tb, mh = cur.mh;
        uint8_t *const grec0 = rec_of(cur);
        const TcUnit nxt = next_unit();  // its loads overlap this unit's work
        if (!tc_wait_all(bar_rec, ph_rec)) {
            timed_out = true;
            break;
        }
        ph_rec ^= 1u;
        rec_pending = false;

        // ---- S_0: record row u = row, reconstructed (FP32, natural scale, transformed domain
        //      with H_32) into tensor-memory lane u; this half's two value blocks ----
        tc_reconstruct<FMT>(p, sb + (uint32_t)kSmRec, rstride, row, ca, cb, tS);

#pragma unroll 1
        for (int p0 = 0; p0 < Tb; p0 += kTcC) {
            const int nt = min(kTcC, Tb - p0);  // live tokens of the piece; the rest are masked
            if (p0 > 0) {
                load_piece(cur, p0);
            } else {  // the first piece's copies (and pi) were issued with the records
                cp_async_wait_all();
                __syncthreads();
            }
            // ---- S_0 as three bf16 parts, MN-major (value columns n x channels), at channel pi(u) ----
            {
                const int ch = (int)(lds_u8(s_perm + row) & 127u);
#pragma unroll 1
                for (int c = ca; c < cb; ++c) {
                    float v[32];
                    tc_ld32(tS + 32 * c, v);
#pragma unroll
                    for (int j8 = 0; j8 < 4; ++j8)
                        split3_store8(sb + kSmB1 + tc_mn_off(32 * c + 8 * j8, ch, 2048), 32768, v + 8 * j8);
                }
            }
            cp_async_wait_all();
            fence_proxy_async_smem();  // the operands written through the generic proxy, before the MMAs
            tc_fence_before();
            __syncthreads();
            tc_fence_after();
            if (tid == 0) {
#pragma unroll 1
                for (int q = 0; q < 3; ++q)
#pragma unroll
                    for (int ks = 0; ks < 8; ++ks)
                        tc_mma(tmem + kColWP, tc_desc(sb + kSmA1 + 256 * ks, 128, 2048),
                               tc_desc(sb + kSmB1 + 32768 * q + 4096 * ks, 2048, 128), kIdWP, (q | ks) != 0);
#pragma unroll
                for (int ks = 0; ks < 8; ++ks)
                    tc_mma(tmem + kColG, tc_desc(sb + kSmA1 + 256 * ks, 128, 2048),
                           tc_desc(sb + kSmA1 + 256 * ks, 128, 2048), kIdG, ks != 0);
                tc_commit(bar_mma);
            }
            // gamma_t = a_0 ... a_t and f_Ct = a_{t+1} ... a_63 (warp 0: lane l holds tokens
            // 2l and 2l + 1; products over the lanes by shuffle scans) while the products run
            if (warp == 0) {
                const float a0 = expf(ldsf(s_g + 8 * lane)), a1 = expf(ldsf(s_g + 8 * lane + 4));
                sts32(s_a + 8 * lane, __float_as_uint(a0));
                sts32(s_a + 8 * lane + 4, __float_as_uint(a1));
                const float tot = a0 * a1;
                float pre = tot, suf = tot;  // inclusive over lanes <= l / >= l
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const float up = __shfl_up_sync(kFull, pre, d), dn = __shfl_down_sync(kFull, suf, d);
                    if (lane >= d) pre *= up;
                    if (lane + d < 32) suf *= dn;
                }
                float ex_pre = __shfl_up_sync(kFull, pre, 1), ex_suf = __shfl_down_sync(kFull, suf, 1);
                if (lane == 0) ex_pre = 1.f;
                if (lane == 31) ex_suf = 1.f;
                sts32(s_gam + 8 * lane, __float_as_uint(ex_pre * a0));
                sts32(s_gam + 8 * lane + 4, __float_as_uint(ex_pre * tot));
                sts32(s_rev + 8 * lane, __float_as_uint(a1 * ex_suf));
                sts32(s_rev + 8 * lane + 4, __float_as_uint(ex_suf));
            }
            if (!tc_wait_all(bar_mma, ph_mma)) {
                timed_out = mma_pending = true;
                break;
            }
            ph_mma ^= 1u;
            tc_fence_after();
            // ---- half 0: rows of L' = beta_t f_ts k_t.k_s (s < t; FP32, for the solve) and of
            //      M = f_ts q_t.k_s (s <= t; rows 64 + t of [.; M], three bf16 parts), and
            //      gamma_t P_t in tensor memory;  half 1: K^T in record-row order and gamma_C
            //      S_0 in tensor memory ----
            if (half == 0) {
                const int t = row & 63;
                const bool qside = row >= 64;
                float gr[64];
                {
                    float g0[32], g1[32];
                    tc_ld32(tG, g0);
                    tc_ld32(tG + 32, g1);
#pragma unroll
                    for (int i = 0; i < 32; ++i) {
                        gr[i] = g0[i];
                        gr[32 + i] = g1[i];
                    }
                }
                const float bt = qside ? 1.f : ldsf(s_beta + 4 * t);
                float f = 1.f;  // f_ts, s running down from t
#pragma unroll
                for (int s2 = 63; s2 >= 0; --s2) {
                    float e = 0.f;
                    if (s2 < t) {
                        f *= ldsf(s_a + 4 * (s2 + 1));
                        e = bt * f * gr[s2];
                    } else if (s2 == t && qside) {
                        e = gr[s2];
                    }
                    gr[s2] = e;
                }
                if (!qside) {  // column t of L'^T (row s holds L'_{., s})
                    const uint32_t colt = sb + (uint32_t)(kSmLP + 4 * t);
#pragma unroll
                    for (int s2 = 0; s2 < 64; ++s2) sts32(colt + (uint32_t)(s2 * kTcRowL * 4), __float_as_uint(gr[s2]));
                } else {
#pragma unroll
                    for (int g = 0; g < 8; ++g) split3_store8(sb + kSmAO + tc_k64_off(64 + t, 8 * g), 16384, gr + 8 * g);
                    // gamma_t P_t: the output product accumulates onto it
                    const float gt = ldsf(s_gam + 4 * t);
#pragma unroll 1
                    for (int c = 0; c < NV; ++c) {
                        float v[32];
                        tc_ld32(tWP + 32 * c, v);
#pragma unroll
                        for (int i = 0; i < 32; ++i) v[i] *= gt;
                        tc_st32(tWP + 32 * c, v);
                    }
                }
            } else {
                // K^T: element (u, s) = k_s[pi(u)]; this thread takes token s = row & 63 and
                // half the rows (its 64 channel indices first, then independent gathers)
                {
                    const int t = row & 63;
                    const uint32_t krow = sb + (uint32_t)(kSmA1 + (t >> 3) * 2048 + (t & 7) * 16);
                    const int u0 = row >= 64 ? 64 : 0;
                    uint32_t pw[16];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const uint4 w4 = lds128(s_perm + (uint32_t)(u0 + 16 * i));
                        pw[4 * i] = w4.x;
                        pw[4 * i + 1] = w4.y;
                        pw[4 * i + 2] = w4.z;
                        pw[4 * i + 3] = w4.w;
                    }
#pragma unroll
                    for (int uc = 0; uc < 8; ++uc) {
                        uint32_t w[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const uint32_t pp = pw[2 * uc + (e >> 1)] >> (16 * (e & 1));  // channels of rows ua, ua + 1
                            const uint32_t ca = pp & 127u, cb = (pp >> 8) & 127u;
                            const uint32_t va = lds_u16(krow + (ca >> 3) * 128u + (ca & 7u) * 2u);
                            const uint32_t vb = lds_u16(krow + (cb >> 3) * 128u + (cb & 7u) * 2u);
                            w[e] = va | (vb << 16);
                        }
                        sts128(sb + kSmA3 + tc_mn_off(u0 + 8 * uc, t, 2048), make_uint4(w[0], w[1], w[2], w[3]));
                    }
                }
                // gamma_C S_0: the state product accumulates onto it
                const float gC = ldsf(s_gam + 4 * (kTcC - 1));
#pragma unroll 1
                for (int c = 0; c < NV; ++c) {
                    float v[32];
                    tc_ld32(tS + 32 * c, v);
#pragma unroll
                    for (int i = 0; i < 32; ++i) v[i] *= gC;
                    tc_st32(tS + 32 * c, v);
                }
            }
            // ---- Y = diag(beta) (v~ - diag(gamma) W), FP32 rows (this half's value blocks) ----
            if (row < 64) {
                const int t = row;
                const float bt = ldsf(s_beta + 4 * t), gt = ldsf(s_gam + 4 * t);
                const uint32_t vrow = sb + (uint32_t)(kSmV + t * kTcRowV + 64 * cur.c0), yrow = sb + (uint32_t)(kSmYU + t * kTcRowY * 4);
#pragma unroll 1
                for (int c = ca; c < cb; ++c) {
                    float w[32];
                    tc_ld32(tWP + 32 * c, w);
                    float2 y[16];
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const uint4 r = lds128(vrow + 64 * c + 16 * q);
                        const uint32_t rw[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            y[4 * q + e] = make_float2(__uint_as_float(rw[e] << 16), __uint_as_float(rw[e] & 0xffff0000u));
                    }
                    if (HAD) hadamard_pairs(y);
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const float2 ya = y[2 * q], yb = y[2 * q + 1];
                        sts128(yrow + 128 * c + 16 * q,
                               make_uint4(__float_as_uint(bt * (ya.x - gt * w[4 * q])), __float_as_uint(bt * (ya.y - gt * w[4 * q + 1])),
                                          __float_as_uint(bt * (yb.x - gt * w[4 * q + 2])),
                                          __float_as_uint(bt * (yb.y - gt * w[4 * q + 3]))));
                    }
                }
            }
            __syncthreads();
            // ---- U = L^-1 Y by forward substitution, in place ----
            tc_solve<kTcThreads / 32, NV>(sb + (uint32_t)kSmYU, sb + (uint32_t)kSmLP, warp, lane);
            __syncthreads();
            // ---- U (half 0) and f_C. U (half 1) as three bf16 parts, K-major (value columns n x
            //      tokens s) ----
            {
                const uint32_t col = sb + (uint32_t)(kSmYU + 4 * row);
                float uc[64];
                if (NV == 4 || row < NC) {
#pragma unroll
                    for (int t = 0; t < 64; ++t) uc[t] = ldsf(col + (uint32_t)(t * kTcRowY * 4));
                }
                __syncthreads();  // every column is read: the parts go over L' and Y / U
                const uint32_t dst = sb + (uint32_t)(half == 0 ? kSmBU : kSmB4);
                if (NV == 4 || row < NC) {
#pragma unroll
                    for (int g = 0; g < 8; ++g) {
                        float x8[8];
#pragma unroll
                        for (int e = 0; e < 8; ++e) x8[e] = half == 0 ? uc[8 * g + e] : ldsf(s_rev + 4 * (8 * g + e)) * uc[8 * g + e];
                        split3_store8(dst + tc_k64_off(row, 8 * g), 16384, x8);
                    }
                }
            }
            fence_proxy_async_smem();
            tc_fence_before();
            __syncthreads();
            tc_fence_after();
            if (tid == 0) {
                // O = gamma P + [.; M] U and S += K^T (f_C. U); six partial products of two
                // split operands (hh, hm, mh, hl, lh, mm), three of an exact one
                constexpr int pa[6] = {0, 0, 1, 0, 2, 1}, pb[6] = {0, 1, 0, 2, 0, 1};
#pragma unroll
                for (int q = 0; q < 6; ++q)
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        tc_mma(tmem + kColWP, tc_desc(sb + kSmAO + 16384 * pa[q] + 256 * ks, 128, 1024),
                               tc_desc(sb + kSmBU + 16384 * pb[q] + 256 * ks, 128, 1024), kIdO, 1u);
#pragma unroll
                for (int q = 0; q < 3; ++q)
#pragma unroll
                    for (int ks = 0; ks < 4; ++ks)
                        tc_mma(tmem + kColS, tc_desc(sb + kSmA3 + 4096 * ks, 2048, 128),
                               tc_desc(sb + kSmB4 + 16384 * q + 256 * ks, 128, 1024), kIdS, 1u);
                tc_commit(bar_mma);
            }
            if (!tc_wait_all(bar_mma, ph_mma)) {
                timed_out = mma_pending = true;
                break;
            }
            ph_mma ^= 1u;
            tc_fence_after();
            if (p0 + kTcC >= Tb && nxt.ok) prefetch(nxt);  // the next unit's loads overlap this one's tail
            // ---- o_t = H (gamma_t P_t + (M U)_t) (lanes 64 + t, this half's value blocks) ----
            if (row >= 64) {
                const int t = row - 64;
                float *orow = p.o + (((int64_t)b * T + p0 + min(t, nt - 1)) * Hm + mh) * 128 + 32 * cur.c0;
#pragma unroll 1
                for (int c = ca; c < cb; ++c) {
                    float ov[32];
                    tc_ld32(tWP + 32 * c, ov);
                    float2 y[16];
                    tc_pairs(ov, y);
                    if (HAD) hadamard_pairs(y);
                    if (t < nt) {
#pragma unroll
                        for (int q = 0; q < 8; ++q)
                            stg128(orow + 32 * c + 4 * q,
                                   make_uint4(__float_as_uint(y[2 * q].x), __float_as_uint(y[2 * q].y),
                                              __float_as_uint(y[2 * q + 1].x), __float_as_uint(y[2 * q + 1].y)));
                    }
                }
            }
        }
        if (timed_out) break;
        // ---- the chunk-final state (tensor-memory lane u = record row u, this half's value
        //      blocks) into the record in place ----
        tc_requantize<FMT>(p, grec0, row, ca, cb, lane, tS);
        cur = nxt;
    }
    // a copy or a product that did not complete in time gets one more bounded wait before
    // the tensor memory and the shared memory go away
    if (rec_pending) mbar_wait_bounded(bar_rec, ph_rec);
    if (mma_pending) mbar_wait_bounded(bar_mma, ph_mma);
    cp_async_wait_all();
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcCols) : "memory");
    }
    if (tid == 0) {
        const uint32_t bits =
            (timed_out ? kDevWaitTimeout : 0u) | (bad_slot ? kDevBadSlot : 0u) | (bad_head ? kDevBadHead : 0u);
        if (bits) atomicOr(p.status, bits);
    }
}

}  // namespace damp
