// convert.cu -- kernels that move whole states in and out of the packed cache.
//
//   quantize_state    natural FP32 state -> packed records (App. A.5 "Prefill
//                     path": the FP32 state is written straight into the packed
//                     cache; rows in pi order, FP16 tier for rows < K_hi, H_32 +
//                     UINT8 affine (Sec. 3.2, Eq. integer_quantizer) for the rest)
//   dequantize_state  packed records -> natural FP32 state (the inverse map)
//   pack_tiers / unpack_tiers
//                     logical tier arrays (S_hi, Q_lo, M_lo of Eq.
//                     packed_state_layout) <-> packed records, bit for bit
//
// quantize and dequantize: an item is 32 packed rows of a (slot, head, value block) record, a
// 32 x 32 FP32 tile whose rows pi scatters over the state.  A warp walks a contiguous range
// of items.  The tile goes through shared memory (rows padded to 36 floats: row-wise and
// lane-per-row accesses are both free of bank conflicts), so that S is read and written in
// whole 128-byte row segments, four per instruction, while lane l quantizes or reconstructs
// row l of the item: with lane l reading its own row from memory every 16-byte access
// touched 32 different lines.  quantize copies the next tile (cp.async) and dequantize loads the
// next item's codes while the current one is computed.  B = 64, H = 32, d = 128, K_hi = 16 (134
// MB FP32 + 41 MB packed): quantize 35.8 us, 4.9 TB/s (B = 256: 128 us, 5.5 TB/s), against 54.8
// and 169 us with a row per lane from memory; dequantize 34 us against 73 us.  HBM-bound.
// pack and unpack, and dequantize at d_k = 32: one warp per record, lane l owns packed rows l, l + 32, ...
#include "damp_common.cuh"
#include "damp_internal.h"
#include "formats.cuh"

#include <algorithm>

namespace damp {

static __device__ uint32_t g_status_convert;

struct ConvParams {
    uint8_t *state;
    int64_t num_slots;
    const int32_t *slot_idx;
    const uint8_t *perm;
    float *S;
    uint16_t *hi;
    uint8_t *codes;
    uint16_t *meta;
    int32_t batch, H, dk, dv, V, K;
    int32_t Hm;                // heads of S: held head h is row head_map[h] (or h)
    const int32_t *head_map;
    int32_t rec_bytes, codes_off, meta_off;
    int64_t slot_bytes, total_tiles;
    uint32_t *status;
};

enum ConvOp { kDequantize = 1, kPackTiers = 2, kUnpackTiers = 3 };

// (batch row, head, value block, row group) of an item, and whether its slot and head are valid
struct ConvItem {
    int b, h, c, i, mh;
    int64_t slot;
    bool ok;
};

constexpr int kCvWarps = 8;
constexpr int kCvRow = 36;                 // floats per row of a staging tile
constexpr int kCvTile = 32 * kCvRow * 4;   // bytes
constexpr int kCvStages = 2;               // quantize: tiles per warp

struct ConvWalk {
    const ConvParams &p;
    int R;
    bool bad_slot = false, bad_head = false;
    __device__ __forceinline__ void look(ConvItem &k) {
        k.slot = p.slot_idx ? (int64_t)p.slot_idx[k.b] : (int64_t)k.b;
        k.mh = p.head_map ? p.head_map[k.h] : k.h;
        const bool slot_ok = k.slot >= 0 && k.slot < p.num_slots, head_ok = k.mh >= 0 && k.mh < p.Hm;
        bad_slot |= !slot_ok;
        bad_head |= slot_ok && !head_ok;
        k.ok = slot_ok && head_ok;
    }
    __device__ __forceinline__ ConvItem at(int64_t item) {
        ConvItem k;
        const int64_t t = item / R, bh = t / p.V;
        k.i = (int)(item - t * R);
        k.c = (int)(t - bh * p.V);
        k.b = (int)(bh / p.H);
        k.h = (int)(bh - (int64_t)k.b * p.H);
        look(k);
        return k;
    }
    // the item after k (k must not be the last item of the last batch row)
    __device__ __forceinline__ void next(ConvItem &k) {
        if (++k.i < R) return;
        k.i = 0;
        if (++k.c < p.V) return;
        k.c = 0;
        if (++k.h == p.H) {
            k.h = 0;
            ++k.b;
        }
        look(k);
    }
    __device__ __forceinline__ uint8_t *record(const ConvItem &k) const {
        return p.state + k.slot * p.slot_bytes + (int64_t)(k.h * p.V + k.c) * p.rec_bytes;
    }
    // this lane's channel: the natural row of packed row 32 i + lane (d_k is a power of two)
    __device__ __forceinline__ int channel(const ConvItem &k, int lane) const {
        return p.perm[(int64_t)k.h * p.dk + 32 * k.i + lane] & (p.dk - 1);
    }
    __device__ __forceinline__ float *rows(const ConvItem &k) const {
        return p.S + ((int64_t)k.b * p.Hm + k.mh) * p.dk * p.dv + k.c * kG;
    }
    __device__ __forceinline__ void report(int lane) const {
        if (lane == 0 && (bad_slot || bad_head))
            atomicOr(p.status, (bad_slot ? (uint32_t)kDevBadSlot : 0u) | (bad_head ? (uint32_t)kDevBadHead : 0u));
    }
};

template <int FMT>
__global__ void __launch_bounds__(32 * kCvWarps, 3) quantize_kernel(const ConvParams p) {
    constexpr bool HAD = fmt_had(FMT), U4 = fmt_u4(FMT);
    extern __shared__ __align__(16) uint8_t cv_tiles[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lr = lane >> 3, lc = lane & 7;  // copies: 8 lanes per 128-byte row segment
    const uint32_t ring = smem_u32(cv_tiles) + (uint32_t)(warp * kCvStages * kCvTile);
    const int K = p.K, lo = p.dk - K, R = p.dk / 32;
    const int64_t n_items = p.total_tiles * R, gw = (int64_t)blockIdx.x * kCvWarps + warp, nw = (int64_t)gridDim.x * kCvWarps;
    const int64_t i0 = n_items * gw / nw, i1 = n_items * (gw + 1) / nw;
    if (i0 >= i1) return;
    ConvWalk w{p, R};
    ConvItem cur = w.at(i0), pre = cur;
    int pch = w.channel(pre, lane);
    int64_t pi = i0;  // the next item to copy in
    auto issue = [&]() {
        if (pi < i1) {
            if (pre.ok) {
                const float *src = w.rows(pre) + 4 * lc;
                const uint32_t dst = ring + (uint32_t)((pi - i0) % kCvStages) * kCvTile + (uint32_t)((lr * kCvRow + 4 * lc) * 4);
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    cp_async16(dst + 16 * q * kCvRow, src + (int64_t)__shfl_sync(kFull, pch, 4 * q + lr) * p.dv);
            }
            if (++pi < i1) {
                w.next(pre);
                pch = w.channel(pre, lane);
            }
        }
        cp_async_commit();  // one group per item, empty past the end
    };
#pragma unroll
    for (int s = 0; s < kCvStages - 1; ++s) issue();
    for (int64_t it = i0;;) {
        __syncwarp();  // every lane is done reading the tile that the next copy overwrites
        issue();
        cp_async_wait<kCvStages - 1>();
        __syncwarp();
        const uint32_t tile = ring + (uint32_t)((it - i0) % kCvStages) * kCvTile;
        if (cur.ok) {
            uint8_t *const rec = w.record(cur);
            const int u0 = 32 * cur.i, u = u0 + lane;
            if (u >= K) {
                const int r = u - K;
                float2 x[16];
#pragma unroll
                for (int m = 0; m < 8; ++m) {
                    const uint4 f = lds128(tile + (uint32_t)(lane * kCvRow * 4 + 16 * m));
                    x[2 * m] = make_float2(__uint_as_float(f.x), __uint_as_float(f.y));
                    x[2 * m + 1] = make_float2(__uint_as_float(f.z), __uint_as_float(f.w));
                }
                if (HAD) hadamard_pairs(x);
                uint32_t cw[8], meta;
                if (FMT == kFmtE4M3) {
                    meta = __float_as_uint(quantize_group_e4m3(x, cw));
                } else {
#pragma unroll
                    for (int m = 0; m < 16; ++m) x[m] = mul2(x[m], splat2(kDown));  // working scale
                    if constexpr (U4) {
                        uint32_t c4[4];
                        meta = quantize_group_u4(x, c4);
#pragma unroll
                        for (int m = 0; m < 4; ++m) cw[m] = c4[m];
                    } else {
                        meta = quantize_group(x, cw);
                    }
                }
                stg128(rec + p.codes_off + lo_chunk_off(r, 0, lo), make_uint4(cw[0], cw[1], cw[2], cw[3]));
                if (!U4) stg128(rec + p.codes_off + lo_chunk_off(r, 1, lo), make_uint4(cw[4], cw[5], cw[6], cw[7]));
                stg32(rec + p.meta_off + 4 * r, meta);
            }
            // FP16 rows, lane = column, two rows per 32-bit word (an odd K leaves the last high half zero)
            const int hi_end = min(K, u0 + 32);
            for (int v = u0; v < hi_end; v += 2) {
                const uint32_t at = tile + (uint32_t)((v - u0) * kCvRow * 4 + 4 * lane);
                stg32(rec + hi_elem_off(v, lane), f2_to_h2(ldsf(at), v + 1 < K ? ldsf(at + kCvRow * 4) : 0.f));
            }
            if (cur.i == R - 1) {  // zero the record padding so packed pools compare bit for bit
                const int used = p.meta_off + 4 * lo;
                if (lane < p.rec_bytes - used) rec[used + lane] = 0;
            }
        }
        if (++it == i1) break;
        w.next(cur);
    }
    cp_async_wait_all();
    w.report(lane);
}

template <int FMT>
__global__ void __launch_bounds__(32 * kCvWarps) dequantize_kernel(const ConvParams p) {
    constexpr bool HAD = fmt_had(FMT), U4 = fmt_u4(FMT);
    extern __shared__ __align__(16) uint8_t cv_tiles[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lr = lane >> 3, lc = lane & 7;
    const uint32_t tile = smem_u32(cv_tiles) + (uint32_t)(warp * kCvTile);
    const int K = p.K, lo = p.dk - K, R = p.dk / 32;
    const int64_t n_items = p.total_tiles * R, gw = (int64_t)blockIdx.x * kCvWarps + warp, nw = (int64_t)gridDim.x * kCvWarps;
    const int64_t i0 = n_items * gw / nw, i1 = n_items * (gw + 1) / nw;
    if (i0 >= i1) return;
    ConvWalk w{p, R};
    ConvItem cur = w.at(i0);
    uint4 c0{}, c1{};
    uint32_t sz = 0;
    int ch = 0;
    auto load = [&](const ConvItem &k) {  // the item's low-tier row of this lane, and its channel
        if (!k.ok) return;
        ch = w.channel(k, lane);
        const int r = 32 * k.i + lane - K;
        if (r < 0) return;
        const uint8_t *rec = w.record(k);
        c0 = *reinterpret_cast<const uint4 *>(rec + p.codes_off + lo_chunk_off(r, 0, lo));
        if (!U4) c1 = *reinterpret_cast<const uint4 *>(rec + p.codes_off + lo_chunk_off(r, 1, lo));
        sz = *reinterpret_cast<const uint32_t *>(rec + p.meta_off + 4 * r);
    };
    load(cur);
    for (int64_t it = i0;;) {
        const ConvItem k = cur;
        const int kch = ch;
        const uint32_t cw[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w}, ksz = sz;
        const bool more = ++it < i1;
        if (more) {
            w.next(cur);
            load(cur);
        }
        if (k.ok) {
            const int u0 = 32 * k.i;
            if (u0 + lane >= K) {
                float2 x[16];
                if constexpr (U4) {
                    const uint32_t c4[4] = {cw[0], cw[1], cw[2], cw[3]};
                    dequantize_group_u4(c4, ksz, 1.0f, x);
                } else if constexpr (FMT == kFmtE4M3) {
                    dequantize_group_e4m3(cw, __uint_as_float(ksz), 1.0f, x);
                } else {
                    dequantize_group(cw, ksz, 1.0f, x);
                }
                if (HAD) hadamard_pairs(x);
#pragma unroll
                for (int m = 0; m < 8; ++m)
                    sts128(tile + (uint32_t)(lane * kCvRow * 4 + 16 * m),
                           make_uint4(__float_as_uint(x[2 * m].x), __float_as_uint(x[2 * m].y), __float_as_uint(x[2 * m + 1].x),
                                      __float_as_uint(x[2 * m + 1].y)));
            }
            const uint8_t *rec = w.record(k);
            // FP16 rows, two per 32-bit word: eight words on their way before the first is used (all rows
            // in FP16: 128 x 128, B = 1 8.8 us, B = 64 38 us; 16.2 and 92 us with one word after the other)
            const int hi_end = min(K, u0 + 32);
#pragma unroll 1
            for (int v0 = u0; v0 < hi_end; v0 += 16) {
                uint32_t hw[8];
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    if (v0 + 2 * j < hi_end) hw[j] = *reinterpret_cast<const uint32_t *>(rec + hi_elem_off(v0 + 2 * j, lane));
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int v = v0 + 2 * j;
                    if (v >= hi_end) break;
                    const float2 f = h2_to_f2(hw[j]);
                    const uint32_t at = tile + (uint32_t)((v - u0) * kCvRow * 4 + 4 * lane);
                    sts32(at, __float_as_uint(f.x));
                    if (v + 1 < K) sts32(at + kCvRow * 4, __float_as_uint(f.y));
                }
            }
            __syncwarp();
            float *const dst = w.rows(k) + 4 * lc;
#pragma unroll
            for (int q = 0; q < 8; ++q)
                stg128(dst + (int64_t)__shfl_sync(kFull, kch, 4 * q + lr) * p.dv,
                       lds128(tile + (uint32_t)(((4 * q + lr) * kCvRow + 4 * lc) * 4)));
            __syncwarp();
        }
        if (!more) break;
    }
    w.report(lane);
}

// pack and unpack, and dequantize at d_k = 32: a record is a single item there, without a next one
// for a warp's loads to run ahead to, and the tile only adds its way through shared memory.
template <int R, int FMT, int OP>
__global__ void __launch_bounds__(256) tiers_kernel(const ConvParams p) {
    constexpr bool HAD = fmt_had(FMT), U4 = fmt_u4(FMT);
    constexpr int CB = U4 ? 16 : 32;  // code bytes per row and value block
    const int lane = threadIdx.x & 31;
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwt = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int K = p.K;
    const int lo = p.dk - K;
    bool bad_slot = false, bad_head = false;
    for (int64_t t = gw; t < p.total_tiles; t += nwt) {
        const int c = (int)(t % p.V);
        const int64_t bh = t / p.V;
        const int h = (int)(bh % p.H);
        const int b = (int)(bh / p.H);
        const int64_t slot = p.slot_idx ? (int64_t)p.slot_idx[b] : (int64_t)b;
        if (slot < 0 || slot >= p.num_slots) {
            bad_slot = true;
            continue;
        }
        // row of S; pack and unpack have no map and always pass, but without the check the compiler orders
        // their accesses worse (pack, H = 32: 128 x 96, B = 64 20.9 us, so 19.1; 128 x 64, B = 100 23.2 / 21.0)
        // and takes 48 registers for 40 at d_k = 32 (32 x 96, B = 64 7.5 / 6.6)
        const int mh = p.head_map ? p.head_map[h] : h;
        if (mh < 0 || mh >= p.Hm) {
            bad_head = true;
            continue;
        }
        uint8_t *rec = p.state + slot * p.slot_bytes + (int64_t)(h * p.V + c) * p.rec_bytes;
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const int u = lane + 32 * i;
            if (u < K) continue;  // FP16 rows: column-mapped loop below
            const int r = u - K;
            uint8_t *crec = rec + p.codes_off + lo_chunk_off(r, 0, lo), *crec1 = rec + p.codes_off + lo_chunk_off(r, 1, lo);
            uint32_t *mrec = reinterpret_cast<uint32_t *>(rec + p.meta_off + 4 * r);
            if (OP == kDequantize) {
                const int n = p.perm[(int64_t)h * p.dk + u] & (p.dk - 1);  // d_k is a power of two
                float *row = p.S + ((((int64_t)b * p.Hm + mh) * p.dk + n) * p.dv + c * kG);
                float2 x[16];
                const uint4 c0 = *reinterpret_cast<const uint4 *>(rec + p.codes_off + lo_chunk_off(r, 0, lo));
                if (U4) {
                    const uint32_t w[4] = {c0.x, c0.y, c0.z, c0.w};
                    dequantize_group_u4(w, *mrec, 1.0f, x);
                } else {
                    const uint4 c1 = *reinterpret_cast<const uint4 *>(rec + p.codes_off + lo_chunk_off(r, 1, lo));
                    const uint32_t w[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
                    if (FMT == kFmtE4M3) dequantize_group_e4m3(w, __uint_as_float(*mrec), 1.0f, x);
                    else dequantize_group(w, *mrec, 1.0f, x);
                }
                if (HAD) hadamard_pairs(x);
#pragma unroll
                for (int m = 0; m < 8; ++m)
                    reinterpret_cast<float4 *>(row)[m] = make_float4(x[2 * m].x, x[2 * m].y, x[2 * m + 1].x, x[2 * m + 1].y);
            } else {
                // logical tiers <-> record, 32-bit words
                const int64_t row_bytes = (int64_t)p.V * CB;
                uint32_t *crow = reinterpret_cast<uint32_t *>(p.codes + ((((int64_t)b * p.H + h) * lo + r) * row_bytes + c * CB));
                uint32_t *mrow = reinterpret_cast<uint32_t *>(p.meta) + (((int64_t)b * p.H + h) * lo + r) * p.V + c;
#pragma unroll
                for (int m = 0; m < CB / 16; ++m) {
                    uint32_t *r4 = reinterpret_cast<uint32_t *>(m ? crec1 : crec);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        if (OP == kPackTiers) r4[e] = crow[4 * m + e];
                        else crow[4 * m + e] = r4[e];
                    }
                }
                if (OP == kPackTiers) *mrec = *mrow;
                else *mrow = *mrec;
            }
        }
        // ---- FP16 rows, lane = column, two rows per 32-bit word ----
        for (int u = 0; u < K; u += 2) {
            const bool two = u + 1 < K;
            uint32_t *word = reinterpret_cast<uint32_t *>(rec + hi_elem_off(u, lane));
            if (OP == kDequantize) {
                float *r0 = p.S + ((((int64_t)b * p.Hm + mh) * p.dk + (p.perm[(int64_t)h * p.dk + u] & (p.dk - 1))) * p.dv + c * kG + lane);
                float *r1 = two ? p.S + ((((int64_t)b * p.Hm + mh) * p.dk + (p.perm[(int64_t)h * p.dk + u + 1] & (p.dk - 1))) * p.dv + c * kG + lane) : nullptr;
                const float2 f = h2_to_f2(*word);
                *r0 = f.x;
                if (two) *r1 = f.y;
            } else {
                uint16_t *t0 = p.hi + ((((int64_t)b * p.H + h) * K + u) * p.dv + c * kG + lane);
                uint16_t *t1 = two ? t0 + p.dv : nullptr;
                if (OP == kPackTiers) {
                    *word = (uint32_t)*t0 | ((uint32_t)(two ? *t1 : 0) << 16);
                } else {
                    const uint32_t w = *word;
                    *t0 = (uint16_t)(w & 0xffffu);
                    if (two) *t1 = (uint16_t)(w >> 16);
                }
            }
        }
        // zero the record padding so packed pools compare bit for bit
        if (OP == kPackTiers) {
            const int used = p.meta_off + 4 * lo;
            if (lane < p.rec_bytes - used) rec[used + lane] = 0;
        }
    }
    if (lane == 0 && (bad_slot || bad_head))
        atomicOr(p.status, (bad_slot ? (uint32_t)kDevBadSlot : 0u) | (bad_head ? (uint32_t)kDevBadHead : 0u));
}

static cudaError_t conv_params(const ConvArgs &a, ConvParams &p) {
    static std::atomic<uint32_t *> cache[64];
    cudaError_t e = symbol_address_cached(&g_status_convert, cache, &p.status);
    if (e != cudaSuccess) return e;
    const RecGeom rg = rec_geom(a.dk, a.K, a.fmt);
    p.state = static_cast<uint8_t *>(a.state);
    p.num_slots = a.num_slots;
    p.slot_idx = a.slot_idx;
    p.perm = a.perm;
    p.S = a.S;
    p.hi = a.hi;
    p.codes = a.codes;
    p.meta = a.meta;
    p.batch = a.batch;
    p.H = a.H;
    p.Hm = a.head_map ? a.Hm : a.H;  // the tiers of pack / unpack are pool-indexed
    p.head_map = a.head_map;
    p.dk = a.dk;
    p.dv = a.dv;
    p.V = a.dv / kG;
    p.K = a.K;
    p.rec_bytes = rg.bytes;
    p.codes_off = rg.codes_off;
    p.meta_off = rg.meta_off;
    p.slot_bytes = (int64_t)a.H * p.V * rg.bytes;
    p.total_tiles = (int64_t)a.batch * a.H * p.V;
    return cudaSuccess;
}

#define DAMP_PICK_FMT(KERN_)                                                                   \
    switch (a.fmt) {                                                                           \
        case kFmtU8H32: kern = KERN_(kFmtU8H32); break;                                        \
        case kFmtU8: kern = KERN_(kFmtU8); break;                                              \
        case kFmtU4H32: kern = KERN_(kFmtU4H32); break;                                        \
        case kFmtU4: kern = KERN_(kFmtU4); break;                                              \
        case kFmtE4M3: kern = KERN_(kFmtE4M3); break;                                          \
        default: break;                                                                        \
    }

template <int OP>
static cudaError_t launch_tiers(const ConvArgs &a, cudaStream_t stream) {
    ConvParams p{};
    const cudaError_t e = conv_params(a, p);
    if (e != cudaSuccess || p.total_tiles == 0) return e;
    const int warps = 8;
    const int64_t want = (p.total_tiles + warps - 1) / warps;
    const int grid = (int)std::min<int64_t>(want, (int64_t)sm_count() * 8);
    void (*kern)(ConvParams) = nullptr;
#define DAMP_TIERS1(F_) tiers_kernel<1, F_, OP>
#define DAMP_TIERS2(F_) tiers_kernel<2, F_, OP>
#define DAMP_TIERS4(F_) tiers_kernel<4, F_, OP>
    if (a.dk == 32) DAMP_PICK_FMT(DAMP_TIERS1)
    if constexpr (OP != kDequantize) {
        if (a.dk == 64) DAMP_PICK_FMT(DAMP_TIERS2)
        if (a.dk == 128) DAMP_PICK_FMT(DAMP_TIERS4)
    }
    if (!kern) return cudaErrorInvalidValue;
    kern<<<grid, 32 * warps, 0, stream>>>(p);
    return cudaGetLastError();
}

template <bool QUANTIZE>
static cudaError_t launch_convert(const ConvArgs &a, cudaStream_t stream) {
    ConvParams p{};
    cudaError_t e = conv_params(a, p);
    if (e != cudaSuccess || p.total_tiles == 0) return e;
    void (*kern)(ConvParams) = nullptr;
#define DAMP_QUANT(F_) quantize_kernel<F_>
#define DAMP_DEQUANT(F_) dequantize_kernel<F_>
    if (QUANTIZE) DAMP_PICK_FMT(DAMP_QUANT)
    else DAMP_PICK_FMT(DAMP_DEQUANT)
    if (!kern) return cudaErrorInvalidValue;
    const int smem = kCvWarps * kCvTile * (QUANTIZE ? kCvStages : 1);
    if ((e = ensure_smem_limit(reinterpret_cast<const void *>(kern), smem)) != cudaSuccess) return e;
    // a warp with work for every record (four items at d_k = 128) up to three resident CTAs per SM
    // (registers; two CTAs with three tiles per warp: quantize 37.4 us against 35.8; four or more
    // for dequantize, whose warps then share the lines that they write: 38 -> 40-52 us)
    const int64_t want = (p.total_tiles + kCvWarps - 1) / kCvWarps;
    const int grid = (int)std::min<int64_t>(want, (int64_t)sm_count() * 3);
    kern<<<grid, 32 * kCvWarps, smem, stream>>>(p);
    return cudaGetLastError();
}

cudaError_t launch_quantize(const ConvArgs &a, cudaStream_t s) { return launch_convert<true>(a, s); }
// d_k = 32, rows straight to S / through the tiles: d_v = 64, H = 32, B = 256 UINT8 25.3 / 29.6 us,
// UINT4 23.6 / 29.9; d_v = 256, B = 1024 421 / 430; one request of 32 x 32 4.2 / 4.6.  From d_k = 64
// the tiles win: 64 x 32, B = 256 24.6 / 20.9.
cudaError_t launch_dequantize(const ConvArgs &a, cudaStream_t s) {
    return a.dk == 32 ? launch_tiers<kDequantize>(a, s) : launch_convert<false>(a, s);
}
cudaError_t launch_pack_tiers(const ConvArgs &a, cudaStream_t s) { return launch_tiers<kPackTiers>(a, s); }
cudaError_t launch_unpack_tiers(const ConvArgs &a, cudaStream_t s) { return launch_tiers<kUnpackTiers>(a, s); }

cudaError_t take_status_convert(uint32_t *bits) {
    uint32_t zero = 0;
    cudaError_t e = cudaMemcpyFromSymbol(bits, g_status_convert, sizeof(uint32_t));
    if (e != cudaSuccess) return e;
    return cudaMemcpyToSymbol(g_status_convert, &zero, sizeof(uint32_t));
}

}  // namespace damp
