// prefill_tc_gdn.cu -- launcher of the GDN prefill chunk on the tensor cores
// (prefill_tc.cuh), d_k = d_v = 128, bf16 q/k/v: the UINT8 tiers (formats 0 and 1).
#include <algorithm>

#include "damp_internal.h"
#include "prefill_tc.cuh"

namespace damp {

cudaError_t launch_prefill_tc_gdn(const PrefillParams &p, int fmt, cudaStream_t stream) {
    const int64_t pairs = (int64_t)p.batch * p.H;
    const int nv = tc_nv(pairs, sm_count());
    void (*kern)(PrefillParams) = nullptr;
    if (fmt == kFmtU8H32) kern = nv == 4 ? prefill_tc_gdn_kernel<kFmtU8H32, 4> : nv == 2 ? prefill_tc_gdn_kernel<kFmtU8H32, 2> : prefill_tc_gdn_kernel<kFmtU8H32, 1>;
    if (fmt == kFmtU8) kern = nv == 4 ? prefill_tc_gdn_kernel<kFmtU8, 4> : nv == 2 ? prefill_tc_gdn_kernel<kFmtU8, 2> : prefill_tc_gdn_kernel<kFmtU8, 1>;
    if (!kern) return cudaErrorNotSupported;
    const int smem = kTcSmem;
    if (p.rec_bytes > kTcMaxRec || smem > max_smem_per_block()) return cudaErrorNotSupported;
    // The CTA allocates all 512 tensor-memory columns of its SM, so a second CTA there
    // would wait in its allocation: the shared memory must keep it off the SM.
    const int per_sm = max_smem_per_sm();
    if (per_sm <= 0 || 2 * smem <= per_sm) return cudaErrorNotSupported;
    cudaError_t e = ensure_smem_limit(reinterpret_cast<const void *>(kern), smem);
    if (e != cudaSuccess) return e;
    const int grid = (int)std::min<int64_t>(pairs * (4 / nv), (int64_t)sm_count());
    kern<<<grid, kTcThreads, smem, stream>>>(p);
    return cudaGetLastError();
}

}  // namespace damp
