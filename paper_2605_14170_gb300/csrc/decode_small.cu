// Single-code launch of the register-resident BP path for small codes (the
// [[72,12,6]] and [[144,12,12]] bivariate bicycle codes of Section IV); the
// per-chunk device code is in bp_small.cuh.  Warps pull
// (chunk of kChunk shots, representation) work items from a global counter.
#include <algorithm>

#include "bp_small.cuh"

namespace mbbp {
namespace {

constexpr int kSmallWarps = 1;  // warps per block: each warp works alone
// Work items: a run of consecutive shots of one representation.  The first
// `s8` shots come in runs of 8, the next `s2` in runs of 2, the rest one by
// one.  A run loads its representation's tables once, so long runs cost least
// per shot (runs of one shot: 13% more time on [[144,12,12]] R = 16, 200,000
// depolarizing shots at p = 0.04), but a shot that does not converge takes 100
// iterations where most take a few, and with runs of 8 the last ones leave
// most of the GPU idle.  So the last kTail1 shots per resident warp go one by
// one and the kTail2 before them in pairs.  With runs of 8 throughout ->
// this: [[72,12,6]] R = 4, 2,000 shots 106 -> 52 us; [[144,12,12]] R = 16 at
// p = 0.0533, 300 / 2,000 / 10,000 shots 296 -> 113 / 443 -> 288 / 1308 -> 1183
// us, 50,000 shots 5.55 -> 5.37 ms; the 200,000 shots above 11.35 -> 11.39 ms.
// Sum-product shots cost ten times as much, their tables nothing beside: runs
// of 2 and 1 only (4,000 shots 3.40 -> 2.76 ms).
//
// ONCE: every item has a warp of its own (short calls, a decoder in a control
// loop), which takes the item of its index: no pull, and no counter to clear
// before the launch.  A kernel of its own: with a test in the loop the one for
// long calls spills 60 bytes.  [[72,12,6]] R = 4, one shot, both in one process,
// 30 pairs taken in turn, each faster: median 17.5 -> 16.3 us a call in a row of
// calls (10% to 90%: 17.2-17.8, 16.1-16.6), 30.5 -> 28.2 us alone, 10.1 -> 4.4 us
// replayed from a graph; 16 shots 30.9 -> 28.7, 50.4 -> 48.4, 29.2 -> 24.1 us.
// (Between processes the host's part scatters by up to 18%.)
struct SmallWork {
    int s8, s2, s1;
};
constexpr long long kTail1 = 8, kTail2 = 8;

template <int VS, int RS, int ORS, int RULE, bool REG, bool OUT, bool ONCE>
__global__ void __launch_bounds__(kSmallWarps * 32, small_min_blocks(RS, RULE))
decode_small_kernel(const DecodeArgs a, const SmallWork work) {
    extern __shared__ __align__(16) float smsg[];
    const DevBases& B = a.B;
    const int lane = threadIdx.x & 31;
    const int warp = kSmallWarps == 1 ? 0 : warp_index();
    const unsigned R = (unsigned)B.R;
    char* smc = reinterpret_cast<char*>(smsg);
    const uint32_t wbase = (uint32_t)(warp * small_bp::warp_floats(B.MP, VS, ORS) * 4);
    const unsigned long long n8 = (unsigned long long)(work.s8 / 8) * R;
    const unsigned long long n2 = n8 + (unsigned long long)(work.s2 / 2) * R;
    const unsigned long long n1 = n2 + (unsigned long long)work.s1 * R;
    for (;;) {
        unsigned long long w = (unsigned long long)blockIdx.x * kSmallWarps + warp;
        if (!ONCE) {
            if (lane == 0) w = atomicAdd(a.counter, 1ull);
            w = __shfl_sync(small_bp::kFull, w, 0);
        }
        if (w >= n1) break;
        const int len = w < n8 ? 8 : (w < n2 ? 2 : 1);
        const int first = w < n8 ? 0 : (w < n2 ? work.s8 : work.s8 + work.s2);
        const unsigned long long l = w - (w < n8 ? 0 : (w < n2 ? n8 : n2));
        const int run = (int)(l / R);
        const int b = (int)(l - (unsigned long long)run * R);
        const int s0 = first + run * len;
        small_bp::run_chunk<VS, RS, ORS, RULE, REG, OUT>(B, a.io, b, s0, s0 + len, smc, wbase);
        if (ONCE) break;
    }
}

template <int VS, int RS, int ORS, int RULE, bool REG>
cudaError_t launch_small_t(const DecodeArgs& a, cudaStream_t s, int sm_count) {
    // calls that ask for posteriors or the message trace take the kernel
    // that writes them; the plain decode has no test for them in its loops
    auto kern = (a.io.c2v || a.io.post) ? decode_small_kernel<VS, RS, ORS, RULE, REG, true, false>
                                        : decode_small_kernel<VS, RS, ORS, RULE, REG, false, false>;
    const int warps = kSmallWarps;
    const size_t smem = (size_t)warps * small_bp::warp_floats(a.B.MP, VS, ORS) * sizeof(float);
    int per_sm = 0;
    cudaError_t e = prepare_kernel(reinterpret_cast<const void*>(kern), warps * 32, smem, &per_sm);
    if (e != cudaSuccess) return e;
    unsigned long long grid = (unsigned long long)per_sm * (unsigned long long)sm_count;
    const long long resident = (long long)grid * warps, batch = a.io.batch, R = a.B.R;
    SmallWork work;
    work.s1 = (int)std::min(batch, (kTail1 * resident + R - 1) / R);
    const long long rest = batch - work.s1;
    work.s8 = RULE == MBBP_RULE_NMS ? (int)(std::max(0ll, rest - (kTail2 * resident + R - 1) / R) / 8 * 8) : 0;
    work.s2 = (int)((rest - work.s8) / 2 * 2);
    work.s1 = (int)(batch - work.s8 - work.s2);
    const unsigned long long items = ((unsigned long long)work.s8 / 8 + work.s2 / 2 + work.s1) * (unsigned long long)R;
    unsigned long long want = (items + warps - 1) / warps;
    if (want <= grid) {
        grid = want;
        if constexpr (RULE == MBBP_RULE_NMS) {
            if (!a.io.c2v && !a.io.post) {
                auto once = decode_small_kernel<VS, RS, ORS, RULE, REG, false, true>;
                e = prepare_kernel(reinterpret_cast<const void*>(once), warps * 32, smem, &per_sm);
                if (e != cudaSuccess) return e;
                once<<<(unsigned)grid, warps * 32, smem, s>>>(a, work);
                return cudaGetLastError();
            }
        }
    }
    e = cudaMemsetAsync(a.counter, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)grid, warps * 32, smem, s>>>(a, work);
    return cudaGetLastError();
}

template <int VS, int RS, int ORS>
cudaError_t launch_shape(const DecodeArgs& a, cudaStream_t s, int sm_count) {
    const bool reg = a.B.regular != 0;
    if (a.rule == MBBP_RULE_NMS)
        return reg ? launch_small_t<VS, RS, ORS, MBBP_RULE_NMS, true>(a, s, sm_count)
                   : launch_small_t<VS, RS, ORS, MBBP_RULE_NMS, false>(a, s, sm_count);
    return reg ? launch_small_t<VS, RS, ORS, MBBP_RULE_SP, true>(a, s, sm_count)
               : launch_small_t<VS, RS, ORS, MBBP_RULE_SP, false>(a, s, sm_count);
}

}  // namespace

cudaError_t launch_decode_small(const DecodeArgs& a, cudaStream_t s, int sm_count) {
    if (a.B.shape == 1) return launch_shape<3, 2, 2>(a, s, sm_count);
    if (a.B.shape == 2) return launch_shape<5, 3, 3>(a, s, sm_count);
    if (a.B.shape == 3) return launch_shape<5, 4, 3>(a, s, sm_count);
    return cudaErrorInvalidValue;
}

}  // namespace mbbp
