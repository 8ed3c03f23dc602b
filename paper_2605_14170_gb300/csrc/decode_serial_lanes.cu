// Serial schedule (Section II-B), one shot per lane, kernel widths 6 and 8, for
// long batches of shots that are not easy (the rule is at serial_route_kernel): a
// block decodes the shots of one representation in two groups of warps, each
// 16 shots in lockstep, two rows of a layer per warp step.  A slot whose shot
// halts takes the next one from the representation's counter, so lanes do not
// wait for slow shots; a block whose representation has none left moves on.
//
// The warp-per-slot kernel of bp_serial.cuh spends 158 instructions per lane
// and edge update on [[288,12,18]]: a layer of 9 to 25 rows fills half a warp,
// every edge pays for the most messages a variable has, and half of its
// shared-memory wavefronts are bank conflicts.  Here lanes hold shots: a layer
// of 20 rows is ten full warp steps, an edge's record is read once for 16
// shots, the rows of a step have their edges sorted by the number of other
// messages (min-sum is symmetric in them) so that only the first few test for
// more than three, and the halting test handles all shots at once: 47
// instructions.  The bound is latency: a group's barrier after every layer
// (issue slots 53% busy), with no more shots per SM than shared memory holds.
// Two groups and 16 shots per step hide it better than one of 32 where two
// blocks fit ([[144]]: 10.3 -> 10.1 ms before the steps were made uniform).
//
// Serial + least metric, p = 0.06, R = 20: [[288,12,18]], 20,000 shots 23.65 ->
// 13.9 ms; [[144,12,12]], 40,000 shots 17.4 -> 8.7 ms.
#include <algorithm>
#include <cmath>

#include "bp_generic.cuh"

namespace mbbp {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kMaxThreads = 768;
constexpr int kRows = 2;             // rows (or variables) of a warp step
constexpr int kShots = 32 / kRows;   // shots of a group of warps
constexpr int kGroups = 2;           // groups of a block (same representation)
constexpr uint32_t kSlots = (1u << kShots) - 1u;
constexpr int kRing = 32;            // tickets (shot numbers) a group holds, at most
constexpr int kPool = kShots;        // tickets kept ahead of need

// Shared memory of fixed size; with the layout below it may fill what a block
// can have.
struct SerialLanesFixed {
    int cls_cnt[16], cls_first[16], cls_pos[16];
    int open;
    uint32_t unsat[kGroups][2];
};
constexpr int kMaxDynamic = 227 * 1024 - (((int)sizeof(SerialLanesFixed) + 127) & ~127);

// Byte offsets in shared memory.
struct SerialLanesLayout {
    int rec, var, cnt, src, hidx, hpos, posof, lptr, group0;  // tables of the block
    int negz, ew, sw, ring, group_bytes;                      // inside a group's area (messages first)
    int total;
    int vwords;  // words of a variable record: mu and its message offsets
};

__host__ __device__ inline int al16(int x) { return (x + 15) & ~15; }

// steps: most row steps of a representation (layers padded to whole steps).
__host__ __device__ inline SerialLanesLayout serial_lanes_layout(int DC, int steps, int m, int n) {
    SerialLanesLayout L;
    const int rows = steps * kRows, npos = n + (DC + 2) * (kRows - 1);
    L.vwords = (DC + 1 + 3) & ~3;
    L.rec = 0;                                   // [rows][DC][8 words]: mu, up to 7 offsets
    L.var = L.rec + rows * DC * 32;              // [npos][vwords]
    L.cnt = L.var + npos * L.vwords * 4;         // [rows] bits 8 + j, 16 + j: edge j has above 3, 5 offsets; row degree << 24
    L.src = L.cnt + 4 * rows;                    // [rows] row of H (0xffff: padding)
    L.hidx = L.src + al16(2 * rows);             // [m] a row with that row of H
    L.hpos = L.hidx + al16(2 * m);               // [DC][m] positions of the columns of H's rows
    L.posof = L.hpos + al16(2 * DC * m);         // [n] position of a variable
    L.lptr = L.posof + al16(2 * n);              // [rows + 1] first step of each layer
    L.group0 = (L.lptr + al16(2 * (rows + 1)) + 127) & ~127;
    L.negz = steps * DC * 128;                   // after the messages: 32 x -0.0f
    L.ew = L.negz + 128;                         // [npos + 1] hard decisions, bit = shot slot
    L.sw = L.ew + 4 * (npos + 1);                // [steps] syndrome bits, bit = lane
    L.ring = L.sw + 4 * steps;
    L.group_bytes = (L.ring + 4 * kRing + 127) & ~127;
    L.total = L.group0 + kGroups * L.group_bytes;
    return L;
}

__device__ __forceinline__ void group_sync(int bar, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(threads) : "memory");
}

// Posterior of a variable of degree D (ascending row).
template <int D>
__device__ __forceinline__ float lane_post(const char* ms, const uint4* rec) {
    constexpr int NV = (D + 1 + 3) / 4;
    uint32_t r[4 * NV];
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        const uint4 x = rec[i];
        r[4 * i] = x.x;
        r[4 * i + 1] = x.y;
        r[4 * i + 2] = x.z;
        r[4 * i + 3] = x.w;
    }
    float m[D > 0 ? D : 1];
#pragma unroll
    for (int i = 0; i < D; ++i) m[i] = *reinterpret_cast<const float*>(ms + r[1 + i]);
    float P = __uint_as_float(r[0]);
#pragma unroll
    for (int i = 0; i < D; ++i) P = __fadd_rn(P, m[i]);
    return P;
}

// Posteriors and hard decisions of the steps of warp wig of nw, in degree order.
template <int D, int DC>
__device__ __forceinline__ void lane_posts(int& st, int nw, const int* cend, const char* ms, const uint4* var,
                                           uint32_t* ew) {
    constexpr int VW = ((DC + 1 + 3) & ~3) / 4;
    const int lane = threadIdx.x & 31, slot = lane % kShots, sub = lane / kShots;
    for (; st + nw < cend[D]; st += 2 * nw) {  // two steps at once: one waits for the other's loads
        const float x = lane_post<D>(ms, var + (st * kRows + sub) * VW);
        const float y = lane_post<D>(ms, var + ((st + nw) * kRows + sub) * VW);
        const uint32_t w = __ballot_sync(kFull, x < 0.f), z = __ballot_sync(kFull, y < 0.f);
        if (slot == 0) {
            ew[st * kRows + sub] = (w >> (sub * kShots)) & kSlots;
            ew[(st + nw) * kRows + sub] = (z >> (sub * kShots)) & kSlots;
        }
    }
    for (; st < cend[D]; st += nw) {
        const uint32_t w = __ballot_sync(kFull, lane_post<D>(ms, var + (st * kRows + sub) * VW) < 0.f);
        if (slot == 0) ew[st * kRows + sub] = (w >> (sub * kShots)) & kSlots;
    }
    if constexpr (D < DC) lane_posts<D + 1, DC>(st, nw, cend, ms, var, ew);
}

// Which of the two serial kernels takes a call.  A shot that halts in this one
// makes its group refill a slot, and the last shots of a representation run at
// its slower pace per iteration (one of 32 shots of a block against one of at
// most 4 of a warp); both are small only beside the iterations of a long batch
// of shots that take several.  How many they take shows in the syndromes, which
// are on the device.  So one block counts the ones of 128 syndromes spread over
// the batch and sets *flag; of the two kernels launched after it the other
// returns at once.  It clears the shot counters too, in place of a memset.  A
// call that stays with the warp-per-slot kernel pays 3 to 8 us for both launches:
// [[72]] R = 4, 20,000 shots at p = 0.001 87 us, 82 without them.
//
// A call takes this kernel when it has at least 16 rounds (32 items per SM each)
// and  rounds * density^2 * min(1, density / 0.12) >= c:  the first factors weigh
// the last shots, whose pace costs up to the iteration limit, so c grows with it,
// 0.2 + 0.008 iters (min-sum) or 0.5 + 0.1 iters (sum-product, which takes longer
// in one lane); the last factor weighs the refills, and below densities of 0.05
// and 0.1 they outweigh all.  Measured at 4,300 points (15 codes of length 60 to
// 288, rows of weight 2 to 8, R = 1 to 20, error rates 0.003 to 0.2, 1 to 200
// iterations, 4 to 768 rounds): at the 2,000 that satisfy the rule this kernel is
// 0.993 to 3.4 times as fast as the warp-per-slot kernel (geometric mean 1.6
// min-sum, 1.5 sum-product).  Slowest and fastest code, min-sum, 100 iterations,
// by error rate, density (rows of weight 6) and rounds; [ ] below the rule:
//      p    density       16             32           96          768
//   0.003   0.018         -              -       [0.69-0.96]  [0.69-0.98]
//   0.01    0.057         -              -       [0.88-1.19]   1.03-1.38
//   0.02    0.11    [0.71-1.12]    [0.84-1.29]    1.04-1.85       -
//   0.04    0.20    [0.90-1.82]     1.03-2.08     1.17-2.52       -
//   0.06    0.27     1.03-2.19      1.21-2.56     1.47-2.90       -
//   0.08    0.32     1.22-2.59      1.28-2.85        -            -
constexpr int kRouteShots = 128;
constexpr int kRouteThreads = 1024;
constexpr int kMinRounds = 16;

// The least density at which a call takes this kernel.
float min_density(int rule, int iters, double rounds) {
    const bool nms = rule == MBBP_RULE_NMS;
    const double x = (nms ? 0.2 + 0.008 * iters : 0.5 + 0.1 * iters) / rounds;
    const double d = x >= 0.12 * 0.12 ? std::sqrt(x) : std::cbrt(0.12 * x);
    return (float)std::max(nms ? 0.05 : 0.1, d);
}

__global__ void __launch_bounds__(kRouteThreads) serial_route_kernel(const uint8_t* __restrict__ synd, int m, int batch,
                                                                     int R, float density, unsigned int* flag,
                                                                     unsigned int* rep_counter) {
    __shared__ int ones;
    if (threadIdx.x == 0) ones = 0;
    if (threadIdx.x < R) rep_counter[threadIdx.x] = 0;
    __syncthreads();
    const int shots = min(batch, kRouteShots), step = batch / shots;
    int c = 0;
    for (int i = threadIdx.x; i < shots * m; i += kRouteThreads) {
        const int k = i / m;
        c += __ldg(synd + (size_t)(k * step) * m + (i - k * m)) & 1;
    }
    c = __reduce_add_sync(kFull, c);
    if ((threadIdx.x & 31) == 0) atomicAdd(&ones, c);
    __syncthreads();
    if (threadIdx.x == 0) *flag = (float)ones >= density * (float)(shots * m);
}

template <int DC, int RULE, bool REG>
__global__ void __launch_bounds__(kMaxThreads, 1) decode_serial_lanes_kernel(const DecodeArgs a) {
    if (!*a.lanes) return;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ SerialLanesFixed fixed;
    int *cls_cnt = fixed.cls_cnt, *cls_first = fixed.cls_first, *cls_pos = fixed.cls_pos;
    const DevBases& B = a.B;
    const ShotIO& io = a.io;
    const int n = B.n, m = B.m, R = B.R, W = B.W, MP = B.MP;
    const SerialLanesLayout L = serial_lanes_layout(DC, B.lsteps, m, n);
    const int lane = threadIdx.x & 31, slot = lane % kShots, sub = lane / kShots;
    const int nw = (int)(blockDim.x >> 5) / kGroups;  // warps of a group
    const int wid = warp_index();
    const int grp = wid / nw, warp = wid - grp * nw;
    const int gthreads = nw * 32, gt = warp * 32 + lane, bar = 1 + grp;
    unsigned char* area = smem + L.group0 + grp * L.group_bytes;
    char* mrow = reinterpret_cast<char*>(area) + 4 * lane;   // a step's own messages
    char* msg = reinterpret_cast<char*>(area) + 4 * slot;    // by record offset
    uint4* rec = reinterpret_cast<uint4*>(smem + L.rec);
    uint4* var = reinterpret_cast<uint4*>(smem + L.var);
    uint32_t* cnt = reinterpret_cast<uint32_t*>(smem + L.cnt);
    uint16_t* src = reinterpret_cast<uint16_t*>(smem + L.src);
    uint16_t* hidx = reinterpret_cast<uint16_t*>(smem + L.hidx);
    uint16_t* hpos = reinterpret_cast<uint16_t*>(smem + L.hpos);
    uint16_t* posof = reinterpret_cast<uint16_t*>(smem + L.posof);
    uint16_t* lptr = reinterpret_cast<uint16_t*>(smem + L.lptr);
    uint32_t* ew = reinterpret_cast<uint32_t*>(area + L.ew);
    uint32_t* sw = reinterpret_cast<uint32_t*>(area + L.sw);
    int* ring = reinterpret_cast<int*>(area + L.ring);
    uint32_t* unsat = fixed.unsat[grp];
    // blocks start spread over the representations by their rows
    if (threadIdx.x == 0) {
        long long total = 0, sum = 0;
        for (int t = 0; t < R; ++t) total += __ldg(B.rows + t);
        const long long at = total * (2 * (long long)blockIdx.x + 1) / (2 * (long long)gridDim.x);
        int t = 0;
        while (t + 1 < R && (sum += __ldg(B.rows + t)) <= at) ++t;
        fixed.open = t;
    }
    __syncthreads();
    const int b0 = fixed.open;

    for (int kb = 0; kb < R; ++kb) {
        __syncthreads();
        const int b = (b0 + kb) % R;
        if (threadIdx.x == 0) {
            fixed.open = *reinterpret_cast<volatile unsigned int*>(a.rep_counter + b) < (unsigned)io.batch;
        }
        if (threadIdx.x < 16) cls_cnt[threadIdx.x] = 0;
        if (gt < 2) unsat[gt] = 0;
        __syncthreads();
        if (!fixed.open) continue;
        // tables of representation b; rows in layer order, layers padded to
        // whole steps.  Until the shots start, the first group's message area
        // holds the row of each position of the chunk layout and, per row, the
        // order of its edges (3 bits each).
        const int Mb = __ldg(B.rows + b), nl = __ldg(B.nlayers + b);
        const uint16_t* lpos = B.lpos + (size_t)b * MP;
        const uint16_t* lp = B.lptr + (size_t)b * (MP + 1);
        const uint32_t* rinfo = B.rinfo_s + (size_t)b * MP;
        const uint4* ed = B.edesc + (size_t)b * DC * MP;
        const uint2* vd = B.vdesc + (size_t)b * n;
        uint16_t* row_at = reinterpret_cast<uint16_t*>(smem + L.group0);
        uint32_t* order = reinterpret_cast<uint32_t*>(smem + L.group0 + al16(2 * MP));
        for (int p = threadIdx.x; p < n; p += blockDim.x) atomicAdd(&cls_cnt[__ldg(&vd[p].y) >> 16], 1);
        if (threadIdx.x == 0) {
            int st = 0;
            for (int l = 0; l < nl; ++l) {
                lptr[l] = (uint16_t)st;
                st += ((int)__ldg(lp + l + 1) - (int)__ldg(lp + l) + kRows - 1) / kRows;
            }
            lptr[nl] = (uint16_t)st;
        }
        __syncthreads();
        const int steps = lptr[nl];
        for (int i = threadIdx.x; i < steps * kRows; i += blockDim.x) src[i] = 0xffffu;
        if (threadIdx.x == 0) {
            int f = 0, q = 0;
            for (int d = 0; d <= DC; ++d) {
                cls_first[d] = f;
                cls_pos[d] = q;
                f += cls_cnt[d];
                q += (cls_cnt[d] + kRows - 1) / kRows * kRows;
            }
            cls_pos[DC + 1] = q;
        }
        // rows: thread t takes the t-th, ... row of the layer order
        for (int t = threadIdx.x; t < Mb; t += blockDim.x) {
            int l = 0;
            while ((int)__ldg(lp + l + 1) <= t) ++l;
            const int i = lptr[l] * kRows + t - (int)__ldg(lp + l);
            const int p = __ldg(lpos + t);
            row_at[p] = (uint16_t)i;
            // edges by the number of other messages, most first (min-sum is
            // symmetric in them; sum-product keeps the column order)
            const int deg = (int)((__ldg(rinfo + p) >> 16) & 0xffu);
            uint32_t no = 0, ord = 0;
            for (int j = 0; j < deg; ++j) {
                const uint4 d = __ldg(ed + generic_bp::row_slot<DC>(p) + 32 * j);
                const uint32_t o[7] = {d.x >> 16, d.y & 0xffffu, d.y >> 16, d.z & 0xffffu,
                                       d.z >> 16, d.w & 0xffffu, d.w >> 16};
                uint32_t c = 0;
                for (int u = 0; u < 7; ++u) c += (o[u] >> 2) < (uint32_t)(DC * MP);
                no |= c << (3 * j);
            }
            for (int j = 0; j < deg; ++j) {
                const uint32_t c = (no >> (3 * j)) & 7u;
                int r = 0;
                for (int u = 0; u < deg; ++u) {
                    const uint32_t cu = (no >> (3 * u)) & 7u;
                    r += (RULE == MBBP_RULE_NMS) ? (cu > c || (cu == c && u < j)) : (u < j);
                }
                ord |= (uint32_t)r << (3 * j);
            }
            order[i] = ord;
        }
        __syncthreads();
        auto off = [&](uint32_t o) -> uint32_t {
            const int s = (int)(o >> 2);
            if (s >= DC * MP) return (uint32_t)L.negz;
            const int p = (s / (32 * DC)) * 32 + (s & 31), j = (s >> 5) % DC, i = row_at[p];
            return (uint32_t)((i / kRows * DC + (int)((order[i] >> (3 * j)) & 7u)) * 128 + i % kRows * (4 * kShots));
        };
        for (int i = threadIdx.x; i < steps * kRows; i += blockDim.x) {
            // padding rows: no edges with messages
            cnt[i] = 0;
            for (int j = 0; j < DC; ++j) {
                rec[(i * DC + j) * 2] = make_uint4(0u, (uint32_t)L.negz, (uint32_t)L.negz, (uint32_t)L.negz);
                rec[(i * DC + j) * 2 + 1] = make_uint4((uint32_t)L.negz, (uint32_t)L.negz, (uint32_t)L.negz, (uint32_t)L.negz);
            }
        }
        __syncthreads();
        for (int t = threadIdx.x; t < Mb; t += blockDim.x) {
            const int p = __ldg(lpos + t), i = row_at[p];
            const uint32_t ri = __ldg(rinfo + p);
            const int deg = (int)((ri >> 16) & 0xffu);
            src[i] = (uint16_t)ri;
            hidx[ri & 0xffffu] = (uint16_t)i;
            uint32_t c = (uint32_t)deg << 24;
            for (int j = 0; j < deg; ++j) {
                const uint4 d = __ldg(ed + generic_bp::row_slot<DC>(p) + 32 * j);
                const uint32_t o[7] = {d.x >> 16, d.y & 0xffffu, d.y >> 16, d.z & 0xffffu,
                                       d.z >> 16, d.w & 0xffffu, d.w >> 16};
                uint32_t f[7], no = 0;
                for (int u = 0; u < 7; ++u) {
                    f[u] = off(o[u]);
                    no += f[u] != (uint32_t)L.negz;
                }
                const int jj = (int)((order[i] >> (3 * j)) & 7u);
                c |= (no > 3 ? 0x100u << jj : 0u) | (no > 5 ? 0x10000u << jj : 0u);
                rec[(i * DC + jj) * 2] = make_uint4(
                    __float_as_uint(__fadd_rn(__ldg(io.llr + (d.x & 0xffffu)), 0.0f)), f[0], f[1], f[2]);
                rec[(i * DC + jj) * 2 + 1] = make_uint4(f[3], f[4], f[5], f[6]);
            }
            cnt[i] = c;
        }
        for (int p = threadIdx.x; p < n; p += blockDim.x) {
            const uint32_t y = __ldg(&vd[p].y);
            const int v = (int)(y & 0xffffu), deg = (int)(y >> 16);
            const uint4 d = __ldg(B.vdesc3 + (size_t)b * n + v);
            const uint32_t o[8] = {d.x & 0xffffu, d.x >> 16, d.y & 0xffffu, d.y >> 16,
                                   d.z & 0xffffu, d.z >> 16, d.w & 0xffffu, d.w >> 16};
            const int idx = p - cls_first[deg];
            int np = cls_pos[deg] + idx;
            posof[v] = (uint16_t)np;
            // a class is padded to whole steps with copies of its last variable
            const int last = (idx == cls_cnt[deg] - 1) ? cls_pos[deg + 1] : np + 1;
            for (; np < last; ++np) {
                uint32_t* r = reinterpret_cast<uint32_t*>(var) + np * L.vwords;
                r[0] = __float_as_uint(__fadd_rn(__ldg(io.llr + v), 0.0f));
                for (int u = 0; u < DC; ++u) r[1 + u] = off(o[u]);
            }
        }
        __syncthreads();
        const int npos = cls_pos[DC + 1];
        int cend[DC + 1];
#pragma unroll
        for (int d = 0; d <= DC; ++d) cend[d] = cls_pos[d + 1] / kRows;
        for (int i = threadIdx.x; i < DC * m; i += blockDim.x) {
            const int j = i / m, r = i - j * m;
            const int v = __ldg(B.hcol + j * B.mpad + r);
            hpos[i] = v < n ? posof[v] : (uint16_t)npos;
        }
        if (gt < 32) reinterpret_cast<float*>(area + L.negz)[gt] = -0.0f;
        if (gt == 0) ew[npos] = 0;
        int head = 0, tail = kShots + kPool;  // ring positions taken / filled
        bool exhausted = false;
        if (warp == 0) {
            int base = 0;
            if (lane == 0) base = (int)atomicAdd(a.rep_counter + b, (unsigned)(kShots + kPool));
            base = __shfl_sync(kFull, base, 0);
            if (lane < kShots + kPool) ring[lane] = base + lane;
        }
        __syncthreads();

        int shot = -1, K = 0, phase = 0;
        uint32_t active = 0, done = 0, conv = 0;
        for (;;) {
            // outputs of the slots that halted
            uint32_t f = done;
            for (int k = 0; f; ++k, f &= f - 1) {
                if (k % nw != warp) continue;
                const int sl = __ffs(f) - 1;
                const int sh = __shfl_sync(kFull, shot, sl);
                const int Ks = __shfl_sync(kFull, K, sl);
                const unsigned long long item = (unsigned long long)sh * R + b;
                for (int w = 0; w < W; ++w) {
                    const int v = 32 * w + lane;
                    const uint32_t word = __ballot_sync(kFull, v < n && ((ew[posof[v < n ? v : 0]] >> sl) & 1u));
                    if (lane == 0) io.cand[item * W + w] = word;
                }
                if (lane == 0) {
                    io.conv[item] = (conv >> sl) & 1u;
                    if (io.iters_run) io.iters_run[item] = (uint16_t)Ks;
                }
            }
            active &= ~done;
            // idle slots take the next tickets
            uint32_t fresh = 0;
            if (active != kSlots && !exhausted) {
                const uint32_t need = kSlots & ~active;
                const int take = min(__popc(need), tail - head);
                const int rank = __popc(need & ((1u << slot) - 1u));
                const bool mine = ((need >> slot) & 1u) && rank < take;
                bool ok = false;
                if (mine) {
                    shot = ring[(head + rank) & (kRing - 1)];
                    ok = (unsigned)shot < (unsigned)io.batch;
                    K = 0;
                }
                fresh = __ballot_sync(kFull, ok) & kSlots;
                if (__any_sync(kFull, mine && !ok)) exhausted = true;
                head += take;
                active |= fresh;
            }
            if (!active) break;
            // tickets for the next refill (read after a barrier)
            if (warp == nw - 1) {
                const int want = exhausted ? 0 : kPool - (tail - head);
                if (want > 0) {
                    int base = 0;
                    if (lane == 0) base = (int)atomicAdd(a.rep_counter + b, (unsigned)want);
                    base = __shfl_sync(kFull, base, 0);
                    if (lane < want) ring[(tail + lane) & (kRing - 1)] = base + lane;
                }
            }
            if (!exhausted) tail = head + kPool;
            if (fresh) {
                if (done) group_sync(bar, gthreads);  // ew has been read
                f = fresh;
                for (int k = 0; f; ++k, f &= f - 1) {
                    if (k % nw != warp) continue;
                    const int sl = __ffs(f) - 1;
                    const uint8_t* sy = io.synd + (size_t)__shfl_sync(kFull, shot, sl) * m;
                    // all loads first, then the bits (padding rows: bit 0)
                    for (int i0 = lane; i0 < steps * kRows; i0 += 8 * 32) {
                        uint32_t bits = 0;
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            const int i = i0 + 32 * u;
                            if (i < steps * kRows && src[i] != 0xffffu) bits |= (uint32_t)(__ldg(sy + src[i]) & 1u) << u;
                        }
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            const int i = i0 + 32 * u;
                            const uint32_t bit = 1u << (i % kRows * kShots + sl);
                            if (i < steps * kRows) {
                                if ((bits >> u) & 1u) atomicOr(sw + i / kRows, bit);
                                else atomicAnd(sw + i / kRows, ~bit);
                            }
                        }
                    }
                }
                if ((fresh >> slot) & 1u)
                    for (int s = warp; s < steps * DC; s += nw) *reinterpret_cast<float*>(mrow + s * 128) = 0.0f;
                for (int p = gt; p < npos; p += gthreads) {
                    const float mu = __uint_as_float(reinterpret_cast<const uint32_t*>(var)[p * L.vwords]);
                    ew[p] = (ew[p] & ~fresh) | (mu < 0.f ? fresh : 0u);
                }
                group_sync(bar, gthreads);
            } else {
                // one serial iteration (slots just filled first test the hard
                // decision of mu)
                for (int l = 0; l < nl; ++l) {
                    const int s1 = lptr[l + 1];
                    for (int st = lptr[l] + warp; st < s1; st += nw) {
                        const int i = st * kRows + sub;
                        const uint4* rr = rec + i * (DC * 2);
                        const uint32_t c = cnt[i];
                        const int deg = REG ? DC : (int)(c >> 24);
                        float q[DC];
#pragma unroll
                        for (int j = 0; j < DC; ++j) {
                            const uint4 d = rr[2 * j];
                            float x = __uint_as_float(d.x);
                            x = __fadd_rn(x, *reinterpret_cast<const float*>(msg + d.y));
                            x = __fadd_rn(x, *reinterpret_cast<const float*>(msg + d.z));
                            q[j] = __fadd_rn(x, *reinterpret_cast<const float*>(msg + d.w));
                        }
                        // further messages where a row of the step has them
                        // (the other row adds the -0.0f slot)
                        const uint32_t more = __reduce_or_sync(kFull, c);
                        if (more & 0xff00u) {
#pragma unroll
                            for (int j = 0; j < DC; ++j) {
                                if (more & (0x100u << j)) {
                                    const uint4 d = rr[2 * j + 1];
                                    q[j] = __fadd_rn(q[j], *reinterpret_cast<const float*>(msg + d.x));
                                    q[j] = __fadd_rn(q[j], *reinterpret_cast<const float*>(msg + d.y));
                                    if (DC > 6 && (more & (0x10000u << j))) {
                                        q[j] = __fadd_rn(q[j], *reinterpret_cast<const float*>(msg + d.z));
                                        q[j] = __fadd_rn(q[j], *reinterpret_cast<const float*>(msg + d.w));
                                    }
                                }
                            }
                        }
                        if (!REG) {
#pragma unroll
                            for (int j = 0; j < DC; ++j)
                                if (j >= deg) q[j] = MBBP_LMAX;
                        }
                        float* row = reinterpret_cast<float*>(mrow + st * (DC * 128));
                        generic_bp::check_out<DC, RULE, REG>(q, row, deg, (sw[st] >> lane) & 1u, io.alpha);
                    }
                    group_sync(bar, gthreads);
                }
                int st = warp;
                lane_posts<0, DC>(st, nw, cend, msg, var, ew);
                group_sync(bar, gthreads);
                ++K;
            }
            // halting rule of all slots: a thread's row is satisfied in the
            // slots whose bit of acc is 0
            uint32_t acc = 0;
            for (int t = gt; t < m; t += gthreads) {
                const int i = hidx[t];
                uint32_t x = (sw[i / kRows] >> (i % kRows * kShots)) & kSlots;
#pragma unroll
                for (int j = 0; j < DC; ++j) x ^= ew[hpos[j * m + t]];
                acc |= x;
            }
            acc = __reduce_or_sync(kFull, acc);
            if (lane == 0 && acc) atomicOr(&unsat[phase], acc);
            group_sync(bar, gthreads);
            conv = active & ~*reinterpret_cast<volatile uint32_t*>(&unsat[phase]);
            done = conv | (active & __ballot_sync(kFull, K >= io.iters));
            phase ^= 1;
            if (gt == 0) unsat[phase] = 0;
        }
    }
}

// Launches the kernel with 24 warps per SM in as many blocks as an SM holds, 1
// to 4: more blocks hide each other's barriers and hold more shots ([[72]] R = 20
// at p = 0.06, 48 rounds, against the warp-per-slot kernel: 1 / 2 / 3 / 4 blocks
// 0.84 / 1.20 / 1.32 / 1.33 times as fast).
template <int DC, int RULE, bool REG>
cudaError_t launch_t(const DecodeArgs& a, cudaStream_t s, int sm_count) {
    auto kern = decode_serial_lanes_kernel<DC, RULE, REG>;
    const SerialLanesLayout L = serial_lanes_layout(DC, a.B.lsteps, a.B.m, a.B.n);
    int blocks = 4, threads = 0, per_sm = 0;
    for (;; --blocks) {
        if (blocks > 1 && (size_t)blocks * L.total > 227 * 1024) continue;
        threads = kMaxThreads / blocks / (32 * kGroups) * (32 * kGroups);
        const cudaError_t e = prepare_kernel(reinterpret_cast<const void*>(kern), threads, (size_t)L.total, &per_sm);
        if (e != cudaSuccess) return e;
        if (per_sm >= blocks) break;  // what a block takes besides can leave room for one less
    }
    const unsigned long long items = (a.total_items + kGroups * kShots - 1) / (kGroups * kShots);
    kern<<<(unsigned)std::min<unsigned long long>((unsigned long long)per_sm * sm_count, items), threads, L.total, s>>>(a);
    return cudaGetLastError();
}

template <int DC>
cudaError_t launch_width(const DecodeArgs& a, cudaStream_t s, int sm_count) {
    const bool reg = a.B.regular != 0;
    if (a.rule == MBBP_RULE_NMS)
        return reg ? launch_t<DC, MBBP_RULE_NMS, true>(a, s, sm_count)
                   : launch_t<DC, MBBP_RULE_NMS, false>(a, s, sm_count);
    return reg ? launch_t<DC, MBBP_RULE_SP, true>(a, s, sm_count)
               : launch_t<DC, MBBP_RULE_SP, false>(a, s, sm_count);
}

}  // namespace

cudaError_t launch_decode_serial_lanes(const DecodeArgs& args, cudaStream_t s, int sm_count, const unsigned int** flag) {
    const DevBases& B = args.B;
    *flag = nullptr;
    const double rounds = (double)args.total_items / (32.0 * sm_count);
    if (rounds < kMinRounds || args.io.post || args.io.llr_stride != 0 ||
        serial_lanes_layout(B.DC, B.lsteps, B.m, B.n).total > kMaxDynamic)
        return cudaMemsetAsync(args.rep_counter, 0, sizeof(unsigned int) * (size_t)B.R, s);
    DecodeArgs a = args;
    unsigned int* word = reinterpret_cast<unsigned int*>(a.counter);  // a work counter that this path does not use
    a.lanes = word;
    serial_route_kernel<<<1, kRouteThreads, 0, s>>>(a.io.synd, B.m, a.io.batch, B.R, min_density(a.rule, a.io.iters, rounds), word,
                                                    a.rep_counter);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    *flag = word;
    return B.DC == 6 ? launch_width<6>(a, s, sm_count) : launch_width<8>(a, s, sm_count);
}

}  // namespace mbbp
