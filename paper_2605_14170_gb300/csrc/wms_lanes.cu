// Weighted min-sum (WMS) training, forward with loss and adjoint, with one shot
// per lane: a block decodes 16 shots of one representation in lockstep, its
// warps taking two rows (or two variables of one degree) per step.  See wms.cu
// for the recursion; every edge and variable is computed by the same
// operations in the same order, so posteriors and messages are the same bits.
//
// Training runs all T iterations of every shot, so lanes never idle, and what
// belongs to an edge (its slot, weight and damping) is shared by the lanes
// that hold a shot each: no bank conflicts in the check pass, uniform
// addresses, and the parameter gradients of 16 shots are summed across lanes
// before one atomic add.  The warp-per-shot kernels of wms.cu spend 80
// (forward) and 216 (backward) instructions per lane and edge iteration and an
// uncoalesced float atomic per parameter and shot; these 49 and 113.
// Messages live in shared memory, the adjoint's recomputed states in the
// workspace (they stay in L2).  Issue slots are 60-65% busy; the rest is
// latency: barriers between the passes and the state loads.  At width 6, 24
// warps per SM at 80 registers: fewer warps with more registers, more with
// spills, 32 shots per block, wider parameter or record loads and a prefetch of
// the next row's state all measured slower or the same.
//
// [[144,12,12]] R = 8, T = 25, checkpoints every 5, batch 4096: forward 0.93 ->
// 0.72 ms, backward 4.58 -> 1.98 ms (0.74 and 2.15 before the warp's index was
// broadcast, which lets the compiler keep what depends on it in uniform
// registers); batch 300 R = 4: 0.091 + 0.336 -> 0.084 +
// 0.201 ms; [[288,12,18]] R = 4, batch 1500: 0.50 + 2.94 -> 0.38 + 1.04 ms.
#include <algorithm>
#include <climits>
#include "bp_generic.cuh"
#include "wms_common.cuh"

namespace mbbp {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kLaneThreads = 768;  // largest block
// Threads of the adjoint by kernel width: a row's edges are in registers
// throughout, and with 80 of them (768 threads) width 8 spills 88 to 112 bytes
// and width 12 408 to 424; with these 8 to 24 and 148 to 168 are left.  A step at
// T = 20, checkpoints every 5, 768 -> these: width 8 (length 96, rows of 8,
// R = 4, batch 300) 0.234 -> 0.213 ms, width 12 (length 96, rows of 10) 0.377 ->
// 0.306 ms; batch 2000, R = 8 1.104 -> 1.053 and 2.108 -> 1.919.  512 and 384:
// 0.207, 0.315; 1.143, 2.354 (12 warps per SM with two blocks of 6).
template <int DC>
constexpr int kBackwardThreads = DC == 12 ? 512 : (DC == 8 ? 640 : kLaneThreads);
constexpr int kLaneRows = 2;       // rows (or variables) of a warp step
constexpr int kLaneShots = 32 / kLaneRows;

// Byte offsets in shared memory.
struct LanesLayout {
    int rsteps, npos;                      // row steps, variable positions
    int vt, e0, sw, et, part, a0, a1, gp;  // tables, two message arrays, the posterior gradients
    int slot_floats, total;                // floats of a message array: the slots, then 32 that are only read
};

// Words of a variable's record: mu, the variable, DC offsets.
__host__ __device__ constexpr int record_words(int DC) { return DC + 2; }

__host__ __device__ inline LanesLayout lanes_layout(int DC, int MP, int n) {
    constexpr int S = kLaneRows;
    LanesLayout L;
    L.rsteps = (MP + S - 1) / S;
    L.npos = (n + (DC + 1) * (S - 1) + S - 1) / S * S;
    L.vt = 0;
    L.e0 = L.vt + L.npos * record_words(DC) * 4;
    L.sw = L.e0 + L.rsteps * S * 4;
    L.et = L.sw + L.rsteps * 4;
    L.part = L.et + L.npos / S * 4;
    L.a0 = (L.part + kLaneThreads * 4 + 127) & ~127;
    L.slot_floats = L.rsteps * DC * 32 + 32;
    L.a1 = L.a0 + L.slot_floats * 4;
    L.gp = L.a1 + L.slot_floats * 4;
    L.total = L.gp + L.npos / S * 128;
    return L;
}

// Sum of N values per lane over the CS lanes of a row: at each step a pair of
// values is split between the two halves of the lanes, so N values take about
// N shuffles in all instead of 5 N.  Afterwards lane l holds the sums of the
// values of index idx[i] (own[i]: this lane stores it).
template <int N, int MASK>
struct LaneSum {
    static constexpr int H = N / 2 + (N & 1);
    static constexpr int OUT = LaneSum<H, MASK / 2>::OUT;
    static __device__ __forceinline__ void run(float (&v)[N], float (&out)[OUT]) {
        const bool up = threadIdx.x & MASK;
        float h[H];
#pragma unroll
        for (int i = 0; i < N / 2; ++i) {
            const float keep = up ? v[2 * i + 1] : v[2 * i];
            const float send = up ? v[2 * i] : v[2 * i + 1];
            h[i] = keep + __shfl_xor_sync(kFull, send, MASK);
        }
        if (N & 1) h[H - 1] = v[N - 1] + __shfl_xor_sync(kFull, v[N - 1], MASK);
        LaneSum<H, MASK / 2>::run(h, out);
    }
    static __device__ __forceinline__ void index(int (&v)[N], bool (&own)[N], int (&out)[OUT], bool (&oown)[OUT]) {
        const bool up = threadIdx.x & MASK;
        int h[H];
        bool o[H];
#pragma unroll
        for (int i = 0; i < N / 2; ++i) {
            h[i] = up ? v[2 * i + 1] : v[2 * i];
            o[i] = up ? own[2 * i + 1] : own[2 * i];
        }
        if (N & 1) {
            h[H - 1] = v[N - 1];
            o[H - 1] = own[N - 1] && !up;
        }
        LaneSum<H, MASK / 2>::index(h, o, out, oown);
    }
};
template <int N>
struct LaneSum<N, 0> {
    static constexpr int OUT = N;
    static __device__ __forceinline__ void run(float (&v)[N], float (&out)[N]) {
#pragma unroll
        for (int i = 0; i < N; ++i) out[i] = v[i];
    }
    static __device__ __forceinline__ void index(int (&v)[N], bool (&own)[N], int (&out)[N], bool (&oown)[N]) {
#pragma unroll
        for (int i = 0; i < N; ++i) {
            out[i] = v[i];
            oown[i] = own[i];
        }
    }
};

template <int DC, bool REG>
struct Block {
    static constexpr int S = kLaneRows, CS = kLaneShots;
    static constexpr int RW = record_words(DC);
    const WmsArgs& a;
    const LanesLayout L;
    unsigned char* smem;
    int lane, warp, nw, slot, sub;
    int b, Mb, rsteps, shot;
    bool live;
    int cend[DC + 1];

    __device__ __forceinline__ Block(const WmsArgs& args, unsigned char* sm)
        : a(args), L(lanes_layout(DC, args.B.MP, args.B.n)), smem(sm) {
        lane = threadIdx.x & 31;
        warp = warp_index();
        nw = blockDim.x >> 5;
        slot = lane & (CS - 1);
        sub = lane / CS;
        b = -1;
    }
    __device__ __forceinline__ uint32_t* vt() const { return reinterpret_cast<uint32_t*>(smem + L.vt); }
    __device__ __forceinline__ int* e0s() const { return reinterpret_cast<int*>(smem + L.e0); }
    __device__ __forceinline__ uint32_t* sw() const { return reinterpret_cast<uint32_t*>(smem + L.sw); }
    __device__ __forceinline__ uint32_t* et() const { return reinterpret_cast<uint32_t*>(smem + L.et); }
    __device__ __forceinline__ char* arr0() const { return reinterpret_cast<char*>(smem) + L.a0; }
    __device__ __forceinline__ char* arr1() const { return reinterpret_cast<char*>(smem) + L.a1; }

    // Tables of representation rep (whole block).
    __device__ void load_rep(int rep, int* cls) {
        const DevBases& B = a.B;
        const int n = B.n, MP = B.MP;
        b = rep;
        Mb = __ldg(B.rows + b);
        rsteps = (Mb + S - 1) / S;
        int *cnt = cls, *first = cls + 16, *pos = cls + 32;
        if (threadIdx.x < 16) cnt[threadIdx.x] = 0;
        __syncthreads();
        const uint2* vd = B.vdesc + (size_t)b * n;
        for (int p = threadIdx.x; p < n; p += blockDim.x) atomicAdd(&cnt[__ldg(&vd[p].y) >> 16], 1);
        __syncthreads();
        if (threadIdx.x == 0) {
            int f = 0, q = 0;
            for (int d = 0; d <= DC; ++d) {
                first[d] = f;
                pos[d] = q;
                f += cnt[d];
                q += (cnt[d] + S - 1) / S * S;
            }
            pos[DC + 1] = q;
        }
        __syncthreads();
        for (int p = threadIdx.x; p < n; p += blockDim.x) {
            const uint2 d = __ldg(vd + p);
            const int v = d.y & 0xffff, deg = (int)(d.y >> 16);
            const float mu = __fadd_rn(__ldg(a.llr + v), 0.0f);
            const int idx = p - first[deg];
            int np = pos[deg] + idx;
            const int last = (idx == cnt[deg] - 1) ? pos[deg + 1] : np + 1;
            // a class is padded to whole warp steps with copies of its last
            // variable, marked by bit 31.  They store nothing and read the row
            // behind the slots, which nobody writes: the two halves of a warp
            // on one variable would read and write its words unordered (the
            // adjoint's gradient could be added twice).  Predicated stores,
            // since a branch around the copies took the step on [[144,12,12]],
            // batch 4096, from 2.72 to 2.82 ms.
            for (uint32_t dup = 0; np < last; ++np, dup = 0x80000000u) {
                uint32_t* rec = vt() + np * RW;
                for (int i = 0; i < DC; ++i) {
                    uint32_t off = (uint32_t)(L.rsteps * (DC * 128));
                    if (i < deg && !dup) {
                        const int s = __ldg(B.vslot + d.x + i);
                        const int r = (s / (32 * DC)) * 32 + (s & 31), j = (s >> 5) % DC;
                        off = (uint32_t)((r / S) * (DC * 128) + j * 128 + (r % S) * (4 * CS));
                    }
                    rec[2 + i] = off;
                }
                rec[0] = __float_as_uint(mu);
                rec[1] = (uint32_t)v | dup;
            }
        }
        for (int r = threadIdx.x; r < rsteps * S; r += blockDim.x) {
            int e = 0;
            if (r < Mb) {
                const int deg = (int)((__ldg(B.rowinfo + (size_t)b * MP + r) >> 16) & 0xffu);
                e = __ldg(B.rowptr + (size_t)b * MP + r) | (deg << 16);
            }
            e0s()[r] = e;
        }
        __syncthreads();
#pragma unroll
        for (int d = 0; d <= DC; ++d) cend[d] = pos[d + 1] / S;
    }

    // Syndrome and error bits of the block's shots (bit = lane of the step).
    __device__ void load_shots(int blk, int batch) {
        const DevBases& B = a.B;
        shot = blk * CS + slot;
        live = shot < batch;
        const int sh = live ? shot : batch - 1;
        const uint8_t* sy = a.synd + (size_t)sh * B.m;
        for (int rs = warp; rs < rsteps; rs += nw) {
            const int r = rs * S + sub;
            const bool bit = r < Mb && (__ldg(sy + (__ldg(B.rowinfo + (size_t)b * B.MP + r) & 0xffffu)) & 1u);
            const uint32_t w = __ballot_sync(kFull, bit);
            if (lane == 0) sw()[rs] = w;
        }
        if (a.etrue) {
            for (int st = warp; st < cend[DC]; st += nw) {
                const uint32_t v = vt()[(st * S + sub) * RW + 1] & 0xffffu;
                const uint32_t w =
                    __ballot_sync(kFull, (__ldg(a.etrue + (size_t)sh * B.W + (v >> 5)) >> (v & 31)) & 1u);
                if (lane == 0) et()[st] = w;
            }
        }
    }

    // The row's weights and damping of one iteration.
    __device__ __forceinline__ void params(const float* wt, const float* gt, int e0, int deg, float (&w)[DC],
                                           float (&g)[DC]) const {
#pragma unroll
        for (int j = 0; j < DC; ++j) {
            w[j] = (REG || j < deg) ? __ldg(wt + e0 + j) : 0.0f;
            g[j] = (REG || j < deg) ? __ldg(gt + e0 + j) : 0.0f;
        }
    }

    // m <- g m + (1 - g) w S mn(q) of every row, q at arr0; m read at src and
    // written to dst (and dst2 unless null), all in the block's slot layout.
    template <class Load>
    __device__ __forceinline__ void check_pass(const float* wt, const float* gt, Load src, char* dst, char* dst2) {
        char* q0 = arr0() + 4 * lane;
        for (int rs = warp; rs < rsteps; rs += nw) {
            const int e = e0s()[rs * S + sub];
            const int e0 = e & 0xffff, deg = REG ? DC : e >> 16;
            const int o = rs * (DC * 128);
            float q[DC], x[DC], w[DC], g[DC], mo[DC];
            params(wt, gt, e0, deg, w, g);
#pragma unroll
            for (int j = 0; j < DC; ++j) {
                q[j] = (REG || j < deg) ? *reinterpret_cast<const float*>(q0 + o + 128 * j) : MBBP_LMAX;
                mo[j] = src(o + 128 * j + 4 * lane);
            }
            const uint32_t sx = (sw()[rs] >> lane) << 31;
            excluded_min<DC>(q, x);
#pragma unroll
            for (int j = 0; j < DC; ++j) {
                const float smn = __uint_as_float(__float_as_uint(x[j]) ^ sx);
                const float c = __fmul_rn(w[j], smn);
                const float mn = __fadd_rn(__fmul_rn(g[j], mo[j]), __fmul_rn(__fsub_rn(1.0f, g[j]), c));
                *reinterpret_cast<float*>(dst + o + 128 * j + 4 * lane) = mn;
                if (dst2) *reinterpret_cast<float*>(dst2 + o + 128 * j + 4 * lane) = mn;
            }
        }
    }

    // q^(t) of one variable of degree D from its messages m (arr0 at off);
    // own: not a padding copy.
    template <int D>
    __device__ __forceinline__ float var_q(const uint32_t (&off)[D > 0 ? D : 1], const float (&m)[D > 0 ? D : 1],
                                           float mu, bool own) const {
        char* q0 = arr0() + 4 * slot;
        float P = mu;
#pragma unroll
        for (int i = 0; i < D; ++i) {
            float q = P;
#pragma unroll
            for (int k = i + 1; k < D; ++k) q = __fadd_rn(q, m[k]);
            if (own) *reinterpret_cast<float*>(q0 + off[i]) = q;
            P = __fadd_rn(P, m[i]);
        }
        return P;
    }

    // f(D, step, offsets, mu, variable word) for every step of this warp, in
    // degree order.
    template <int D, class F>
    __device__ __forceinline__ void var_class(int& st, F&& f) {
        for (; st < cend[D]; st += nw) {
            const uint32_t* rec = vt() + (st * S + sub) * RW;
            uint32_t off[D > 0 ? D : 1];
#pragma unroll
            for (int i = 0; i < D; ++i) off[i] = rec[2 + i];
            f.template operator()<D>(st, off, __uint_as_float(rec[0]), rec[1]);
        }
        if constexpr (D < DC) var_class<D + 1>(st, f);
    }
    template <class F>
    __device__ __forceinline__ void var_pass(F&& f) {
        int st = warp;
        var_class<0>(st, f);
    }
};

template <int DC, bool REG>
__global__ void __launch_bounds__(kLaneThreads, 1) wms_forward_lanes_kernel(const WmsArgs a, int batch, int blocks) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int cls[48];
    __shared__ int s_item;
    using Blk = Block<DC, REG>;
    Blk k(a, smem);
    const DevBases& B = a.B;
    char* M = k.arr1();
    float* part = reinterpret_cast<float*>(smem + k.L.part);
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_item = (int)atomicAdd(a.counter, 1ull);
        __syncthreads();
        const int item = s_item;
        if (item >= blocks * B.R) break;
        const int b = item / blocks, blk = item - b * blocks;
        if (b != k.b) k.load_rep(b, cls);
        k.load_shots(blk, batch);
        // q^(0) = mu, m^(0) = 0
        k.var_pass([&]<int D>(int, const uint32_t(&off)[D > 0 ? D : 1], float mu, uint32_t v) {
            char* q0 = k.arr0() + 4 * k.slot;
#pragma unroll
            for (int i = 0; i < D; ++i)
                if (!(v >> 31)) *reinterpret_cast<float*>(q0 + off[i]) = mu;
        });
        for (int i = threadIdx.x; i < k.rsteps * (DC * 32); i += blockDim.x) reinterpret_cast<float*>(M)[i] = 0.0f;
        __syncthreads();
        float lacc = 0.0f;
        for (int it = 0; it < a.T; ++it) {
            const float* wt = a.w + ((size_t)b * a.T + it) * a.E;
            const float* gt = a.g + ((size_t)b * a.T + it) * a.E;
            const bool last = it + 1 == a.T;
            char* ck = nullptr;
            if (a.ckpt_buf && (it + 1) % a.ckpt == 0 && !last)
                ck = reinterpret_cast<char*>(a.ckpt_buf +
                                             ((size_t)item * a.nckpt + ((it + 1) / a.ckpt - 1)) * k.L.slot_floats);
            k.check_pass(wt, gt, [&](int o) { return *reinterpret_cast<const float*>(M + o); }, M, ck);
            __syncthreads();
            const bool bce = a.etrue && a.loss && (a.all_iters || last);
            k.var_pass([&]<int D>(int st, const uint32_t(&off)[D > 0 ? D : 1], float mu, uint32_t v) {
                const char* m0 = M + 4 * k.slot;
                float m[D > 0 ? D : 1];
#pragma unroll
                for (int i = 0; i < D; ++i) m[i] = *reinterpret_cast<const float*>(m0 + off[i]);
                const float post = k.template var_q<D>(off, m, mu, !(v >> 31));
                if (bce) {
                    const float x = bce_neg_sigmoid(post, (int)((k.et()[st] >> k.lane) & 1u));
                    if (!(v >> 31)) lacc += x;
                }
                if (last && a.post && k.live && !(v >> 31)) a.post[((size_t)k.shot * B.R + b) * B.n + v] = post;
            });
            __syncthreads();
        }
        if (a.loss && a.etrue) {
            part[threadIdx.x] = lacc;
            __syncthreads();
            if (threadIdx.x < Blk::CS) {
                float acc = 0.0f;
                for (int i = threadIdx.x; i < (int)blockDim.x; i += Blk::CS) acc += part[i];
                if (k.live) a.loss[(size_t)k.shot * B.R + b] = a.scale * acc * (a.all_iters ? 1.0f / a.T : 1.0f);
            }
        }
    }
}

template <int DC, bool REG>
__global__ void __launch_bounds__(kBackwardThreads<DC>, 1) wms_backward_lanes_kernel(const WmsArgs a, int batch, int blocks) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int cls[48];
    __shared__ int s_item;
    using Blk = Block<DC, REG>;
    Blk k(a, smem);
    const DevBases& B = a.B;
    char* GM = k.arr1();
    float* GP = reinterpret_cast<float*>(smem + k.L.gp) + k.lane;
    using Sum = LaneSum<2 * DC, Blk::CS / 2>;
    int sidx[Sum::OUT];
    bool sown[Sum::OUT];
    {
        int id[2 * DC];
        bool ow[2 * DC];
#pragma unroll
        for (int i = 0; i < 2 * DC; ++i) {
            id[i] = i;
            ow[i] = true;
        }
        Sum::index(id, ow, sidx, sown);
    }
    const float lw = a.scale * (a.all_iters ? 1.0f / a.T : 1.0f);
    float* seg = a.seg_buf + (size_t)blockIdx.x * a.ckpt * k.L.slot_floats;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_item = (int)atomicAdd(a.counter, 1ull);
        __syncthreads();
        const int item = s_item;
        if (item >= blocks * B.R) break;
        const int b = item / blocks, blk = item - b * blocks;
        if (b != k.b) k.load_rep(b, cls);
        k.load_shots(blk, batch);
        __syncthreads();
        // dL/dm^(T)_e = lw (e_v - sigmoid(-post_v)) on every edge of v
        const float lwl = k.live ? lw : 0.0f;
        const int sh = k.live ? k.shot : batch - 1;
        k.var_pass([&]<int D>(int st, const uint32_t(&off)[D > 0 ? D : 1], float, uint32_t v) {
            char* g0 = GM + 4 * k.slot;
            const float pv = __ldg(a.post + ((size_t)sh * B.R + b) * B.n + (v & 0xffffu));
            const float sig = 1.0f / (1.0f + expf(pv));
            const float gp = lwl * ((float)((k.et()[st] >> k.lane) & 1u) - sig);
#pragma unroll
            for (int i = 0; i < D; ++i)
                if (!(v >> 31)) *reinterpret_cast<float*>(g0 + off[i]) = gp;
        });
        const int nseg = (a.T + a.ckpt - 1) / a.ckpt;
        for (int sg = nseg - 1; sg >= 0; --sg) {
            const int t0 = sg * a.ckpt, t1 = min(a.T, t0 + a.ckpt);
            // state i = m^(t0 + i): the checkpoint (or zero), then recomputed
            auto state = [&](int i) -> char* {
                if (i == 0 && t0 > 0)
                    return reinterpret_cast<char*>(a.ckpt_buf + ((size_t)item * a.nckpt + (sg - 1)) * k.L.slot_floats);
                return reinterpret_cast<char*>(seg + (size_t)i * k.L.slot_floats);
            };
            if (t0 == 0) {
                float* z = seg;
                for (int i = threadIdx.x; i < k.rsteps * (DC * 32); i += blockDim.x) z[i] = 0.0f;
            }
            __syncthreads();
            for (int t = t0 + 1; t < t1; ++t) {
                const char* mp = state(t - 1 - t0);
                k.var_pass([&]<int D>(int, const uint32_t(&off)[D > 0 ? D : 1], float mu, uint32_t v) {
                    const char* m0 = mp + 4 * k.slot;
                    float m[D > 0 ? D : 1];
#pragma unroll
                    for (int i = 0; i < D; ++i) m[i] = *reinterpret_cast<const float*>(m0 + off[i]);
                    k.template var_q<D>(off, m, mu, !(v >> 31));
                });
                __syncthreads();
                const float* wt = a.w + ((size_t)b * a.T + (t - 1)) * a.E;
                const float* gt = a.g + ((size_t)b * a.T + (t - 1)) * a.E;
                k.check_pass(wt, gt, [&](int o) { return *reinterpret_cast<const float*>(mp + o); }, state(t - t0),
                             nullptr);
                __syncthreads();
            }
            // q^(t-1) (and the gradient of post^(t-1)) from m^(t-1); with VG
            // first the adjoint of the variable pass of iteration t + 1's q,
            // which the same thread owns
            auto var_both = [&](const char* mp, bool adjoint, bool forward) {
                k.var_pass([&]<int D>(int st, const uint32_t(&off)[D > 0 ? D : 1], float mu, uint32_t v) {
                    constexpr int DD = D > 0 ? D : 1;
                    const char* q0 = k.arr0() + 4 * k.slot;
                    char* g0 = GM + 4 * k.slot;
                    float m[DD];
                    if (forward) {
                        const char* m0 = mp + 4 * k.slot;
#pragma unroll
                        for (int i = 0; i < D; ++i) m[i] = *reinterpret_cast<const float*>(m0 + off[i]);
                    }
                    if (adjoint) {
                        float gq[DD], G = 0.0f;
#pragma unroll
                        for (int i = 0; i < D; ++i) {
                            gq[i] = *reinterpret_cast<const float*>(q0 + off[i]);
                            G += gq[i];
                        }
                        const float gp = a.all_iters ? GP[32 * st] : 0.0f;
#pragma unroll
                        for (int i = 0; i < D; ++i) {
                            float* gm = reinterpret_cast<float*>(g0 + off[i]);
                            const float x = *gm + (G - gq[i] + gp);
                            if (!(v >> 31)) *gm = x;
                        }
                    }
                    if (forward) {
                        const float post = k.template var_q<D>(off, m, mu, !(v >> 31));
                        if (a.all_iters)
                            GP[32 * st] =
                                lwl * ((float)((k.et()[st] >> k.lane) & 1u) - 1.0f / (1.0f + expf(post)));
                    }
                });
            };
            var_both(state(t1 - 1 - t0), false, true);
            __syncthreads();
            for (int t = t1; t > t0; --t) {
                const char* mp = state(t - 1 - t0) + 4 * k.lane;
                const float* wt = a.w + ((size_t)b * a.T + (t - 1)) * a.E;
                const float* gt = a.g + ((size_t)b * a.T + (t - 1)) * a.E;
                float* gwt = a.gw + ((size_t)b * a.T + (t - 1)) * a.E;
                float* ggt = a.gg + ((size_t)b * a.T + (t - 1)) * a.E;
                for (int rs = k.warp; rs < k.rsteps; rs += k.nw) {
                    const int e = k.e0s()[rs * Blk::S + k.sub];
                    const int e0 = e & 0xffff, deg = e >> 16;
                    const int o = rs * (DC * 128);
                    char* qr = k.arr0() + 4 * k.lane + o;
                    char* gr = GM + 4 * k.lane + o;
                    float w[DC], g[DC], q[DC], x[DC];
                    k.params(wt, gt, e0, deg, w, g);
#pragma unroll
                    for (int j = 0; j < DC; ++j)
                        q[j] = (REG || j < deg) ? *reinterpret_cast<const float*>(qr + 128 * j) : MBBP_LMAX;
                    const uint32_t sx = (k.sw()[rs] >> k.lane) << 31;
                    excluded_min<DC>(q, x);
                    // the edge a1 of the smallest |q| below LMAX (lowest index on
                    // ties) and a2 of the smallest of the others: dL/dq goes to
                    // these two only
                    float min1 = MBBP_LMAX, min2 = MBBP_LMAX;
                    int a1 = -1, a2 = -1;
#pragma unroll
                    for (int j = 0; j < DC; ++j) {
                        const float y = fabsf(q[j]);
                        const bool p1 = y < min1, p2 = y < min2;
                        a2 = p1 ? a1 : (p2 ? j : a2);
                        min2 = p1 ? min1 : (p2 ? y : min2);
                        a1 = p1 ? j : a1;
                        min1 = p1 ? y : min1;
                    }
                    float v[2 * DC];
                    float G1 = 0.0f, G2 = 0.0f;
#pragma unroll
                    for (int j = 0; j < DC; ++j) {
                        const float smn = __uint_as_float(__float_as_uint(x[j]) ^ sx);
                        const float gmj = *reinterpret_cast<const float*>(gr + 128 * j);
                        const float mo = *reinterpret_cast<const float*>(mp + o + 128 * j);
                        const float ag = gmj * (1.0f - g[j]);
                        v[2 * j] = ag * smn;
                        v[2 * j + 1] = gmj * (mo - w[j] * smn);
                        *reinterpret_cast<float*>(gr + 128 * j) = gmj * g[j];
                        const float gmn =
                            __uint_as_float(__float_as_uint(ag * w[j]) ^ (__float_as_uint(smn) & 0x80000000u));
                        if (REG || j < deg) {
                            if (j == a1) G2 = gmn;
                            else G1 += gmn;
                        }
                    }
#pragma unroll
                    for (int j = 0; j < DC; ++j) {
                        const float gj = (j == a1) ? G1 : ((j == a2) ? G2 : 0.0f);
                        const float gs = __uint_as_float(__float_as_uint(gj) ^ (__float_as_uint(q[j]) & 0x80000000u));
                        if (REG || j < deg) *reinterpret_cast<float*>(qr + 128 * j) = gs;
                    }
                    float sum[Sum::OUT];
                    Sum::run(v, sum);
#pragma unroll
                    for (int i = 0; i < Sum::OUT; ++i)
                        if (sown[i] && (sidx[i] >> 1) < deg)
                            atomicAdd(((sidx[i] & 1) ? ggt : gwt) + e0 + (sidx[i] >> 1), sum[i]);
                }
                __syncthreads();
                const bool fwd = t - 1 > t0;
                if (t >= 2) var_both(fwd ? state(t - 2 - t0) : nullptr, true, fwd);
                __syncthreads();
            }
        }
    }
}

template <int DC>
cudaError_t launch_lanes(const WmsArgs& a, int batch, bool backward, cudaStream_t s, int sm_count) {
    const LanesLayout L = lanes_layout(DC, a.B.MP, a.B.n);
    const bool reg = a.B.regular != 0;
    const void* kern = backward ? (reg ? reinterpret_cast<const void*>(wms_backward_lanes_kernel<DC, true>)
                                       : reinterpret_cast<const void*>(wms_backward_lanes_kernel<DC, false>))
                                : (reg ? reinterpret_cast<const void*>(wms_forward_lanes_kernel<DC, true>)
                                       : reinterpret_cast<const void*>(wms_forward_lanes_kernel<DC, false>));
    // all warps that registers allow: two blocks of half of them when their
    // shared memory fits twice and there is work for both, else one
    const int most = backward ? kBackwardThreads<DC> : kLaneThreads;
    int threads = most / 2, per_sm = 0;
    cudaError_t e = prepare_kernel(kern, threads, L.total, &per_sm);
    if (e == cudaSuccess && (per_sm < 2 || wms_lanes_grid(a.B, batch, sm_count) <= (size_t)sm_count)) {
        threads = most;
        e = prepare_kernel(kern, threads, L.total, &per_sm);
    }
    if (e != cudaSuccess) return e;
    WmsArgs aa = a;
    int blocks = (int)(((long long)batch + kLaneShots - 1) / kLaneShots);
    const size_t grid = std::min((size_t)sm_count * per_sm, wms_lanes_grid(a.B, batch, sm_count));
    void* args[] = {&aa, &batch, &blocks};
    return cudaLaunchKernel(kern, dim3((unsigned)grid), dim3(threads), args, L.total, s);
}

}  // namespace

bool wms_lanes_fit(const DevBases& B, int batch) {
    // From 256 (shot, representation) pairs on: 64 shots at R = 2 of
    // [[144,12,12]] took 0.284 ms a step here and 0.276 ms warp per shot, 64 at
    // R = 8 0.284 and 0.322 ms; 128 at R = 2 of codes of length 96 with rows of 8
    // and 10 (T = 20) 0.213 and 0.260, 0.305 and 0.362.  The block's two message
    // arrays must fit shared memory (the length-882 code's do not).
    const long long blocks = ((long long)batch + kLaneShots - 1) / kLaneShots;
    return (long long)batch * B.R >= 256 && blocks * B.R <= INT_MAX / 2 &&
           lanes_layout(B.DC, B.MP, B.n).total <= 226 * 1024 + 256;  // and 256 static
}

size_t wms_lanes_grid(const DevBases& B, int batch, int sm_count) {
    const long long blocks = ((long long)batch + kLaneShots - 1) / kLaneShots;
    return (size_t)std::min(blocks * B.R, 2ll * sm_count);
}

size_t wms_lanes_ckpt_floats(const DevBases& B, int batch) {
    const long long blocks = ((long long)batch + kLaneShots - 1) / kLaneShots;
    return (size_t)(blocks * B.R) * lanes_layout(B.DC, B.MP, B.n).slot_floats;
}

size_t wms_lanes_state_floats(const DevBases& B) { return (size_t)lanes_layout(B.DC, B.MP, B.n).slot_floats; }

cudaError_t launch_wms_lanes(const WmsArgs& a, int batch, bool backward, cudaStream_t s, int sm_count) {
    if (a.B.DC == 6) return launch_lanes<6>(a, batch, backward, s, sm_count);
    if (a.B.DC == 8) return launch_lanes<8>(a, batch, backward, s, sm_count);
    if (a.B.DC == 12) return launch_lanes<12>(a, batch, backward, s, sm_count);
    return cudaErrorInvalidValue;
}

}  // namespace mbbp
