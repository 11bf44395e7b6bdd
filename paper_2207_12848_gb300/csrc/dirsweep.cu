// The batched sweep with one block per direction, and the operator it streams.
//
// The dependency graphs of different directions share nothing, so a direction that one block sweeps
// alone needs no readiness test and no grid barrier: its wavefront levels are separated by
// __syncthreads, and the intensities its tasks have just written are read back from a ring in shared
// memory instead of through L2.
//
// Order. The tasks of a level, sorted by the entries they have, are laid out in slices of 32, one lane per
// task; a round is up to W slices of one level, one for each worker warp. A task's place is
// 32 slice + lane along its direction; the ring keeps the last R places.
//
// A task with n entries (its inflow sides) sums them as (n + 2) / 2 elements, counted from its last entry:
// element 0 is the unpaired last entry (n odd) or empty, every other element a pair w1 |x1| + w0 |x0|; the
// elements are added in a binary tree aligned at element 0. This is the order of summation of the warp
// packets that all directions share. Two elements (four entries) make a quad.
//
// Operator. Per direction two contiguous byte streams, read once per sweep in order:
//   E, per slice the quads of its longest task, each {four weights, four 16-bit sources} per lane (768
//     bytes a quad in FP32, 1280 in FP64);
//   C, per round: header, per slice {quads, E offset in the round}, per task {cell, P_c}, and the list of its
//     far sources {kind << 30 | index}: values older than the ring (this sweep's array), the
//     periodic partner's (the previous iteration's array), the boundary inflow. A round ends early where its
//     far sources would exceed their staging slots.
// A 16-bit source indexes the block's value array: the ring, then the staging slots of the far sources, then
// a slot that holds 0.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstddef>
#include <cstring>

#include "common.cuh"

namespace sw {
namespace {

constexpr uint32_t PAD_CELL = 0xffffffffu;
constexpr int MAX_SLOTS = 8;  // rounds of a stream in shared memory at most
constexpr int MAX_Q = 16;   // quads of the longest task (63 entries)
enum { FAR_THIS = 0, FAR_PREV = 1, FAR_BC = 2 };

// quads of a task with n entries
__host__ __device__ __forceinline__ int quads_of(int n) { return ((n + 2) / 2 + 1) / 2; }
__host__ __device__ __forceinline__ uint32_t up16(uint32_t x) { return (x + 15u) & ~15u; }

template <typename real>
constexpr uint32_t quad_bytes() { return 32u * (4u * sizeof(real) + 8u); }

// header of a round in C
struct RoundHdr {
    uint32_t ns, nfar, pad, ring0;  // slices, far sources, ring slot of its first place
};
// a task in C
template <typename real>
struct TaskRec {
    uint32_t cell;
    float P;
};
template <>
struct alignas(16) TaskRec<double> {
    double P;
    uint32_t cell, pad;
};
__host__ __device__ __forceinline__ uint32_t c_tasks(uint32_t ns) { return 16u + up16(4u * ns); }
template <typename real>
__host__ __device__ __forceinline__ uint32_t c_far(uint32_t ns) { return c_tasks(ns) + 32u * ns * (uint32_t)sizeof(TaskRec<real>); }
template <typename real>
__host__ __device__ __forceinline__ uint32_t c_bytes(uint32_t ns, uint32_t nfar) { return c_far<real>(ns) + up16(4u * nfar); }

// ---------------------------------------------------------------------------------------------
// Building the operator
// ---------------------------------------------------------------------------------------------
struct DirBuild {
    const int32_t *dcnt, *dbase, *depth;  // [nd][cap] cells and list start of each level; [nd]
    int cap, lcap, nd, W, R, A, Fs;
    int transposed;
    int64_t N;
    int SC, RC;                // slices and rounds a direction's tables hold
    const uint32_t* list;      // [nd][N] cells in level order
    int32_t *sbase, *rbase;    // [nd][lcap] first slice and first round of each level in sweep order
    uint32_t* place;           // [nd][N] place of each cell
    uint32_t* ord;             // [nd][SC * 32] cell of each place
    uint64_t* msk;             // [nd][SC * 32] entries of each place (bit k: row position k)
    float* P;                  // [nd][SC * 32] P_c of each place (FP32)
    uint32_t* nq;              // [nd][SC] quads of each slice
    uint32_t* eoff;            // [nd][SC + 1] E offset / 256
    uint32_t* sfar;            // [nd][SC] far sources of each slice
    uint32_t* lend;            // [nd][SC] end of its level (place)
    int32_t* nround;           // [nd][lcap] rounds of each level
    uint2* rinfo;              // [nd][RC] {first slice, slices} of each round
    uint32_t* nfar;            // [nd][RC]
    uint32_t* coff;            // [nd][RC + 1] C offset / 16
    uint2* rtab;               // [nd][RC + 1] {C offset / 16, E offset / 256} of each round
    int2* tot;                 // [nd] slices, rounds
    DirMeta* meta;             // [nd]
    int32_t* stat;             // [0] does not apply, [1] most far sources of a slice, [2] bound on a round's E bytes, [3] a level
                               // is too wide for the ring
    uint32_t e_slot, quad_b;   // E bytes of a round's slot, bytes of a quad
    unsigned char *E, *C;
    const uint32_t* rowptr;
    const SideRec* side;
    const d4* side64;
    const float4 *om32, *om32lo;
    const double* om64;
    const int4* info;
    const uint64_t* dc_inm;
    const float* dc_share32;
    const double* dc_share64;
};

// The sides of a task's row that are its entries (bit k: row position k; rows of at most 64 sides): the
// inflow sides, or the effective inflow sides of scheme (b), or, transposed, the outflow sides that lead
// to a cell. Signs as in the classification. P: the task's P_c.
__device__ uint64_t entry_mask(const DirBuild& a, uint32_t c, int d, float* P) {
    const int4 info = a.info[(int64_t)c * a.nd + d];
    *P = __int_as_float(info.y & 0x7fffffff);
    if (a.dc_inm) return a.dc_inm[(int64_t)c * a.nd + d];
    if (!a.transposed && info.y >= 0) return (uint32_t)info.z;  // a row of up to 32 sides
    const uint32_t r0 = a.rowptr[c], r1 = a.rowptr[c + 1];
    const float4 om = a.om32[d];
    const double* o64 = a.om64 + 3 * d;
    uint64_t m = a.transposed ? 0ull : (uint32_t)info.z;
    for (uint32_t s = a.transposed ? r0 : r0 + 32; s < r1; ++s) {
        const int4 r = a.side[s].hi;
        if (a.transposed && r.x < 0) continue;
        const float ax = __int_as_float(r.y), ay = __int_as_float(r.z), az = __int_as_float(r.w);
        const int sg = classify_side(dot32(ax, ay, az, om), ax, ay, az, a.side64, s, o64);
        if (a.transposed ? sg > 0 : sg < 0) m |= 1ull << (s - r0);
    }
    return m;
}

// Raises *p to v, by an atomic only where it would change it: of the hundreds of thousands of blocks and slices few do, and
// atomics on one address come one after the other.
__device__ __forceinline__ void raise_stat(int32_t* p, int v) {
    if (v > *(volatile int32_t*)p) atomicMax(p, v);
}
// The plan is over: its slots are too small for the E of a round, and the host plans again with the bound (a second count of
// 2^18 cells, 128 directions costs 2.1 ms of a 15 ms solve), or a level is too wide for the ring (found after the count
// it cost 90 us of a 0.7 ms solve: 8,000 cells, scheme (b), FP64).
__device__ __forceinline__ bool plan_over(const DirBuild& a) { return a.stat[3] || (uint32_t)a.stat[2] > a.e_slot; }

__device__ __forceinline__ int level_slices(int n) { return (n + 31) >> 5; }
// A level of n slices has ceil(n / W) rounds of equal size, so its last round is not a small remainder.
__device__ __forceinline__ int round_slices(int ns, int W) {
    const int nr = (ns + W - 1) / W;
    return nr ? (ns + nr - 1) / nr : 0;
}

// Exclusive sums of v over the levels of a direction in sweep order (transposed: last level first), by one
// block of 1024 threads; returns the total.
template <typename F>
__device__ int level_scan(int nl, int reverse, F v, int32_t* out) {
    __shared__ int s_w[32], s_carry;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_carry = 0;
    __syncthreads();
    for (int b = 0; b < nl; b += 1024) {
        const int i = b + (int)threadIdx.x, L = reverse ? nl - 1 - i : i;
        const int x = i < nl ? v(L) : 0;
        int inc = x;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane == 31) s_w[warp] = inc;
        __syncthreads();
        int pre = s_carry;
        for (int w = 0; w < warp; ++w) pre += s_w[w];
        if (i < nl) out[L] = pre + inc - x;
        __syncthreads();
        if (threadIdx.x == 1023) s_carry = pre + inc;
        __syncthreads();
    }
    return s_carry;
}

// A source that is not in the ring at its level's end was summed A rounds before any round of the level or earlier: the
// fetch of the round, A iterations ahead of its sums, finds it in memory.
__device__ __forceinline__ bool ring_too_short(const DirBuild& a, int ns) { return (ns + a.A * a.W) * 32 > a.R; }

// First slice of every level, and whether the ring is long enough for it.
__global__ void __launch_bounds__(1024) k_dir_slices(DirBuild a) {
    const int d = blockIdx.x;
    for (int L = threadIdx.x; L < a.depth[d]; L += 1024)
        if (ring_too_short(a, level_slices(a.dcnt[(size_t)d * a.cap + L]))) atomicOr(&a.stat[3], 1);
    const int32_t* cnt = a.dcnt + (size_t)d * a.cap;
    const int n = level_scan(a.depth[d], a.transposed, [&](int L) { return level_slices(cnt[L]); }, a.sbase + (size_t)d * a.lcap);
    if (threadIdx.x == 0) {
        a.tot[d].x = n;
        if (n > a.SC) atomicOr(&a.stat[0], 1);
    }
}

// First round of every level.
__global__ void __launch_bounds__(1024) k_dir_rounds(DirBuild a) {
    if (plan_over(a)) return;
    const int d = blockIdx.x;
    const int32_t* nr = a.nround + (size_t)d * a.lcap;
    const int n = level_scan(a.depth[d], a.transposed, [&](int L) { return nr[L]; }, a.rbase + (size_t)d * a.lcap);
    if (threadIdx.x == 0) {
        a.tot[d].y = n;
        if (n > a.RC) atomicOr(&a.stat[0], 1);
    }
}

// Rounds of a level, one thread: up to `per` slices each, ended where the far sources would exceed Fs.
template <typename F>
__device__ int cut_rounds(const uint32_t* sfar, int ns, int per, uint32_t Fs, F put) {
    int n = 0, first = 0;
    uint32_t far = 0;
    for (int i = 0; i < ns; ++i) {
        if (i > first && (i - first == per || far + sfar[i] > Fs)) {
            put(n++, first, i - first, far);
            first = i;
            far = 0;
        }
        far += sfar[i];
    }
    if (ns > first) put(n++, first, ns - first, far);
    return n;
}
template <bool WRITE>
__global__ void __launch_bounds__(128) k_dir_cut(DirBuild a) {
    const int L = blockIdx.x * 128 + threadIdx.x, d = blockIdx.y;
    if (L >= a.depth[d] || plan_over(a)) return;
    const int ns = level_slices(a.dcnt[(size_t)d * a.cap + L]), s0 = a.sbase[(size_t)d * a.lcap + L];
    if (s0 + ns > a.SC) return;
    const uint32_t* sf = a.sfar + (size_t)d * a.SC + s0;
    const int per = round_slices(ns, a.W);
    if (!WRITE) {
        a.nround[(size_t)d * a.lcap + L] = cut_rounds(sf, ns, per, (uint32_t)a.Fs, [](int, int, int, uint32_t) {});
    } else {
        const int r0 = a.rbase[(size_t)d * a.lcap + L];
        if (r0 + a.nround[(size_t)d * a.lcap + L] > a.RC) return;
        cut_rounds(sf, ns, per, (uint32_t)a.Fs, [&](int i, int first, int n, uint32_t far) {
            a.rinfo[(size_t)d * a.RC + r0 + i] = make_uint2((uint32_t)(s0 + first), (uint32_t)n);
            a.nfar[(size_t)d * a.RC + r0 + i] = far;
        });
    }
}

// One block per (level, direction): the tasks sorted by their quads (counting sort, longest first) and put
// into slices. A round's slices follow one another, so none has more quads than a level's first round.
constexpr int PLACE_THREADS = 128;
__global__ void __launch_bounds__(PLACE_THREADS) k_dir_place(DirBuild a) {
    __shared__ int s_bin[MAX_Q + 1], s_end[MAX_Q + 1], s_first;
    const int L = blockIdx.x, d = blockIdx.y;
    if (L >= a.depth[d] || a.stat[3]) return;
    const int n = a.dcnt[(size_t)d * a.cap + L];
    const uint32_t* src = a.list + (size_t)d * a.N + a.dbase[(size_t)d * a.cap + L];
    const int s0 = a.sbase[(size_t)d * a.lcap + L], ns = level_slices(n);
    if (s0 + ns > a.SC) return;
    const size_t o = ((size_t)d * a.SC + s0) * 32;
    if (threadIdx.x <= MAX_Q) s_bin[threadIdx.x] = 0;
    if (threadIdx.x == 0) s_first = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += PLACE_THREADS) {
        float P;
        const int k = __popcll(entry_mask(a, src[i], d, &P));
        if (k > 63) atomicOr(&a.stat[0], 1);
        atomicAdd(&s_bin[quads_of(min(k, 63))], 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int at = 0;
        for (int k = MAX_Q; k >= 1; --k) {
            const int c = s_bin[k];
            s_bin[k] = at;
            at += c;
            s_end[k] = at;
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += PLACE_THREADS) {
        const uint32_t c = src[i];
        float P;
        const uint64_t m = entry_mask(a, c, d, &P);
        const int p = atomicAdd(&s_bin[quads_of(min(63, __popcll(m)))], 1);
        a.ord[o + p] = c;
        a.msk[o + p] = m;
        a.P[o + p] = P;
        a.place[(size_t)d * a.N + c] = (uint32_t)(s0 * 32 + p);
    }
    for (int i = n + threadIdx.x; i < ns * 32; i += PLACE_THREADS) {
        a.ord[o + i] = PAD_CELL;
        a.msk[o + i] = 0ull;
        a.P[o + i] = 1.f;
    }
    for (int i = threadIdx.x; i < ns; i += PLACE_THREADS) {  // a slice's longest task is its first
        int q = MAX_Q;
        while (q > 1 && s_end[q] <= i * 32) --q;
        a.nq[(size_t)d * a.SC + s0 + i] = (uint32_t)q;
        if (i < round_slices(ns, a.W)) atomicAdd(&s_first, q);
    }
    __syncthreads();
    if (threadIdx.x == 0) raise_stat(&a.stat[2], s_first * (int)a.quad_b);
}

// ring slot of an entry's source, or ~0 where the value has to be staged. level_end: the place after the
// level's last; by then the ring has lost what is R places older.
__device__ __forceinline__ uint32_t near_slot(const DirBuild& a, int d, int32_t nb, uint32_t level_end) {
    if (nb < 0 || (nb & NBR_PERIODIC)) return ~0u;
    const uint32_t p = a.place[(size_t)d * a.N + (uint32_t)nb];
    return level_end - p <= (uint32_t)a.R ? p % (uint32_t)a.R : ~0u;
}

// Far entries of each slice (one block per level of a direction, a warp per slice).
__global__ void __launch_bounds__(128) k_dir_count(DirBuild a) {
    const int L = blockIdx.x, d = blockIdx.y;
    if (L >= a.depth[d] || plan_over(a)) return;
    const int ns = level_slices(a.dcnt[(size_t)d * a.cap + L]), s0 = a.sbase[(size_t)d * a.lcap + L];
    if (s0 + ns > a.SC) return;
    const uint32_t end = (uint32_t)(s0 + ns) * 32u;
    if (threadIdx.x == 0 && ring_too_short(a, ns)) atomicOr(&a.stat[0], 1);  // a plan made again may have a shorter ring
    const int lane = threadIdx.x & 31;
    for (int k = threadIdx.x >> 5; k < ns; k += 4) {
        const size_t t = ((size_t)d * a.SC + s0 + k) * 32 + lane;
        uint64_t m = a.msk[t];
        int far = 0;
        if (m) {
            const uint32_t r0 = a.rowptr[a.ord[t]];
            for (; m; m &= m - 1)
                far += near_slot(a, d, a.side[r0 + (uint32_t)(__ffsll((long long)m) - 1)].hi.x, end) == ~0u;
        }
        far = __reduce_add_sync(0xffffffffu, far);
        if (lane == 0) {
            a.sfar[(size_t)d * a.SC + s0 + k] = (uint32_t)far;
            a.lend[(size_t)d * a.SC + s0 + k] = end;
            raise_stat(&a.stat[1], far);
        }
    }
}

// exclusive scan of n values v(i) by one block of 1024 threads into out[0..n]; returns the total
template <typename F>
__device__ uint32_t block_scan(int n, F v, uint32_t* out) {
    __shared__ uint32_t s_w[32], s_c;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (threadIdx.x == 0) s_c = 0;
    __syncthreads();
    for (int b = 0; b < n; b += 1024) {
        const int i = b + (int)threadIdx.x;
        const uint32_t x = i < n ? v(i) : 0u;
        uint32_t inc = x;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane == 31) s_w[warp] = inc;
        __syncthreads();
        uint32_t pre = s_c;
        for (int w = 0; w < warp; ++w) pre += s_w[w];
        if (i < n) out[i] = pre + inc - x;
        __syncthreads();
        if (threadIdx.x == 1023) s_c = pre + inc;
        __syncthreads();
    }
    if (threadIdx.x == 0) out[n] = s_c;
    return s_c;
}

// Offsets of every slice in E and of every round in C, per direction.
template <typename real>
__global__ void __launch_bounds__(1024) k_dir_offsets(DirBuild a) {
    const int d = blockIdx.x;
    const int2 t = a.tot[d];
    if (t.x > a.SC || t.y > a.RC || plan_over(a)) return;
    const uint32_t* nq = a.nq + (size_t)d * a.SC;
    uint32_t* eoff = a.eoff + (size_t)d * (a.SC + 1);
    uint32_t* coff = a.coff + (size_t)d * (a.RC + 1);
    const uint2* ri = a.rinfo + (size_t)d * a.RC;
    const uint32_t* nf = a.nfar + (size_t)d * a.RC;
    const uint32_t e = block_scan(t.x, [&](int i) { return nq[i] * (quad_bytes<real>() / 256u); }, eoff);
    const uint32_t c = block_scan(t.y, [&](int i) { return c_bytes<real>(ri[i].y, nf[i]) / 16u; }, coff);
    __syncthreads();
    for (int i = threadIdx.x; i <= t.y; i += 1024)
        a.rtab[(size_t)d * (a.RC + 1) + i] = make_uint2(coff[i], i < t.y ? eoff[ri[i].x] : e);
    if (threadIdx.x == 0) {
        if (e >= (1u << 24) || c >= (1u << 28)) atomicOr(&a.stat[0], 1);  // offsets are kept in 32 bits
        a.meta[d].e_bytes = (int64_t)e * 256;
        a.meta[d].c_bytes = (int64_t)c * 16;
        a.meta[d].rounds = t.y;
    }
}

// Start of every direction's streams (128-byte aligned), and their sizes; one block.
__global__ void __launch_bounds__(1024) k_dir_bases(DirMeta* meta, int nd, int64_t* total, uint32_t* scan) {
    uint32_t* se = scan;
    uint32_t* sc = scan + nd + 1;
    const uint32_t e = block_scan(nd, [&](int i) { return (uint32_t)((meta[i].e_bytes + 127) / 128); }, se);
    const uint32_t c = block_scan(nd, [&](int i) { return (uint32_t)((meta[i].c_bytes + 127) / 128); }, sc);
    __syncthreads();
    for (int i = threadIdx.x; i < nd; i += 1024) {
        meta[i].e_base = (int64_t)se[i] * 128;
        meta[i].c_base = (int64_t)sc[i] * 128;
    }
    if (threadIdx.x == 0) {
        total[0] = (int64_t)e * 128;
        total[1] = (int64_t)c * 128;
    }
}

// weight of entry s of a task (the line form's and the packets' FP32 weight; FP64: A |n.Omega|)
template <typename real>
__device__ __forceinline__ real entry_weight(const DirBuild& a, int d, uint32_t s, const int4& r, const float4& om,
                                             const float4& oml) {
    if (a.dc_inm && r.x >= 0) {  // scheme (b): the upwind cell's share
        const int64_t i = (int64_t)(r.x & NBR_MASK) * a.nd + d;
        return sizeof(real) == 8 ? (real)a.dc_share64[i] : (real)a.dc_share32[i];
    }
    if (sizeof(real) == 8) {
        const d4 n = a.side64[s];
        return (real)__dmul_rn(n.w, fabs(exact_t(n, a.om64 + 3 * d)));
    }
    return (real)side_weight(r, a.side[s].lo, om, oml);
}

// Writes E and C: one block per round of a direction, a warp per slice.
template <typename real>
__global__ void __launch_bounds__(128) k_dir_write(DirBuild a) {
    __shared__ int s_far;
    const int r = blockIdx.x, d = blockIdx.y;
    if (r >= a.tot[d].y) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) s_far = 0;
    __syncthreads();
    const uint2 ri = a.rinfo[(size_t)d * a.RC + r];
    const uint32_t ns = ri.y, end = a.lend[(size_t)d * a.SC + ri.x], nfar = a.nfar[(size_t)d * a.RC + r];
    const uint32_t* eoff = a.eoff + (size_t)d * (a.SC + 1) + ri.x;
    const uint32_t* coff = a.coff + (size_t)d * (a.RC + 1) + r;
    const DirMeta m = a.meta[d];
    unsigned char* C = a.C + m.c_base + (size_t)coff[0] * 16;
    uint32_t* tab = reinterpret_cast<uint32_t*>(C + 16);
    TaskRec<real>* tasks = reinterpret_cast<TaskRec<real>*>(C + c_tasks(ns));
    uint32_t* fars = reinterpret_cast<uint32_t*>(C + c_far<real>(ns));
    const uint32_t far0 = (uint32_t)a.R + (uint32_t)(r % (a.A + 1)) * (uint32_t)a.Fs;
    const uint32_t zero = (uint32_t)a.R + (uint32_t)(a.A + 1) * (uint32_t)a.Fs;
    if (threadIdx.x == 0)
        *reinterpret_cast<RoundHdr*>(C) = RoundHdr{ns, nfar, 0u, ri.x * 32u % (uint32_t)a.R};
    const float4 om = a.om32[d], oml = a.om32lo[d];
    for (uint32_t k = warp; k < ns; k += 4) {
        const int nq = (int)a.nq[(size_t)d * a.SC + ri.x + k];
        if (lane == 0) tab[k] = (uint32_t)nq | (eoff[k] - eoff[0]) << 8;
        const size_t t = ((size_t)d * a.SC + ri.x + k) * 32 + lane;
        const uint32_t c = a.ord[t], r0 = c != PAD_CELL ? a.rowptr[c] : 0u;
        uint64_t left = a.msk[t];
        TaskRec<real> rec;
        rec.cell = c;
        rec.P = (real)a.P[t];
        if (sizeof(real) == 8 && c != PAD_CELL) {
            // P_c in FP64, in row order. The FP64 pipe bounds this build, so the sides that the classification calls
            // inflow are left out.
            double P = 0.0;
            const auto add = [&](uint32_t s) {
                const d4 nn = a.side64[s];
                const double tt = exact_t(nn, a.om64 + 3 * d);
                if (tt > 0.0) P = __dadd_rn(P, __dmul_rn(nn.w, tt));
            };
            const uint32_t r1 = a.rowptr[c + 1], n = r1 - r0;
            uint32_t m = ~(uint32_t)a.info[(int64_t)c * a.nd + d].z & (n >= 32u ? ~0u : (1u << n) - 1u);
            for (; m; m &= m - 1) add(r0 + (uint32_t)(__ffs((int)m) - 1));
            for (uint32_t s = r0 + 32; s < r1; ++s) add(s);
            rec.P = (real)P;
        }
        tasks[k * 32u + lane] = rec;
        unsigned char* e = a.E + m.e_base + (size_t)eoff[k] * 256;
        const int odd = __popcll(left) & 1;
        for (int q = 0; q < nq; ++q, e += quad_bytes<real>()) {
            real w[4];
            uint32_t ix[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {  // elements 2 q and 2 q + 1 as {slot 1, slot 0} each, last entry first
                w[j] = 0;
                ix[j] = zero;
                // element 0 holds the unpaired entry in slot 0, or nothing
                if (!left || (q == 0 && (j == 0 || (j == 1 && !odd)))) continue;
                const int b = 63 - __clzll((long long)left);
                left &= ~(1ull << b);
                const uint32_t s = r0 + (uint32_t)b;
                const int4 sd = a.side[s].hi;
                w[j] = entry_weight<real>(a, d, s, sd, om, oml);
                const uint32_t slot = near_slot(a, d, sd.x, end);
                if (slot != ~0u) {
                    ix[j] = slot;
                } else {
                    const uint32_t f = (uint32_t)atomicAdd(&s_far, 1);
                    ix[j] = far0 + f;
                    fars[f] = sd.x < 0 ? ((uint32_t)FAR_BC << 30 | (uint32_t)(-1 - sd.x))
                                       : ((sd.x & NBR_PERIODIC) ? (uint32_t)FAR_PREV << 30 : 0u) | (uint32_t)(sd.x & NBR_MASK);
                }
                if (w[j] == (real)0) ix[j] = zero;  // an entry of weight 0 takes no value
            }
            real* ew = reinterpret_cast<real*>(e) + 4 * lane;
#pragma unroll
            for (int j = 0; j < 4; ++j) ew[j] = w[j];
            reinterpret_cast<uint2*>(e + 128 * sizeof(real))[lane] = make_uint2(ix[0] | ix[1] << 16, ix[2] | ix[3] << 16);
        }
    }
}

// ---------------------------------------------------------------------------------------------
// The sweep
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* b, unsigned n) {
    asm volatile("mbarrier.init.shared.b64 [%0], %1;" ::"r"(smem_addr(b)), "r"(n) : "memory");
}
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar, uint64_t pol) {
    asm volatile("mbarrier.arrive.expect_tx.shared.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar)), "l"(pol)
        : "memory");
}
// bounded wait for a phase of an mbarrier; false on giving up
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, long long budget) {
    for (long long n = 0; n <= budget; ++n) {
        uint32_t ok;
        asm volatile(
            "{ .reg .pred p; mbarrier.try_wait.parity.shared.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
            : "=r"(ok) : "r"(smem_addr(bar)), "r"(parity) : "memory");
        if (ok) return true;
    }
    return false;
}
template <int B>
__device__ __forceinline__ void async_copy(uint32_t dst, const void* src) {
    if constexpr (B == 32) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16), "l"((const char*)src + 16) : "memory");
    } else if constexpr (B == 64) {
        async_copy<32>(dst, src);
        async_copy<32>(dst + 32, (const char*)src + 32);
    } else if constexpr (B == 16) {
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
    } else {
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(B) : "memory");
    }
}
__device__ __forceinline__ void async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// all but the last LEFT groups of this thread have arrived
template <int LEFT>
__device__ __forceinline__ void async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory");
}

__device__ __forceinline__ float fma_(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float mul_(float a, float b) { return __fmul_rn(a, b); }  // never fused with a later add
__device__ __forceinline__ double mul_(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float div_(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double div_(double a, double b) { return __ddiv_rn(a, b); }
__device__ __forceinline__ float signed_(float v, int par) { return __uint_as_float(__float_as_uint(v) ^ (par ? 0x80000000u : 0u)); }
__device__ __forceinline__ double signed_(double v, int par) { return par ? -v : v; }

template <typename real, int GC>
struct alignas(sizeof(real) * GC <= 16 ? sizeof(real) * GC : 16) Vals {
    real v[GC];
};

// four entries of one lane
template <typename real>
struct Quad {
    real w[4];
    uint2 ix;
};
// quads of a slice held in registers: tasks of up to 23 entries in FP32, 15 in FP64
template <typename real> constexpr int NQ = sizeof(real) == 8 ? 4 : 6;

// quad q of the slice at e, for this lane
template <typename real>
__device__ __forceinline__ void get_quad(Quad<real>& t, const unsigned char* e, int q, int lane) {
    const unsigned char* w = e + q * quad_bytes<real>() + lane * 4u * sizeof(real);
    if constexpr (sizeof(real) == 4) {
        const float4 v = *reinterpret_cast<const float4*>(w);
        t.w[0] = v.x; t.w[1] = v.y; t.w[2] = v.z; t.w[3] = v.w;
    } else {
        const double2 u = *reinterpret_cast<const double2*>(w), v = *reinterpret_cast<const double2*>(w + 16);
        t.w[0] = u.x; t.w[1] = u.y; t.w[2] = v.x; t.w[3] = v.y;
    }
    t.ix = *reinterpret_cast<const uint2*>(e + q * quad_bytes<real>() + 128u * sizeof(real) + 8u * lane);
}

// the sum of a quad's two elements
template <typename real, int GC>
__device__ __forceinline__ void quad_sum(const Vals<real, GC>* val, const Quad<real>& t, real (&s)[GC]) {
    const Vals<real, GC> a1 = val[t.ix.x & 0xffffu], a0 = val[t.ix.x >> 16], b1 = val[t.ix.y & 0xffffu], b0 = val[t.ix.y >> 16];
#pragma unroll
    for (int g = 0; g < GC; ++g)
        s[g] = fma_(t.w[0], (real)fabs(a1.v[g]), mul_(t.w[1], (real)fabs(a0.v[g]))) +
               fma_(t.w[2], (real)fabs(b1.v[g]), mul_(t.w[3], (real)fabs(b0.v[g])));
}

// Sum of a task's entries: quads (q0 + q1) + (q2 + q3), plus (q4 + q5) + (q6 + q7), plus quads 8..15 likewise. The
// quads past those in registers come straight from E.
template <typename real, int GC>
__device__ __noinline__ void sum_tail(const Vals<real, GC>* val, const unsigned char* e, int nq, int lane, real (&s45)[GC], real (&acc)[GC]) {
    auto four = [&](int q0, real (&s)[GC]) {  // (quad q0 + quad q0+1) + (quad q0+2 + quad q0+3); those in registers and absent ones 0
        real u[GC];
#pragma unroll
        for (int g = 0; g < GC; ++g) s[g] = 0;
        for (int h = 0; h < 2; ++h) {
            real v[GC];
#pragma unroll
            for (int g = 0; g < GC; ++g) v[g] = 0;
            for (int i = 0; i < 2; ++i) {
                const int q = q0 + 2 * h + i;
                if (q < NQ<real> || q >= nq) continue;
                Quad<real> t;
                get_quad<real>(t, e, q, lane);
                quad_sum<real, GC>(val, t, u);
#pragma unroll
                for (int g = 0; g < GC; ++g) v[g] += u[g];
            }
#pragma unroll
            for (int g = 0; g < GC; ++g) s[g] += v[g];
        }
    };
    real x[GC], y[GC];
    four(4, x);
#pragma unroll
    for (int g = 0; g < GC; ++g) acc[g] += s45[g] + x[g];
    if (nq > 8) {
        four(8, x);
        four(12, y);
#pragma unroll
        for (int g = 0; g < GC; ++g) acc[g] += x[g] + y[g];
    }
}
template <typename real, int GC>
__device__ __forceinline__ void task_sum(const Vals<real, GC>* val, const Quad<real> (&t)[NQ<real>], const unsigned char* e, int nq,
                                         int lane, real (&acc)[GC]) {
    quad_sum<real, GC>(val, t[0], acc);
    if (nq > 1) {
        real u[GC];
        quad_sum<real, GC>(val, t[1], u);
#pragma unroll
        for (int g = 0; g < GC; ++g) acc[g] += u[g];
        if (nq > 2) {
            quad_sum<real, GC>(val, t[2], u);
            if (nq > 3) {
                real v[GC];
                quad_sum<real, GC>(val, t[3], v);
#pragma unroll
                for (int g = 0; g < GC; ++g) u[g] += v[g];
            }
#pragma unroll
            for (int g = 0; g < GC; ++g) acc[g] += u[g];
            if (nq > 4) {
#pragma unroll
                for (int g = 0; g < GC; ++g) u[g] = 0;
                if constexpr (NQ<real> > 4) {
                    quad_sum<real, GC>(val, t[4], u);
                    if (nq > 5) {
                        real v[GC];
                        quad_sum<real, GC>(val, t[5], v);
#pragma unroll
                        for (int g = 0; g < GC; ++g) u[g] += v[g];
                    }
                }
                if (nq <= NQ<real>) {
#pragma unroll
                    for (int g = 0; g < GC; ++g) acc[g] += u[g];
                } else {
                    sum_tail<real, GC>(val, e, nq, lane, u, acc);
                }
            }
        }
    }
}

struct DirArgs {
    const unsigned char *E, *C;
    const DirMeta* meta;
    const uint2* rtab;
    int rstride;                    // rounds + 1 that the table holds per direction
    int R, Fs, W;
    uint32_t off_cm, off_c, off_e;  // byte offsets of the shared-memory regions
    uint32_t c_slot, e_slot;        // bytes of a round's slot
};

// Two forms, by the width of the levels: worker warps at most, rounds whose sources are fetched ahead, rounds of C
// and of E in shared memory.
enum { NARROW = 0, MID = 1 };
template <int FORM> struct Form;
template <> struct Form<NARROW> { static constexpr int W = 4, A = 3, NC = 8, NE = 6; };
template <> struct Form<MID> { static constexpr int W = 7, A = 2, NC = 4, NE = 4; };

// Threads a block is compiled for: 112 registers each. It has 64 + 64 W, 512 at most, but with the registers of 512
// the compiler's order of the loads made the forms of seven workers a third slower (1.66 against 1.21 ms, 2^18 cells,
// 64 directions, 2 groups), and with those of 672 four groups spill (3.2 against 1.65 ms).
constexpr int DIR_BOUND = 576;

// Iteration r of a direction: the sums of round r, while E and the sources of the next rounds come in. One
// barrier ends it.
//   worker warps: the sums; control words and E of round r + 1 into registers;
//   fetcher warps, as many: cell sources and far sources of round r + A into shared memory;
//   two copying warps: bulk copies of the rounds of C and of E to come, into the slots that have fallen free.
// What bounds it is the longest chain of instructions of any warp between two barriers, so the work of an
// iteration is spread over kinds of warps: with the workers fetching their own sources a 55,000-cell periodic box of
// 84 directions took 0.92 ms per sweep, with one copying warp for both streams 0.56 ms, as it stands 0.52 ms (the
// packets of all directions: 0.88 ms). 3000 cells, 16 directions, 2 groups: 0.12 against 0.20 ms; 2^18 cells, 64
// directions, 2 groups: 1.21 against 1.60 ms.
// STOPS (tests only): a form of its own, because the copying warps are part of every level's chain and a condition
// more in their loop costs 0.5 to 1% of a sweep.
template <typename real, int GC, int MODE, int FORM, bool STOPS = false>
__global__ void __launch_bounds__(DIR_BOUND)
    k_sweep_dir(const __grid_constant__ SweepArgs a, const __grid_constant__ DirArgs p) {
    extern __shared__ __align__(128) unsigned char sm[];
    __shared__ __align__(8) uint64_t bars[2 * MAX_SLOTS];  // slots of C, slots of E
    __shared__ int s_fail;  // a wait gave up before this iteration, else INT_MAX
    constexpr int A = Form<FORM>::A, NST = A + 1, NC = Form<FORM>::NC, NE = Form<FORM>::NE;
    static_assert(NC >= A + 1 && NE >= 3 && NC <= MAX_SLOTS && NE <= MAX_SLOTS, "rounds in use at any time");
    using V = Vals<real, GC>;
    struct alignas(16 < 2 * sizeof(real) * GC ? 16 : 2 * sizeof(real) * GC) Src {
        real v[2 * GC];  // {q, kappa_t V} per group
    };
    V* val = reinterpret_cast<V*>(sm);
    Src* cms = reinterpret_cast<Src*>(sm + p.off_cm);
    unsigned char* const C = sm + p.off_c;
    unsigned char* const Es = sm + p.off_e;
    const int T = 32 * p.W, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool worker = tid < T;
    const uint32_t R = (uint32_t)p.R;
    if (tid == 0) {
        for (int i = 0; i < 2 * MAX_SLOTS; ++i) mbar_init(&bars[i], 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_fail = INT_MAX;
        for (int g = 0; g < GC; ++g) val[R + NST * p.Fs].v[g] = 0;
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    const volatile int* fail = &s_fail;
    uint32_t base = 0;  // rounds of the earlier directions of this block
    for (int d = blockIdx.x; d < a.nd; d += gridDim.x) {
        const DirMeta m = p.meta[d];
        const int nr = m.rounds;
        if (nr == 0) continue;
        const size_t slab = (size_t)d * a.N;
        V* const I = reinterpret_cast<V*>(a.I) + slab;
        auto c_of = [&](int r) { return C + (base + (uint32_t)r) % (uint32_t)NC * p.c_slot; };
        if (tid < 2 * T) {
            const int ft = tid - T;  // thread among the fetchers
            const Src* cm = reinterpret_cast<const Src*>(a.cm);
            // cell sources and far sources of round r + A
            auto fetch = [&](int r) {
                const unsigned char* c = c_of(r);
                const uint4 h = *reinterpret_cast<const uint4*>(c);
                const uint32_t st = (uint32_t)r % NST;
                if ((uint32_t)ft < 32u * h.x) {
                    const uint32_t cell = reinterpret_cast<const TaskRec<real>*>(c + c_tasks(h.x))[ft].cell;
                    if (cell != PAD_CELL) async_copy<sizeof(Src)>(smem_addr(&cms[st * T + ft]), cm + cell);
                }
                if (h.y) {
                    const uint32_t* far = reinterpret_cast<const uint32_t*>(c + c_far<real>(h.x));
                    V* dst = &val[R + st * p.Fs];
                    for (uint32_t k = ft; k < h.y; k += T) {
                        const uint32_t f = far[k], kind = f >> 30, i = f & 0x3fffffffu;
                        const V* from = reinterpret_cast<const V*>(kind == FAR_BC ? a.bc : a.Iprev);
                        if (kind == FAR_THIS) {
                            async_copy<sizeof(V)>(smem_addr(dst + k), I + i);
                        } else if (from) {
                            async_copy<sizeof(V)>(smem_addr(dst + k), from + (kind == FAR_BC ? 0 : slab) + i);
                        } else {
#pragma unroll
                            for (int g = 0; g < GC; ++g) dst[k].v[g] = 0;
                        }
                    }
                }
            };
            const real wd = MODE == PK_TRANSPOSED ? (sizeof(real) == 8 ? (real)a.w64[d] : (real)(float)a.w64[d]) : (real)1;
            // round r of this warp's slice: quads (0: no slice), E, the task's ring slot, cell and P_c
            int nq = 0;
            uint32_t e = 0;
            uint32_t slot = 0, cell = PAD_CELL;
            real P = 1;
            Quad<real> quad[NQ<real>];
            __syncthreads();  // the first round's control words have arrived
            for (int r = -A; r < nr && *fail > r; ++r) {
                if (worker) {
                    int nq1 = 0;
                    uint32_t e1 = 0, slot1 = 0, cell1 = PAD_CELL;
                    real P1 = 1;
                    if (r + 1 >= 0 && r + 1 < nr) {  // control words of round r + 1
                        const unsigned char* c = c_of(r + 1);
                        const uint4 h = *reinterpret_cast<const uint4*>(c);
                        if ((uint32_t)warp < h.x) {
                            const uint32_t w = reinterpret_cast<const uint32_t*>(c + 16)[warp];
                            const TaskRec<real> t = reinterpret_cast<const TaskRec<real>*>(c + c_tasks(h.x))[tid];
                            nq1 = (int)(w & 0xffu);
                            e1 = p.off_e + (base + (uint32_t)(r + 1)) % (uint32_t)NE * p.e_slot + (w >> 8) * 256u;
                            slot1 = h.w + (uint32_t)tid;
                            slot1 -= slot1 >= R ? R : 0u;
                            cell1 = t.cell;
                            P1 = t.P;
                        }
                    }
                    real acc[GC];
                    Src qr;
                    if (nq) {
                        qr = cms[(uint32_t)r % NST * T + tid];
                        task_sum<real, GC>(val, quad, sm + e, nq, lane, acc);
                    }
#pragma unroll
                    for (int j = 0; j < NQ<real>; ++j)
                        if (j < nq1) get_quad<real>(quad[j], sm + e1, j, lane);
                    if (nq) {
                        V v, o, mean;
#pragma unroll
                        for (int g = 0; g < GC; ++g) {
                            if constexpr (MODE == PK_EXP) {
                                exp_update_lanes(acc[g], qr.v[2 * g], qr.v[2 * g + 1], P, v.v[g], mean.v[g]);
                            } else if constexpr (MODE == PK_TRANSPOSED) {
                                v.v[g] = div_(fma_(wd, qr.v[2 * g], acc[g]), P + qr.v[2 * g + 1]);
                            } else {
                                v.v[g] = div_(qr.v[2 * g] + acc[g], P + qr.v[2 * g + 1]);
                            }
                            o.v[g] = signed_(v.v[g], a.parity);
                        }
                        val[slot] = v;
                        if (cell != PAD_CELL) {
                            I[cell] = o;
                            if constexpr (MODE == PK_EXP) reinterpret_cast<V*>(a.Imean)[slab + cell] = mean;
                        }
                    }
                    nq = nq1; e = e1; slot = slot1; cell = cell1; P = P1;
                } else {
                    if (r + A < nr) fetch(r + A);
                    async_commit();
                    async_wait<A - 1>();
                }
                __syncthreads();
            }
            async_wait<0>();
        } else {
            // one warp copies C, the other E, round by round (its first lane; the others only meet the barriers)
            const bool is_c = tid < 2 * T + 32, on = lane == 0;
            const uint2* tab = p.rtab + (size_t)d * p.rstride;
            const uint32_t depth = is_c ? NC : NE;
            const unsigned char* src = is_c ? p.C + m.c_base : p.E + m.e_base;
            unsigned char* ring = is_c ? C : Es;
            const uint32_t slot_bytes = is_c ? p.c_slot : p.e_slot, unit = is_c ? 16u : 256u;
            uint64_t* bar = bars + (is_c ? 0 : MAX_SLOTS);
            const uint64_t pol = policy_evict_first();
            int iss = 0, wt = 0;  // rounds copied, rounds waited for; their slots, and the phase of the latter
            uint32_t is = base % depth, ws = is, ph = base / depth & 1u;
            bool ok = true;
            // offsets of round iss and of the next one (read an iteration before they are used)
            uint32_t at = is_c ? tab[0].x : tab[0].y, to = is_c ? tab[1].x : tab[1].y;
            // STOPS: the copies of one stream of direction 0 end at a round, whose wait then gives up at once
            int stop = nr;
            if (STOPS && d == 0 && (a.debug_stall & 1) == (is_c ? 0 : 1)) stop = min(nr, (a.debug_stall - 2) >> 1);
            auto issue = [&](int lim) {  // rounds below lim
                if (iss < min(lim, stop)) {
                    bulk_load(ring + is * slot_bytes, src + (size_t)at * unit, (to - at) * unit, &bar[is], pol);
                    at = to;
                    is = is + 1 == depth ? 0u : is + 1;
                    if (++iss < nr) to = is_c ? tab[iss + 1].x : tab[iss + 1].y;
                }
            };
            auto need = [&](int lim) {  // rounds below lim have arrived
                for (; ok && wt < min(lim, nr); ++wt) {
                    ok = wt < iss && mbar_wait(&bar[ws], ph, a.spin_budget);
                    ws = ws + 1 == depth ? 0u : ws + 1;
                    ph ^= ws == 0 ? 1u : 0u;
                }
            };
            if (on) {
                for (int i = 0; i < (int)depth; ++i) issue(i + 1);
                need(is_c ? 1 : 0);
                if (!ok) s_fail = -A;
            }
            __syncwarp();
            __syncthreads();
            for (int r = -A; r < nr && *fail > r; ++r) {
                if (on) {
                    // C of rounds up to r (in registers) and E of rounds before r are done with
                    issue(is_c ? r + 1 + NC : r + NE);
                    need(is_c ? r + A + 2 : r + 3);
                    if (!ok) s_fail = r + 1;
                }
                __syncwarp();
                __syncthreads();
            }
            if (on && *fail <= nr) {  // a bounded wait gave up: report, let the copies in flight land (the one waited for first)
                atomicCAS(a.err, DEV_OK, DEV_TIMEOUT);
                for (int w = ok ? wt : wt - 1; w < iss; ++w) {  // from the round whose wait gave up
                    const uint32_t q = base + (uint32_t)w;
                    mbar_wait(&bar[q % depth], q / depth & 1u, a.spin_budget);
                }
            }
            __syncwarp();
        }
        if (*fail <= nr) return;  // all threads, after the barrier that ended the loop
        base += (uint32_t)nr;
        __syncthreads();
    }
}

template <typename real, int FORM>
const void* dir_kernel(int GC, int mode) {
    if (mode == PK_TRANSPOSED) return GC == 2 ? (const void*)k_sweep_dir<real, 2, PK_TRANSPOSED, FORM>
                                              : (const void*)k_sweep_dir<real, 4, PK_TRANSPOSED, FORM>;
    if constexpr (sizeof(real) == 4) {
        if (mode == PK_EXP) {
            switch (GC) {
                case 1: return (const void*)k_sweep_dir<real, 1, PK_EXP, FORM>;
                case 2: return (const void*)k_sweep_dir<real, 2, PK_EXP, FORM>;
                default: return (const void*)k_sweep_dir<real, 4, PK_EXP, FORM>;
            }
        }
    }
    switch (GC) {
        case 1: return (const void*)k_sweep_dir<real, 1, PK_BALANCE, FORM>;
        case 2: return (const void*)k_sweep_dir<real, 2, PK_BALANCE, FORM>;
        default: return (const void*)k_sweep_dir<real, 4, PK_BALANCE, FORM>;
    }
}
template <typename real>
const void* dir_kernel(int GC, int mode, int form, bool stops) {
    if (stops) {
        if constexpr (sizeof(real) == 4)
            if (form == MID) return (const void*)k_sweep_dir<real, 2, PK_BALANCE, MID, true>;
        return (const void*)k_sweep_dir<real, 2, PK_BALANCE, NARROW, true>;
    }
    if constexpr (sizeof(real) == 4)
        if (form == MID) return dir_kernel<real, MID>(GC, mode);
    return dir_kernel<real, NARROW>(GC, mode);
}

constexpr uint32_t SMEM_BLOCK = 227u * 1024u - 1024u;  // dynamic shared memory of a block that has an SM alone

// Shared-memory layout for the present form, W, Fs and slot sizes; the value ring takes what is left.
bool layout(DirOp& P) {
    const uint32_t vb = (uint32_t)(P.real_bytes * P.GC), T = 32u * (uint32_t)P.W;
    const bool narrow = P.form == NARROW;
    const uint32_t NC = narrow ? Form<NARROW>::NC : Form<MID>::NC, NE = narrow ? Form<NARROW>::NE : Form<MID>::NE;
    P.A = narrow ? Form<NARROW>::A : Form<MID>::A;
    const uint32_t nst = (uint32_t)P.A + 1u, cm = nst * T * 2u * vb;
    const int64_t fixed = (int64_t)NE * P.e_slot + (int64_t)NC * P.c_slot + cm + (int64_t)nst * P.Fs * vb + vb + 256;
    int64_t R = ((int64_t)SMEM_BLOCK - fixed) / vb;
    R = std::min<int64_t>(R, 65535 - (int64_t)nst * P.Fs) / 32 * 32;
    if (R < (int64_t)nst * T + 32) return false;
    P.R = (int)R;
    const uint64_t values = (uint64_t)(R + (int64_t)nst * P.Fs + 1) * vb;
    P.off_cm = (uint32_t)((values + 127) & ~127ull);
    P.off_c = (P.off_cm + cm + 127u) & ~127u;
    P.off_e = P.off_c + NC * P.c_slot;
    P.smem = P.off_e + NE * P.e_slot;
    return P.smem <= SMEM_BLOCK;
}

}  // namespace

// Plans the operator of the levels L for values of GC numbers of real_bytes: places, slices, rounds, offsets.
// *ok = false where this form does not apply; P.e_bytes and P.c_bytes are what the streams need.
cudaError_t dir_plan(const DevMesh& m, Levels& L, DirOp& P, bool transposed, int real_bytes, int GC, const double* om64_all,
                     const float4* om32_all, const float4* om32lo_all, int sms, cudaStream_t st, bool* ok, int w_max) {
    *ok = false;
    const int nd = L.nd, nl = L.n_levels;
    if (nl < 1 || m.max_row > 64 || m.NB >= (1ll << 30) || !L.by_dir) return cudaSuccess;
    double dsum = 0;
    for (int x : L.depth) dsum += x;
    const double width = (double)m.N * nd / std::max(1.0, dsum);  // tasks of a mean level
    // Where the line lies. A direction's rounds follow one another on one SM, so what counts is how much of a level a
    // round takes. FP32: 204 tasks per level (2^18 cells, 64 directions) 1.21 against 1.60 ms for the packets of
    // all directions, 196 (scheme (b), 60 directions) 0.08 against 0.11 ms; 584 (2^21 cells, 128 directions) 9.7
    // against 10.6 ms, which the longer build does not earn back; 957 (25 meshes, 2 groups) 7.1 against
    // 5.6 ms. Four values are bound by the sums of one SM sooner than the packets by few directions: 1.01 against 1.13 ms
    // (156 tasks, 12 directions), 1.71 against 1.57 (249, 12), 1.82 against 1.85 (247, 32). With more than two
    // directions per SM the directions that wait cost more than the levels gain.
    // FP64 has the mesh-row kernel to beat: 350 (the 32^3 lattice) 0.40 against 0.54 ms. A level costs the FP64 pipe of
    // one SM time in proportion to its values and their entries, however few directions there are, while the mesh
    // rows' level gets cheaper with fewer. Solves, ms by direction / over the mesh rows (tasks per level, directions), of
    // 8,000 to 250,000 cells of 15.4 sides unless stated:
    //   1 value   4.1 / 4.3 (263, 1)    4.3 / 5.4 (270, 4)    scheme (b) 0.58 / 0.58 (300, 1)    0.59 / 0.64 (331, 4)
    //   2 values  4.87 / 4.86 (163, 1)  10.0 / 6.4 (263, 1)   5.3 / 6.0 (169, 4)   10.4 / 8.4 (270, 4)
    //             5.3 / 7.2 (156, 12)   11.5 / 10.0 (249, 12)   11.1 / 13.9 (247, 32)
    //             lattice 0.35 / 0.48 (197, 1)   scheme (b), n = 3 0.97 / 0.81 (300, 1)   1.02 / 1.15 (315, 12)
    //   4 values  6.16 / 6.21 (74, 7)   8.4 / 7.4 (96, 7)   11.1 / 11.5 (114, 32)   13.2 / 12.4 (128, 32)
    //             19.4 / 27.5 (154, 96)   scheme (b), n = 1 0.41 / 0.39 (151, 7)   0.42 / 0.50 (159, 32)
    // Four values leave room for three workers and a short ring. The mesh rows' transposed sweep takes twice as long:
    // gradients of two groups 22.8 / 23.7 (148, 7). The caps are the widest levels measured.
    double line = GC == 4 && !transposed ? std::min(256.0, 180.0 + 2.0 * nd) : 256.0;
    if (real_bytes == 8) {
        const double sides = std::min((double)m.S / m.N, L.transport > 0 ? std::max(8.0, 2.0 * L.transport + 2.0) : 64.0);
        const double weight = (GC == 4 ? 5.2 : (GC == 2 ? 2.0 : 1.1)) * (sides + 5.0), slow = transposed ? 2.0 : 1.0;
        line = std::min(GC == 4 ? 160.0 : std::min(512.0, slow * (280.0 + 20.0 * nd)), slow * (6400.0 + 210.0 * nd) / weight);
    }
    if (width > line || nd > 2 * sms) return cudaSuccess;
    // one round per level where the workers suffice (FP64 sums are bound by the FP64 pipe: four warps fill it)
    P.W = std::min(real_bytes == 8 ? Form<NARROW>::W : Form<MID>::W, std::max(1, (int)(1.2 * (width / 32.0 + 0.5) + 0.5)));
    P.W = std::min(P.W, w_max);
    const auto narrower = [&]() -> cudaError_t {  // the regions of a round leave no ring (FP64, four values): fewer workers
        if (P.W <= 1) return cudaSuccess;
        return dir_plan(m, L, P, transposed, real_bytes, GC, om64_all, om32_all, om32lo_all, sms, st, ok, P.W - 1);
    };
    P.form = P.W <= Form<NARROW>::W ? NARROW : MID;
    P.Fs = std::max(256, 128 + 64 * P.W);
    const uint32_t cb = real_bytes == 8 ? c_bytes<double>((uint32_t)P.W, (uint32_t)P.Fs) : c_bytes<float>((uint32_t)P.W, (uint32_t)P.Fs);
    P.c_slot = (cb + 127u) & ~127u;
    // E of a round: a guess at its longest slices' quads, corrected below by the bound that placing the tasks gives
    P.e_slot = (uint32_t)((P.W == 1 ? 6.0 : (P.W == 2 ? 5.0 : (P.W <= 4 ? 4.0 : 3.4))) * P.W) * (uint32_t)(32 * (4 * real_bytes + 8));
    if (!layout(P)) return narrower();
    DirBuild a;
    a.cap = L.dlev_cap;
    a.dcnt = L.dlev;
    a.dbase = a.dcnt + (int64_t)nd * a.cap;
    a.depth = a.dbase + (int64_t)nd * a.cap + nd;
    a.nd = nd;
    a.W = P.W;
    a.transposed = transposed ? 1 : 0;
    a.N = m.N;
    a.lcap = nl;
    // a level of n tasks has at most n / 32 + 1 slices; its rounds are of W of them, or fewer where many sources are far
    a.SC = (int)std::min<int64_t>(m.N / 32 + nl + 1, m.N);
    a.RC = (int)std::min<int64_t>(2 * (int64_t)a.SC / P.W + 2 * nl + 64, a.SC);
    const size_t nN = (size_t)nd * m.N, nS = (size_t)nd * (a.SC + 1), nR = (size_t)nd * (a.RC + 1), nL = (size_t)nd * nl;
    size_t off = 0;
    auto part = [&](size_t bytes) {
        const size_t o = off;
        off += (bytes + 255) & ~(size_t)255;
        return o;
    };
    const size_t o_sb = part(4 * nL), o_rb = part(4 * nL), o_nr = part(4 * nL), o_pl = part(4 * nN), o_or = part(128 * nS),
                 o_ms = part(256 * nS), o_P = part(128 * nS), o_nq = part(4 * nS), o_eo = part(4 * nS), o_sf = part(4 * nS),
                 o_le = part(4 * nS), o_ri = part(8 * nR), o_nf = part(4 * nR), o_co = part(4 * nR), o_to = part(8 * (size_t)nd),
                 o_st = part(16), o_tt = part(16), o_sc = part(8 * ((size_t)nd + 1));
    cudaError_t e;
    if (off > L.dir_ws_bytes) {
        if (L.dir_ws) dev_free(L.dir_ws);
        L.dir_ws = nullptr;
        L.dir_ws_bytes = 0;
        // no room: the packets take their place
        P.room = off;
        if (!dev_room(off + ((size_t)2 << 30))) return cudaSuccess;
        if (dev_alloc(&L.dir_ws, off) != cudaSuccess) {
            cudaGetLastError();
            return cudaSuccess;
        }
        P.room = 0;
        L.dir_ws_bytes = off;
    }
    const size_t keep = ((sizeof(DirMeta) * nd + 255) & ~(size_t)255) + 8 * nR;
    if (keep > P.meta_bytes) {
        if (P.meta) dev_free(P.meta);
        P.meta = nullptr;
        P.meta_bytes = 0;
        if (dev_alloc(&P.meta, keep) != cudaSuccess) {
            cudaGetLastError();
            P.room = keep;
            return cudaSuccess;
        }
        P.meta_bytes = keep;
    }
    P.rtab = (uint2*)((char*)P.meta + ((sizeof(DirMeta) * nd + 255) & ~(size_t)255));
    P.rstride = a.RC + 1;
    char* ws = (char*)L.dir_ws;
    int64_t* total = (int64_t*)(ws + o_tt);
    a.list = L.raw;
    a.sbase = (int32_t*)(ws + o_sb); a.rbase = (int32_t*)(ws + o_rb); a.nround = (int32_t*)(ws + o_nr);
    a.place = (uint32_t*)(ws + o_pl); a.ord = (uint32_t*)(ws + o_or); a.msk = (uint64_t*)(ws + o_ms); a.P = (float*)(ws + o_P);
    a.nq = (uint32_t*)(ws + o_nq); a.eoff = (uint32_t*)(ws + o_eo); a.sfar = (uint32_t*)(ws + o_sf); a.lend = (uint32_t*)(ws + o_le);
    a.rinfo = (uint2*)(ws + o_ri); a.nfar = (uint32_t*)(ws + o_nf); a.coff = (uint32_t*)(ws + o_co); a.rtab = P.rtab;
    a.tot = (int2*)(ws + o_to); a.meta = P.meta; a.stat = (int32_t*)(ws + o_st);
    a.E = nullptr; a.C = nullptr;
    a.rowptr = m.rowptr; a.side = m.side; a.side64 = m.side64;
    a.om32 = om32_all + L.d0; a.om32lo = om32lo_all + L.d0; a.om64 = om64_all + 3 * (int64_t)L.d0;
    a.info = L.info;
    const bool dc = L.transport > 0 && !transposed;
    a.dc_inm = dc ? L.dc_inm : nullptr; a.dc_share32 = dc ? L.dc_share32 : nullptr; a.dc_share64 = dc ? L.dc_share64 : nullptr;
    a.R = P.R; a.A = P.A; a.Fs = P.Fs;
    a.quad_b = (uint32_t)(32 * (4 * real_bytes + 8));
    if ((e = cudaMemsetAsync(a.stat, 0, 16, st))) return e;
    const dim3 lev((unsigned)nl, (unsigned)nd), levt((unsigned)((nl + 127) / 128), (unsigned)nd);
    for (int attempt = 0; attempt < 5; ++attempt) {
        a.R = P.R; a.A = P.A; a.Fs = P.Fs; a.e_slot = P.e_slot;
        if (attempt == 0) {
            k_dir_slices<<<nd, 1024, 0, st>>>(a);
            k_dir_place<<<lev, PLACE_THREADS, 0, st>>>(a);
        }
        if ((e = cudaMemsetAsync(a.stat + 1, 0, 4, st))) return e;
        k_dir_count<<<lev, 128, 0, st>>>(a);
        k_dir_cut<false><<<levt, 128, 0, st>>>(a);
        k_dir_rounds<<<nd, 1024, 0, st>>>(a);
        k_dir_cut<true><<<levt, 128, 0, st>>>(a);
        if (real_bytes == 8) k_dir_offsets<double><<<nd, 1024, 0, st>>>(a);
        else k_dir_offsets<float><<<nd, 1024, 0, st>>>(a);
        k_dir_bases<<<1, 1024, 0, st>>>(P.meta, nd, total, (uint32_t*)(ws + o_sc));
        P.launches += attempt == 0 ? 8 : 6;
        int32_t stat[4] = {};
        int64_t tt[2] = {};
        if ((e = cudaMemcpyAsync(stat, a.stat, sizeof stat, cudaMemcpyDeviceToHost, st))) return e;
        if ((e = cudaMemcpyAsync(tt, total, sizeof tt, cudaMemcpyDeviceToHost, st))) return e;
        if ((e = cudaStreamSynchronize(st))) return e;
        P.e_bytes = tt[0];
        P.c_bytes = tt[1];
        if (stat[0] || stat[3]) return cudaSuccess;
        // a round's E, and a slice's far sources, must fit their slots
        bool fits = true;
        if (stat[1] > P.Fs) {
            P.Fs = (stat[1] + 31) & ~31;
            const uint32_t cbn = real_bytes == 8 ? c_bytes<double>((uint32_t)P.W, (uint32_t)P.Fs) : c_bytes<float>((uint32_t)P.W, (uint32_t)P.Fs);
            P.c_slot = (cbn + 127u) & ~127u;
            fits = false;
        }
        if ((uint32_t)stat[2] > P.e_slot) {
            P.e_slot = ((uint32_t)stat[2] + 127u) & ~127u;
            fits = false;
        }
        if (fits) {
            *ok = true;
            P.args.resize(sizeof a);
            memcpy(P.args.data(), &a, sizeof a);
            return cudaGetLastError();
        }
        if (!layout(P)) return narrower();
    }
    return cudaSuccess;
}

// Writes the planned operator into P.E and P.C (directly after dir_plan).
cudaError_t dir_write(DirOp& P, cudaStream_t st) {
    DirBuild a;
    memcpy(&a, P.args.data(), sizeof a);
    a.E = P.E;
    a.C = P.C;
    const dim3 g((unsigned)a.RC, (unsigned)a.nd);
    if (P.real_bytes == 8) k_dir_write<double><<<g, 128, 0, st>>>(a);
    else k_dir_write<float><<<g, 128, 0, st>>>(a);
    P.launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_sweep_dir(const SweepArgs& a, const DirOp& P, int mode, int sms, cudaStream_t st) {
    DirArgs p;
    p.E = P.E; p.C = P.C; p.meta = P.meta; p.rtab = P.rtab; p.rstride = P.rstride; p.R = P.R; p.Fs = P.Fs; p.W = P.W;
    p.off_cm = P.off_cm; p.off_c = P.off_c; p.off_e = P.off_e; p.c_slot = P.c_slot; p.e_slot = P.e_slot;
    const void* f = P.real_bytes == 8 ? dir_kernel<double>(P.GC, mode, P.form, a.debug_stall >= 2)
                                      : dir_kernel<float>(P.GC, mode, P.form, a.debug_stall >= 2);
    // the most that any plan takes, not this plan's: the attribute belongs to the kernel, and a context of another
    // thread may set it between here and the launch
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BLOCK);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)std::min(a.nd, sms));
    cfg.blockDim = dim3(64u * (unsigned)P.W + 64u);
    cfg.dynamicSmemBytes = P.smem;
    cfg.stream = st;
    void* args[] = {(void*)&a, (void*)&p};
    return cudaLaunchKernelExC(&cfg, f, args);
}

}  // namespace sw
