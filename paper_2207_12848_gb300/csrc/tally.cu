// FP64 tallies and the per-iteration updates around the sweep (K4, K5, K6) and the
// adjoint's gradient accumulation. Every sum runs in a fixed order, so results are
// reproducible run to run. All sums are FP64, on a part with two FP64 lanes per SM and clock: a pass over
// the intensities is bound by the FP64 pipe as soon as it spends more than one or two FP64 instructions per
// value. So FP32 intensities are widened by integer instructions, products are accumulated by one fused
// multiply-add (one rounding less than a product and a sum), and factors and divisions that
// do not depend on the direction stand outside the sums.
//
//   mean intensity  J_c = (1/4pi) sum_d w_d I_c,d                     (Sec. 3.2, photon rate up to 1/13.6 eV)
//   absorbed rate   Gamma_c = kappa_a,c V_c sum_d w_d I_c,d
//   escaped         sum_d w_d sum_{boundary outflow sides} |a_f| I_c,d
//   source update   q_c = eps_c/4pi + kappa_s,c V_c J_c                (Alg. 1, scattering as a fixed source)
//   periodic source j_c = sum_d w_d sum_{periodic inflow sides} |a_f| I_partner,d   (Sec. 2.7)
//   relative change E_c = |j^n - j^(n-1)| / (j^n + j^(n-1))             (Eq. relativeErrorPbc)
#include <cooperative_groups.h>

#include <type_traits>

#include "adjoint.cuh"
#include "common.cuh"

namespace cg = cooperative_groups;

namespace sw {
namespace {

__device__ __forceinline__ double dmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double dadd(double a, double b) { return __dadd_rn(a, b); }

// |x| in FP64. An FP32 value is widened by integer instructions (exact): its exponent re-biased, its fraction
// shifted into place; only denormals, infinities and NaN take the conversion instruction.
__device__ __forceinline__ double widen(float x) {
    const uint32_t u = __float_as_uint(x) & 0x7fffffffu;
    if (u - 0x00800000u >= 0x7f000000u && u) return (double)__uint_as_float(u);
    return __hiloint2double(u ? (int)((u >> 3) + 0x38000000u) : 0, (int)(u << 29));
}
__device__ __forceinline__ double widen(double x) { return fabs(x); }
template <typename real>
__device__ __forceinline__ double mag(const real* p) { return widen(*p); }

// x / 4 pi: the product with the rounded reciprocal, corrected by its residual (Markstein's correction of a
// quotient, correctly rounded for a correctly rounded reciprocal), in three FP64 instructions
__device__ __forceinline__ double over_4pi(double x) {
    const uint32_t h = (uint32_t)__double2hiint(x) & 0x7fffffffu;
    // tiny (the residual could underflow), infinite or NaN
    if (h - 0x06000000u >= 0x79000000u && (h | (uint32_t)__double2loint(x))) return x / FOURPI;
    constexpr double r = 1.0 / FOURPI;
    const double q = x * r;
    return fma(fma(-q, FOURPI, x), r, q);
}

// sum over the directions of w_d |I_d| of one (cell, group); the loads of eight directions are in flight together
template <typename real>
__device__ __forceinline__ double weighted_sum(const real* I, size_t stride, int nd, const double* w64) {
    double s = 0.0;
    int d = 0;
    for (; d + 8 <= nd; d += 8) {
        real v[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) v[k] = I[(size_t)(d + k) * stride];
#pragma unroll
        for (int k = 0; k < 8; ++k) s = fma(__ldg(w64 + d + k), widen(v[k]), s);
    }
    for (; d < nd; ++d) s = fma(__ldg(w64 + d), widen(I[(size_t)d * stride]), s);
    return s;
}

// Largest of a non-negative value over the block, into *dmax by one atomic per block (one per value serialises in L2:
// 0.50 ms for 10^6 values). A NaN (the change between two infinite values) counts as none; it is told by its bits, the FP64
// pipe being the bound. Blocks of 256 threads.
__device__ __forceinline__ void block_max(double v, unsigned long long* dmax) {
    __shared__ unsigned long long s_max[8];
    unsigned long long x = (unsigned long long)__double_as_longlong(v);
    if (x > 0x7ff0000000000000ull) x = 0ull;
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long y = __shfl_xor_sync(0xffffffffu, x, o);
        x = y > x ? y : x;
    }
    __syncthreads();  // s_max may still be read from an earlier call
    if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) x = s_max[w] > x ? s_max[w] : x;
        if (x) atomicMax(dmax, x);
    }
}

// deterministic block sum of two values per thread into out[blockIdx][0..1]
__device__ void block_sum2(double a, double b, double* out) {
    __shared__ double s0[256], s1[256];
    s0[threadIdx.x] = a;
    s1[threadIdx.x] = b;
    __syncthreads();
    for (int off = blockDim.x / 2; off > 0; off >>= 1) {
        if (threadIdx.x < off) {
            s0[threadIdx.x] += s0[threadIdx.x + off];
            s1[threadIdx.x] += s1[threadIdx.x + off];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[2 * blockIdx.x] = s0[0];
        out[2 * blockIdx.x + 1] = s1[0];
    }
}

__global__ void k_prep_material(int64_t N, int G, const double* vol, const double* ka, const double* ks,
                                const double* em, const double* J, float2* cm32, double2* cm64) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N * G) return;
    int64_t c = i / G;
    double V = vol[c];
    double kscat = ks ? ks[i] : 0.0;
    double q = over_4pi(em[i]);
    if (ks && J) q = dadd(q, dmul(dmul(kscat, V), J[i]));
    double dnm = dmul(dadd(ka[i], kscat), V);
    if (cm64) cm64[i] = make_double2(q, dnm);
    if (cm32) cm32[i] = make_float2((float)q, (float)dnm);
}

// adjoint sources split into non-negative parts: groups [0,G) carry g+, [G,2G) carry g-
__global__ void k_prep_adjoint(int64_t N, int G, const double* vol, const double* ka, const double* ks,
                               const double* dlj, const double* dlg, float2* cm32, double2* cm64) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N * G) return;
    int64_t c = i / G;
    int g = (int)(i - c * G);
    double V = vol[c];
    double gd = dlg ? dmul(dmul(dlg[i], ka[i]), V) : 0.0;
    double gj = dlj ? over_4pi(dlj[i]) : 0.0;
    double src = dadd(gd, gj);
    double dnm = dmul(dadd(ka[i], ks ? ks[i] : 0.0), V);
    double gp = src > 0.0 ? src : 0.0, gm = src < 0.0 ? -src : 0.0;
    int64_t o = c * (2 * G);
    if (cm64) {
        cm64[o + g] = make_double2(gp, dnm);
        cm64[o + G + g] = make_double2(gm, dnm);
    }
    if (cm32) {
        cm32[o + g] = make_float2((float)gp, (float)dnm);
        cm32[o + G + g] = make_float2((float)gm, (float)dnm);
    }
}

template <typename real>
__global__ void k_tally(const real* I, int64_t N, int G, int nd, const double* w64, double wsum, const double* vol,
                        const double* ka, const double* em, double* J, double* Gam, double* partial) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double absorbed = 0.0, emitted = 0.0;
    if (i < N * G) {
        const double j = over_4pi(weighted_sum(I + i, (size_t)N * G, nd, w64));
        int64_t c = i / G;
        double gam = dmul(dmul(dmul(ka[i], vol[c]), FOURPI), j);
        J[i] = j;
        if (Gam) Gam[i] = gam;
        absorbed = gam;
        emitted = over_4pi(dmul(em[i], wsum));
    }
    block_sum2(absorbed, emitted, partial);
}

// Sums over the rows of a few cells (boundary or periodic cells) for every direction: one block per
// cell, its threads over directions, so the FP64 classification and the strided intensity reads of
// the D directions run in parallel; the block's partial sums are then combined in a fixed order
// (warp shuffles, then the warps in index order), so results do not depend on timing.
constexpr int ROW_THREADS = 128;

__device__ __forceinline__ double block_sum_fixed(double v, double* sh) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();  // sh may still be read from the previous call
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    for (int w = 0; w < ROW_THREADS / 32; ++w) t += sh[w];
    return t;
}

// Escaped (outflow through vacuum faces) and injected (boundary inflow) photon rates of one boundary
// cell, into partial[2k], partial[2k+1]. Bound by the FP64 pipe: a direction's flux factor sum A n.Omega over the
// cell's outflow faces is formed first (three fused multiply-adds a face, none for a face whose FP32 sign says inflow
// of a vacuum boundary) and meets the G intensities once; n.Omega per face and group took 3.3 ms for the
// 110,000 boundary cells of 25 meshes, 128 directions, 2 groups. The fused n.Omega may differ in sign from the
// classification's where it is all rounding; with scheme (a) such a face carries next to nothing, under scheme (b) a
// chosen face carries its share whatever n.Omega is, so there the mask alone decides.
template <typename real>
__global__ void __launch_bounds__(ROW_THREADS) k_boundary_tally(const int32_t* bcells, const uint32_t* rowptr,
                                                                const SideRec* side, const d4* side64, const real* I,
                                                                int64_t N, int G, int nd, const double* om64,
                                                                const double* w64, const double* bc,
                                                                double* partial, DcTabs dc) {
    __shared__ double sh[ROW_THREADS / 32];
    const int64_t k = blockIdx.x;
    const int32_t c = bcells[k];
    const uint32_t r0 = rowptr[c], r1 = rowptr[c + 1];
    double esc = 0.0, inj = 0.0;
    for (int d = threadIdx.x; d < nd; d += ROW_THREADS) {
        const double ox = om64[3 * d], oy = om64[3 * d + 1], oz = om64[3 * d + 2], w = w64[d];
        const float fx = (float)ox, fy = (float)oy, fz = (float)oz;
        const uint64_t chosen = dc.mask ? dc.mask[(int64_t)c * nd + d] : 0ull;
        double out = 0.0;  // flux factor of the outflow through vacuum faces
        for (uint32_t s = r0; s < r1; ++s) {
            const int4 rec = side[s].hi;
            if (rec.x >= 0) continue;
            if (!bc) {
                const float ax = __int_as_float(rec.y), ay = __int_as_float(rec.z), az = __int_as_float(rec.w);
                if (ax * fx + ay * fy + az * fz < -BAND_REL * (fabsf(ax) + fabsf(ay) + fabsf(az))) continue;
            }
            // scheme (b): the outflow leaves through a vacuum face only if the cell chose it, with its share
            if (dc.mask && ((chosen >> (s - r0)) & 1ull)) {
                out = dadd(out, dc.share64[(int64_t)c * nd + d]);
                continue;
            }
            const d4 n = side64[s];
            const double t = fma(n.z, oz, fma(n.y, oy, dmul(n.x, ox)));
            if (t > 0.0) {
                if (!dc.mask) out = fma(n.w, t, out);
            } else if (bc) {
                const double wa = dmul(w, dmul(n.w, -t));
                for (int g = 0; g < G; ++g) inj = fma(wa, bc[(size_t)(-1 - rec.x) * G + g], inj);
            }
        }
        if (out != 0.0) {
            double I0 = 0.0;
            for (int g = 0; g < G; ++g) I0 = dadd(I0, mag(I + ((size_t)d * N + c) * G + g));
            esc = fma(dmul(w, out), I0, esc);
        }
    }
    esc = block_sum_fixed(esc, sh);
    if (bc) inj = block_sum_fixed(inj, sh);
    if (threadIdx.x == 0) {
        partial[2 * k] = esc;
        partial[2 * k + 1] = inj;
    }
}

// Periodic-inflow weight table, fixed for a solve: for every periodic side of every periodic cell (in
// row order) and every direction, w_d A |n.Omega| in FP64 where the side is an inflow side, else 0.
// Built once per solve; each iteration then needs one FP64 multiply-add per inflow side and direction
// instead of recomputing n.Omega and the weight on this part's narrow FP64 pipe. Beside the weights stand the
// partner of each side and, per periodic cell, its number and its range of sides, so that an iteration reads
// one record and consecutive lists instead of searching the cell's row for its periodic sides.
__global__ void k_pside_count(const int32_t* pcells, int64_t np, const uint32_t* rowptr, const SideRec* side,
                              int32_t* cnt) {
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= np) return;
    const int32_t c = pcells[k];
    int n = 0;
    for (uint32_t s = rowptr[c]; s < rowptr[c + 1]; ++s) {
        const int32_t x = side[s].hi.x;
        if (x >= 0 && (x & NBR_PERIODIC)) ++n;
    }
    cnt[k] = n;
}

// exclusive scan of n counts by one block of 1024 threads; off[n] = total
__global__ void k_scan_counts(const int32_t* cnt, int64_t n, int32_t* off) {
    __shared__ int32_t s_sum[1024];
    const int64_t per = (n + blockDim.x - 1) / blockDim.x;
    const int64_t i0 = threadIdx.x * per;
    int32_t loc = 0;
    for (int64_t i = i0; i < i0 + per && i < n; ++i) loc += cnt[i];
    s_sum[threadIdx.x] = loc;
    __syncthreads();
    if (threadIdx.x == 0) {
        int32_t run = 0;
        for (int t = 0; t < (int)blockDim.x; ++t) {
            const int32_t v = s_sum[t];
            s_sum[t] = run;
            run += v;
        }
        off[n] = run;
    }
    __syncthreads();
    int32_t run = s_sum[threadIdx.x];
    for (int64_t i = i0; i < i0 + per && i < n; ++i) {
        off[i] = run;
        run += cnt[i];
    }
}

__global__ void __launch_bounds__(ROW_THREADS) k_pside_weights(const int32_t* pcells, const int32_t* off,
                                                               const uint32_t* rowptr, const SideRec* side,
                                                               const d4* side64, int nd, const double* om64,
                                                               const double* w64, double* wa, int32_t* partner, int4* rec,
                                                               DcTabs dc) {
    const int64_t k = blockIdx.x;
    const int32_t c = pcells[k];
    const uint32_t r0 = rowptr[c], r1 = rowptr[c + 1];
    if (threadIdx.x == 0) rec[k] = make_int4(c, off[k], off[k + 1], 0);
    for (int d = threadIdx.x; d < nd; d += ROW_THREADS) {
        int64_t j = off[k];
        for (uint32_t s = r0; s < r1; ++s) {
            const int32_t x = side[s].hi.x;
            if (x < 0 || !(x & NBR_PERIODIC)) continue;
            const d4 n = side64[s];
            const double t = exact_t(n, om64 + 3 * d);
            double v = t < 0.0 ? dmul(w64[d], dmul(n.w, fabs(t))) : 0.0;
            if (dc.mask && t < 0.0) {  // scheme (b): the partner's share, if the partner chose this face
                const int64_t i = (int64_t)(x & NBR_MASK) * nd + d;
                v = ((dc.mask[i] >> dc.twin[s]) & 1ull) ? dmul(w64[d], dc.share64[i]) : 0.0;
            }
            wa[j * nd + d] = v;
            if (d == 0) partner[j] = x & NBR_MASK;
            ++j;
        }
    }
}

// Periodic iteration (Sec. 2.7): the inflow j^n of one periodic cell, per group, summed over the directions and its
// periodic sides of the partner cells' intensities, and the relative change E = |j^n - j^(n-1)| / (j^n + j^(n-1))
// (Eq. relativeErrorPbc). Writes jn1, and the sum over groups and the largest of the cell's E into partial[2k],
// partial[2k+1]. One block per cell, a direction per thread; what bounds it is the chain of dependent loads (record,
// partners and weights, intensities) and the FP64 pipe, so four sides are in flight per thread, groups are a template
// argument (GC = 0: a number up to 8 known at run time) read as one vector, and the sum over the threads is taken by
// one warp from shared memory (8 FP64 instructions a group, 20 with a butterfly in every warp). With its
// reduction, per iteration of 2,097,344 cells, 128 directions: 0.75 ms before, 0.37 now; of 108,027 cells, 48 directions, 2 groups: 0.16 ms before, 0.075 now.
template <typename real, int GC>
__global__ void __launch_bounds__(ROW_THREADS) k_periodic_source(const int4* rec, const int32_t* partner, const double* wa,
                                                                 const real* I, int64_t N, int G, int nd, double* jn1,
                                                                 const double* jn, double* partial) {
    constexpr int M = GC > 0 ? GC : 8;
    constexpr int U = GC > 0 ? 4 : 1;
    const int Gn = GC > 0 ? GC : G;
    struct alignas(GC > 0 && sizeof(real) * M <= 16 ? sizeof(real) * M : sizeof(real)) Vec {
        real x[M];
    };
    __shared__ double sh[M][ROW_THREADS];
    const int64_t k = blockIdx.x;
    const int4 r = rec[k];
    const int lane = threadIdx.x;
    const double jold = lane < Gn ? jn[(size_t)r.x * Gn + lane] : 0.0;
    double j[M];
#pragma unroll
    for (int g = 0; g < M; ++g) j[g] = 0.0;
    for (int d = threadIdx.x; d < nd; d += blockDim.x) {
        const real* Id = I + (size_t)d * N * Gn;
        for (int q = r.y; q < r.z; q += U) {
            double w[U];
            int32_t nb[U];
            Vec v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const bool in = q + u < r.z;
                w[u] = in ? wa[(size_t)(q + u) * nd + d] : 0.0;
                nb[u] = in ? partner[q + u] : 0;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (!__double_as_longlong(w[u])) continue;  // no inflow side for this direction
                const real* src = Id + (size_t)nb[u] * Gn;
                if constexpr (GC > 0) {
                    v[u] = *reinterpret_cast<const Vec*>(src);
                } else {
#pragma unroll
                    for (int g = 0; g < M; ++g) v[u].x[g] = g < Gn ? src[g] : (real)0;
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (!__double_as_longlong(w[u])) continue;
#pragma unroll
                for (int g = 0; g < M; ++g) j[g] = fma(w[u], widen(v[u].x[g]), j[g]);
            }
        }
    }
#pragma unroll
    for (int g = 0; g < M; ++g) sh[g][threadIdx.x] = j[g];
    __syncthreads();
    if (threadIdx.x >= 32) return;
    double jt = 0.0;  // lane g: the sum of group g
#pragma unroll
    for (int g = 0; g < M; ++g) {
        if (g >= Gn) break;
        double t = sh[g][lane];
        for (int i = lane + 32; i < (int)blockDim.x; i += 32) t += sh[g][i];
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == g) jt = t;
    }
    double e = 0.0;
    if (lane < Gn) {
        const double s = jt + jold;
        e = s > 0.0 ? fabs(jt - jold) / s : 0.0;
        jn1[(size_t)r.x * Gn + lane] = jt;
    }
    double esum = 0.0, emax = 0.0;
#pragma unroll
    for (int g = 0; g < M; ++g) {
        const double x = __shfl_sync(0xffffffffu, e, g);
        if (g >= Gn) break;
        esum += x;
        if (x > emax) emax = x;
    }
    if (lane == 0) *reinterpret_cast<double2*>(partial + 2 * k) = make_double2(esum, emax);
}

// One source iteration's update (Alg. 1): J from the sweep's intensities, its largest relative change against
// the last J (0/0 none, x/0 infinite), and the source of the next sweep, q = eps/4pi + kappa_s V J. The FP64
// sum over the directions bounds it (see the head of this file); J is read and written once, where the
// tally, the change and the source in three kernels took 1.19 ms for 2^18 cells, 4 groups, 96 directions; now 0.42 ms.
template <typename real>
__global__ void __launch_bounds__(256) k_scat_update(const real* I, int64_t N, int G, int nd, const double* w64, const double* vol,
                                                     const double* ks, const double* em, double* Jold, float2* cm32,
                                                     double2* cm64, unsigned long long* dmax) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double e = 0.0;
    if (i < N * G) {
        const double J = over_4pi(weighted_sum(I + i, (size_t)N * G, nd, w64));
        const double dj = fabs(J - Jold[i]);
        if (dj != 0.0) e = J > 0.0 ? dj / J : (double)INFINITY;
        Jold[i] = J;
        const double q = dadd(over_4pi(em[i]), dmul(dmul(ks[i], vol[i / G]), J));
        if (cm64) cm64[i].x = q;
        if (cm32) cm32[i].x = (float)q;
    }
    block_max(e, dmax);
}

// Sums of n pairs in a fixed order, or with MAX the sum of the first and the largest of the (non-negative) second,
// raised into *dmax. A cluster of blocks of 1024 threads, two accumulators per thread and pair, a shared-memory tree per
// block; rank 0 adds the blocks' results in their order through distributed shared memory: one
// block of 1024 threads took 66 us for 100,000 pairs, bound by the loads it can have in flight. From 2049 pairs on
// a cluster of eight is launched; below, one block holds all pairs in two loads a thread (up to 1024 pairs: 256 threads
// in four).
constexpr int RED_THREADS = 1024, RED_CLUSTER = 8;
template <bool MAX>
__global__ void __launch_bounds__(RED_THREADS) k_reduce_pairs(const double* partial, int n, double* out,
                                                              unsigned long long* dmax) {
    __shared__ double s0[RED_THREADS], s1[RED_THREADS];
    const int T = (int)(gridDim.x * blockDim.x);
    const double2* p = reinterpret_cast<const double2*>(partial);
    double a[4] = {0.0, 0.0, 0.0, 0.0}, b[4] = {0.0, 0.0, 0.0, 0.0};
    const auto join = [](double x, double y) { return MAX ? (x > y ? x : y) : x + y; };
    for (int i = (int)(blockIdx.x * blockDim.x + threadIdx.x); i < n; i += 4 * T) {
        double2 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = i + u * T < n ? p[i + u * T] : make_double2(0.0, 0.0);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            a[u] += v[u].x;
            b[u] = join(b[u], v[u].y);
        }
    }
    s0[threadIdx.x] = (a[0] + a[1]) + (a[2] + a[3]);
    s1[threadIdx.x] = join(join(b[0], b[1]), join(b[2], b[3]));
    __syncthreads();
    for (int off = (int)blockDim.x / 2; off >= 32; off >>= 1) {
        if (threadIdx.x < off) {
            s0[threadIdx.x] += s0[threadIdx.x + off];
            s1[threadIdx.x] = join(s1[threadIdx.x], s1[threadIdx.x + off]);
        }
        __syncthreads();
    }
    if (threadIdx.x < 32) {
        double x = s0[threadIdx.x], y = s1[threadIdx.x];
        for (int o = 16; o > 0; o >>= 1) {
            x += __shfl_xor_sync(0xffffffffu, x, o);
            y = join(y, __shfl_xor_sync(0xffffffffu, y, o));
        }
        if (threadIdx.x == 0) {
            s0[0] = x;
            s1[0] = y;
        }
    }
    const cg::cluster_group cl = cg::this_cluster();
    if (gridDim.x > 1) cl.sync();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        double x = s0[0], y = s1[0];
        for (unsigned r = 1; r < gridDim.x; ++r) {
            x += *cl.map_shared_rank(&s0[0], r);
            y = join(y, *cl.map_shared_rank(&s1[0], r));
        }
        out[0] = x;
        out[1] = MAX ? 0.0 : y;
        if (MAX && y > 0.0) atomicMax(dmax, (unsigned long long)__double_as_longlong(y));
    }
    if (gridDim.x > 1) cl.sync();  // rank 0 has read the others' shared memory
}

// lambda of group g = lambda+ (group g) - lambda- (group G+g) of the split adjoint sweep. With
// scattering (J != nullptr) also dL/dkappa_s = V sum_d lambda_d (J - I_d).
template <typename real>
__global__ void k_grad(const real* I, const real* lam, int64_t N, int G, int nd, const double* w64, const double* vol,
                       const double* dlg, const double* J, double* gk, double* ge, double* gks) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N * G) return;
    int64_t c = i / G;
    int g = (int)(i - c * G);
    const double V = vol[c], rg = dlg ? dlg[i] : 0.0, Jc = J ? J[i] : 0.0;
    // sums over the directions of I (w dL/dGamma - lambda), lambda and lambda (J - I); V and 4 pi stand outside
    double sk = 0.0, se = 0.0, ss = 0.0;
    const size_t N2 = (size_t)N * G, o = (size_t)c * (2 * G) + g;
#pragma unroll 4
    for (int d = 0; d < nd; ++d) {
        const double Icd = mag(I + (size_t)d * N2 + i);
        const real* lp = lam + (size_t)d * (2 * N2) + o;
        const double lcd = mag(lp) - mag(lp + G);
        sk = fma(Icd, fma(__ldg(w64 + d), rg, -lcd), sk);
        se = dadd(se, lcd);
        if (J) ss = fma(lcd, Jc - Icd, ss);
    }
    gk[i] = dadd(gk[i], dmul(V, sk));
    ge[i] = dadd(ge[i], over_4pi(se));
    if (J && gks) gks[i] = dmul(V, ss);
}

// Transposed iteration: mu+- = sum_d lambda+-_d (no direction weight: the reverse sweep puts w_d on
// its source), the largest change and the largest magnitude of mu = mu+ - mu- (dmax[0], dmax[1]), and
// the split sources of the next transposed sweep, g+- + kappa_s V mu+- / 4pi (ks may be null).
template <typename real>
__global__ void k_adj_mu(const real* lam, int64_t N, int G, int nd, const double* vol, const double* ka,
                         const double* ks, const double* dlj, const double* dlg, double* mu, float2* cm32,
                         double2* cm64, unsigned long long* dmax) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    double change = 0.0, size = 0.0;
    if (i < N * G) {
        const int64_t c = i / G;
        const int g = (int)(i - c * G);
        const size_t G2 = 2 * (size_t)G, o = (size_t)c * G2;
        double sp = 0.0, sm = 0.0;
#pragma unroll 8
        for (int d = 0; d < nd; ++d) {
            const real* lp = lam + (size_t)d * N * G2 + o;
            sp = dadd(sp, mag(lp + g));
            sm = dadd(sm, mag(lp + G + g));
        }
        change = fabs((sp - sm) - (mu[o + g] - mu[o + G + g]));
        size = fabs(sp - sm);
        mu[o + g] = sp;
        mu[o + G + g] = sm;
        double V = vol[c];
        double src = dadd(dlg ? dmul(dmul(dlg[i], ka[i]), V) : 0.0, dlj ? over_4pi(dlj[i]) : 0.0);
        double gp = src > 0.0 ? src : 0.0, gm = src < 0.0 ? -src : 0.0;
        double kv = ks ? dmul(ks[i], V) : 0.0;
        double qp = dadd(gp, over_4pi(dmul(kv, sp))), qm = dadd(gm, over_4pi(dmul(kv, sm)));
        double dnm = dmul(dadd(ka[i], ks ? ks[i] : 0.0), V);
        if (cm64) {
            cm64[o + g] = make_double2(qp, dnm);
            cm64[o + G + g] = make_double2(qm, dnm);
        }
        if (cm32) {
            cm32[o + g] = make_float2((float)qp, (float)dnm);
            cm32[o + G + g] = make_float2((float)qm, (float)dnm);
        }
    }
    block_max(change, dmax);
    block_max(size, dmax + 1);
}

__global__ void k_fill_u32(uint32_t* p, uint32_t v, int64_t n) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = v;
}

template <typename real>
__global__ void k_to_f64(const real* I, int64_t n, double* out) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = fabs((double)I[i]);
}

inline unsigned nb(int64_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

}  // namespace

cudaError_t launch_prep_material(int64_t N, int G, const double* vol, const double* ka, const double* ks,
                                 const double* em, const double* J, float2* cm32, double2* cm64, cudaStream_t st) {
    if (N * G > 0) k_prep_material<<<nb(N * G), 256, 0, st>>>(N, G, vol, ka, ks, em, J, cm32, cm64);
    return cudaGetLastError();
}

cudaError_t launch_prep_adjoint_src(int64_t N, int G, const double* vol, const double* ka, const double* ks,
                                    const double* dl_dJ, const double* dl_dG, float2* cm32, double2* cm64,
                                    cudaStream_t st) {
    if (N * G > 0) k_prep_adjoint<<<nb(N * G), 256, 0, st>>>(N, G, vol, ka, ks, dl_dJ, dl_dG, cm32, cm64);
    return cudaGetLastError();
}

cudaError_t launch_tally(int precision, const void* I, int64_t N, int G, int nd, int d0, const double* w64,
                         double wsum, const double* vol, const double* ka, const double* em, double* J, double* Gam,
                         double* partial, cudaStream_t st) {
    unsigned b = nb(N * G);
    if (b == 0) b = 1;
    if (precision == 64)
        k_tally<double><<<b, 256, 0, st>>>((const double*)I, N, G, nd, w64 + d0, wsum, vol, ka, em, J, Gam, partial);
    else
        k_tally<float><<<b, 256, 0, st>>>((const float*)I, N, G, nd, w64 + d0, wsum, vol, ka, em, J, Gam, partial);
    return cudaGetLastError();
}

cudaError_t launch_boundary_tally(int precision, const DevMesh& m, const void* I, int G, int nd, int d0,
                                  const double* om64, const double* w64, const double* bc, double* partial,
                                  cudaStream_t st, const DcTabs* dc) {
    const DcTabs tabs = dc ? *dc : DcTabs();
    if (m.n_bcells <= 0) return cudaSuccess;
    const unsigned b = (unsigned)m.n_bcells;
    if (precision == 64)
        k_boundary_tally<double><<<b, ROW_THREADS, 0, st>>>(m.bcells, m.rowptr, m.side, m.side64, (const double*)I,
                                                            m.N, G, nd, om64 + 3 * d0, w64 + d0, bc, partial, tabs);
    else
        k_boundary_tally<float><<<b, ROW_THREADS, 0, st>>>(m.bcells, m.rowptr, m.side, m.side64, (const float*)I,
                                                           m.N, G, nd, om64 + 3 * d0, w64 + d0, bc, partial, tabs);
    return cudaGetLastError();
}

cudaError_t launch_scat_update(int precision, const void* I, int64_t N, int G, int nd, const double* w64, const double* vol,
                               const double* ks, const double* em, double* Jold, float2* cm32, double2* cm64,
                               unsigned long long* d_max, cudaStream_t st) {
    if (N * G <= 0) return cudaSuccess;
    if (precision == 64)
        k_scat_update<double><<<nb(N * G), 256, 0, st>>>((const double*)I, N, G, nd, w64, vol, ks, em, Jold, nullptr, cm64, d_max);
    else
        k_scat_update<float><<<nb(N * G), 256, 0, st>>>((const float*)I, N, G, nd, w64, vol, ks, em, Jold, cm32, nullptr, d_max);
    return cudaGetLastError();
}

cudaError_t build_periodic_table(const DevMesh& m, int nd, const double* om64, const double* w64, PeriodicTable* t,
                                 cudaStream_t st, const DcTabs* dc) {
    if (m.n_pcells <= 0) return cudaSuccess;
    const int64_t np = m.n_pcells;
    cudaError_t e;
    if (t->off_cap < (size_t)(2 * (np + 1))) {
        if (t->off) dev_free(t->off);
        t->off = nullptr;
        t->off_cap = 0;
        if ((e = dev_alloc(&t->off, sizeof(int32_t) * 2 * (np + 1)))) return e;
        t->off_cap = 2 * (np + 1);
    }
    if (t->rec_cap < (size_t)np) {
        if (t->rec) dev_free(t->rec);
        t->rec = nullptr;
        t->rec_cap = 0;
        if ((e = dev_alloc(&t->rec, sizeof(int4) * np))) return e;
        t->rec_cap = (size_t)np;
    }
    int32_t* cnt = t->off + (np + 1);
    k_pside_count<<<nb(np), 256, 0, st>>>(m.pcells, np, m.rowptr, m.side, cnt);
    k_scan_counts<<<1, 1024, 0, st>>>(cnt, np, t->off);
    int32_t total = 0;
    if ((e = cudaMemcpyAsync(&total, t->off + np, sizeof total, cudaMemcpyDeviceToHost, st))) return e;
    if ((e = cudaStreamSynchronize(st))) return e;
    const size_t sides = (size_t)(total > 0 ? total : 1), need = sides * nd;
    if (t->partner_cap < sides) {
        if (t->partner) dev_free(t->partner);
        t->partner = nullptr;
        t->partner_cap = 0;
        if ((e = dev_alloc(&t->partner, sizeof(int32_t) * sides))) return e;
        t->partner_cap = sides;
    }
    if (t->wa_cap < need) {
        if (t->wa) dev_free(t->wa);
        t->wa = nullptr;
        t->wa_cap = 0;
        if ((e = dev_alloc(&t->wa, sizeof(double) * need))) return e;
        t->wa_cap = need;
    }
    k_pside_weights<<<(unsigned)np, ROW_THREADS, 0, st>>>(m.pcells, t->off, m.rowptr, m.side, m.side64, nd, om64, w64,
                                                          t->wa, t->partner, t->rec, dc ? *dc : DcTabs());
    return cudaGetLastError();
}

namespace {
template <typename real>
cudaError_t periodic_source(const DevMesh& m, const real* I, int G, int nd, double* jn1, const double* jn, double* partial,
                            cudaStream_t st, const PeriodicTable& t) {
    const unsigned b = (unsigned)m.n_pcells;
    const int threads = nd >= ROW_THREADS ? ROW_THREADS : (nd + 31) / 32 * 32;
    auto go = [&](auto gc) {
        k_periodic_source<real, decltype(gc)::value>
            <<<b, threads, 0, st>>>(t.rec, t.partner, t.wa, I, m.N, G, nd, jn1, jn, partial);
    };
    if (G == 1) go(std::integral_constant<int, 1>());
    else if (G == 2) go(std::integral_constant<int, 2>());
    else if (G == 4) go(std::integral_constant<int, 4>());
    else go(std::integral_constant<int, 0>());
    return cudaGetLastError();
}
template <bool MAX>
cudaError_t reduce_pairs(const double* partial, int n, double* out, unsigned long long* dmax, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = n > 2 * RED_THREADS ? RED_CLUSTER : 1;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(at[0].val.clusterDim.x);
    cfg.blockDim = dim3(n > RED_THREADS ? RED_THREADS : RED_THREADS / 4);
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_reduce_pairs<MAX>, partial, n, out, dmax);
}
}  // namespace

cudaError_t launch_periodic_source(int precision, const DevMesh& m, const void* I, int G, int nd, double* jn1,
                                   const double* jn, double* partial, cudaStream_t st, const PeriodicTable& tab) {
    if (m.n_pcells <= 0) return cudaSuccess;
    if (precision == 64) return periodic_source(m, (const double*)I, G, nd, jn1, jn, partial, st, tab);
    return periodic_source(m, (const float*)I, G, nd, jn1, jn, partial, st, tab);
}

cudaError_t launch_reduce_sum(const double* partial, int n, double* out, cudaStream_t st) {
    return reduce_pairs<false>(partial, n, out, nullptr, st);
}

cudaError_t launch_reduce_change(const double* partial, int n, double* out, unsigned long long* d_max, cudaStream_t st) {
    return reduce_pairs<true>(partial, n, out, d_max, st);
}

cudaError_t launch_grad_accum(int precision, const void* I, const void* lam, int64_t N, int G, int nd, int d0,
                              const double* w64, const double* vol, const double* dl_dG, double* gk, double* ge,
                              cudaStream_t st) {
    return launch_grad_scat(precision, I, lam, N, G, nd, d0, w64, vol, dl_dG, nullptr, gk, ge, nullptr, st);
}

cudaError_t launch_grad_scat(int precision, const void* I, const void* lam, int64_t N, int G, int nd, int d0,
                             const double* w64, const double* vol, const double* dl_dG, const double* J, double* gk,
                             double* ge, double* gks, cudaStream_t st) {
    if (N * G <= 0) return cudaSuccess;
    if (precision == 64)
        k_grad<double><<<nb(N * G), 256, 0, st>>>((const double*)I, (const double*)lam, N, G, nd, w64 + d0, vol,
                                                  dl_dG, J, gk, ge, gks);
    else
        k_grad<float><<<nb(N * G), 256, 0, st>>>((const float*)I, (const float*)lam, N, G, nd, w64 + d0, vol, dl_dG,
                                                 J, gk, ge, gks);
    return cudaGetLastError();
}

cudaError_t launch_adjoint_mu(int precision, const void* lam, int64_t N, int G, int nd, const double* vol,
                              const double* ka, const double* ks, const double* dl_dJ, const double* dl_dG,
                              double* mu, float2* cm32, double2* cm64, unsigned long long* d_max, cudaStream_t st) {
    if (N * G <= 0) return cudaSuccess;
    if (precision == 64)
        k_adj_mu<double><<<nb(N * G), 256, 0, st>>>((const double*)lam, N, G, nd, vol, ka, ks, dl_dJ, dl_dG, mu,
                                                    cm32, cm64, d_max);
    else
        k_adj_mu<float><<<nb(N * G), 256, 0, st>>>((const float*)lam, N, G, nd, vol, ka, ks, dl_dJ, dl_dG, mu, cm32,
                                                   cm64, d_max);
    return cudaGetLastError();
}

cudaError_t launch_fill_u32(uint32_t* p, uint32_t v, int64_t n, cudaStream_t st) {
    if (n > 0) k_fill_u32<<<nb(n), 256, 0, st>>>(p, v, n);
    return cudaGetLastError();
}

cudaError_t launch_to_f64(int precision, const void* I, int64_t n, double* out, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    if (precision == 64) k_to_f64<double><<<nb(n), 256, 0, st>>>((const double*)I, n, out);
    else k_to_f64<float><<<nb(n), 256, 0, st>>>((const float*)I, n, out);
    return cudaGetLastError();
}

}  // namespace sw

// ---------------------------------------------------------------------------------------------
// Rotation of the direction set (the rotation paragraph of Sec. 2.6): the remap coefficients
// c_ij = dS_ij / dS_i between the bins of the new directions i and the old directions j, by a
// quadrature of equal-weight points on the unit sphere, and the remap of the stored intensities
// I(Omega'_i) = sum_j c_ij I(Omega_j).
// ---------------------------------------------------------------------------------------------
namespace sw {
namespace {

// the direction (of n_dir) nearest to p: largest ((px Ox) + (py Oy)) + (pz Oz), ties to the lower index
__device__ __forceinline__ int nearest_dir(const double3 p, const double* om, int n_dir) {
    int best = 0;
    double bd = -2.0;
    for (int d = 0; d < n_dir; ++d) {
        const double t = __dadd_rn(__dadd_rn(__dmul_rn(p.x, om[3 * d]), __dmul_rn(p.y, om[3 * d + 1])),
                                   __dmul_rn(p.z, om[3 * d + 2]));
        if (t > bd) {
            bd = t;
            best = d;
        }
    }
    return best;
}

__global__ void k_remap_count(const double3* pts, int64_t n, const double* om_old, const double* om_new, int n_dir,
                              unsigned long long* cnt) {
    extern __shared__ double s_om[];  // [2][n_dir][3]
    for (int i = threadIdx.x; i < 6 * n_dir; i += blockDim.x) s_om[i] = i < 3 * n_dir ? om_new[i] : om_old[i - 3 * n_dir];
    __syncthreads();
    const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= n) return;
    const double3 p = pts[m];
    const int i = nearest_dir(p, s_om, n_dir);
    const int j = nearest_dir(p, s_om + 3 * n_dir, n_dir);
    atomicAdd(&cnt[(int64_t)i * n_dir + j], 1ull);
}

// out[i][c][g] = sum over the nonzeros (j, c_ij) of row i of c_ij |in[j][c][g]|, written with the sign
// bit `par` (the parity the buffer's values carry); one thread per (cell, group) element
template <typename real>
__global__ void k_remap(const real* in, real* out, int64_t NG, int n_dir, const int32_t* rp, const int32_t* col,
                        const double* val, int par) {
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= NG) return;
    for (int i = 0; i < n_dir; ++i) {
        double acc = 0.0;
        for (int k = rp[i]; k < rp[i + 1]; ++k)
            acc = __dadd_rn(acc, __dmul_rn(val[k], fabs((double)in[(int64_t)col[k] * NG + e])));
        const real v = (real)acc;
        out[(int64_t)i * NG + e] = par ? -v : v;
    }
}

}  // namespace

cudaError_t launch_remap_count(const double3* pts, int64_t n, const double* om_old, const double* om_new, int n_dir,
                               unsigned long long* cnt, cudaStream_t st) {
    if (n > 0)
        k_remap_count<<<(unsigned)((n + 255) / 256), 256, sizeof(double) * 6 * n_dir, st>>>(pts, n, om_old, om_new,
                                                                                            n_dir, cnt);
    return cudaGetLastError();
}

cudaError_t launch_remap(int precision, const void* in, void* out, int64_t NG, int n_dir, const int32_t* rp,
                         const int32_t* col, const double* val, int par, cudaStream_t st) {
    if (NG <= 0) return cudaSuccess;
    const unsigned b = (unsigned)((NG + 255) / 256);
    if (precision == 64)
        k_remap<double><<<b, 256, 0, st>>>((const double*)in, (double*)out, NG, n_dir, rp, col, val, par);
    else
        k_remap<float><<<b, 256, 0, st>>>((const float*)in, (float*)out, NG, n_dir, rp, col, val, par);
    return cudaGetLastError();
}

}  // namespace sw
