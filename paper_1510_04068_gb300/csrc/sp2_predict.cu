// sp2_predict.cu -- O(N) kernels around the pairwise passes: the copy
// (scatter) kernel and the Taylor predictor of Sec. 2.2.4, the record packing
// for the all-pairs entry points, and the element-wise parts of the shared
// time-step Hermite-4 step and its reverse.
//
// The predictor is memory bound (it reads ~116-140 B and writes 48-96 B per
// particle).  It evaluates each Taylor sum left to right with explicitly
// rounded multiplies and adds (no fused multiply-add), dt^k/k! formed as dt^k
// times the double nearest 1/k!, so the predicted FP64 values are those of a
// plain IEEE evaluation of the polynomial.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "sp2_ds.cuh"
#include "sp2_internal.h"
#include "sp2_launch.cuh"

namespace sp2 {
namespace {

constexpr int kThreads = 256;
// The per-particle kernels with FP64 arithmetic and conversions (an SM retires
// 2 FP64 operations a clock) take small CTAs, so that a few thousand particles
// reach every SM.
constexpr int kSmallThreads = 64;
constexpr double kBlockDtMin = 1.0 / (1ll << 50);  // smallest block step (2^-50)

inline unsigned grid_small(int64_t n) { return static_cast<unsigned>((n + kSmallThreads - 1) / kSmallThreads); }
inline unsigned grid_for(int64_t n) { return static_cast<unsigned>((n + kThreads - 1) / kThreads); }
// FP64-heavy per-particle kernels over a few hundred active particles: one
// warp per CTA spreads them over the SMs (an SM retires 2 FP64 FMAs a clock)
constexpr int kWarpCta = 32;
// (256, 2048 or as many CTAs as the particles need: block runs of 4096 and 65536
// particles differ by less than two runs of one of them)
constexpr unsigned kCorrectMaxCtas = 2048;
inline unsigned grid_for_warps(int64_t n) { return static_cast<unsigned>((n + kWarpCta - 1) / kWarpCta); }

__device__ __forceinline__ double dmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double dadd(double a, double b) { return __dadd_rn(a, b); }


__device__ __forceinline__ void store_mixed(unsigned char *rec, int rb, int64_t j, const double *xp,
                                            const double *vp, const double *ap, double m, int id) {
    float xh[3], xl[3];
    for (int c = 0; c < 3; ++c) {
        const ds q = ds_split(xp[c]);  // hi = fl32(x), lo = fl32(x - hi)
        xh[c] = q.h;
        xl[c] = q.l;
    }
    float4 *o = reinterpret_cast<float4 *>(rec + j * rb);
    o[0] = make_float4(xh[0], xh[1], xh[2], __double2float_rn(m));
    o[1] = make_float4(xl[0], xl[1], xl[2], __int_as_float(id));
    o[2] = make_float4(__double2float_rn(vp[0]), __double2float_rn(vp[1]), __double2float_rn(vp[2]), 0.f);
    if (ap) o[3] = make_float4(__double2float_rn(ap[0]), __double2float_rn(ap[1]), __double2float_rn(ap[2]), 0.f);
}

__device__ __forceinline__ void store_fp64(unsigned char *rec, int rb, int64_t j, const double *xp,
                                           const double *vp, const double *ap, double m, int id) {
    double2 *o = reinterpret_cast<double2 *>(rec + j * rb);
    o[0] = make_double2(xp[0], xp[1]);
    o[1] = make_double2(xp[2], m);
    o[2] = make_double2(vp[0], vp[1]);
    o[3] = make_double2(vp[2], __longlong_as_double(static_cast<long long>(id)));
    if (ap) {
        o[4] = make_double2(ap[0], ap[1]);
        o[5] = make_double2(ap[2], 0.0);
    }
}

__device__ __forceinline__ void write_dscache(const JStore &d, int64_t s) {
    float4 *o = d.dsc + s * ((d.sn != nullptr) ? 8 : 7);
    const ds x0 = ds_split(d.x[3 * s]), x1 = ds_split(d.x[3 * s + 1]), x2 = ds_split(d.x[3 * s + 2]);
    const ds v0 = ds_split(d.v[3 * s]), v1 = ds_split(d.v[3 * s + 1]), v2 = ds_split(d.v[3 * s + 2]);
    const ds a0 = ds_split(d.a[3 * s]), a1 = ds_split(d.a[3 * s + 1]), a2 = ds_split(d.a[3 * s + 2]);
    const ds tt = ds_split(d.t[s]);
    o[0] = make_float4(x0.h, x1.h, x2.h, __double2float_rn(d.m[s]));
    o[1] = make_float4(x0.l, x1.l, x2.l, tt.h);
    o[2] = make_float4(v0.h, v1.h, v2.h, tt.l);
    o[3] = make_float4(v0.l, v1.l, v2.l, __int_as_float(d.id[s]));
    o[4] = make_float4(a0.h, a1.h, a2.h, 0.f);
    o[5] = make_float4(a0.l, a1.l, a2.l, 0.f);
    o[6] = make_float4(__double2float_rn(d.jk[3 * s]), __double2float_rn(d.jk[3 * s + 1]),
                       __double2float_rn(d.jk[3 * s + 2]), 0.f);
    if (d.sn)
        o[7] = make_float4(__double2float_rn(d.sn[3 * s]), __double2float_rn(d.sn[3 * s + 1]),
                           __double2float_rn(d.sn[3 * s + 2]), 0.f);
}

// The copy and the cache refresh take four threads per particle: threads 0-2
// one component of every vector, thread 3 the scalars (m, t, id).  Each loads
// all its values before its first store (the arrays may alias for all the
// compiler knows, so a loop over the components would put a memory round trip
// behind every store), the FP64 conversions of a particle run in four lanes
// at once, and a warp's cache stores are whole 16-byte words.  Small CTAs
// spread a block of a few hundred particles over the SMs.
// Latency bound; a block step of one particle on 131072 sources 28.2 -> 25.5 us,
// of 1000 on 100003 190 -> 182 us (the copy of 1000 took 13 us under ncu).
constexpr int kLanesPerParticle = 4;
inline unsigned grid_for_store(int64_t n) {
    return static_cast<unsigned>((n * kLanesPerParticle + kSmallThreads - 1) / kSmallThreads);
}

// one lane's column of the particle's cache words (layout: write_dscache)
__device__ __forceinline__ void write_dscache_vec(const JStore &d, int64_t s, int c, double x, double v, double a,
                                                  double jk, double sn) {
    float *o = reinterpret_cast<float *>(d.dsc + s * ((d.sn != nullptr) ? 8 : 7)) + c;
    const ds X = ds_split(x), V = ds_split(v), A = ds_split(a);
    o[0] = X.h;
    o[4] = X.l;
    o[8] = V.h;
    o[12] = V.l;
    o[16] = A.h;
    o[20] = A.l;
    o[24] = __double2float_rn(jk);
    if (d.sn) o[28] = __double2float_rn(sn);
}
__device__ __forceinline__ void write_dscache_scalars(const JStore &d, int64_t s, double m, double t, int id) {
    float *o = reinterpret_cast<float *>(d.dsc + s * ((d.sn != nullptr) ? 8 : 7)) + 3;
    const ds T = ds_split(t);
    o[0] = __double2float_rn(m);
    o[4] = T.h;
    o[8] = T.l;
    o[12] = __int_as_float(id);
    o[16] = 0.f;
    o[20] = 0.f;
    o[24] = 0.f;
    if (d.sn) o[28] = 0.f;
}

__global__ void __launch_bounds__(kSmallThreads) dscache_kernel(JStore d, int64_t first, int64_t n) {
    grid_wait();
    const int64_t g = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    const int64_t s = first + g / kLanesPerParticle;
    const int c = static_cast<int>(g % kLanesPerParticle);
    if (s >= first + n) return;
    if (c == 3) {
        write_dscache_scalars(d, s, d.m[s], d.t[s], d.id[s]);
        return;
    }
    const int64_t q = 3 * s + c;
    write_dscache_vec(d, s, c, d.x[q], d.v[q], d.a[q], d.jk[q], d.sn ? d.sn[q] : 0.0);
}

// Block times are compared through an unsigned key that orders like the
// doubles (negative times included): the sign bit flipped for t >= 0, every bit
// for t < 0; all ones (the empty minimum) decodes to NaN.
__device__ __forceinline__ unsigned long long time_key(double t) {
    const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(t));
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double key_time(unsigned long long k) {
    const unsigned long long b = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
    return __longlong_as_double(static_cast<long long>(b));
}

// minimum over a warp's lanes into *dst (all ones: nothing to add)
__device__ __forceinline__ void warp_min_to(unsigned long long *dst, unsigned long long v) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, off));
    if ((threadIdx.x & 31) == 0 && v != ~0ull) atomicMin(dst, v);
}

// Block time-steps: the start of block b, run by every thread of the
// prediction (slot j; threads past n take part in the warp's minimum).  The
// block time is in slot b % 4 of the run state; particles due then are
// appended to the active list, and the next due time of all others goes into
// slot (b + 1) % 4, to which the corrector adds the active particles' new
// times: no pass over the particles is spent on finding the next block time.
// The slots of the blocks after that are reset on the way (nothing reads or
// writes them during block b).  Returns false when the run has stopped or the
// block time is past t_end (which stops it: the counts stay 0 and every later
// kernel does nothing).
__device__ __forceinline__ bool block_select(const BlockStep &b, int64_t j, int64_t n, double *t1) {
    BlockDev *bd = b.bd;
    if (j == 0) bd->count[(b.slot + 1) & 3] = 0u;  // (also once stopped: every count must be 0 then)
    if (bd->stop) return false;
    *t1 = key_time(bd->t1bits[b.slot]);
    if (!(*t1 <= b.t_end)) {
        if (j == 0) bd->stop = 1u;
        return false;
    }
    if (j == 0) bd->t1bits[(b.slot + 2) & 3] = ~0ull;
    unsigned long long next = ~0ull;
    if (j < n) {
        const double due = b.t[j] + b.dt[j];
        if (due == *t1) b.active[atomicAdd(&bd->count[b.slot], 1u)] = static_cast<int32_t>(j);
        else next = time_key(due);
    }
    warp_min_to(&bd->t1bits[(b.slot + 1) & 3], next);
    return true;
}

// Mixed-precision predictor on the double-single cache (predict_ds_record).
// BLOCK: to the time of the current block, whose active set it selects.
template <int ORDER, bool BLOCK>
__global__ void predict_ds_kernel(const float4 *dsc, int64_t n, float t_hi, float t_lo, unsigned char *rec,
                                  const BlockStep b) {
    grid_wait();
    const int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if constexpr (BLOCK) {
        double t;
        if (!block_select(b, j, n, &t)) return;
        t_hi = __double2float_rn(t);
        t_lo = __double2float_rn(t - static_cast<double>(t_hi));
    }
    if (j >= n) return;
    float4 o[4];
    predict_ds_record<ORDER>(dsc, j, t_hi, t_lo, o);
    float4 *dst = reinterpret_cast<float4 *>(rec + j * (ORDER == 6 ? 64 : 48));
    dst[0] = o[0];
    dst[1] = o[1];
    dst[2] = o[2];
    if (ORDER == 6) dst[3] = o[3];
}

__global__ void __launch_bounds__(kSmallThreads)
scatter_kernel(JStore d, const int32_t *slots, int64_t n, int64_t n_loaded, unsigned int *err, const int32_t *id,
               const double *m, const double *x, const double *v, const double *a, const double *jk, const double *sn,
               const double *t) {
    grid_wait();
    const int64_t g = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    const int64_t k = g / kLanesPerParticle;
    const int c = static_cast<int>(g % kLanesPerParticle);
    if (k >= n) return;
    // v, a, jk, t may be absent for leap-frog (order 2) sources
    if (c == 3) {
        const int64_t s = slots[k];
        const double mm = m[k], tt = t ? t[k] : 0.0;
        const int32_t ii = id[k];
        if (s < 0 || s >= n_loaded) {  // reported by sp2_sync; the particle is not stored
            atomicOr(err, 1u);
            return;
        }
        d.id[s] = ii;
        d.m[s] = mm;
        d.t[s] = tt;
        if (d.dsc) write_dscache_scalars(d, s, mm, tt, ii);
        return;
    }
    const int64_t p = 3 * k + c;
    const int64_t s = slots[k];
    const double xx = x[p], vv = v ? v[p] : 0.0, aa = a ? a[p] : 0.0, jj = jk ? jk[p] : 0.0, ss = sn ? sn[p] : 0.0;
    if (s < 0 || s >= n_loaded) return;
    const int64_t q = 3 * s + c;
    d.x[q] = xx;
    d.v[q] = vv;
    d.a[q] = aa;
    d.jk[q] = jj;
    if (sn) d.sn[q] = ss;
    if (d.dsc) write_dscache_vec(d, s, c, xx, vv, aa, jj, ss);
}

template <int ORDER, bool MIXED, bool BLOCK>
__global__ void predict_kernel(JStore js, int64_t n, double t, unsigned char *rec, const BlockStep b) {
    grid_wait();
    const int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if constexpr (BLOCK) {
        if (!block_select(b, j, n, &t)) return;
    }
    if (j >= n) return;
    const double c2 = 0.5, c3 = 1.0 / 6.0, c4 = 1.0 / 24.0;
    const double dt = dadd(t, -js.t[j]);
    const double dt2 = dmul(dt, dt);
    const double dt3 = dmul(dt2, dt);
    const double dt4 = dmul(dt3, dt);
    const double h2 = dmul(dt2, c2), h3 = dmul(dt3, c3), h4 = dmul(dt4, c4);
    double xp[3], vp[3], ap[3];
    // Mixed-precision records: Horner form with fused multiply-adds (the
    // double-single split keeps ~48 bits, far more than the evaluation order
    // changes).  FP64 records: left-to-right sums of explicitly rounded
    // products, exactly the plain IEEE evaluation of the Taylor polynomial.
    const double d2 = 0.5 * dt, d3 = dt * (1.0 / 6.0), d4 = dt * (1.0 / 24.0);
    for (int c = 0; c < 3; ++c) {
        const int64_t q = 3 * j + c;
        const double x = js.x[q], v = js.v[q], a = js.a[q], jk = js.jk[q];
        if (ORDER == 2) {  // leap-frog (GRAPE-5): sources are used where they are
            xp[c] = x;
            vp[c] = 0.0;
        } else if (ORDER == 6 && js.cr) {
            // 6th-order block steps: the crackle term too (x to dt^5, v to
            // dt^4, a to dt^3), Horner form in both precisions
            const double s = js.sn[q], cr = js.cr[q];
            const double d5 = dt * (1.0 / 120.0);
            xp[c] = fma(fma(fma(fma(fma(cr, d5, s * (1.0 / 24.0)), dt, jk * (1.0 / 6.0)), dt, 0.5 * a), dt, v), dt, x);
            vp[c] = fma(fma(fma(fma(cr, d4, s * (1.0 / 6.0)), dt, 0.5 * jk), dt, a), dt, v);
            ap[c] = fma(fma(fma(cr, d3, 0.5 * s), dt, jk), dt, a);
        } else if (MIXED && ORDER == 6) {
            const double s = js.sn[q];
            xp[c] = fma(fma(fma(fma(s, d4, jk * (1.0 / 6.0)), dt, 0.5 * a), dt, v), dt, x);
            vp[c] = fma(fma(fma(s, d3, 0.5 * jk), dt, a), dt, v);
            ap[c] = fma(fma(s, d2, jk), dt, a);
        } else if (MIXED) {
            xp[c] = fma(fma(fma(jk, d3, 0.5 * a), dt, v), dt, x);
            vp[c] = fma(fma(jk, d2, a), dt, v);
        } else if (ORDER == 6) {
            const double s = js.sn[q];
            xp[c] = dadd(dadd(dadd(dadd(x, dmul(v, dt)), dmul(a, h2)), dmul(jk, h3)), dmul(s, h4));
            vp[c] = dadd(dadd(dadd(v, dmul(a, dt)), dmul(jk, h2)), dmul(s, h3));
            ap[c] = dadd(dadd(a, dmul(jk, dt)), dmul(s, h2));
        } else {
            xp[c] = dadd(dadd(dadd(x, dmul(v, dt)), dmul(a, h2)), dmul(jk, h3));
            vp[c] = dadd(dadd(v, dmul(a, dt)), dmul(jk, h2));
        }
    }
    const int rb = MIXED ? (ORDER == 6 ? 64 : 48) : (ORDER == 6 ? 96 : 64);
    if (MIXED) store_mixed(rec, rb, j, xp, vp, ORDER == 6 ? ap : nullptr, js.m[j], js.id[j]);
    else store_fp64(rec, rb, j, xp, vp, ORDER == 6 ? ap : nullptr, js.m[j], js.id[j]);
}

template <bool MIXED>
__global__ void pack_state_kernel(int64_t n, const double *m, const double *x, const double *v, unsigned char *rec) {
    grid_wait();
    const int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const double xp[3] = {x[3 * j], x[3 * j + 1], x[3 * j + 2]};
    const double vp[3] = {v[3 * j], v[3 * j + 1], v[3 * j + 2]};
    if (MIXED) store_mixed(rec, 48, j, xp, vp, nullptr, m[j], static_cast<int>(j));
    else store_fp64(rec, 64, j, xp, vp, nullptr, m[j], static_cast<int>(j));
}

// Neighbour lists after the pass: stored slots become ids and each list is
// sorted by id, so a list without overflow has one defined order.  A warp per
// sink: lists of up to kNbShared entries (the usual tens) are read once into
// shared memory and every entry is written straight to its rank (the entries
// below it, counted with broadcast reads; equal ids keep their order); longer
// ones are sorted in place by a bitonic network whose comparators all point
// the same way, so that entries past the end need no padding.  An insertion
// sort by one thread per sink, in place, took 187 us for 16384 lists.
constexpr int kNbShared = 256;
constexpr int kNbWarps = 4;

__global__ void __launch_bounds__(32 * kNbWarps)
nb_finish_kernel(const int32_t *ids, int64_t n_i, int nb_max, const int32_t *count, int32_t *list) {
    grid_wait();
    __shared__ int32_t buf[kNbWarps][kNbShared];
    const int lane = threadIdx.x & 31;
    const int64_t i = static_cast<int64_t>(blockIdx.x) * kNbWarps + (threadIdx.x >> 5);
    if (i >= n_i) return;  // uniform across the warp
    const int c = min(count[i], nb_max);
    int32_t *l = list + i * nb_max;
    if (c <= kNbShared) {
        int32_t *sh = buf[threadIdx.x >> 5];
        for (int k = lane; k < c; k += 32) sh[k] = ids[l[k]];
        __syncwarp();
        for (int k = lane; k < c; k += 32) {
            const int32_t v = sh[k];
            int rank = 0;
            for (int q = 0; q < c; ++q) rank += (sh[q] < v || (sh[q] == v && q < k)) ? 1 : 0;
            l[rank] = v;
        }
        return;
    }
    for (int k = lane; k < c; k += 32) l[k] = ids[l[k]];
    __syncwarp();
    auto order = [&](int p, int q) {
        if (q >= c) return;
        const int32_t a = l[p], b = l[q];
        if (a > b) {
            l[p] = b;
            l[q] = a;
        }
    };
    int half = 1;
    for (int size = 2; half < c; size *= 2, half *= 2) {
        // mirrored step: position p of a block's lower half against the mirror position
        for (int k = lane; k < (c + size - 1) / size * half; k += 32) {
            const int blk = k / half, p = k - blk * half;
            order(blk * size + p, blk * size + size - 1 - p);
        }
        __syncwarp();
        for (int d = half / 2; d > 0; d /= 2) {
            for (int k = lane; k < (c + 2 * d - 1) / (2 * d) * d; k += 32) {
                const int blk = k / d, p = k - blk * d;
                order(blk * 2 * d + p, blk * 2 * d + p + d);
            }
            __syncwarp();
        }
    }
}

// ---- block time-steps (Sec. 3.7: Hermite integration with individual,
// power-of-two time-steps; the integrator around the force pass) ----------
//
// Aarseth's criterion (Aarseth 2003) with the higher derivatives of the
// Hermite interpolation over the last step [t0, t1] (Makino & Aarseth 1992):
//   a2(t0) = (-6 (a0 - a1) - dt (4 j0 + 2 j1)) / dt^2
//   a3     = (12 (a0 - a1) + 6 dt (j0 + j1)) / dt^3
//   a2(t1) = a2(t0) + dt a3
//   dt'    = sqrt(eta (|a1| |a2(t1)| + |j1|^2) / (|j1| |a3| + |a2(t1)|^2))
// quantised to the largest power of two not above dt', at most twice the last
// step and dt_max, and dividing t1 (so the blocks stay synchronised).
__device__ __forceinline__ double norm3(const double *p) { return sqrt(p[0] * p[0] + p[1] * p[1] + p[2] * p[2]); }

__device__ __forceinline__ double quantise_dt(double want, double cap, double t1) {
    double d = cap;
    while (d > want && d > kBlockDtMin) d *= 0.5;
    // d = cap 2^-k divides t1 exactly iff fmod(t1, d) == 0.  With r = t1 / cap
    // (one correctly rounded division), a multiple t1 = m d gives r = m 2^-k
    // exactly for m < 2^53, so q = r 2^k (an exact scaling) is the integer m;
    // above 2^53 every double is an integer.  A fractional q therefore rules d
    // out, and the candidate that survives is confirmed exactly: t1 - q d by
    // one fused multiply-add (zero iff t1 = q d) below 2^53, fmod above.
    double q = (t1 / cap) * (cap / d);
    while (d > kBlockDtMin) {
        if (q == trunc(q)) {
            const bool exact = (fabs(q) < 9007199254740992.0) ? (fma(-q, d, t1) == 0.0) : (fmod(t1, d) == 0.0);
            if (exact) break;
        }
        d *= 0.5;
        q *= 2.0;
    }
    return d;
}

// initial steps at t0 from |a| / |j| (the usual start of a Hermite run)
__global__ void block_init_kernel(JStore js, double *dt, int64_t n, double eta_s, double dt_max, double t0) {
    const int64_t s = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (s >= n) return;
    const double an = norm3(js.a + 3 * s), jn = norm3(js.jk + 3 * s);
    const double want = (jn > 0.0) ? eta_s * an / jn : dt_max;
    dt[s] = quantise_dt(want, dt_max, t0);
    js.t[s] = t0;
}

// Hermite-4 corrector and the next step for the active particles (a1, j1 at
// the predicted state, position k of the active list); the double-single
// cache follows the store.  Four lanes take a particle (FP64 runs at 2 lanes
// a clock per SM, so a few hundred particles are spread over as many lanes as
// there are): lanes c = 0..2 correct component c and lane q forms the norm
// of the q-th of the vectors (a, j, a2, a3); every lane then has all four norms
// and the same new step, which it returns.  Whole groups of four take part.
// (One thread per particle took 15 us for a few hundred particles under ncu:
// one dependent chain of some 250 FP64 operations and seven memory round trips.)
__device__ __forceinline__ double group_get(double v, int src) { return __shfl_sync(0xffffffffu, v, src, 4); }

__device__ __forceinline__ double correct_one(const JStore &js, double *dt, int64_t s, int64_t k, int c, bool valid,
                                              double t1, const double *a1, const double *j1, double eta,
                                              double dt_max) {
    const bool vec = valid && c < 3, scal = valid && c == 3;
    const int64_t q = 3 * s + c, p = 3 * k + c;
    const double t0 = valid ? js.t[s] : 0.0;
    const double x0 = vec ? js.x[q] : 0.0, v0 = vec ? js.v[q] : 0.0;
    const double a0 = vec ? js.a[q] : 0.0, j0 = vec ? js.jk[q] : 0.0;
    const double aa = vec ? a1[p] : 0.0, jj = vec ? j1[p] : 0.0;
    const double m = scal ? js.m[s] : 0.0;
    const int32_t id = scal ? js.id[s] : 0;
    const double h = t1 - t0;
    const double h2 = h * h;
    const double v1 = v0 + (a0 + aa) * (h / 2) + (j0 - jj) * (h2 / 12);
    const double x1 = x0 + (v0 + v1) * (h / 2) + (a0 - aa) * (h2 / 12);
    const double a2_0 = (-6.0 * (a0 - aa) - h * (4.0 * j0 + 2.0 * jj)) / h2;
    const double a3 = (12.0 * (a0 - aa) + 6.0 * h * (j0 + jj)) / (h2 * h);
    const double a2 = a2_0 + h * a3;
    double w[3];
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        const double g0 = group_get(aa, e), g1 = group_get(jj, e), g2 = group_get(a2, e), g3 = group_get(a3, e);
        w[e] = (c == 0) ? g0 : (c == 1) ? g1 : (c == 2) ? g2 : g3;
    }
    const double mine = norm3(w);
    const double A = group_get(mine, 0), J = group_get(mine, 1), A2 = group_get(mine, 2), A3 = group_get(mine, 3);
    const double den = J * A3 + A2 * A2;
    const double want = (den > 0.0) ? sqrt(eta * (A * A2 + J * J) / den) : dt_max;
    const double dn = valid ? quantise_dt(want, fmin(2.0 * h, dt_max), t1) : 0.0;
    if (vec) {
        js.x[q] = x1;
        js.v[q] = v1;
        js.a[q] = aa;
        js.jk[q] = jj;
        if (js.dsc) write_dscache_vec(js, s, c, x1, v1, aa, jj, 0.0);
    }
    if (scal) {
        js.t[s] = t1;
        dt[s] = dn;
        if (js.dsc) write_dscache_scalars(js, s, m, t1, id);
    }
    return dn;
}

// A step at the 2^-50 floor means the criterion has collapsed (Sec. 3.7 notes
// that noisy jerk and snap can drive the step to zero): the run stops after
// this block and the host reports it.
__device__ __forceinline__ void check_underflow(double dt, BlockDev *bd) {
    if (dt <= kBlockDtMin) {
        bd->underflow = 1u;
        bd->stop = 1u;
    }
}

// Explicit sinks (sp2_compute_ext): positions / velocities [/ accelerations]
// given by the caller, packed in the context's record format.
template <int ORDER, bool MIXED>
__global__ void pack_sinks_kernel(int64_t n, const double *x, const double *v, const double *a, unsigned char *rec) {
    const int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (j >= n) return;
    double xp[3], vp[3], ap[3];
    for (int c = 0; c < 3; ++c) {
        xp[c] = x[3 * j + c];
        vp[c] = v ? v[3 * j + c] : 0.0;
        ap[c] = (ORDER == 6) ? a[3 * j + c] : 0.0;
    }
    const int rb = MIXED ? (ORDER == 6 ? 64 : 48) : (ORDER == 6 ? 96 : 64);
    if (MIXED) store_mixed(rec, rb, j, xp, vp, ORDER == 6 ? ap : nullptr, 0.0, -1);
    else store_fp64(rec, rb, j, xp, vp, ORDER == 6 ? ap : nullptr, 0.0, -1);
}

// ---- the same block time-steps driven from the device: the block time,
// the active count and a stop flag live in a BlockDev, so the host can queue
// many blocks without reading anything back.
// The first block time of a run: the smallest t + dt, into slot 0.
__global__ void block_first_kernel(const double *t, const double *dt, int64_t n, BlockDev *bd) {
    const int64_t s = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    warp_min_to(&bd->t1bits[0], s < n ? time_key(t[s] + dt[s]) : ~0ull);
}

// The run's statistics (first thread of a corrector).
__device__ __forceinline__ void count_block(BlockDev *bd, unsigned int n_act, double t1) {
    bd->steps += 1;
    bd->active_sum += n_act;
    bd->max_active = max(bd->max_active, n_act);
    bd->min_active = min(bd->min_active, n_act);
    bd->t_last = t1;
}

__global__ void __launch_bounds__(kWarpCta)
block_correct_dev_kernel(JStore js, const BlockStep b, const double *a1, const double *j1, double eta, double dt_max) {
    grid_wait();
    constexpr int kPer = kWarpCta / kLanesPerParticle;  // particles of a CTA (one warp) at a time
    const unsigned int n_act = b.bd->count[b.slot];
    const double t1 = key_time(b.bd->t1bits[b.slot]);
    if (blockIdx.x == 0 && threadIdx.x == 0 && n_act > 0) count_block(b.bd, n_act, t1);
    const int c = threadIdx.x % kLanesPerParticle;
    unsigned long long next = ~0ull;
    for (unsigned int k0 = blockIdx.x * kPer; k0 < n_act; k0 += gridDim.x * kPer) {  // uniform across the warp
        const unsigned int k = k0 + threadIdx.x / kLanesPerParticle;
        const bool valid = k < n_act;
        const int64_t s = valid ? b.active[k] : 0;
        const double dn = correct_one(js, b.dt, s, k, c, valid, t1, a1, j1, eta, dt_max);
        if (valid) {
            if (c == 3) check_underflow(dn, b.bd);
            next = min(next, time_key(t1 + dn));
        }
    }
    warp_min_to(&b.bd->t1bits[(b.slot + 1) & 3], next);
}

// 6th-order Hermite corrector (Nitadori & Makino 2008) for slot s, position k
// of the active list: the quintic Hermite interpolant of the acceleration
// through (a, j, s) at both ends, integrated once for v and, with (v, a, j),
// for x; its 3rd to 5th derivatives at t1 (crackle, pop, and the constant
// fifth derivative q) follow from the three matching conditions at t1:
//   c1 h^3 = 60 (a1 - a0) - 24 h j0 - 36 h j1 - 3 h^2 s0 + 9 h^2 s1
//   p1 h^4 = 360 (a1 - a0) - 168 h j0 - 192 h j1 - 24 h^2 s0 + 36 h^2 s1
//   q  h^5 = 720 (a1 - a0) - 360 h (j0 + j1) - 60 h^2 (s0 - s1).
// The next step is the mean of Aarseth's criterion (eta4 inside the root),
// evaluated as the 4th-order scheme does from a and jerk at both ends (the
// 2nd and 3rd derivatives at t1 of their cubic Hermite interpolant), and its
// 6th-order generalisation (eta6 times the sixth root) with the pass's snap
// and the quintic interpolant's crackle, pop and 5th derivative, quantised
// like the 4th-order step.  Only the 6th-order half sees the h^-5
// amplification of force noise in the interpolated derivatives.
__device__ __forceinline__ void correct6_one(const JStore &js, double *dt, int64_t s, int64_t k, double t1,
                                             const double *a1, const double *j1, const double *s1, double eta4,
                                             double eta6, double dt_max) {
    const double h = t1 - js.t[s];
    const double h2 = h * h, h3 = h2 * h;
    const double ih3 = 1.0 / h3, ih4 = ih3 / h, ih5 = ih4 / h;
    double an[3], jn[3], sn[3], cn[3], pn[3], qn[3], a2[3], a3[3];
    for (int c = 0; c < 3; ++c) {
        const int64_t q = 3 * s + c;
        const double x0 = js.x[q], v0 = js.v[q], a0 = js.a[q], j0 = js.jk[q], s0 = js.sn[q];
        const double aa = a1[3 * k + c], jj = j1[3 * k + c], ss = s1[3 * k + c];
        const double v1 = v0 + (a0 + aa) * (h / 2) - (jj - j0) * (h2 / 10) + (s0 + ss) * (h3 / 120);
        const double x1 = x0 + (v0 + v1) * (h / 2) - (aa - a0) * (h2 / 10) + (j0 + jj) * (h3 / 120);
        const double da = aa - a0;
        cn[c] = (60.0 * da - h * (24.0 * j0 + 36.0 * jj) + h2 * (9.0 * ss - 3.0 * s0)) * ih3;
        pn[c] = (360.0 * da - h * (168.0 * j0 + 192.0 * jj) + h2 * (36.0 * ss - 24.0 * s0)) * ih4;
        qn[c] = (720.0 * da - 360.0 * h * (j0 + jj) - 60.0 * h2 * (s0 - ss)) * ih5;
        a3[c] = (12.0 * (a0 - aa) + 6.0 * h * (j0 + jj)) / h3;
        a2[c] = (-6.0 * (a0 - aa) - h * (4.0 * j0 + 2.0 * jj)) / h2 + h * a3[c];
        an[c] = aa;
        jn[c] = jj;
        sn[c] = ss;
        js.x[q] = x1;
        js.v[q] = v1;
        js.a[q] = aa;
        js.jk[q] = jj;
        js.sn[q] = ss;
        js.cr[q] = cn[c];
    }
    js.t[s] = t1;
    const double A = norm3(an), J = norm3(jn), S = norm3(sn), C = norm3(cn), P = norm3(pn), Q = norm3(qn);
    const double A2 = norm3(a2), A3 = norm3(a3);
    const double d4 = J * A3 + A2 * A2, d6 = C * Q + P * P;
    const double want = (d4 > 0.0 && d6 > 0.0)
                            ? 0.5 * (sqrt(eta4 * (A * A2 + J * J) / d4) + eta6 * pow((A * S + J * J) / d6, 1.0 / 6.0))
                            : dt_max;
    dt[s] = quantise_dt(want, fmin(2.0 * h, dt_max), t1);
    if (js.dsc) write_dscache(js, s);
}

__global__ void block_correct6_dev_kernel(JStore js, const BlockStep b, const double *a1, const double *j1,
                                          const double *s1, double eta4, double eta6, double dt_max) {
    const int64_t k = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    const unsigned int n_act = b.bd->count[b.slot];
    const double t1 = key_time(b.bd->t1bits[b.slot]);
    if (k == 0 && n_act > 0) count_block(b.bd, n_act, t1);
    unsigned long long next = ~0ull;
    if (k < n_act) {
        const int64_t s = b.active[k];
        correct6_one(js, b.dt, s, k, t1, a1, j1, s1, eta4, eta6, dt_max);
        check_underflow(b.dt[s], b.bd);
        next = time_key(t1 + b.dt[s]);
    }
    warp_min_to(&b.bd->t1bits[(b.slot + 1) & 3], next);
}

__global__ void iota_kernel(int32_t *dst, int64_t n) {
    const int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (j < n) dst[j] = static_cast<int32_t>(j);
}

// Hermite-4 predictor of the shared-step scheme (to t + dt), packed as records.
template <bool MIXED>
__global__ void h4_predict_pack_kernel(int64_t n, double dt, const double *m, const double *x, const double *v,
                                       const double *a, const double *jk, unsigned char *rec) {
    grid_wait();
    const int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const double h2 = dt * dt * 0.5, h3 = dt * dt * dt * (1.0 / 6.0);
    double xp[3], vp[3];
    for (int c = 0; c < 3; ++c) {
        const int64_t q = 3 * j + c;
        xp[c] = x[q] + v[q] * dt + a[q] * h2 + jk[q] * h3;
        vp[c] = v[q] + a[q] * dt + jk[q] * h2;
    }
    if (MIXED) store_mixed(rec, 48, j, xp, vp, nullptr, m[j], static_cast<int>(j));
    else store_fp64(rec, 64, j, xp, vp, nullptr, m[j], static_cast<int>(j));
}

// Hermite-4 corrector (Makino & Aarseth 1992), in place; a1, j1 at the predicted state.
__global__ void h4_correct_kernel(int64_t n3, double dt, double *x, double *v, double *a, double *jk,
                                  const double *a1, const double *j1) {
    grid_wait();
    const int64_t q = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (q >= n3) return;
    const double h = 0.5 * dt, h12 = dt * dt / 12.0;
    const double v1 = v[q] + (a[q] + a1[q]) * h + (jk[q] - j1[q]) * h12;
    x[q] = x[q] + (v[q] + v1) * h + (a[q] - a1[q]) * h12;
    v[q] = v1;
    a[q] = a1[q];
    jk[q] = j1[q];
}

__device__ __forceinline__ void store_vjp(bool mixed, unsigned char *rec, int64_t j, const double *xp, const double *vp,
                                          const double *ab, const double *jb, double pb, double m) {
    if (mixed) {
        float xh[3], xl[3];
        for (int c = 0; c < 3; ++c) {
        const ds q = ds_split(xp[c]);  // hi = fl32(x), lo = fl32(x - hi)
        xh[c] = q.h;
        xl[c] = q.l;
    }
        float4 *o = reinterpret_cast<float4 *>(rec + j * 80);
        o[0] = make_float4(xh[0], xh[1], xh[2], __double2float_rn(m));
        o[1] = make_float4(xl[0], xl[1], xl[2], __double2float_rn(pb));
        o[2] = make_float4(__double2float_rn(vp[0]), __double2float_rn(vp[1]), __double2float_rn(vp[2]), 0.f);
        o[3] = make_float4(__double2float_rn(ab[0]), __double2float_rn(ab[1]), __double2float_rn(ab[2]), 0.f);
        o[4] = make_float4(__double2float_rn(jb[0]), __double2float_rn(jb[1]), __double2float_rn(jb[2]), 0.f);
    } else {
        double2 *o = reinterpret_cast<double2 *>(rec + j * 112);
        o[0] = make_double2(xp[0], xp[1]);
        o[1] = make_double2(xp[2], m);
        o[2] = make_double2(vp[0], vp[1]);
        o[3] = make_double2(vp[2], pb);
        o[4] = make_double2(ab[0], ab[1]);
        o[5] = make_double2(ab[2], jb[0]);
        o[6] = make_double2(jb[1], jb[2]);
    }
}

template <bool MIXED>
__global__ void pack_vjp_kernel(int64_t n, const double *m, const double *x, const double *v, const double *abar,
                                const double *jbar, const double *pbar, unsigned char *rec) {
    grid_wait();
    const int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const double zero[3] = {0.0, 0.0, 0.0};
    const double *ab = abar ? abar + 3 * j : zero;
    const double *jb = jbar ? jbar + 3 * j : zero;
    store_vjp(MIXED, rec, j, x + 3 * j, v + 3 * j, ab, jb, pbar ? pbar[j] : 0.0, m[j]);
}

// Reverse of the corrector for the output cotangents (gx, gv, ga, gj):
//   gv1 = gv + gx dt/2,  ga1 = ga + gv1 dt/2 - gx dt^2/12,  gj1 = gj - gv1 dt^2/12
// are the cotangents of the force outputs (a1, j1) at the predicted state,
// which is recomputed here and packed with them into VJP records.
template <bool MIXED>
__global__ void h4_vjp_pre_kernel(int64_t n, double dt, const double *m, const double *x, const double *v,
                                  const double *a, const double *jk, const double *gx, const double *gv,
                                  const double *ga, const double *gj, unsigned char *rec) {
    grid_wait();
    const int64_t j = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const double h2 = dt * dt * 0.5, h3 = dt * dt * dt * (1.0 / 6.0), h12 = dt * dt / 12.0;
    double xp[3], vp[3], ab[3], jb[3];
    for (int c = 0; c < 3; ++c) {
        const int64_t q = 3 * j + c;
        xp[c] = x[q] + v[q] * dt + a[q] * h2 + jk[q] * h3;
        vp[c] = v[q] + a[q] * dt + jk[q] * h2;
        const double gv1 = gv[q] + gx[q] * (0.5 * dt);
        ab[c] = ga[q] + gv1 * (0.5 * dt) - gx[q] * h12;
        jb[c] = gj[q] - gv1 * h12;
    }
    store_vjp(MIXED, rec, j, xp, vp, ab, jb, 0.0, m[j]);
}

// Combine: cotangents of the step inputs from the output cotangents and the
// force VJP (xpbar, vpbar) at the predicted state.
__global__ void h4_vjp_post_kernel(int64_t n3, double dt, const double *xpbar, const double *vpbar, double *gx,
                                   double *gv, double *ga, double *gj) {
    grid_wait();
    const int64_t q = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (q >= n3) return;
    const double h = 0.5 * dt, h2 = dt * dt * 0.5, h3 = dt * dt * dt * (1.0 / 6.0), h12 = dt * dt / 12.0;
    const double gx1 = gx[q];
    const double gv1 = gv[q] + gx1 * h;
    const double xb = xpbar[q], vb = vpbar[q];
    gx[q] = gx1 + xb;
    gv[q] = gx1 * h + gv1 + xb * dt + vb;
    ga[q] = gx1 * h12 + gv1 * h + xb * h2 + vb * dt;
    gj[q] = gv1 * h12 + xb * h3 + vb * h2;
}

__global__ void scan_finite_kernel(const double *p, int64_t n, unsigned int *flag) {
    const int64_t q = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (q < n && !isfinite(p[q])) atomicOr(flag, 1u);
}

}  // namespace

cudaError_t launch_scatter_j(const JStore &dst, const int32_t *slots, int64_t n, int64_t n_loaded, unsigned int *err,
                             const int32_t *id, const double *m, const double *x, const double *v, const double *a,
                             const double *jk, const double *sn, const double *t, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    return launch_overlapped(scatter_kernel, grid_for_store(n), kSmallThreads, 0, s, dst, slots, n, n_loaded, err, id, m, x, v, a, jk, sn, t);
}

cudaError_t launch_dscache(int order, const JStore &js, int64_t first, int64_t n, cudaStream_t s) {
    if (n <= 0 || !js.dsc) return cudaSuccess;
    (void)order;
    return launch_overlapped(dscache_kernel, grid_for_store(n), kSmallThreads, 0, s, js, first, n);
}

namespace {
template <bool BLOCK>
cudaError_t launch_predict_form(int order, int mixed, const JStore &js, int64_t n, double t, unsigned char *rec,
                                cudaStream_t s, const BlockStep &b) {
    const unsigned g = grid_for(n);
    if (mixed && js.dsc) {
        const float th = static_cast<float>(t);
        const float tl = static_cast<float>(t - static_cast<double>(th));
        if (order == 6) return launch_overlapped(predict_ds_kernel<6, BLOCK>, g, kThreads, 0, s, js.dsc, n, th, tl, rec, b);
        else if (order == 2) return launch_overlapped(predict_ds_kernel<2, BLOCK>, g, kThreads, 0, s, js.dsc, n, th, tl, rec, b);
        return launch_overlapped(predict_ds_kernel<4, BLOCK>, g, kThreads, 0, s, js.dsc, n, th, tl, rec, b);
    }
    // the FP64 predictor is FP64-bound: 64-thread CTAs spread it over the SMs
    const unsigned g64 = static_cast<unsigned>((n + 63) / 64);
    if (order == 6) {
        if (mixed) return launch_overlapped(predict_kernel<6, true, BLOCK>, g64, 64, 0, s, js, n, t, rec, b);
        return launch_overlapped(predict_kernel<6, false, BLOCK>, g64, 64, 0, s, js, n, t, rec, b);
    } else if (order == 2) {
        if (mixed) return launch_overlapped(predict_kernel<2, true, BLOCK>, g64, 64, 0, s, js, n, t, rec, b);
        return launch_overlapped(predict_kernel<2, false, BLOCK>, g64, 64, 0, s, js, n, t, rec, b);
    } else {
        if (mixed) return launch_overlapped(predict_kernel<4, true, BLOCK>, g64, 64, 0, s, js, n, t, rec, b);
        return launch_overlapped(predict_kernel<4, false, BLOCK>, g64, 64, 0, s, js, n, t, rec, b);
    }
}
}  // namespace

cudaError_t launch_predict(int order, int mixed, const JStore &js, int64_t n, double t, unsigned char *rec,
                           cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    return launch_predict_form<false>(order, mixed, js, n, t, rec, s, BlockStep{});
}

cudaError_t launch_block_predict(int order, int mixed, const JStore &js, int64_t n, unsigned char *rec,
                                 const BlockStep &b, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    return launch_predict_form<true>(order, mixed, js, n, 0.0, rec, s, b);
}

cudaError_t launch_pack_state(int mixed, int64_t n, const double *m, const double *x, const double *v,
                              unsigned char *rec, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    if (mixed) return launch_overlapped(pack_state_kernel<true>, grid_small(n), kSmallThreads, 0, s, n, m, x, v, rec);
    return launch_overlapped(pack_state_kernel<false>, grid_small(n), kSmallThreads, 0, s, n, m, x, v, rec);
}

cudaError_t launch_pack_sinks(int order, int mixed, int64_t n, const double *x, const double *v, const double *a,
                              unsigned char *rec, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const unsigned g = grid_small(n);
    if (order == 6) {
        if (mixed) pack_sinks_kernel<6, true><<<g, kSmallThreads, 0, s>>>(n, x, v, a, rec);
        else pack_sinks_kernel<6, false><<<g, kSmallThreads, 0, s>>>(n, x, v, a, rec);
    } else {
        if (mixed) pack_sinks_kernel<4, true><<<g, kSmallThreads, 0, s>>>(n, x, v, a, rec);
        else pack_sinks_kernel<4, false><<<g, kSmallThreads, 0, s>>>(n, x, v, a, rec);
    }
    return cudaGetLastError();
}

cudaError_t launch_iota(int32_t *dst, int64_t n, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    iota_kernel<<<grid_for(n), kThreads, 0, s>>>(dst, n);
    return cudaGetLastError();
}

cudaError_t launch_block_first(const double *t, const double *dt, int64_t n, BlockDev *bd, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    block_first_kernel<<<grid_for(n), kThreads, 0, s>>>(t, dt, n, bd);
    return cudaGetLastError();
}

cudaError_t launch_block_correct_dev(const JStore &js, const BlockStep &b, int64_t n_max, const double *a1,
                                     const double *j1, double eta, double dt_max, cudaStream_t s) {
    if (n_max <= 0) return cudaSuccess;
    // (most blocks hold a small part of the particles: the grid is capped, and strides)
    const unsigned g = std::min(grid_for_warps(kLanesPerParticle * n_max), kCorrectMaxCtas);
    return launch_overlapped(block_correct_dev_kernel, g, kWarpCta, 0, s, js, b, a1, j1, eta, dt_max);
}

cudaError_t launch_block_correct6_dev(const JStore &js, const BlockStep &b, int64_t n_max, const double *a1,
                                      const double *j1, const double *s1, double eta4, double eta6, double dt_max,
                                      cudaStream_t s) {
    if (n_max <= 0) return cudaSuccess;
    block_correct6_dev_kernel<<<grid_for_warps(n_max), kWarpCta, 0, s>>>(js, b, a1, j1, s1, eta4, eta6, dt_max);
    return cudaGetLastError();
}

cudaError_t launch_block_init(const JStore &js, double *dt, int64_t n, double eta_s, double dt_max, double t0,
                              cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    block_init_kernel<<<grid_for(n), kThreads, 0, s>>>(js, dt, n, eta_s, dt_max, t0);
    return cudaGetLastError();
}

cudaError_t launch_nb_finish(const int32_t *ids, int64_t n_i, int nb_max, const int32_t *count, int32_t *list,
                             cudaStream_t s) {
    if (n_i <= 0) return cudaSuccess;
    return launch_overlapped(nb_finish_kernel, static_cast<unsigned>((n_i + kNbWarps - 1) / kNbWarps), 32 * kNbWarps, 0, s, ids, n_i, nb_max, count, list);
}

cudaError_t launch_h4_predict_pack(int mixed, int64_t n, double dt, const double *m, const double *x,
                                   const double *v, const double *a, const double *jk, unsigned char *rec,
                                   cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    if (mixed) return launch_overlapped(h4_predict_pack_kernel<true>, grid_small(n), kSmallThreads, 0, s, n, dt, m, x, v, a, jk, rec);
    return launch_overlapped(h4_predict_pack_kernel<false>, grid_small(n), kSmallThreads, 0, s, n, dt, m, x, v, a, jk, rec);
}

cudaError_t launch_h4_correct(int64_t n, double dt, double *x, double *v, double *a, double *jk, const double *a1,
                              const double *j1, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    return launch_overlapped(h4_correct_kernel, grid_small(3 * n), kSmallThreads, 0, s, 3 * n, dt, x, v, a, jk, a1, j1);
}

cudaError_t launch_h4_vjp_pre(int mixed, int64_t n, double dt, const double *m, const double *x, const double *v,
                              const double *a, const double *jk, const double *gx, const double *gv,
                              const double *ga, const double *gj, unsigned char *vrec, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    if (mixed) return launch_overlapped(h4_vjp_pre_kernel<true>, grid_small(n), kSmallThreads, 0, s, n, dt, m, x, v, a, jk, gx, gv, ga, gj, vrec);
    return launch_overlapped(h4_vjp_pre_kernel<false>, grid_small(n), kSmallThreads, 0, s, n, dt, m, x, v, a, jk, gx, gv, ga, gj, vrec);
}

cudaError_t launch_h4_vjp_post(int64_t n, double dt, const double *xpbar, const double *vpbar, double *gx,
                               double *gv, double *ga, double *gj, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    return launch_overlapped(h4_vjp_post_kernel, grid_small(3 * n), kSmallThreads, 0, s, 3 * n, dt, xpbar, vpbar, gx, gv, ga, gj);
}

cudaError_t launch_pack_vjp(int mixed, int64_t n, const double *m, const double *x, const double *v,
                            const double *abar, const double *jbar, const double *pbar, unsigned char *vrec,
                            cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    if (mixed) return launch_overlapped(pack_vjp_kernel<true>, grid_small(n), kSmallThreads, 0, s, n, m, x, v, abar, jbar, pbar, vrec);
    return launch_overlapped(pack_vjp_kernel<false>, grid_small(n), kSmallThreads, 0, s, n, m, x, v, abar, jbar, pbar, vrec);
}

cudaError_t launch_scan_finite(const double *p, int64_t n, unsigned int *flag, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    scan_finite_kernel<<<grid_for(n), kThreads, 0, s>>>(p, n, flag);
    return cudaGetLastError();
}

}  // namespace sp2
