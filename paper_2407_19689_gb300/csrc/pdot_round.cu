// pdot_round.cu -- Algorithm 3 of arXiv 2407.19689 (rounding onto the
// transportation polytope, after Altschuler et al.) and the weak-duality
// bound, on the device.
//
// Rounding: with x = min(f / X1, 1), y = min(g / (diag(x) X)^T 1, 1), the plan
// diag(x) X diag(y) + err_r err_c^T / ||err_r||_1.  Four sweeps over X, each
// sum in a fixed order:
//   rows   r = X1 -> x
//   cols   c = (diag(x) X)^T 1, by row groups, then one thread per column adds
//          the groups -> y and err_c = g - y c (the column sums of
//          diag(x) X diag(y) are y_j c_j: no sweep of their own)
//   rows   X y -> err_r = f - x (X y); the last block adds ||err_r||_1
//   write  the plan, and <C, plan> when a cost is given
// All scalars stay on the device: the old form copied them to the host and
// back three times and took the write through 64 blocks (1313 us at 4096 x
// 4096, FP32; here 133 us; 2 x 67 MB take 20 us).
//
// FP64 is a narrow pipe on this part (two lanes per cycle and SM: one FP64
// operation per entry of a 4096 x 4096 plan takes 27 us), so FP32 plans are
// summed as unevaluated FP32 pairs: Knuth's TwoSum keeps each addition's
// rounding error, an FMA each product's, and the pairs are added up in FP64
// at the end of a lane's run.  Scales are kept as FP32 pairs too (48 bits).
// The sums' error (about 1e-13) stays far below the FP32 rounding of the
// written entries; measured against 64 bits the plan's error is unchanged
// (2.5e-8).  Where FP32's range would not hold a sum or a scale, the sweeps
// that follow take FP64 arithmetic and the FP64 scales, which are kept beside
// the pairs: row sums or errors of 1e30 and more or not finite, and scales below RTINY
// that are multiplied by more than 1 (a pair's absolute error is 2^-150, so a
// product with at most 1 is off by one or two of FP32's smallest steps).  The objective
// <C, plan> is an FP64 sum of FP64 products (once per solve that asks for it).
// FP64 plans use FP64 throughout.
#include <cuda_runtime.h>
#include <math_constants.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "pdot_internal.h"

namespace pdot {

namespace {

constexpr int RB = 256;           // threads per block
constexpr int RPARTS = 64;        // most row groups of the column sums
constexpr int RU = 4;             // rows a thread of the write has in flight
constexpr int RROWS = 64;         // rows whose scales a block of the write holds at a time
constexpr double RWIDE = 1e30;    // row sums and column errors from here on: FP64 arithmetic
constexpr double RTINY = 0x1p-100;   // scales below: an FP32 pair has lost bits (its low part is subnormal from 2^-102 on)

// Words of RoundScratch::state: the ticket; FP32's range does not hold a row
// sum or scale (from the first sweep), a column's or the error's scale (from
// the sweeps behind the column sums); a column's error exceeds 1.
constexpr int RS_TICKET = 0, RS_WIDE = 1, RS_LATE = 2, RS_ERR = 3, RS_WORDS = 4;

// v >= 1 (or not a number), in integer arithmetic: an FP64 comparison takes the
// FP64 pipe.
__device__ __forceinline__ bool from_one(double v) { return __double2hiint(v) >= 0x3ff00000; }

// A scale as the sweeps use it: an FP32 pair for FP32 plans, FP64 otherwise.
template <typename T>
struct __align__(8) Scale {
    float h, l;
    __device__ __forceinline__ void set(double v) {
        h = (float)v;
        l = (float)(v - (double)h);
    }
};
template <>
struct Scale<double> {
    double v;
    __device__ __forceinline__ void set(double w) { v = w; }
};

// Running sum: FP32 pair (value plus the additions' errors) or FP64.
template <typename T>
struct __align__(8) Acc {
    float s = 0.f, e = 0.f;
    __device__ __forceinline__ void two_sum(float x) {
        const float t = s + x, b = t - s;
        e += (s - (t - b)) + (x - b);
        s = t;
    }
    __device__ __forceinline__ void add(float x) { two_sum(x); }
    __device__ __forceinline__ void add(float x, const Scale<float>& w) {
        const float p = x * w.h;
        e += fmaf(x, w.l, fmaf(x, w.h, -p));
        two_sum(p);
    }
    __device__ __forceinline__ void merge(const Acc& o) {
        two_sum(o.s);
        e += o.e;
    }
    __device__ __forceinline__ Acc shfl_xor(int m) const {
        Acc r;
        r.s = __shfl_xor_sync(0xffffffffu, s, m);
        r.e = __shfl_xor_sync(0xffffffffu, e, m);
        return r;
    }
    __device__ __forceinline__ double get() const { return (double)s + (double)e; }
    // The errors folded into the value, before they grow in number.
    __device__ __forceinline__ void fold() {
        const float t = s + e;
        e = (s - t) + e;
        s = t;
    }
};
template <>
struct __align__(8) Acc<double> {
    double s = 0.0;
    __device__ __forceinline__ void merge(const Acc& o) { s += o.s; }
    __device__ __forceinline__ Acc shfl_xor(int m) const {
        Acc r;
        r.s = __shfl_xor_sync(0xffffffffu, s, m);
        return r;
    }
    __device__ __forceinline__ void fold() {}
    __device__ __forceinline__ void add(double x) { s += x; }
    __device__ __forceinline__ void add(double x, const Scale<double>& w) { s = fma(x, w.v, s); }
    __device__ __forceinline__ double get() const { return s; }
};

// min(b / s, 1), 1 for a sum of zero; a marginal that is not a number makes its
// scale one too (fmin would return 1 and leave the rest of the plan finite).
__device__ __forceinline__ double scale_to(double b, double s) {
    const double t = b / s;
    return !(s > 0.0) ? 1.0 : t > 1.0 ? 1.0 : t;
}

template <typename T>
__device__ __forceinline__ void warp_merge(Acc<T>& a) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a.merge(a.shfl_xor(o));
}
__device__ __forceinline__ double warp_add(double s) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// Four consecutive entries (VEC: 16-byte aligned rows), `cnt` of which exist.
template <typename T, bool VEC>
__device__ __forceinline__ void load4(const T* p, long long cnt, T (&v)[4]) {
    if (VEC && cnt >= 4) {
        if constexpr (sizeof(T) == 4) {
            const float4 t = *reinterpret_cast<const float4*>(p);
            v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
        } else {
            const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
            v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
        }
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = e < cnt ? p[e] : T(0);
    }
}

// Sweep by rows: a block has RB / 32 warps, WPR of which share RPW rows
// (every entry's scale is then read once for RPW rows).  WEIGHTED: sum_j X_ij
// y_j -> out = err_r, and the last block the inverse of ||err_r||_1; else sum_j
// X_ij -> out.  A lane's four entries are consecutive (16-byte loads), or 32
// columns apart where rows are not aligned and where scales are read (their
// loads then are consecutive over the lanes).
template <typename T, bool VEC, int WPR, int RPW, bool WEIGHTED>
__global__ void __launch_bounds__(RB) k_round_rows(const T* __restrict__ X, long long m, long long n, long long ldx,
                                                   const double* __restrict__ f, const Scale<T>* __restrict__ ys,
                                                   const double* __restrict__ yd, const double* __restrict__ xs, double* out,
                                                   double* inv_l1, unsigned* state) {
    constexpr int RPB = (RB / 32) / WPR * RPW;
    constexpr bool V4 = VEC && !WEIGHTED;
    __shared__ Acc<T> part[RB / 32][RPW];
    __shared__ double red[RB / 32];
    __shared__ unsigned last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long i0 = (long long)blockIdx.x * RPB + warp / WPR * RPW;
    const bool wide = sizeof(T) == 4 && WEIGHTED && (state[RS_WIDE] | state[RS_LATE]) != 0u;
    const int w0 = (warp % WPR) * 128, step = 128 * WPR;
    Acc<T> a[RPW][2];
    const T* row[RPW];
#pragma unroll
    for (int u = 0; u < RPW; ++u) row[u] = X + (i0 + u < m ? i0 + u : 0) * ldx + (V4 ? lane * 4 : lane);
    auto chunk = [&](long long j0, auto tail_c) {
        constexpr bool TAIL = decltype(tail_c)::value;
        Scale<T> y[4];
        if (WEIGHTED) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const long long j = j0 + e * 32 + lane;
                y[e] = ys[!TAIL || j < n ? j : n - 1];
            }
        }
        T v[RPW][4];
#pragma unroll
        for (int u = 0; u < RPW; ++u) {
            if (V4) {
                load4<T, true>(row[u] + j0, TAIL ? n - j0 - lane * 4 : 4, v[u]);
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) v[u][e] = !TAIL || j0 + e * 32 + lane < n ? row[u][j0 + e * 32] : T(0);
            }
        }
#pragma unroll
        for (int u = 0; u < RPW; ++u) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (WEIGHTED) a[u][e & 1].add(v[u][e], y[e]);
                else a[u][e & 1].add(v[u][e]);
            }
        }
    };
    if (!wide) {
        constexpr int UN = RPW == 1 ? 8 : 2;   // chunks in flight
        long long j0 = w0;
        int run = 0;
        for (; j0 + (UN - 1) * step + 128 <= n; j0 += UN * step) {
#pragma unroll
            for (int k = 0; k < UN; ++k) chunk(j0 + k * step, std::false_type());
            if (++run == 8) {   // long rows
                run = 0;
#pragma unroll
                for (int u = 0; u < RPW; ++u) { a[u][0].fold(); a[u][1].fold(); }
            }
        }
        for (; j0 < n; j0 += step) chunk(j0, std::true_type());
    }
#pragma unroll
    for (int u = 0; u < RPW; ++u) {
        a[u][0].merge(a[u][1]);
        warp_merge(a[u][0]);
        if (WPR > 1 && lane == 0) part[warp][u] = a[u][0];
    }
    if (WPR > 1) {
        __syncthreads();
        if (warp % WPR == 0) {
#pragma unroll
            for (int u = 0; u < RPW; ++u)
                for (int w = 1; w < WPR; ++w) a[u][0].merge(part[warp + w][u]);
        }
    }
    if (warp % WPR == 0) {
#pragma unroll
        for (int u = 0; u < RPW; ++u) {
            const long long i = i0 + u;
            if (i >= m) break;
            // Sums that leave FP32's range: again, in FP64 by one warp.
            const bool big = sizeof(T) == 4 && (wide || (!WEIGHTED && !(fabsf((float)a[u][0].s) < (float)RWIDE)));
            double sum = 0.0;
            if (big) {
                for (long long j = lane; j < n; j += 32)
                    sum += WEIGHTED ? (double)X[i * ldx + j] * yd[j] : (double)X[i * ldx + j];
                sum = warp_add(sum);
            }
            if (lane == 0) {
                if (!big) sum = a[u][0].get();
                if (!WEIGHTED) {
                    out[i] = sum;
                    if (big || (sizeof(T) == 4 && from_one(sum) && f[i] > 0.0 && f[i] < RTINY * sum)) atomicOr(state + RS_WIDE, 1u);
                } else {
                    out[i] = f[i] - xs[i] * sum;
                }
            }
        }
    }
    if (!WEIGHTED) return;
    // The last block adds |err_r| (each thread a strided run, then in order).
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(state + RS_TICKET, 1u) == gridDim.x - 1 ? 1u : 0u;
    __syncthreads();
    if (!last) return;
    __threadfence();
    double l1 = 0.0;
    for (long long r = threadIdx.x; r < m; r += RB) l1 += fabs(__ldcg(out + r));
    l1 = warp_add(l1);
    if (lane == 0) red[warp] = l1;
    __syncthreads();
    if (threadIdx.x == 0) {
        l1 = 0.0;
        for (int w = 0; w < RB / 32; ++w) l1 += red[w];
        *inv_l1 = l1 > 0.0 ? 1.0 / l1 : 0.0;
        red[0] = l1;
    }
    if (sizeof(T) == 8 || state[RS_ERR] == 0u) return;
    __syncthreads();
    bool tiny = false;   // the scales |err_r| / ||err_r||_1 of the error term
    for (long long r = threadIdx.x; r < m; r += RB) {
        const double e = fabs(__ldcg(out + r));
        tiny |= e > 0.0 && e < RTINY * red[0];
    }
    if (tiny) atomicOr(state + RS_LATE, 1u);
}

// The sweeps' FP64 forms for FP32 plans whose sums or scales leave FP32's
// range, out of line: they would only take registers from the others.
template <typename T>
__device__ __noinline__ void cols_wide(const T* X, long long r0, long long r1, long long ldx, const double* f,
                                       const double* r_sum, long long n, long long j, long long es, double* part) {
    for (int e = 0; e < 4; ++e) {
        if (j + e * es >= n) break;
        double c = 0.0;
        for (long long i = r0; i < r1; ++i)
            c += (double)X[i * ldx + j + e * es] * scale_to(f[i], r_sum[i]);
        part[j + e * es] = c;
    }
}

// x_i = min(f_i / r_i, 1) (a zero sum keeps scale 1; the blocks of the first
// columns write it), and colpart[g][j] = sum over the rows i of group g of
// x_i X_ij: four columns per thread.
template <typename T, bool VEC>
__global__ void __launch_bounds__(RB) k_round_cols(const T* __restrict__ X, long long m, long long n, long long ldx,
                                                   const double* __restrict__ f, const double* __restrict__ r_sum, double* xs,
                                                   Acc<T>* __restrict__ colpart, int parts, const unsigned* __restrict__ state) {
    const long long j = VEC ? ((long long)blockIdx.x * RB + threadIdx.x) * 4 : (long long)blockIdx.x * RB * 4 + threadIdx.x;
    constexpr long long ES = VEC ? 1 : RB;   // distance of a thread's columns
    const int grp = blockIdx.y;
    const long long r0 = m * grp / parts, r1 = m * (grp + 1) / parts;
    const bool wide = sizeof(T) == 4 && state[RS_WIDE] != 0u;
    __shared__ Scale<T> sx[64];
    if (wide && j < n) cols_wide(X, r0, r1, ldx, f, r_sum, n, j, ES, reinterpret_cast<double*>(colpart) + (long long)grp * n);
    Acc<T> a[4];
    for (long long b = r0; b < r1; b += 64) {
        const int cnt = (int)(b + 64 < r1 ? 64 : r1 - b);
        __syncthreads();
        if ((int)threadIdx.x < cnt) {
            const double x = scale_to(f[b + threadIdx.x], r_sum[b + threadIdx.x]);
            sx[threadIdx.x].set(x);
            if (blockIdx.x == 0) xs[b + threadIdx.x] = x;
        }
        __syncthreads();
        if (j >= n || wide) continue;
#pragma unroll 8
        for (int r = 0; r < cnt; ++r) {
            const T* row = X + (b + r) * ldx + j;
            T v[4];
            if (VEC) {
                load4<T, true>(row, n - j, v);
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) v[e] = j + e * ES < n ? row[e * ES] : T(0);
            }
            const Scale<T> w = sx[r];
#pragma unroll
            for (int e = 0; e < 4; ++e) a[e].add(v[e], w);
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) a[e].fold();
    }
    if (j >= n || wide) return;
#pragma unroll
    for (int e = 0; e < 4; ++e)
        if (j + e * ES < n) colpart[(long long)grp * n + j + e * ES] = a[e];
}

// c_j = the groups' sums -> y_j, err_c (FP32 plans: in FP64 too).  Bound by the
// groups' loads: sixteen of them are requested before any is added.
template <typename T>
__global__ void __launch_bounds__(64) k_round_colscale(const Acc<T>* __restrict__ colpart, int parts, long long n, const double* __restrict__ g,
                                 Scale<T>* ys, Scale<T>* ec, double* yd, double* ed, unsigned* state) {
    const bool wide = sizeof(T) == 4 && state[RS_WIDE] != 0u;
    const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    double c = 0.0;
    if (wide) {
        for (int k = 0; k < parts; ++k) c += *reinterpret_cast<const double*>(colpart + (long long)k * n + j);
    } else {
        Acc<T> a;
        for (int k = 0; k < parts; k += 16) {
            Acc<T> v[16];
#pragma unroll
            for (int u = 0; u < 16; ++u)
                if (k + u < parts) v[u] = colpart[(long long)(k + u) * n + j];
#pragma unroll
            for (int u = 0; u < 16; ++u)
                if (k + u < parts) a.merge(v[u]);
        }
        c = a.get();
    }
    const double y = scale_to(g[j], c);
    const double e = g[j] - y * c;
    ys[j].set(y);
    ec[j].set(e);
    if (sizeof(T) == 4) {
        yd[j] = y;
        ed[j] = e;
        if (from_one(c) && y > 0.0 && y < RTINY) atomicOr(state + RS_LATE, 1u);
        if (from_one(e)) {
            atomicOr(state + RS_ERR, 1u);
            if (!(e < RWIDE)) atomicOr(state + RS_LATE, 1u);
        }
    }
}

struct Bf16 {
    unsigned short b;
    __device__ operator float() const { return __uint_as_float(((unsigned)b) << 16); }
};

// Cost entry (i, j) for the objective of the rounded plan: a stored matrix
// (null: no objective) or the generated cost.
template <typename TC>
struct StoredCost {
    const TC* C;
    long long ldc;
    __device__ __forceinline__ bool on() const { return C != nullptr; }
    __device__ __forceinline__ double operator()(long long i, long long j) const { return (double)C[i * ldc + j]; }
    __device__ __forceinline__ float f32(long long i, long long j) const { return (float)C[i * ldc + j]; }
};
struct PointsCost {
    GenSpec g;
    __device__ __forceinline__ bool on() const { return true; }
    __device__ __forceinline__ float f32(long long i, long long j) const {
        return gen_cost(g.kind, g.d, g.xs + i * g.d, g.ys + j * g.d, g.div, g.inv);
    }
    __device__ __forceinline__ double operator()(long long i, long long j) const { return (double)f32(i, j); }
};

// The entry x y v + a e of the rounded plan (a = err_r / ||err_r||_1), rounded
// once to the plan's type.
__device__ __forceinline__ float rounded(float v, const Scale<float>& x, const Scale<float>& y, const Scale<float>& a,
                                         const Scale<float>& e) {
    const float t = v * x.h;
    const float tl = fmaf(v, x.l, fmaf(v, x.h, -t));
    const float p = t * y.h;
    const float pl = fmaf(tl, y.h, fmaf(t, y.l, fmaf(t, y.h, -p)));
    const float c = a.h * e.h;
    const float cl = fmaf(a.l, e.h, fmaf(a.h, e.l, fmaf(a.h, e.h, -c)));
    const float s = p + c, b = s - p;
    return s + (((p - (s - b)) + (c - b)) + (pl + cl));
}
__device__ __forceinline__ double rounded(double v, const Scale<double>& x, const Scale<double>& y, const Scale<double>& a,
                                          const Scale<double>& e) {
    return fma(v * x.v, y.v, a.v * e.v);
}

template <typename T, typename CA>
__device__ __noinline__ double write_wide(const T* X, long long r0, long long r1, long long ldx, const double* xs,
                                          const double* yd, const double* er, const double* ed, double inv, T* out,
                                          long long ldo, const CA& C, long long n, long long j, long long es) {
    double obj = 0.0;
    for (long long i = r0; i < r1; ++i) {
        for (int e = 0; e < 4; ++e) {
            const long long c = j + e * es;
            if (c >= n) break;
            const T w = (T)((double)X[i * ldx + c] * xs[i] * yd[c] + er[i] * ed[c] * inv);
            out[i * ldo + c] = w;
            if (C.on()) obj += C(i, c) * (double)w;
        }
    }
    return obj;
}

template <typename T, bool VEC, typename CA>
__global__ void __launch_bounds__(RB) k_round_write(const T* X, long long m, long long n, long long ldx,
                                                    const double* __restrict__ xs, const Scale<T>* __restrict__ ys,
                                                    const double* __restrict__ er, const Scale<T>* __restrict__ ec,
                                                    const double* __restrict__ yd, const double* __restrict__ ed,
                                                    const double* __restrict__ inv_l1, T* out, long long ldo, CA C,
                                                    double* objpart, const unsigned* __restrict__ state) {
    __shared__ double red[RB / 32];
    __shared__ Scale<T> sx[RROWS], sa[RROWS];
    const long long j = VEC ? ((long long)blockIdx.x * RB + threadIdx.x) * 4 : (long long)blockIdx.x * RB * 4 + threadIdx.x;
    constexpr long long ES = VEC ? 1 : RB;
    const int grp = blockIdx.y, parts = gridDim.y;
    const long long r0 = m * grp / parts, r1 = m * (grp + 1) / parts;
    const double inv = *inv_l1;
    const bool wide = sizeof(T) == 4 && (state[RS_WIDE] | state[RS_LATE]) != 0u;
    double obj = 0.0;
    if (wide) {
        if (j < n) obj = write_wide(X, r0, r1, ldx, xs, yd, er, ed, inv, out, ldo, C, n, j, ES);
    } else {
        auto load = [&](long long i, T (&v)[4]) {
            const T* row = X + i * ldx + j;
            if (VEC) {
                load4<T, true>(row, n - j, v);
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) v[e] = j + e * ES < n ? row[e * ES] : T(0);
            }
        };
        Scale<T> y[4], e4[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const bool in = j + e * ES < n;
            y[e] = ys[in ? j + e * ES : 0];
            e4[e] = ec[in ? j + e * ES : 0];
        }
        for (long long b = r0; b < r1; b += RROWS) {
            const int cnt = (int)(b + RROWS < r1 ? RROWS : r1 - b);
            // RU rows are read before the ones before them are written (out may
            // be X itself: an entry is read and written by one thread).
            T v[RU][4];
            if (j < n) {
#pragma unroll
                for (int u = 0; u < RU; ++u)
                    if (u < cnt) load(b + u, v[u]);
            }
            __syncthreads();
            if ((int)threadIdx.x < cnt) {   // the rows' scales
                sx[threadIdx.x].set(xs[b + threadIdx.x]);
                sa[threadIdx.x].set(er[b + threadIdx.x] * inv);
            }
            __syncthreads();
            if (j >= n) continue;
            for (int rb = 0; rb < cnt; rb += RU) {
#pragma unroll
                for (int u = 0; u < RU; ++u) {
                    const int r = rb + u;
                    if (r >= cnt) break;
                    const Scale<T> x = sx[r], a = sa[r];
                    T w[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) w[e] = rounded(v[u][e], x, y[e], a, e4[e]);
                    if (r + RU < cnt) load(b + r + RU, v[u]);
                    T* o = out + (b + r) * ldo + j;
                    if (VEC && j + 4 <= n) {
                        if constexpr (sizeof(T) == 4) {
                            *reinterpret_cast<float4*>(o) = make_float4(w[0], w[1], w[2], w[3]);
                        } else {
                            reinterpret_cast<double2*>(o)[0] = make_double2(w[0], w[1]);
                            reinterpret_cast<double2*>(o)[1] = make_double2(w[2], w[3]);
                        }
                    } else {
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            if (j + e * ES < n) o[e * ES] = w[e];
                    }
                    if (C.on()) {
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            if (j + e * ES < n) obj += C(b + r, j + e * ES) * (double)w[e];
                    }
                }
            }
        }
    }
    if (!C.on()) return;
    obj = warp_add(obj);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = obj;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < RB / 32; ++w) t += red[w];
        objpart[(long long)blockIdx.y * gridDim.x + blockIdx.x] = t;
    }
}

// Weak-duality bound of Eq. (1) from a row dual p (no counterpart in the
// paper; it certifies a result): q_j = min_i (C_ij - p_i) is the largest
// column dual with p_i + q_j <= C_ij for all i, and f^T p + g^T q <= OPT.  The
// minimum is exact, so the result does not depend on the grouping.
//
// FP64 C: one sweep.  Otherwise the difference, the comparison and the
// conversion in FP64 would bound the sweep (106 us at 4096 x 4096): a first
// sweep takes the minimum of C - RN32(p) in FP32, a second one forms the FP64
// difference only where the FP32 one is within its rounding error of that
// minimum -- a handful of entries per column (two sweeps, 42 us).  |RN32(c - RN32(p)) - (c - p)| is
// at most 2^-24 (|p| + |c - p|) (and 2^-149 below the normal range), so the
// entry that attains the minimum lies within 2^-22 (max|p| + |min|) + 2^-125.
// Row duals of 1e30 and more make every entry a candidate.
__device__ __forceinline__ unsigned key32(float v) {   // order-preserving
    const unsigned u = __float_as_uint(v);
    return u & 0x80000000u ? ~u : u | 0x80000000u;
}
__device__ __forceinline__ float unkey32(unsigned k) { return __uint_as_float(k & 0x80000000u ? k & 0x7fffffffu : ~k); }
__device__ __forceinline__ unsigned long long key64(double v) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(v);
    return u >> 63 ? ~u : u | 0x8000000000000000ull;
}
__device__ __forceinline__ double unkey64(unsigned long long k) {
    return __longlong_as_double((long long)(k >> 63 ? k & 0x7fffffffffffffffull : ~k));
}

// Four cost entries of a row (columns j + e ES).
template <bool VEC, typename CA>
__device__ __forceinline__ void cost4(const CA& C, long long i, long long j, long long es, long long n, float (&c)[4]) {
#pragma unroll
    for (int e = 0; e < 4; ++e) c[e] = j + e * es < n ? C.f32(i, j + e * es) : 0.f;
}
template <bool VEC>
__device__ __forceinline__ void cost4(const StoredCost<float>& C, long long i, long long j, long long es, long long n,
                                      float (&c)[4]) {
    if (VEC) {
        load4<float, true>(C.C + i * C.ldc + j, n - j, c);
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) c[e] = j + e * es < n ? C.f32(i, j + e * es) : 0.f;
    }
}
template <bool VEC>
__device__ __forceinline__ void cost4(const StoredCost<Bf16>& C, long long i, long long j, long long es, long long n,
                                      float (&c)[4]) {
    if (VEC && j + 4 <= n) {
        const uint2 t = *reinterpret_cast<const uint2*>(C.C + i * C.ldc + j);
        c[0] = __uint_as_float(t.x << 16); c[1] = __uint_as_float(t.x & 0xffff0000u);
        c[2] = __uint_as_float(t.y << 16); c[3] = __uint_as_float(t.y & 0xffff0000u);
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) c[e] = j + e * es < n ? C.f32(i, j + e * es) : 0.f;
    }
}

// EXACT false: qmin[j] <- min of the FP32 differences (as keys), pmax <- the
// complement of the bits of max |RN32(p)| (all of these start as all ones).  EXACT true: qkey[j] <- min of the FP64 differences of
// the candidates.
template <bool EXACT, bool VEC, typename CA>
__global__ void __launch_bounds__(RB) k_bound_cols(CA C, const double* __restrict__ p, long long m, long long n,
                                                   unsigned* qmin, unsigned* pmax, unsigned long long* qkey) {
    const long long j = VEC ? ((long long)blockIdx.x * RB + threadIdx.x) * 4 : (long long)blockIdx.x * RB * 4 + threadIdx.x;
    constexpr long long ES = VEC ? 1 : RB;
    const long long r0 = m * blockIdx.y / gridDim.y, r1 = m * (blockIdx.y + 1) / gridDim.y;
    __shared__ float sp[64];
    float lim[4];
    double best[4];
    bool any[4] = {false, false, false, false};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        lim[e] = CUDART_INF_F;
        best[e] = CUDART_INF;
        if (EXACT && j + e * ES < n) {
            const float v = unkey32(qmin[j + e * ES]), pm = __uint_as_float(~*pmax);
            lim[e] = pm < 1e30f ? v + (0x1p-22f * (pm + fabsf(v)) + 0x1p-125f) : CUDART_NAN_F;
        }
    }
    float pm = 0.f;
    for (long long b = r0; b < r1; b += 64) {
        const int cnt = (int)(b + 64 < r1 ? 64 : r1 - b);
        __syncthreads();
        if ((int)threadIdx.x < cnt) {
            sp[threadIdx.x] = (float)p[b + threadIdx.x];
            pm = fmaxf(pm, fabsf(sp[threadIdx.x]));
        }
        __syncthreads();
        if (j >= n) continue;
#pragma unroll 8
        for (int r = 0; r < cnt; ++r) {
            float c[4];
            cost4<VEC>(C, b + r, j, ES, n, c);
            const float ph = sp[r];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float t = c[e] - ph;
                if (!EXACT) {
                    lim[e] = fminf(lim[e], t);
                } else if (!(t > lim[e])) {   // (also where the limit is not a number)
                    const double d = (double)c[e] - p[b + r];
                    any[e] = true;
                    if (d < best[e]) best[e] = d;
                }
            }
        }
    }
    if (!EXACT && blockIdx.x == 0 && threadIdx.x < 64) {
        // (NaN duals leave the maximum alone: their differences are never minima)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) pm = fmaxf(pm, __shfl_xor_sync(0xffffffffu, pm, o));
        if ((threadIdx.x & 31) == 0) atomicMin(pmax, ~__float_as_uint(pm));
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        if (j + e * ES >= n) continue;
        if (!EXACT) atomicMin(qmin + j + e * ES, key32(lim[e]));
        else if (any[e]) atomicMin(qkey + j + e * ES, key64(best[e]));
    }
}

// FP64 differences throughout: FP64 costs, and matrices too small for the
// screen's second launch to pay.
template <typename CA>
__global__ void __launch_bounds__(RB) k_bound_cols64(CA C, const double* __restrict__ p, long long m, long long n,
                                                     unsigned long long* qkey) {
    const long long j = (long long)blockIdx.x * RB + threadIdx.x;
    if (j >= n) return;
    const long long r0 = m * blockIdx.y / gridDim.y, r1 = m * (blockIdx.y + 1) / gridDim.y;
    double v = CUDART_INF;
#pragma unroll 8
    for (long long i = r0; i < r1; ++i) {
        const double t = C(i, j) - p[i];
        if (t < v) v = t;
    }
    atomicMin(qkey + j, key64(v));
}

// q from its keys (into q_out, where wanted) and out[0] = f^T p + g^T q: fixed
// runs per block, the last block adds the blocks' sums in order.  ticket starts
// as all ones.  (q_out may be the keys' own memory: an entry has one thread.)
__global__ void __launch_bounds__(RB) k_bound_value(const double* __restrict__ f, const double* __restrict__ p, long long m,
                                                    const double* __restrict__ g,
                                                    const unsigned long long* qkey, double* q_out, long long n,
                                                    double* part, double* out, unsigned* ticket) {
    __shared__ double red[RB / 32];
    __shared__ unsigned last;
    double s = 0.0;
    for (long long e = (long long)blockIdx.x * RB + threadIdx.x; e < m + n; e += (long long)gridDim.x * RB) {
        if (e < m) {
            s = fma(f[e], p[e], s);
        } else {
            const double q = unkey64(qkey[e - m]);
            if (q_out) q_out[e - m] = q;
            s = fma(g[e - m], q, s);
        }
    }
    s = warp_add(s);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        s = 0.0;
        for (int w = 0; w < RB / 32; ++w) s += red[w];
        part[blockIdx.x] = s;
        __threadfence();
        last = atomicAdd(ticket, 1u) + 1u == gridDim.x - 1 ? 1u : 0u;
    }
    __syncthreads();
    if (!last || threadIdx.x >= 32) return;
    __threadfence();
    s = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += 32) s += __ldcg(part + b);
    s = warp_add(s);
    if (threadIdx.x == 0) out[0] = s;
}

// Below 2M entries the bound takes one sweep of FP64 differences: the FP32
// screen's second launch and its keys' round trip take 15 us of a call, the
// FP64 pipe less.  Whole calls, screened -> direct: 64 x 64 55.7 -> 38.4 us,
// 1053 x 439 59.1 -> 43.0, 1000 x 1000 59.6 -> 44.9, 1400 x 1400 59.3 -> 55.7;
// 2000 x 2000 59.4 -> 69.2.
constexpr long long BOUND_DIRECT = 1LL << 21;

// Row groups of a sweep over `cb` blocks of columns: four blocks per SM, of at
// least 16 rows.
long long bound_parts(long long cb, long long m, int sm) {
    long long parts = (4LL * sm + cb - 1) / cb;
    if (parts > (m + 15) / 16) parts = (m + 15) / 16;
    return parts > 65535 ? 65535 : parts;
}

// (Row groups as above, but up to 64 of any size: a thread's FP64 differences
// are one chain.  With 64 groups at most, 100000 x 10 from 8 coordinates took
// 632 us; here 119.)
template <typename CA>
void launch_bound_cols64(CA C, const double* p, long long m, long long n, unsigned long long* qkey, int sm, cudaStream_t st) {
    const long long parts = std::max(bound_parts((n + RB - 1) / RB, m, sm), std::min(64LL, m));
    k_bound_cols64<CA><<<dim3((unsigned)((n + RB - 1) / RB), (unsigned)parts), RB, 0, st>>>(C, p, m, n, qkey);
}

// Costs generated from 4 or 8 coordinates take one sweep at any size: the
// columns' coordinates are then 16 or 32 bytes apart, a warp's loads of them
// conflict in the banks, and the screen's second sweep reads them again (8191 x
// 8191, direct / screened: 4 coordinates 460 / 467 us, 8 602 / 1056; 3: 464 /
// 333, 6: 465 / 400).
bool bound_direct(const PointsCost& C) { return C.g.d % 4 == 0; }
template <typename CA>
bool bound_direct(const CA&) { return false; }

// Returns the number of launches.
template <typename CA>
int launch_bound_cols(CA C, bool vec, const double* p, long long m, long long n, unsigned* qmin, unsigned* pmax,
                      unsigned long long* qkey, int sm, cudaStream_t st) {
    if (m * n < BOUND_DIRECT || bound_direct(C)) {
        launch_bound_cols64(C, p, m, n, qkey, sm, st);
        return 1;
    }
    const long long cb = (n + 4 * RB - 1) / (4 * RB);
    const dim3 grid((unsigned)cb, (unsigned)bound_parts(cb, m, sm));
    if (vec) {
        k_bound_cols<false, true, CA><<<grid, RB, 0, st>>>(C, p, m, n, qmin, pmax, qkey);
        k_bound_cols<true, true, CA><<<grid, RB, 0, st>>>(C, p, m, n, qmin, pmax, qkey);
    } else {
        k_bound_cols<false, false, CA><<<grid, RB, 0, st>>>(C, p, m, n, qmin, pmax, qkey);
        k_bound_cols<true, false, CA><<<grid, RB, 0, st>>>(C, p, m, n, qmin, pmax, qkey);
    }
    return 2;
}

constexpr int BOUND_BLOCKS = 64;

}  // namespace

// Scratch of the bound in bytes: the keys, the FP32 minima, max |p| and the
// ticket (all ones at the start), the block sums, the value.
long long bound_scratch_bytes(long long n) { return 8 * n + 4 * ((n + 1) / 2 * 2) + 8 + 8 * (BOUND_BLOCKS + 1); }

// The bound above: q_out (n, or null) and *value = f^T p + g^T q.
// ctype: 0 FP32, 1 BF16, 2 FP64 (row-major with leading dimension ldc), 3
// generated (gen).  *launches: how many kernels it took.
int launch_dual_bound(const void* C, int ctype, long long ldc, const GenSpec* gen, const double* p,
                      const double* f, const double* g, long long m, long long n, void* scratch, double* q_out,
                      double** value, int sm, int* launches, void* stream) {
    const cudaStream_t st = (cudaStream_t)stream;
    unsigned long long* qkey = static_cast<unsigned long long*>(scratch);
    unsigned* qmin = reinterpret_cast<unsigned*>(qkey + n);
    unsigned* pmax = qmin + (n + 1) / 2 * 2;
    double* part = reinterpret_cast<double*>(pmax + 2);
    *value = part + BOUND_BLOCKS;
    const cudaError_t e = cudaMemsetAsync(scratch, 0xff, (size_t)(reinterpret_cast<char*>(part) - static_cast<char*>(scratch)), st);
    if (e != cudaSuccess) return (int)e;
    const bool a16 = reinterpret_cast<uintptr_t>(C) % 16 == 0;
    int k = 1;
    if (ctype == 3) {
        k = launch_bound_cols(PointsCost{*gen}, false, p, m, n, qmin, pmax, qkey, sm, st);
    } else if (ctype == 2) {
        launch_bound_cols64(StoredCost<double>{(const double*)C, ldc}, p, m, n, qkey, sm, st);
    } else if (ctype == 1) {
        k = launch_bound_cols(StoredCost<Bf16>{(const Bf16*)C, ldc}, a16 && ldc % 4 == 0, p, m, n, qmin, pmax, qkey, sm, st);
    } else {
        k = launch_bound_cols(StoredCost<float>{(const float*)C, ldc}, a16 && ldc % 4 == 0, p, m, n, qmin, pmax, qkey, sm, st);
    }
    *launches = k + 1;
    // One block per 256 entries where that is fewer.
    long long vb = (m + n + RB - 1) / RB;
    if (vb > BOUND_BLOCKS) vb = BOUND_BLOCKS;
    k_bound_value<<<(unsigned)vb, RB, 0, st>>>(f, p, m, g, qkey, q_out, n, part, *value, pmax + 1);
    return (int)cudaGetLastError();
}

namespace {

// Scratch of a rounding, in doubles (scales take one each).
struct RoundScratch {
    double *rs, *xs, *er, *ys, *ec, *yd, *ed, *colpart, *inv, *obj;   // yd, ed: ys and ec in FP64
    unsigned* state;
    long long words;
};
int round_parts(long long m, long long n, int sm) {
    // Row groups: enough blocks for four per SM, of at least 16 rows.
    const long long cb = (n + 4 * RB - 1) / (4 * RB);
    long long p = (4LL * sm + cb - 1) / cb;
    if (p > (m + 15) / 16) p = (m + 15) / 16;
    if (p > 65535) p = 65535;
    return (int)(p < 1 ? 1 : p);
}
RoundScratch round_scratch(double* base, long long m, long long n, int sm) {
    const int parts = round_parts(m, n, sm);
    const int cparts = parts < RPARTS ? parts : RPARTS;
    const long long cb = (n + 4 * RB - 1) / (4 * RB);
    RoundScratch r;
    r.rs = base;
    r.xs = r.rs + m;
    r.er = r.xs + m;
    r.ys = r.er + m;
    r.ec = r.ys + n;
    r.yd = r.ec + n;
    r.ed = r.yd + n;
    r.colpart = r.ed + n;
    r.inv = r.colpart + (long long)cparts * n;
    r.state = reinterpret_cast<unsigned*>(r.inv + 1);
    r.obj = r.inv + 1 + (RS_WORDS + 1) / 2;
    r.words = 3 * m + (4 + (long long)cparts) * n + 1 + (RS_WORDS + 1) / 2 + cb * parts;
    return r;
}

template <typename T, bool VEC, typename CA>
int run_round(const T* X, long long m, long long n, long long ldx, const double* f, const double* g, T* out, long long ldo,
              CA C, const RoundScratch& w, int sm, cudaStream_t st) {
    double* xs = w.xs;
    Scale<T>* ys = reinterpret_cast<Scale<T>*>(w.ys);
    Scale<T>* ec = reinterpret_cast<Scale<T>*>(w.ec);
    const int parts = round_parts(m, n, sm), cparts = parts < RPARTS ? parts : RPARTS;
    const unsigned cb = (unsigned)((n + 4 * RB - 1) / (4 * RB));
    const cudaError_t e = cudaMemsetAsync(w.state, 0, RS_WORDS * sizeof(unsigned), st);
    if (e != cudaSuccess) return (int)e;
    // By rows: a block per row where there are few rows, else a warp per row
    // (the weighted sweep: four rows per warp where that leaves eight warps per
    // SM, for one read of the columns' scales).
    Acc<T>* cpart = reinterpret_cast<Acc<T>*>(w.colpart);
    const bool few = m < 16LL * sm && n >= 1024;
    if (few)
        k_round_rows<T, VEC, 8, 1, false><<<(unsigned)m, RB, 0, st>>>(X, m, n, ldx, f, nullptr, nullptr, nullptr, w.rs, nullptr, w.state);
    else
        k_round_rows<T, VEC, 1, 1, false><<<(unsigned)((m + 7) / 8), RB, 0, st>>>(X, m, n, ldx, f, nullptr, nullptr, nullptr,
                                                                                  w.rs, nullptr, w.state);
    k_round_cols<T, VEC><<<dim3(cb, (unsigned)cparts), RB, 0, st>>>(X, m, n, ldx, f, w.rs, xs, cpart, cparts, w.state);
    k_round_colscale<T><<<(unsigned)((n + 63) / 64), 64, 0, st>>>(cpart, cparts, n, g, ys, ec, w.yd, w.ed, w.state);
    if (few && m >= 4LL * sm)
        k_round_rows<T, VEC, 8, 4, true><<<(unsigned)((m + 3) / 4), RB, 0, st>>>(X, m, n, ldx, f, ys, w.yd, xs, w.er, w.inv, w.state);
    else if (few)
        k_round_rows<T, VEC, 8, 1, true><<<(unsigned)m, RB, 0, st>>>(X, m, n, ldx, f, ys, w.yd, xs, w.er, w.inv, w.state);
    else if (m < 64LL * sm && n >= 1024)
        k_round_rows<T, VEC, 4, 4, true><<<(unsigned)((m + 7) / 8), RB, 0, st>>>(X, m, n, ldx, f, ys, w.yd, xs, w.er, w.inv, w.state);
    else
        k_round_rows<T, VEC, 1, 4, true><<<(unsigned)((m + 31) / 32), RB, 0, st>>>(X, m, n, ldx, f, ys, w.yd, xs, w.er, w.inv, w.state);
    k_round_write<T, VEC, CA><<<dim3(cb, (unsigned)parts), RB, 0, st>>>(X, m, n, ldx, xs, ys, w.er, ec, w.yd, w.ed, w.inv, out, ldo, C,
                                                                        w.obj, w.state);
    return (int)cudaGetLastError();
}

template <typename T, typename CA>
int run_round_v(const T* X, long long m, long long n, long long ldx, const double* f, const double* g, T* out, long long ldo,
                CA C, const RoundScratch& w, int sm, cudaStream_t st) {
    // 16-byte accesses where the rows of both plans start on 16-byte boundaries.
    const long long q = 16 / (long long)sizeof(T);
    const bool vec = reinterpret_cast<uintptr_t>(X) % 16 == 0 && reinterpret_cast<uintptr_t>(out) % 16 == 0 &&
                     ldx % q == 0 && ldo % q == 0;
    return vec ? run_round<T, true>(X, m, n, ldx, f, g, out, ldo, C, w, sm, st)
               : run_round<T, false>(X, m, n, ldx, f, g, out, ldo, C, w, sm, st);
}

}  // namespace

// Doubles of scratch a rounding takes, and the objective partials in it.
long long round_scratch_words(long long m, long long n, int sm) { return round_scratch(nullptr, m, n, sm).words; }
double* round_obj_parts(double* base, long long m, long long n, int sm, long long* count) {
    *count = (n + 4 * RB - 1) / (4 * RB) * round_parts(m, n, sm);
    return round_scratch(base, m, n, sm).obj;
}

// Algorithm 3 on X (m x n, leading dimension ldx) into out (ldo); with a cost,
// the partials of <C, out> too.
int launch_round(const void* X, int xtype, long long m, long long n, long long ldx, const double* f, const double* g,
                 void* out, long long ldo, const void* C, int ctype, long long ldc, const GenSpec* gen, double* scratch,
                 int sm, void* stream) {
    const cudaStream_t st = (cudaStream_t)stream;
    const RoundScratch w = round_scratch(scratch, m, n, sm);
    if (xtype == 2)
        return run_round_v((const double*)X, m, n, ldx, f, g, (double*)out, ldo, StoredCost<double>{(const double*)C, ldc}, w,
                           sm, st);
    if (ctype == 3) return run_round_v((const float*)X, m, n, ldx, f, g, (float*)out, ldo, PointsCost{*gen}, w, sm, st);
    if (ctype == 1)
        return run_round_v((const float*)X, m, n, ldx, f, g, (float*)out, ldo, StoredCost<Bf16>{(const Bf16*)C, ldc}, w, sm,
                           st);
    return run_round_v((const float*)X, m, n, ldx, f, g, (float*)out, ldo, StoredCost<float>{(const float*)C, ldc}, w, sm, st);
}

}  // namespace pdot
