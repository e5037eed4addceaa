// pdot_persist.cuh -- passes of one instance in one cooperative launch
// (included by pdot_kernels.cu after pdot_pass.cuh).
//
// What bounded an iteration as two kernels (plan pass, dual update) was not
// the memory: at 64 x 64 the two took 17 us for a few KB, at 4096 x 4096 about
// 12 us of 70 were launches, ramp-up, the first loads' chain (descriptor,
// controller, duals, plan) and the dual update's own chain.  Here every warp
// keeps its plan tile for all passes of a check period:
//   tile    as pdot_pass.cuh (deferred plan writes, the same sums), but the
//           ring of shared-memory stages is not refilled at a pass's end: the
//           passes alternate their row order, so the next pass starts with the
//           groups the last one ended with.  A tile of up to 12 rows (8 with
//           the compensated reduced cost) stays in shared memory for the whole
//           launch, a taller one saves as many rows of C and X per pass;
//   barrier (all row and column partial sums are written);
//   dual    the arithmetic of dual_tile, one CTA per vector tile;
//   barrier (the tiles' step scalars are written);
//   control every CTA adds the scalars in the order of the last tile of
//           dual_tile and runs finalize_step on its own copy of the controller:
//           the same inputs, so the same decision in every CTA.
// FP64 is the serial part (64 cycles per warp instruction and scheduler), so
// conversions are integer operations (widen) and the dual update's FP64 is
// spread over the CTA's schedulers.  Measured per iteration of a whole call
// (its start and end included), before deferred writes and this kernel ->
// here: constant steps, 64 x 64 15.7 -> 8.8 us, 517 x 301 20.2 -> 12.4,
// 16384 x 16384 904 -> 592; adaptive steps with their checks, 1024 x 1024 27.3
// -> 16.0, 4096 x 4096 74.0 -> 43.8 (two kernels with deferred writes: 53).
// The two barriers are one counter each way (release add, acquire poll), with
// a poll limit; all CTAs are co-resident (cooperative launch, one tile per
// warp).  A CTA that gives up sets the counter's fail bit, which every other
// waiter reads, and the instance's status becomes ST_DEVICE.
#pragma once

namespace pdot {
namespace pers {

typedef lagp::Packed f2;
typedef lagp::Two<f2> f4;
__device__ __forceinline__ f2 pack(float lo, float hi) { return lagp::make2<f2>(lo, hi); }
constexpr int R = lagp::R;
constexpr int ARR = lagp::ARR;
constexpr int SB = 2 * ARR;                  // a stage: four rows of X and C
// Shared memory of a warp: NS stages; 256 bytes of
// scratch (a group's row duals and coordinates during a pass, the warp's group
// sums in the dual update); the pending steps' column duals.  The plain
// reduced cost has three stages, the compensated one two (its duals are pairs;
// it serves plans of less than 4M entries, whose tiles are short).
template <bool CP>
struct Lay {
    static constexpr int NS = CP ? 2 : 3;
    static constexpr int SCR = NS * SB;
    static constexpr int PHI = SCR;              // float4 per step: the high parts of the four rows' duals
    static constexpr int PLO = PHI + 64;         // the low parts
    static constexpr int XS = PLO + 64;          // the rows' coordinates (generated cost), 8 floats per row
    static constexpr int Q = SCR + 256;          // [step][128] high parts, then the low parts
    static constexpr int WARP = (Q + LAG * 512 * (CP ? 2 : 1) + 127) / 128 * 128;
    static constexpr int CTA = TWARPS * WARP;
};

constexpr int HALVE_MIN = 32;               // partial sums per column from which a vector tile is halved
// Grid barrier: thread 0 of a CTA adds and polls, `polls` times at most (the
// library's BARRIER_POLLS: seconds).  Returns false (in every thread of the
// CTA) when it, or another CTA, gave up.
__device__ __forceinline__ bool grid_sync(unsigned* c, unsigned target, int* s_ok, int polls) {
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(c) : "memory");
        unsigned v = 0;
        int it = 0;
        do {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(c) : "memory");
        } while (v < target && ++it < polls);
        if (v < target) atomicOr(c, BARRIER_FAIL);
        *s_ok = v >= target && v < BARRIER_FAIL;
    }
    __syncthreads();
    return *s_ok != 0;
}

// One step's primal update and the sums of the candidate, for RR of a
// group's four rows.  x and c come in the order the rows are taken in; a row
// or column that does not exist has x = 0 and a dual of -inf, which leaves
// every sum as it is.  All of a lane's entries go through a step together
// (4 or 8 independent chains: four warps per scheduler do not hide the packed
// instructions' latency by themselves).
struct Sums {
    f2 csa[2];      // column sums of X+ - X, four columns per lane
    float dxa;      // ||X+ - X||^2
    int rows;       // rows since the sums were last added into FP64
};
// Shared-memory accesses by 32-bit address, for data that only this kernel's
// asm touches between the warp barriers (which carry the compiler fences; a
// clobber on each access made the compiler reload every shared field).
__device__ __forceinline__ f4 lds2(unsigned a) {
    f4 v;
    asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(v.x.v), "=l"(v.y.v) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts2(unsigned a, f2 x, f2 y) {
    asm volatile("st.shared.v2.u64 [%0], {%1, %2};" ::"r"(a), "l"(x.v), "l"(y.v));
}
__device__ __forceinline__ f2 lds1(unsigned a) {
    f2 v;
    asm volatile("ld.shared.u64 %0, [%1];" : "=l"(v.v) : "r"(a));
    return v;
}
__device__ __forceinline__ float lds(unsigned a) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts(unsigned a, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v)); }
// RR consecutive floats (8- or 16-byte aligned).
template <int RR>
__device__ __forceinline__ void ld_rows(unsigned a, float (&v)[RR]) {
    if constexpr (RR == 4) {
        const f4 t = lds2(a);
        lagp::unpack(t.x, v[0], v[1]);
        lagp::unpack(t.y, v[2], v[3]);
    } else {
        lagp::unpack(lds1(a), v[0], v[1]);
    }
}

// A step of RR rows from the given duals: x <- its projection (phi / plo: the
// rows' duals, qs: the lane's columns').
template <int RR, bool CP>
__device__ __forceinline__ void step_rows(f2 (&x)[RR][2], const f2 (&c)[RR][2], unsigned phi, unsigned plo, f2 q0, f2 q1,
                                          f2 l0, f2 l1, f2 nt) {
    float ph[RR], pl[RR];
    ld_rows<RR>(phi, ph);
    if (CP) ld_rows<RR>(plo, pl);
#pragma unroll
    for (int r = 0; r < RR; ++r) {
        const f2 hh = pack(ph[r], ph[r]), ll = CP ? pack(pl[r], pl[r]) : hh;
        x[r][0] = lagp::primal2<CP>(x[r][0], c[r][0], hh, ll, q0, l0, nt);
        x[r][1] = lagp::primal2<CP>(x[r][1], c[r][1], hh, ll, q1, l1, nt);
    }
}
// The sums of a candidate's change (MID: rows in order behind a ragged first
// group -- the sums' 32 rows can end inside a group; rows lo .. hi exist).
template <int RR, bool MID, typename FLUSH>
__device__ __forceinline__ void sum_rows(const f2 (&d)[RR][2], Sums& a, float* rs, int lo, int hi, FLUSH&& flush) {
#pragma unroll
    for (int r = 0; r < RR; ++r) {
        float e[4];
        lagp::unpack(d[r][0], e[0], e[1]);
        lagp::unpack(d[r][1], e[2], e[3]);
        a.csa[0] = lagp::add2(a.csa[0], d[r][0]);
        a.csa[1] = lagp::add2(a.csa[1], d[r][1]);
#pragma unroll
        for (int k = 0; k < 4; ++k) a.dxa = fmaf(e[k], e[k], a.dxa);
        rs[r] = ((e[0] + e[1]) + e[2]) + e[3];
        if (MID && r >= lo && r < hi && ++a.rows == FLUSH_ROWS) flush();
    }
}

// What a vector tile's update needs besides the partial sums, per lane
// (loaded by the warps that use it, before the barrier where it can be).
struct DualPre {
    double b, r, y, ybar;
};
// A vector tile is updated by one CTA (half < 0), or its entries of even and
// of odd index by one CTA each (half 0 and 1; lanes 0 .. 15 hold them, and 16 ..
// 31 the same ones in the sums' upper four groups).
__device__ __forceinline__ int vec_entry(int lvt, int half, int lane) {
    return lvt * VE + (half < 0 ? lane : (lane & 15) * 2 + half);
}
__device__ __forceinline__ void dual_pre(const Inst& I, const Ctrl& S, int lvt, int half, DualPre& d) {
    const long long m = I.m, n = I.n, e = vec_entry(lvt, half, threadIdx.x & 31);
    d.b = d.r = d.y = d.ybar = 0.0;
    if (e >= m + n) return;
    const double* Vc = slot_v(I, S.cur);
    d.b = e < m ? I.f[e] : I.g[e - m];
    d.r = Vc[m + n + e];
    d.y = Vc[e];
    if (S.k != 0) d.ybar = slot_v(I, S.bar)[e];
}

// dual_tile on the CTA's copy of the controller, with FP32 row partials and
// no ticket: the tile's scalars go to vpart (an odd half's four words on).
// FP64 takes 64 cycles per warp instruction on each scheduler, so what
// follows the partial sums is spread over four warps (four schedulers): each adds the eight group sums, then
// warp 0 forms the duals and ||dy||^2, warp 1 dy^T A dx, warp 2 the tile's
// slice of ||dX||^2, warp 3 the new sums and averages.
// A column's partial sums are one per tile of rows, up to 570 in eight groups:
// two warps per scheduler take turns for 64 cycles each.  Halves of a tile
// take four warps of full lanes (16 entries x 2 groups), one per scheduler,
// and the scalars' tree over a tile's 32 lanes ends with even + odd, so its
// bits are those of a whole tile.
__device__ __forceinline__ void dual_part(const Inst& I, const Ctrl& S, int lvt, int half, const DualPre& d, int t0, int t1,
                                          unsigned char* scr, int pitch) {
    // scr: 256 bytes per warp, `pitch` bytes apart
    const int m = (int)I.m, n = (int)I.n;
    const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5;
    const int off = half < 0 ? 0 : lane >> 4 << 2, at = half < 0 ? lane : lane & 15;
    auto sgrp = [&](int g2) -> double& { return reinterpret_cast<double*>(scr + g2 * pitch)[at]; };
    const int e = vec_entry(lvt, half, lane);
    const bool row = e < m, col = !row && e < m + n;
    if (half < 0 || grp < 4) {
        double s = 0.0;
        if (lvt * VE < m) s = group_sum<4>(reinterpret_cast<const float*>(I.rowpart) + e, m, I.nstrips, grp, row, off);
        if (lvt * VE + VE > m) {
            const double c = group_sum<16>(I.colpart + (e - m), (int)I.ldx, I.nchunks, grp, col, off);
            if (col) s = c;
        }
        sgrp(grp + off) = s;
    }
    if (grp == (half < 0 ? 2 : 4) && half <= 0) {
        double a2 = 0.0;
        for (int tt = t0 + lane; tt < t1; tt += 32) a2 += __ldcg(I.tpart + (long long)tt * TP);
        a2 = warp_sum(a2);
        if (lane == 0) I.vpart[(long long)lvt * VP + 2] = a2;
    }
    __syncthreads();
    if (grp == 0 || grp == 1 || grp == 3) {
        double t = sgrp(0);
#pragma unroll
        for (int g2 = 1; g2 < VG; ++g2) t += sgrp(g2);
        const bool in = (row || col) && lane == at;
        const double yn = d.y + S.sigma * (d.b - (d.r + 2.0 * t));
        if (grp == 3) {
            if (in) {
                slot_v(I, S.nxt)[m + n + e] = d.r + t;
                slot_v(I, S.barn)[e] = S.k == 0 ? yn : d.ybar + S.wavg * (yn - d.ybar);
            }
        } else {
            const double dy = yn - d.y;
            double a = 0.0;
            if (in) a = grp == 0 ? dy * dy : dy * t;
            if (grp == 0 && in) {
                slot_v(I, S.nxt)[e] = yn;
                float2 v;
                split_dual(yn, v.x, v.y);
                I.yf[(long long)((S.h0 + S.npend + 1) % YRING) * I.yslot + e] = v;
            }
            a = warp_sum(a);
            if (lane == 0) I.vpart[(long long)lvt * VP + (half > 0 ? 4 : 0) + grp] = a;
        }
    }
}

}  // namespace pers

// npass passes of an instance, then the pending steps applied and written.
// refs: the instance of every CTA and its place among that instance's CTAs
// (null: all CTAs serve insts[0]).  Instances of one launch only share the
// launch: each has its own barrier counter.
// TC float also serves a generated cost whose tiles stay in shared memory
// (ctype 3: the entries are computed once, when a tile is loaded).
template <typename TC, bool CP>
__global__ void __launch_bounds__(TWARPS * 32, 2)
k_persist(const Inst* __restrict__ insts, const CtaRef* __restrict__ refs, GridSync* gs, int epoch, int npass, int roworder,
          int polls) {
    using namespace pers;
    using pers::pack; using lagp::unpack; using lagp::widen;
    constexpr int DM = GenDims<TC>::value;
    constexpr bool GEN = DM > 0;
    constexpr int DA = GEN ? DM : 1;
    __shared__ Ctrl S;
    __shared__ Inst I;
    __shared__ double s_sum[3], s_wn;
    __shared__ SchedFactors s_fac;
    __shared__ StepPre s_pre;
    __shared__ float s_nt[LAG], s_w[LAG];   // -tau and averaging weight of the pending steps
    __shared__ int s_ok;
    typedef Lay<CP> L;
    constexpr int NS = L::NS;
    extern __shared__ __align__(128) unsigned char dsm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ CtaRef me;
    if (threadIdx.x == 0) me = refs == nullptr ? CtaRef{0, (int)blockIdx.x, (int)gridDim.x} : refs[blockIdx.x];
    __syncthreads();
    insts += me.inst;
    gs += me.inst;
    for (int w = threadIdx.x; w < (int)(sizeof(Inst) / 4); w += blockDim.x)
        reinterpret_cast<int*>(&I)[w] = reinterpret_cast<const int*>(insts)[w];
    __syncthreads();
    for (int w = threadIdx.x; w < (int)(sizeof(Ctrl) / 4); w += blockDim.x)
        reinterpret_cast<int*>(&S)[w] = reinterpret_cast<const int*>(I.ctrl)[w];
    __shared__ unsigned* bar_count;
    if (threadIdx.x == 0) bar_count = &gs->count[epoch & 1];
    if (me.cta == 0 && threadIdx.x == 0) gs->count[(epoch & 1) ^ 1] = 0u;   // for the next launch
    __syncthreads();
    if (S.status != ST_RUNNING) return;

    // ---- this warp's tile ----
    unsigned char* wbase = dsm + warp * L::WARP;
    const unsigned wbase_s = smem_u32(wbase);
    const int per_cta = (I.ntiles + me.count - 1) / me.count;   // at most TWARPS
    const int lt = me.cta * per_cta + warp;
    const bool active = warp < per_cta && lt < I.ntiles;
    const unsigned strip = (unsigned)lt % (unsigned)I.nstrips, chunk = (unsigned)lt / (unsigned)I.nstrips;
    const int n = (int)I.n, m = (int)I.m;
    const int r0 = (int)chunk * I.tile_rows;
    const int nrows = active ? min(I.tile_rows, m - r0) : 0;
    const int NG = (nrows + R - 1) / R;                    // groups of four rows, at r0 + 4 g
    const int j0 = (int)strip * STRIP + lane * 4;
    const bool on = j0 < n;
    const bool gen_fill = !GEN && I.ctype == 3;            // generated cost, computed once into the stages
    const long long ldx = I.ldx, ldc = I.ldc;
    const TC* Ct = GEN ? nullptr : reinterpret_cast<const TC*>(I.C) + (long long)r0 * ldc + j0;   // C at the tile's first row
    float* const X0 = reinterpret_cast<float*>(I.X) + (long long)r0 * ldx + j0;                   // slot 0 there
    const long long xslot = I.xslot;
    const float2* const yf0 = I.yf;
    const long long yslot = I.yslot;
    float* const rowp = reinterpret_cast<float*>(I.rowpart) + (long long)strip * m + r0;
    const int l_row = lane & 3, l_slot = lane >> 2;        // the row dual this lane fetches: step l_slot's of row l_row
    // Group g into stage g % NS: every lane copies the 16 bytes (BF16: 8) of X
    // and of C that it will read itself, so no other lane waits for them.
    // Rows and columns that do not exist are zero-filled.
    const unsigned cbytes = GEN || gen_fill || !on ? 0u : (unsigned)min(4, n - j0) * (unsigned)(GEN ? 0 : sizeof(TC));
    const bool slow_last = nrows % R != 0 || (!GEN && !gen_fill && n % 4 != 0 && r0 + nrows == m && (int)strip == I.nstrips - 1);
    auto issue = [&](int g, unsigned st, const float* Xt) {   // st: g % NS; Xt: X at the tile's first row, column j0
        const unsigned dst = wbase_s + st * SB + (unsigned)lane * 16u;
        const float* xp = Xt + (long long)(g * R) * ldx;
        const TC* cp = GEN ? nullptr : Ct + (long long)(g * R) * ldc;
        if (g != NG - 1 || !slow_last) {
            if (on) {   // (columns that do not exist stay as they were zeroed)
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    lagp::cp16(dst + r * (STRIP * 4), xp, 16u);
                    xp += ldx;
                }
                if constexpr (!GEN) {
                    if (!gen_fill) {
                        // A lane with fewer than four columns copies the row's
                        // padding too (its duals are -inf there).
#pragma unroll
                        for (int r = 0; r < R; ++r) {
                            if constexpr (sizeof(TC) == 4) lagp::cp16(dst + ARR + r * (STRIP * 4), cp, 16u);
                            else lagp::cp8(dst - lane * 8u + ARR + r * (STRIP * 4), cp, 8u);
                            cp += ldc;
                        }
                    }
                }
            }
        } else if (on) {
            // Rows that do not exist are zero-filled; the last matrix row may
            // end with the caller's allocation.
#pragma unroll 1
            for (int r = 0; r < R; ++r) {
                const bool in = g * R + r < nrows;
                lagp::cp16(dst + r * (STRIP * 4), in ? xp + r * ldx : xp, in ? 16u : 0u);
                if constexpr (!GEN) {
                    if (!gen_fill) {
                        if constexpr (sizeof(TC) == 4)
                            lagp::cp16(dst + ARR + r * (STRIP * 4), in ? cp + r * ldc : cp, in ? cbytes : 0u);
                        else
                            lagp::cp8(dst - lane * 8u + ARR + r * (STRIP * 4), in ? cp + r * ldc : cp, in ? cbytes : 0u);
                    }
                }
            }
        }
    };
    // Columns that do not exist: zeros in every stage, once.
    if (!on)
        for (int o = 0; o < NS * SB; o += STRIP * 4) *reinterpret_cast<float4*>(wbase + o + lane * 16) = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncwarp();

    // Generated cost: the lane's four columns' coordinates.
    float gy[4][DA];
    int g_kind = 0, g_d = 0;
    float g_div = 1.f, g_inv = 1.f;
    if constexpr (GEN) {
        g_kind = I.gen.kind;
        g_d = I.gen.d;
        g_div = I.gen.div;
        g_inv = I.gen.inv;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
#pragma unroll
            for (int k = 0; k < DA; ++k)
                gy[e][k] = (active && k < g_d && j0 + e < n) ? __ldg(I.gen.ys + (long long)(j0 + e) * g_d + k) : 0.f;
        }
    }
    if (gen_fill && active) {
        // (The columns' coordinates are read once: eight floats apart, a warp's
        // loads of them conflict in every bank.  Read for each row, a launch at
        // 1500 x 1400 from 8 coordinates took 52 us more.)
        const GenSpec gp = I.gen;
        float y[4][GEN_DMAX];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
#pragma unroll
            for (int k = 0; k < GEN_DMAX; ++k)
                y[e][k] = (k < gp.d && j0 + e < n) ? __ldg(gp.ys + (long long)(j0 + e) * gp.d + k) : 0.f;
        }
        for (int r = 0; r < nrows; ++r) {
            const float* x = gp.xs + (long long)(r0 + r) * gp.d;
            float c[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) c[e] = j0 + e < n ? gen_cost<GEN_DMAX>(gp.kind, gp.d, x, y[e], gp.div, gp.inv) : 0.f;
            st4(reinterpret_cast<float*>(wbase + (r / R) * SB + ARR + (r % R) * (STRIP * 4)) + lane * 4, c);
        }
        __syncwarp();
    }

    // ---- pass state ----
    const unsigned phi = wbase_s + L::PHI, plo = wbase_s + L::PLO, xsb = wbase_s + L::XS;
    const unsigned qs = wbase_s + L::Q + (unsigned)lane * 16u;
    const unsigned nt_s = smem_u32(s_nt), w_s = smem_u32(s_w);
    f2 qc[2] = {}, qcl[CP ? 2 : 1] = {}, ntc = {};   // the current step's column duals and -tau
    Sums a = {};
    double cs[4] = {0.0, 0.0, 0.0, 0.0}, dx2 = 0.0;
    int np = 0;
    bool dfirst = false, flushed = false;
    auto load_q = [&](int ring, f2 (&h)[2], f2 (&l)[CP ? 2 : 1]) {
        const float2* y = yf0 + ring * yslot + m + j0;
        float2 v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = (active && j0 + e < n) ? y[e] : make_float2(-CUDART_INF_F, 0.f);
        h[0] = pack(v[0].x, v[1].x);
        h[1] = pack(v[2].x, v[3].x);
        if (CP) {
            l[0] = pack(v[0].y, v[1].y);
            l[CP ? 1 : 0] = pack(v[2].y, v[3].y);
        }
    };
    auto flush_sums = [&]() {
        float v[4];
        unpack(a.csa[0], v[0], v[1]);
        unpack(a.csa[1], v[2], v[3]);
        if (flushed) {
#pragma unroll
            for (int e = 0; e < 4; ++e) cs[e] += widen(v[e]);
            dx2 += widen(a.dxa);
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) cs[e] = widen(v[e]);
            dx2 = widen(a.dxa);
        }
        flushed = true;
        a = Sums{};
    };
    // Rows RB .. RB + RR of a group (in the order they are taken in: DESC, the
    // stage's rows from the last to the first).  WRITE: apply the pending steps
    // to X and D and write both (Dg, Xg: D and the written X at the group's
    // first row); fin: no candidate.
    auto rows = [&](auto rr_c, auto rb_c, auto write_c, auto desc_c, auto mid_c, unsigned sl, int count, bool fin, float* Dg,
                    float* Xg, const float4 (&dn)[2], float* rs) {
        constexpr int RR = decltype(rr_c)::value, RB = decltype(rb_c)::value;
        constexpr bool WRITE = decltype(write_c)::value, DESC = decltype(desc_c)::value, MID = decltype(mid_c)::value;
        constexpr int ROW0 = DESC ? R - 1 - RB : RB, DR = DESC ? -1 : 1;   // the stage's rows
        f2 x[RR][2], c[RR][2];
        float4 dv[WRITE ? RR : 1];
        if (WRITE) {
#pragma unroll
            for (int r = 0; r < RR; ++r) dv[WRITE ? r : 0] = dn[WRITE ? r : 0];
        }
#pragma unroll
        for (int r = 0; r < RR; ++r) {
            const int o = (ROW0 + DR * r) * (STRIP * 4);
            const f4 tx = lds2(sl + o);
            x[r][0] = tx.x; x[r][1] = tx.y;
            if constexpr (GEN) {
                float cc[4];
                lagp::gen_row<DA>(reinterpret_cast<const float*>(wbase + L::XS) + (ROW0 + DR * r) * 8, gy, g_kind, g_div,
                                  g_inv, cc);
                c[r][0] = pack(cc[0], cc[1]);
                c[r][1] = pack(cc[2], cc[3]);
            } else if constexpr (sizeof(TC) == 4) {
                const f4 t = lds2(sl + ARR + o);
                c[r][0] = t.x; c[r][1] = t.y;
            } else {
                const unsigned long long t = lds1(sl - (unsigned)lane * 8u + ARR + o).v;
                const unsigned lo = (unsigned)t, hi = (unsigned)(t >> 32);
                c[r][0] = pack(__uint_as_float(lo << 16), __uint_as_float(lo & 0xffff0000u));
                c[r][1] = pack(__uint_as_float(hi << 16), __uint_as_float(hi & 0xffff0000u));
            }
        }
#pragma unroll 1
        for (int s = 0; s < np; ++s) {
            const f4 qh = lds2(qs + s * (STRIP * 4));
            f4 ql = qh;
            if (CP) ql = lds2(qs + (LAG + s) * (STRIP * 4));
            const float nt = lds(nt_s + 4 * s);
            f2 old[WRITE ? RR : 1][2];
            if (WRITE) {
#pragma unroll
                for (int r = 0; r < RR; ++r) { old[WRITE ? r : 0][0] = x[r][0]; old[WRITE ? r : 0][1] = x[r][1]; }
            }
            step_rows<RR, CP>(x, c, phi + 16 * s + 4 * RB, plo + 16 * s + 4 * RB, qh.x, qh.y, ql.x, ql.y, pack(nt, nt));
            if (WRITE) {
                const float w = lds(w_s + 4 * s);
                const bool first = s == 0 && dfirst;
#pragma unroll
                for (int r = 0; r < RR; ++r) {
                    float4& v = dv[WRITE ? r : 0];
                    float d0, d1, d2, d3;
                    unpack(lagp::sub2(x[r][0], old[WRITE ? r : 0][0]), d0, d1);
                    unpack(lagp::sub2(x[r][1], old[WRITE ? r : 0][1]), d2, d3);
                    v.x = avg_dev_next(v.x, d0, w, first);
                    v.y = avg_dev_next(v.y, d1, w, first);
                    v.z = avg_dev_next(v.z, d2, w, first);
                    v.w = avg_dev_next(v.w, d3, w, first);
                }
            }
        }
        if (WRITE) {
#pragma unroll
            for (int r = 0; r < RR; ++r) {
                const int rr = ROW0 + DR * r;
                if (rr < count && on) {
                    f4 t;
                    t.x = x[r][0]; t.y = x[r][1];
                    *reinterpret_cast<f4*>(Xg + rr * ldx) = t;
                    *reinterpret_cast<float4*>(Dg + rr * ldx) = dv[WRITE ? r : 0];
                    sts2(sl + rr * (STRIP * 4), x[r][0], x[r][1]);   // the stage holds the written plan
                }
            }
            if (fin) return;
        }
        f2 d[RR][2];
#pragma unroll
        for (int r = 0; r < RR; ++r) { d[r][0] = x[r][0]; d[r][1] = x[r][1]; }
        step_rows<RR, CP>(d, c, phi + 16 * LAG + 4 * RB, plo + 16 * LAG + 4 * RB, qc[0], qc[1], qcl[0], qcl[CP ? 1 : 0], ntc);
#pragma unroll
        for (int r = 0; r < RR; ++r) {
            d[r][0] = lagp::sub2(d[r][0], x[r][0]);
            d[r][1] = lagp::sub2(d[r][1], x[r][1]);
        }
        sum_rows<RR, MID>(d, a, rs + RB, (DESC ? R - count : 0) - RB, (DESC ? R : count) - RB, flush_sums);
    };
    // D of two rows (rb and rb + 1 in the order they are taken in).  A stored
    // cost's are requested two rows ahead of their use: 4096 x 4096, 55.0K ->
    // 52.4K cycles per traversal.  A generated cost and the compensated one
    // have no registers to hold them and load them in place (they spilled, and
    // a spilled value is read from L2 after a barrier: generated, 4096 x 4096,
    // 88K -> 92K cycles per pass; compensated, 64 x 64, 18.0K -> 19.7K).
    constexpr bool AHEAD = !GEN && !CP;
    auto load_d = [&](const float* Dg, int count, int rb, bool desc, float4 (&d)[2]) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int rr = desc ? R - 1 - rb - r : rb + r;
            d[r] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (rr < count && on && !dfirst) d[r] = __ldcg(reinterpret_cast<const float4*>(Dg + rr * ldx));
        }
    };
    float4 dn[2];   // (writing passes) D of the next two rows
    // ncount, Dn: the next group's rows and D (0: none).
    auto group = [&](auto desc_c, auto mid_c, bool wr, unsigned sl, int count, bool fin, float* Dg, float* Xg, int ncount,
                     const float* Dn, float* rs) {
        typedef std::integral_constant<int, 0> I0;
        typedef std::integral_constant<int, 2> I2;
        typedef std::integral_constant<int, 4> I4;
        constexpr bool DESC = decltype(desc_c)::value;
        if (!wr && CP) {   // (the compensated cost's pairs leave registers for two rows at a time)
            rows(I2(), I0(), std::false_type(), desc_c, mid_c, sl, count, false, nullptr, nullptr, dn, rs);
            rows(I2(), I2(), std::false_type(), desc_c, mid_c, sl, count, false, nullptr, nullptr, dn, rs);
        } else if (!wr) {
            rows(I4(), I0(), std::false_type(), desc_c, mid_c, sl, count, false, nullptr, nullptr, dn, rs);
        } else {
            if (!AHEAD) load_d(Dg, count, 0, DESC, dn);
            float4 d[2] = {dn[0], dn[1]};
            if (AHEAD) load_d(Dg, count, 2, DESC, dn);
            rows(I2(), I0(), std::true_type(), desc_c, mid_c, sl, count, fin, Dg, Xg, d, rs);
            if (!AHEAD) load_d(Dg, count, 2, DESC, dn);
            d[0] = dn[0];
            d[1] = dn[1];
            if (AHEAD && ncount > 0) load_d(Dn, ncount, 0, DESC, dn);
            rows(I2(), I2(), std::true_type(), desc_c, mid_c, sl, count, fin, Dg, Xg, d, rs);
        }
    };

    // Row duals of a group, one per lane: this lane's step (pending steps in
    // slots 0.., the current one in slot LAG) of row l_row.
    const float2 none = make_float2(-CUDART_INF_F, 0.f);   // a row that does not exist
    auto row_dual = [&](int ring, int g) -> float2 {
        return g * R + l_row < nrows ? yf0[ring * yslot + r0 + g * R + l_row] : none;
    };

    // One traversal of the tile.  pw: the first group's row duals; fin: only
    // apply and write the pending steps.
    auto traverse = [&](bool fin, float2 pw) {
        const bool rev = (S.passes & 1) != 0;
        const bool desc = rev && roworder, mid = desc && nrows % R != 0;
        const bool wr = fin || np == LAG;
        const int g0 = rev ? NG - 1 : 0, dg = rev ? -1 : 1;
        const int ring = l_slot < np ? (S.h0 + l_slot) % YRING : l_slot == LAG && !fin ? (S.h0 + np) % YRING : -1;
        const unsigned at = 4u * (unsigned)(l_slot * 4 + (desc ? R - 1 - l_row : l_row));
        float xw = 0.f;
        auto fetch_x = [&](int g) {
            if constexpr (GEN) {
                const int r = lane >> 3, k = lane & 7;
                xw = (k < g_d && g * R + r < nrows) ? __ldg(I.gen.xs + (long long)(r0 + g * R + r) * g_d + k) : 0.f;
            }
        };
        fetch_x(g0);
        const float* Xt = X0 + S.xcur * xslot;
        float* Dt = X0 + S.xbar * xslot;
        float* Xo = X0 + S.xdst * xslot;
        const float2* py = ring >= 0 ? yf0 + ring * yslot + r0 + l_row : nullptr;
        float* rp = rowp + (desc ? R - 1 - (lane >> 3) : lane >> 3);
        unsigned st = (unsigned)g0 % NS;
        if (AHEAD && wr) load_d(Dt + (long long)(g0 * R) * ldx, min(R, nrows - g0 * R), 0, desc, dn);
#pragma unroll 1
        for (int t = 0, g = g0; t < NG; ++t, g += dg) {
            const int count = min(R, nrows - g * R);
            if (l_slot <= LAG) {
                sts(phi + at, pw.x);
                if (CP) sts(plo + at, pw.y);
            }
            if constexpr (GEN) sts(xsb + 4u * (unsigned)lane, xw);
            if (t + 1 < NG) {
                if (py != nullptr) pw = (g + dg) * R + l_row < nrows ? py[(g + dg) * R] : none;
                fetch_x(g + dg);
            }
            lagp::cp_wait<NS - 1>();   // (one commit per group taken, empty or not: the oldest is this group)
            __syncwarp();
            float rsv[R] = {0.f, 0.f, 0.f, 0.f};
            const unsigned sl = wbase_s + st * SB + (unsigned)lane * 16u;
            float* Dg = Dt + (long long)(g * R) * ldx;
            float* Xg = Xo + (long long)(g * R) * ldx;
            const int ncount = t + 1 < NG ? min(R, nrows - (g + dg) * R) : 0;
            const float* Dn = Dg + (long long)(dg * R) * ldx;
            if (!desc) group(std::false_type(), std::false_type(), wr, sl, count, fin, Dg, Xg, ncount, Dn, rsv);
            else if (!mid) group(std::true_type(), std::false_type(), wr, sl, count, fin, Dg, Xg, ncount, Dn, rsv);
            else group(std::true_type(), std::true_type(), wr, sl, count, fin, Dg, Xg, ncount, Dn, rsv);
            __syncwarp();
            if (t + NS < NG) issue(g + NS * dg, st, Xt);   // (the same stage)
            lagp::cp_commit();
            st = rev ? (st == 0 ? NS - 1 : st - 1) : (st == NS - 1 ? 0 : st + 1);
            if (!fin) {
                const float tot = lagp::rows4_sum(rsv, lane);
                const int r = desc ? R - 1 - (lane >> 3) : lane >> 3;
                if ((lane & 7) == 0 && r < count) rp[g * R] = tot;
                if (!mid) {
                    a.rows += count;
                    if (a.rows >= FLUSH_ROWS) flush_sums();
                }
            }
        }
    };

    // First loads: the groups the first pass starts with.
    {
        const bool rev = (S.passes & 1) != 0;
        const float* Xt = X0 + S.xcur * xslot;
        for (int t = 0; t < NS; ++t) {
            const int g = rev ? NG - 1 - t : t;
            if (t < NG) issue(g, (unsigned)g % NS, Xt);
            lagp::cp_commit();
        }
    }
    bool ok = true;
    float2 pw = none;
    if (active) {
        const int h = (S.h0 + S.npend) % YRING;
        load_q(h, qc, qcl);
        if (l_slot == LAG) pw = row_dual(h, (S.passes & 1) ? NG - 1 : 0);
    }
    // The CTA's first vector tile (its slice of the plan tiles' ||dX||^2).  Tiles
    // with column duals are halved where there are CTAs for all halves and the
    // columns' sums are long enough to pay for the halves' extra additions
    // (0.5K cycles in every CTA).  The longest vector tile, whole -> halved:
    // 64 x 64 (32 partial sums per column) 5.2K -> 3.9K cycles, 1024 x 1024
    // (256) 11.2K -> 8.5K, 1137 x 155 (569) 19.2K -> 14.7K.  Only the
    // compensated kernels: the plain ones serve plans whose vector tiles fill
    // the CTAs, and lost 2.7 % at 4096 x 4096 to the spills of the unused code.
    constexpr bool HALVES = CP;
    __shared__ int s_sl[2], s_half, s_rows;
    int vt0 = me.cta;
    if constexpr (HALVES) {
        const int nr = (int)(I.m / VE);   // tiles of row duals only
        const bool halve = I.nchunks >= HALVE_MIN && 2 * I.nvt - nr <= me.count;
        const bool mine = halve && vt0 >= nr;
        if (threadIdx.x == 0) {
            s_rows = halve ? nr : I.nvt;
            s_half = mine ? (vt0 - nr) & 1 : -1;
        }
        if (mine) vt0 = nr + (vt0 - nr) / 2;
        __syncthreads();
    }
    if (threadIdx.x < 2 && vt0 < I.nvt) s_sl[threadIdx.x] = (int)((long long)I.ntiles * (vt0 + (int)threadIdx.x) / I.nvt);
    for (int ps = 0; ps < npass; ++ps) {
        if (active) {
            const float t0 = -(float)S.tau;
            ntc = pack(t0, t0);
            flushed = false;
            a = Sums{};
            traverse(false, pw);
            flush_sums();
            if (on) {
                double* cp = I.colpart + (long long)chunk * ldx + j0;
                reinterpret_cast<double2*>(cp)[0] = make_double2(cs[0], cs[1]);
                reinterpret_cast<double2*>(cp)[1] = make_double2(cs[2], cs[3]);
            }
            const double t = warp_sum(dx2);
            if (lane == 0) I.tpart[(long long)lt * TP] = t;
        }
        DualPre d;
        if (warp < 4 && vt0 < I.nvt) dual_pre(I, S, vt0, HALVES ? s_half : -1, d);   // (arrives during the barrier)
        if (!grid_sync(bar_count, (unsigned)(me.count * (2 * ps + 1)), &s_ok, polls)) { ok = false; break; }
        if (vt0 < I.nvt) dual_part(I, S, vt0, HALVES ? s_half : -1, d, s_sl[0], s_sl[1], dsm + L::SCR, L::WARP);
        if (threadIdx.x == 5 * 32) {
            // What the controller needs besides the sums, by a warp that has
            // done its part of the dual update.
            if (S.adaptive_step) s_fac = sched_factors(&S, S.total);
            s_wn = 1.0 / (double)(S.k + 2);
            s_pre = step_pre(&S);
        }
        for (int vt = (HALVES ? me.cta : vt0) + me.count; vt < (HALVES ? s_rows : I.nvt); vt += me.count) {
            __syncthreads();   // the scratch is reused
            if (warp < 4) dual_pre(I, S, vt, -1, d);
            dual_part(I, S, vt, -1, d, (int)((long long)I.ntiles * vt / I.nvt), (int)((long long)I.ntiles * (vt + 1) / I.nvt), dsm + L::SCR,
                      L::WARP);
        }
        if (!grid_sync(bar_count, (unsigned)(me.count * (2 * ps + 2)), &s_ok, polls)) { ok = false; break; }
        // The step scalars, one warp each; meanwhile all warps request what
        // the next pass starts with, for either decision.
        const int h_old = (S.h0 + S.npend) % YRING, np_old = S.npend;
        const bool wrote = np_old == LAG;
        const int np_base = wrote ? 0 : np_old, h_base = wrote ? h_old : S.h0;
        const long long total_old = S.total;
        if (warp < 3) {
            const int nvt = I.nvt;
            double b = 0.0;
#pragma unroll 1
            for (int v0 = lane; v0 - lane < nvt; v0 += 32 * 8) {
                double t[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) t[u] = ld_part(I.vpart + (long long)(v0 + 32 * u) * VP + warp, v0 + 32 * u < nvt);
                if (HALVES && warp < 2 && s_rows < nvt) {   // halved tiles: even + odd
                    double o[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int v = v0 + 32 * u;
                        o[u] = ld_part(I.vpart + (long long)v * VP + 4 + warp, v >= s_rows && v < nvt);
                    }
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        if (v0 - lane + 32 * u >= nvt) break;
                        t[u] += o[u];
                    }
                }
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    if (v0 - lane + 32 * u >= nvt) break;
                    b = v0 == lane && u == 0 ? t[u] : b + t[u];
                }
            }
            b = warp_sum(b);
            if (lane == 0) s_sum[warp] = b;
        }
        f2 qn[2], qnl[CP ? 2 : 1];
        float2 pa = none, pr = none;   // row duals of the next pass's first group: accepted, rejected
        if (active) {
            load_q((h_old + 1) % YRING, qn, qnl);
            const int g = (S.passes & 1) ? 0 : NG - 1;
            if (l_slot == LAG) {
                pa = row_dual((h_old + 1) % YRING, g);
                pr = row_dual(h_old, g);
            } else if (l_slot <= np_base && l_slot < LAG) {
                pa = pr = row_dual((h_base + l_slot) % YRING, g);
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            finalize_step(&S, s_pre, s_sum[2], s_sum[0], s_sum[1], s_fac, s_wn);
            if (S.total != total_old) {
                s_nt[np_base] = -s_pre.tau;
                s_w[np_base] = s_pre.wavg;
            }
        }
        __syncthreads();
        np = S.npend;
        dfirst = S.pfirst != 0;
        pw = pr;
        if (S.total != total_old) {   // accepted
            sts2(qs + np_base * (STRIP * 4), qc[0], qc[1]);
            if (CP) sts2(qs + (LAG + np_base) * (STRIP * 4), qcl[0], qcl[CP ? 1 : 0]);
            qc[0] = qn[0]; qc[1] = qn[1];
            qcl[0] = qnl[0]; qcl[CP ? 1 : 0] = qnl[CP ? 1 : 0];
            pw = pa;
        }
        if (S.status != ST_RUNNING) break;
    }
    // The pending steps, written.
    if (ok && active && np > 0) traverse(true, pw);
    if (!ok && lane == 0) atomicExch(&I.ctrl->status, ST_DEVICE);   // a barrier gave up
    if (me.cta != 0) return;
    __syncthreads();
    if (threadIdx.x == 0 && S.npend > 0) {
        S.h0 = (S.h0 + S.npend) % YRING;
        S.npend = 0;
        S.xcur = S.xdst;
        S.xdst = plan_dst(S.xcur, S.xbar, S.xanc);
    }
    __syncthreads();
    const int sw = (int)(offsetof(Ctrl, status) / 4);   // a running status stays as it is (a CTA may have failed)
    for (int w = threadIdx.x; w < (int)(sizeof(Ctrl) / 4); w += blockDim.x)
        if (w != sw || S.status != ST_RUNNING)
            reinterpret_cast<int*>(I.ctrl)[w] = reinterpret_cast<const int*>(&S)[w];
}

// Self-test of the barrier's failure path: every CTA waits for one arrival
// more than there are CTAs, gives up after `polls` polls or when another one
// has, and records the status k_persist records then.
__global__ void k_watchdog_selftest(unsigned* count, int polls, int* status) {
    __shared__ int s_ok;
    const bool ok = pers::grid_sync(count, gridDim.x + 1, &s_ok, polls);
    if (threadIdx.x == 0) atomicExch(status, ok ? ST_OK : ST_DEVICE);
}

}  // namespace pdot
