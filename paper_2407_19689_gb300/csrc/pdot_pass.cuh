// pdot_pass.cuh -- the plan pass of FP32 plans (included by pdot_kernels.cu).
//
// Deferred plan writes.  A pass needs the current plan X only to form the
// candidate X+ = max(0, X - tau (C - p 1^T - 1 q^T)) and the row and column
// sums of X+ - X; the next pass needs X+ only if the step was accepted.  So a
// pass does not write X+.  The plan buffer keeps an earlier iterate, the
// instance keeps the (tau, p, q) of the accepted steps since then (at most
// LAG), and a pass recomputes those steps on the entries it has just read:
// the same FP32 operations on the same operands, so the same bits.  When LAG
// steps are pending the pass also reads the average's deviation D, applies
// the steps to both and writes them back (in place, unless the buffer is the
// restart anchor).  Per entry a pass then reads C and X (8 B with an FP32
// cost) and every LAG-th pass moves 20 B, instead of 20 B every pass; and
// because X and D are updated in place, C and X of a 4096 x 4096 plan
// (134 MB) nearly fit in L2 from pass to pass.  The price is arithmetic: four
// FP32 operations per entry and pending step.  Measured, the pass alone, FP32
// cost: 4096 x 4096 58.4 -> 37.1 us, 16384 x 16384 820 -> 519 us; BF16 cost
// 16384 x 16384 717 -> 476 us; cost from coordinates 729 -> 503 us.  With LAG
// = 3 a cycle moves 12 B per entry and pass; beyond that the recomputed steps
// cost what the bytes save (the kernel is bound by its instructions and their
// latency at four warps per scheduler, not by HBM any more).
//
// Work split: one warp per tile of 128 columns x tile_rows rows (16-byte
// accesses, four consecutive columns per lane).  Rows are streamed in groups
// of four through a ring of shared-memory stages per warp.  Every lane copies
// the 16 bytes it will read itself (cp.async): the same rows by cp.async.bulk
// took 40 cycles of an SM's bulk-copy engine per 512-byte row, 3.9 TB/s for
// the device whatever the kernel did besides.  The same 12 KB hold three
// stages of C and X, or two of C, X and D.  The group's row duals come with
// its copies, so no load is waited for between groups.
#pragma once

namespace pdot {
namespace lagp {

constexpr int R = 4;                        // rows per group
constexpr int ARR = R * STRIP * 4;          // bytes of one array's rows in a stage (rows 512 B apart)
constexpr int RING = 6 * ARR;               // bytes of stages per warp
constexpr int SMAX = 3;                     // most stages in the ring
constexpr int PSLOT = LAG + 1;              // duals per row: LAG pending steps, then the current step
static_assert(PSLOT == 4, "a row's duals are read as one float4");

constexpr int OFF_REFS = RING;                         // tile of the group in a stage
constexpr int OFF_PHI = OFF_REFS + 16;                 // float4 per stage and row: the high parts of its duals
constexpr int OFF_PLO = OFF_PHI + SMAX * R * 16;       // the low parts (compensated reduced cost)
constexpr int OFF_XS = OFF_PLO + SMAX * R * 16;        // the rows' coordinates (generated cost), 8 floats per row
__host__ __device__ constexpr int warp_smem() { return (OFF_XS + SMAX * R * 32 + 127) / 128 * 128; }
__host__ __device__ constexpr int smem_bytes() { return TWARPS * warp_smem(); }

// A lane's columns in pairs.  Pair: two scalars.  Packed: one 64-bit register
// pair for the f32x2 instructions, each half of which rounds as the scalar
// instruction does.  Packed halves the FP32 instructions but takes moves to
// form its pairs: the cooperative kernel gains from it (4096 x 4096 pass 54.9k
// against 58.2k cycles), this kernel, which runs out of registers, does not
// (39.2 against 37.1 us a pass).
struct __align__(8) Pair {
    float a, b;
};
struct Packed {
    unsigned long long v;
};
template <typename V>
struct __align__(16) Two {
    V x, y;
};
template <typename V>
__device__ __forceinline__ V make2(float lo, float hi) {
    V r;
    if constexpr (std::is_same<V, Pair>::value) {
        r.a = lo;
        r.b = hi;
    } else {
        asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    }
    return r;
}
__device__ __forceinline__ void unpack(Pair v, float& lo, float& hi) { lo = v.a; hi = v.b; }
__device__ __forceinline__ void unpack(Packed v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v.v));
}
__device__ __forceinline__ Pair fma2(Pair a, Pair b, Pair c) { return Pair{fmaf(a.a, b.a, c.a), fmaf(a.b, b.b, c.b)}; }
__device__ __forceinline__ Pair add2(Pair a, Pair b) { return Pair{a.a + b.a, a.b + b.b}; }
__device__ __forceinline__ Pair sub2(Pair a, Pair b) { return Pair{a.a - b.a, a.b - b.b}; }
__device__ __forceinline__ Packed fma2(Packed a, Packed b, Packed c) {
    Packed r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ Packed add2(Packed a, Packed b) {
    Packed r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ Packed sub2(Packed a, Packed b) { return fma2(b, make2<Packed>(-1.f, -1.f), a); }   // one rounding
typedef Pair f2;
typedef Two<Pair> f4;
__device__ __forceinline__ f2 pack(float lo, float hi) { return make2<f2>(lo, hi); }

// Asynchronous copies of 16, 8 and 4 bytes; the bytes past `bytes` are
// zero-filled.
__device__ __forceinline__ void cp16(unsigned dst, const void* src, unsigned bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes));
}
// The same without a byte count: all 16 (8) bytes, or zeros.
__device__ __forceinline__ void cp16z(unsigned dst, const void* src, bool zero) {
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %2, 0; cp.async.cg.shared.global [%0], [%1], 16, p; }" ::"r"(dst), "l"(src),
                 "r"((unsigned)zero)
                );
}
__device__ __forceinline__ void cp8z(unsigned dst, const void* src, bool zero) {
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %2, 0; cp.async.ca.shared.global [%0], [%1], 8, p; }" ::"r"(dst), "l"(src),
                 "r"((unsigned)zero)
                );
}
__device__ __forceinline__ void cp8(unsigned dst, const void* src, unsigned bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(bytes));
}
__device__ __forceinline__ void cp4(unsigned dst, const void* src, unsigned bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes));
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Sum v[r] over the 32 lanes for R = 4 rows with 6 shuffles.  The total of
// row r ends in lanes 8r .. 8r+7.
__device__ __forceinline__ float rows4_sum(const float (&v)[4], int lane) {
    const bool hi16 = lane & 16;
    const float s0 = __shfl_xor_sync(0xffffffffu, hi16 ? v[0] : v[2], 16);
    const float s1 = __shfl_xor_sync(0xffffffffu, hi16 ? v[1] : v[3], 16);
    const float a0 = (hi16 ? v[2] : v[0]) + s0;   // row 0 (low half) / row 2 (high half)
    const float a1 = (hi16 ? v[3] : v[1]) + s1;   // row 1 / row 3
    const bool hi8 = lane & 8;
    const float t = __shfl_xor_sync(0xffffffffu, hi8 ? a0 : a1, 8);
    float b = (hi8 ? a1 : a0) + t;
    b += __shfl_xor_sync(0xffffffffu, b, 4);
    b += __shfl_xor_sync(0xffffffffu, b, 2);
    b += __shfl_xor_sync(0xffffffffu, b, 1);
    return b;
}

// Four generated cost entries of a row with coordinates xr (zero beyond the
// instance's dimension, as are the columns': a zero difference changes none
// of the sums or maxima).  The operations of gen_cost, with the distance kind
// resolved once per row.
template <int DM>
__device__ __forceinline__ void gen_row(const float* xr, const float (&gy)[4][DM], int kind, float div, float inv,
                                        float (&c)[4]) {
    float x[DM];
    if constexpr (DM >= 4) {
#pragma unroll
        for (int k = 0; k < DM; k += 4) {
            const float4 t = *reinterpret_cast<const float4*>(xr + k);
            x[k] = t.x; x[k + 1] = t.y; x[k + 2] = t.z; x[k + 3] = t.w;
        }
    } else {
        const float2 t = *reinterpret_cast<const float2*>(xr);
        x[0] = t.x; x[1] = t.y;
    }
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    if (kind == GK_L1) {
#pragma unroll
        for (int k = 0; k < DM; ++k)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[e] = acc[e] + fabsf(x[k] - gy[e][k]);
    } else if (kind == GK_LINF) {
#pragma unroll
        for (int k = 0; k < DM; ++k)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[e] = fmaxf(acc[e], fabsf(x[k] - gy[e][k]));
    } else {
#pragma unroll
        for (int k = 0; k < DM; ++k)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float t = x[k] - gy[e][k];
                acc[e] = fmaf(t, t, acc[e]);
            }
        if (kind == GK_L2) {
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[e] = sqrtf(acc[e]);
        }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) c[e] = gen_div(acc[e], div, inv);
}

// FP32 -> FP64 without the FP64 pipe (64 cycles per warp instruction and
// scheduler on this part): rebias the exponent in integer arithmetic;
// subnormals, infinities and NaN take the conversion instruction.
__device__ __forceinline__ double widen(float x) {
    const unsigned u = __float_as_uint(x), e = (u >> 23) & 255u;
    if (e - 1u < 254u || (u << 1) == 0u) {
        const unsigned hi = (u & 0x80000000u) | ((u << 1) == 0u ? 0u : ((u & 0x7fffffffu) >> 3) + (896u << 20));
        return __hiloint2double((int)hi, (int)(u << 29));
    }
    return (double)x;
}

__device__ __forceinline__ float at4(const float4& v, int k) { return k == 0 ? v.x : k == 1 ? v.y : k == 2 ? v.z : v.w; }

// reduced_cost on a pair of entries.
template <bool CP, typename V>
__device__ __forceinline__ V reduced2(V c, V ph, V pl, V qh, V ql) {
    if (!CP) return sub2(sub2(c, ph), qh);
    const V s = sub2(c, ph), bv = sub2(s, c);
    const V e = add2(sub2(c, sub2(s, bv)), sub2(sub2(make2<V>(0.f, 0.f), ph), bv));
    return add2(sub2(s, qh), sub2(e, add2(pl, ql)));
}

// One primal step on a pair of entries: projection of x - tau (c - p - q)
// (ntau = -tau).  A column past the matrix has q = -inf, so its reduced cost
// is +inf (or NaN where the caller's padding holds one) and the entry stays 0.
template <bool CP, typename V>
__device__ __forceinline__ V primal2(V x, V c, V ph, V pl, V qh, V ql, V ntau) {
    float a, b;
    unpack(fma2(ntau, reduced2<CP>(c, ph, pl, qh, ql), x), a, b);
    return make2<V>(fmaxf(a, 0.f), fmaxf(b, 0.f));
}

}  // namespace lagp

// FINAL: no candidate step -- apply the pending steps and write X and D (before
// a check, and at the end of a fixed number of steps).
// roworder: a bottom-up pass takes the rows strictly in descending order
// instead of descending groups of four ascending rows (the order of the FP32
// column sums, nothing else).
template <typename TC, bool CP, bool FINAL>
__global__ void __launch_bounds__(TWARPS * 32, 2)
k_pass_lag(const Inst* __restrict__ insts, const TileRef* __restrict__ tmap, const int* __restrict__ Tp,
           unsigned* wctr, int wc, int dir_xor, int roworder) {
    using namespace lagp;
    constexpr int DM = GenDims<TC>::value;
    constexpr bool GEN = DM > 0;                         // C generated, not copied
    constexpr int DA = GEN ? DM : 1;                     // coordinate array size
    constexpr int NRO = GEN ? 1 : 2;                     // arrays of a reading pass: X (, C); a writing pass adds D
    constexpr int S_RO = RING / (NRO * ARR) < SMAX ? RING / (NRO * ARR) : SMAX;
    constexpr int S_WR = RING / ((NRO + 1) * ARR);
    // (Tile count and maps are host-written: read before the wait.)
    const int T = *Tp;
    extern __shared__ __align__(128) unsigned char dsm[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned char* wbase = dsm + warp * warp_smem();
    int* refs = reinterpret_cast<int*>(wbase + OFF_REFS);
    const unsigned wbase_s = smem_u32(wbase);
    prefetch_first_tile(insts, tmap, T);
    pdl_enter();
    reset_other_counters(wctr, wc);

    // ---- producer: a tile's groups ----
    const int l_row = lane & 3, l_slot = lane >> 2;      // lane k < 16 fetches step k / 4's dual of row k % 4
    int p_tile = T, p_left = 0, p_first = 0;             // rows left, rows of the first group
    int p_row = 0, p_drow = 0, p_step = 1;               // the group's first row, its change per group; the rows' order
    int p_d = 0, p_slow = -1;                            // p_left of the group with a ragged last matrix row (-1: none)
    bool p_wr = false, p_rd = false;                     // the tile writes X and D; the stored D is read
    const float* p_x = nullptr;                          // X (and C) at the group's first row, this lane's columns
    const TC* p_c = nullptr;
    long long p_ldx = 0, p_ldc = 0, p_doff = 0;          // row strides; D's offset from X
    unsigned p_xb = 0, p_cb = 0;                         // bytes of X and of C that this lane has in a row
    const float2* p_y = nullptr;                         // this lane's step of the row duals
    const float* p_xs = nullptr;
    bool q_first = true;
    auto next_tile = [&]() {
        for (;;) {
            p_tile = tile_next(&wctr[wc], q_first);
            if (p_tile >= T) return;
            const TileRef tr = tmap[p_tile];
            const Inst& I = insts[tr.inst];
            const Ctrl& Sc = *I.ctrl;
            const int np = Sc.npend;
            if (FINAL ? (np == 0 || (Sc.status != ST_RUNNING && Sc.status != ST_NUMERIC)) : Sc.status != ST_RUNNING)
                continue;
            const unsigned strip = (unsigned)tr.local % (unsigned)I.nstrips, chunk = (unsigned)tr.local / (unsigned)I.nstrips;
            const long long c0 = (long long)strip * STRIP;
            const int ncols = (int)min((long long)STRIP, I.n - c0);
            const int r0 = (int)chunk * I.tile_rows;
            const int r1 = min(r0 + I.tile_rows, (int)I.m);
            const bool rev = pass_reversed(Sc, dir_xor);
            p_left = r1 - r0;
            p_step = 1;
            p_first = min(R, p_left);
            p_drow = R;
            int start = r0;
            if (rev) {
                p_drow = -R;
                if (roworder) {
                    start = r1 - 1;
                    p_step = -1;
                } else {
                    start = r0 + (p_left - 1) / R * R;
                    p_first = r1 - start;                // the ragged group comes first
                }
            }
            p_row = start;
            // The group that holds the last matrix row of a ragged strip: the
            // first one of a bottom-up pass, the last one of a top-down pass.
            p_slow = -1;
            if (!GEN && ncols % 4 != 0 && r1 == (int)I.m) p_slow = rev ? p_left : (p_left - 1) % R + 1;
            p_wr = FINAL || np == LAG;
            p_rd = p_wr && !Sc.pfirst;
            const bool on = lane * 4 < ncols;
            p_xb = on ? 16u : 0u;
            p_ldx = I.ldx;
            p_x = reinterpret_cast<const float*>(I.X) + (long long)Sc.xcur * I.xslot + start * p_ldx + c0 + (on ? lane * 4 : 0);
            p_doff = (long long)(Sc.xbar - Sc.xcur) * I.xslot;
            if constexpr (!GEN) {
                p_cb = on ? (unsigned)min(4, ncols - lane * 4) * (unsigned)sizeof(TC) : 0u;
                p_ldc = I.ldc;
                p_c = reinterpret_cast<const TC*>(I.C) + start * p_ldc + c0 + (on ? lane * 4 : 0);
            }
            // Duals of the pending steps in slots 0.., of the current step in slot LAG.
            p_y = nullptr;
            if (l_slot < np) p_y = I.yf + (long long)((Sc.h0 + l_slot) % YRING) * I.yslot;
            else if (l_slot == LAG && !FINAL) p_y = I.yf + (long long)((Sc.h0 + np) % YRING) * I.yslot;
            if constexpr (GEN) {
                p_d = I.gen.d;
                p_xs = I.gen.xs;
            }
            return;
        }
    };
    // The ring: `ns` stages of `sb` bytes, the next stage to fill and to read.
    // Its form follows the tile (reading or writing); it changes only when the
    // ring is empty.  One commit group per group of rows.
    int in_flight = 0, st_i = 0, st_c = 0, ns = S_RO;
    unsigned sb = NRO * ARR;
    bool r_wr = false;
    auto issue = [&]() {
        const int count = p_first;
        const unsigned dst = wbase_s + st_i * sb + (unsigned)lane * 16u;
        const long long sx = p_step * p_ldx, sc = p_step * p_ldc;
        if (count == R && p_left != p_slow) {
            const bool off = p_xb == 0u;
            const float* xr = p_x;
            const TC* cr = p_c;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                cp16z(dst + r * (STRIP * 4), xr, off);
                if (p_rd) cp16z(dst + NRO * ARR + r * (STRIP * 4), xr + p_doff, off);
                xr += sx;
                if constexpr (!GEN) {
                    // A lane with fewer than four columns copies the row's
                    // padding too (its duals are -inf there), except on the
                    // last matrix row, which may end with the allocation.
                    if constexpr (sizeof(TC) == 4) cp16z(dst + ARR + r * (STRIP * 4), cr, off);
                    else cp8z(dst - lane * 8u + ARR + r * (STRIP * 4), cr, off);
                    cr += sc;
                }
            }
        } else {
#pragma unroll 1
            for (int r = 0; r < R; ++r) {
                const bool in = r < count;
                const float* xr = in ? p_x + r * sx : p_x;
                cp16(dst + r * (STRIP * 4), xr, in ? p_xb : 0u);
                if (p_rd) cp16(dst + NRO * ARR + r * (STRIP * 4), xr + p_doff, in ? p_xb : 0u);
                if constexpr (!GEN) {
                    const TC* cr = in ? p_c + r * sc : p_c;
                    if constexpr (sizeof(TC) == 4) cp16(dst + ARR + r * (STRIP * 4), cr, in ? p_cb : 0u);
                    else cp8(dst - lane * 8u + ARR + r * (STRIP * 4), cr, in ? p_cb : 0u);
                }
            }
        }
        if constexpr (!GEN) p_c += p_drow * p_ldc;
        const bool there = l_row < count;
        const int row = p_row + l_row * p_step;
        if (there && p_y != nullptr) {
            const unsigned o = (unsigned)(st_i * R + l_row) * 16u + (unsigned)l_slot * 4u;
            cp4(wbase_s + OFF_PHI + o, &p_y[row].x, 4u);
            if (CP) cp4(wbase_s + OFF_PLO + o, &p_y[row].y, 4u);
        }
        if constexpr (GEN) {
            const int k = l_slot;                        // up to 8 coordinates x 4 rows
            const bool in = there && k < p_d;
            if (k < (DA < 4 ? 4 : DA))
                cp4(wbase_s + OFF_XS + (unsigned)(st_i * R + l_row) * 32u + (unsigned)k * 4u,
                    in ? p_xs + (long long)row * p_d + k : p_xs, in ? 4u : 0u);
        }
        cp_commit();
        if (lane == 0) refs[st_i] = p_tile;
        if (++st_i == ns) st_i = 0;
        ++in_flight;
        p_left -= count;
        p_first = min(R, p_left);
        p_row += p_drow;
        p_x += p_drow * p_ldx;
        if (p_left == 0) next_tile();
    };
    auto refill = [&]() {
        while (p_tile < T && in_flight < ns) {
            if (p_wr != r_wr) {
                if (in_flight > 0) return;
                r_wr = p_wr;
                ns = r_wr ? S_WR : S_RO;
                sb = (NRO + (r_wr ? 1 : 0)) * ARR;
                st_i = st_c = 0;
            }
            issue();
        }
    };
    next_tile();
    refill();

    // ---- consumer ----
    int c_tile = -1, c_local = 0, np = 0, c_chunk = 0, c_left = 0, c_count = 0, rows_in_batch = 0;
    int c_row = 0, c_drow = 0, c_step = 1;               // the group's first row, its change per group; the rows' order
    const Inst* CI = nullptr;
    long long c_ldx = 0, c_n = 0, j0 = 0;
    float* c_xo = nullptr;      // where X and D (matrix row 0, column j0) are written
    float* c_do = nullptr;
    double* c_rowpart = nullptr;
    bool on = false, dfirst = false, flushed = false;
    f2 qc[2], qcl[2], qp[LAG][2], qpl[LAG][2], ntc = {}, ntp[LAG];
    float wp[LAG];
    double cs[4] = {0.0, 0.0, 0.0, 0.0}, dx2 = 0.0;
    f2 csa[2] = {};
    float dxa = 0.f;
    int g_kind = 0;
    float g_div = 1.f, g_inv = 1.f, gy[4][DA];
    auto flush_sums = [&]() {
        float v[4];
        unpack(csa[0], v[0], v[1]);
        unpack(csa[1], v[2], v[3]);
        if (flushed) {
#pragma unroll
            for (int e = 0; e < 4; ++e) cs[e] += widen(v[e]);
            dx2 += widen(dxa);
        } else {   // the first 32 rows: the sums start as these values
#pragma unroll
            for (int e = 0; e < 4; ++e) cs[e] = widen(v[e]);
            dx2 = widen(dxa);
        }
        flushed = true;
        csa[0] = csa[1] = f2{};
        dxa = 0.f;
        rows_in_batch = 0;
    };
    auto flush_tile = [&]() {
        if (FINAL) return;
        flush_sums();
        if (on) {
            double* cp = CI->colpart + (long long)c_chunk * CI->ldx + j0;
            reinterpret_cast<double2*>(cp)[0] = make_double2(cs[0], cs[1]);
            reinterpret_cast<double2*>(cp)[1] = make_double2(cs[2], cs[3]);
        }
        const double d = warp_sum(dx2);
        if (lane == 0) CI->tpart[(long long)c_local * TP + 0] = d;
    };
    auto open_consumer = [&](int t) {
        const TileRef tr = tmap[t];
        CI = &insts[tr.inst];
        const Ctrl& Sc = *CI->ctrl;
        c_local = tr.local;
        const unsigned strip = (unsigned)tr.local % (unsigned)CI->nstrips, chunk = (unsigned)tr.local / (unsigned)CI->nstrips;
        const long long c0 = (long long)strip * STRIP;
        c_chunk = (int)chunk;
        c_n = CI->n;
        c_ldx = CI->ldx;
        const int r0 = (int)chunk * CI->tile_rows;
        const int r1 = min(r0 + CI->tile_rows, (int)CI->m);
        c_left = r1 - r0;
        c_step = 1;
        c_drow = R;
        c_row = r0;
        c_count = min(R, c_left);
        if (pass_reversed(Sc, dir_xor)) {
            c_drow = -R;
            if (roworder) {
                c_row = r1 - 1;
                c_step = -1;
            } else {
                c_row = r0 + (c_left - 1) / R * R;
                c_count = r1 - c_row;
            }
        }
        j0 = c0 + lane * 4;
        on = j0 < c_n;
        np = Sc.npend;
        dfirst = Sc.pfirst != 0;
        float* Xb = reinterpret_cast<float*>(CI->X);
        c_xo = Xb + (long long)Sc.xdst * CI->xslot + j0;
        c_do = Xb + (long long)Sc.xbar * CI->xslot + j0;
        c_rowpart = CI->rowpart + (long long)strip * CI->m;
        if constexpr (GEN) {
            const GenSpec& gs = CI->gen;
            g_kind = gs.kind;
            g_div = gs.div;
            g_inv = gs.inv;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
#pragma unroll
                for (int k = 0; k < DA; ++k)
                    gy[e][k] = (k < gs.d && j0 + e < c_n) ? __ldg(gs.ys + (j0 + e) * gs.d + k) : 0.f;
            }
        }
        const int h0 = Sc.h0;
#pragma unroll
        for (int s = 0; s <= LAG; ++s) {
            if (s < LAG ? s >= np : FINAL) continue;
            const int ring = (h0 + (s == LAG ? np : s)) % YRING;
            const float2* y = CI->yf + (long long)ring * CI->yslot + CI->m + j0;
            float2 v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = j0 + e < c_n ? y[e] : make_float2(-CUDART_INF_F, 0.f);
            const f2 h[2] = {pack(v[0].x, v[1].x), pack(v[2].x, v[3].x)}, l[2] = {pack(v[0].y, v[1].y), pack(v[2].y, v[3].y)};
            if (s < LAG) {
                qp[s % LAG][0] = h[0]; qp[s % LAG][1] = h[1];
                qpl[s % LAG][0] = l[0]; qpl[s % LAG][1] = l[1];
                ntp[s % LAG] = pack(-Sc.ptau[ring], -Sc.ptau[ring]);
                wp[s % LAG] = Sc.pw[ring];
            } else {
                qc[0] = h[0]; qc[1] = h[1];
                qcl[0] = l[0]; qcl[1] = l[1];
            }
        }
        const float t0 = -(float)Sc.tau;
        ntc = pack(t0, t0);
        flushed = false;
        csa[0] = csa[1] = f2{};
        dxa = 0.f;
        rows_in_batch = 0;
    };

    // One group.  FULL: all four rows exist (columns that do not exist hold
    // zeros and have a dual of -inf).  NP: the number
    // of pending steps (-1: read from np).  Which of them runs changes no
    // arithmetic.
    auto group = [&](auto full_c, auto np_c, float (&rsv)[R]) {
        constexpr bool FULL = decltype(full_c)::value;
        constexpr int NP = decltype(np_c)::value;
        const bool wr = FINAL || (NP >= 0 ? NP == LAG : np == LAG);
        const unsigned char* stage = wbase + st_c * sb + lane * 16;
        const float4* phi = reinterpret_cast<const float4*>(wbase + OFF_PHI) + st_c * R;
        const float4* plo = reinterpret_cast<const float4*>(wbase + OFF_PLO) + st_c * R;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            rsv[r] = 0.f;
            if (FULL || r < c_count) {
                const int i = c_row + r * c_step;
                f2 c[2] = {}, x[2] = {};
                float db[4] = {0.f, 0.f, 0.f, 0.f};
                const float4 ph = phi[r];
                float4 pl = make_float4(0.f, 0.f, 0.f, 0.f);
                if (CP) pl = plo[r];
                if constexpr (GEN) {
                    float cc[4];
                    gen_row<DA>(reinterpret_cast<const float*>(wbase + OFF_XS) + (st_c * R + r) * 8, gy, g_kind, g_div,
                                g_inv, cc);
                    c[0] = pack(cc[0], cc[1]);
                    c[1] = pack(cc[2], cc[3]);
                }
                {
                    const f4 tx = *reinterpret_cast<const f4*>(stage + r * (STRIP * 4));
                    x[0] = tx.x; x[1] = tx.y;
                    if constexpr (!GEN) {
                        if constexpr (sizeof(TC) == 4) {
                            const f4 t = *reinterpret_cast<const f4*>(stage + ARR + r * (STRIP * 4));
                            c[0] = t.x; c[1] = t.y;
                        } else {
                            const uint2 t = *reinterpret_cast<const uint2*>(stage - lane * 8 + ARR + r * (STRIP * 4));
                            c[0] = pack(bf16_bits_to_f32(t.x & 0xffffu), bf16_bits_to_f32(t.x >> 16));
                            c[1] = pack(bf16_bits_to_f32(t.y & 0xffffu), bf16_bits_to_f32(t.y >> 16));
                        }
                    }
                    if (wr && !dfirst) {
                        const float4 tb = *reinterpret_cast<const float4*>(stage + NRO * ARR + r * (STRIP * 4));
                        db[0] = tb.x; db[1] = tb.y; db[2] = tb.z; db[3] = tb.w;
                    }
                }
#pragma unroll
                for (int s = 0; s < LAG; ++s) {
                    if (NP >= 0 ? s < NP : s < np) {
                        const f2 hh = pack(at4(ph, s), at4(ph, s)), ll = pack(at4(pl, s), at4(pl, s));
#pragma unroll
                        for (int k = 0; k < 2; ++k) {
                            const f2 v = primal2<CP>(x[k], c[k], hh, ll, qp[s][k], qpl[s][k], ntp[s]);
                            if (wr) {
                                float d0, d1;
                                unpack(sub2(v, x[k]), d0, d1);
                                db[2 * k] = avg_dev_next(db[2 * k], d0, wp[s], s == 0 && dfirst);
                                db[2 * k + 1] = avg_dev_next(db[2 * k + 1], d1, wp[s], s == 0 && dfirst);
                            }
                            x[k] = v;
                        }
                    }
                }
                if (wr && on) {
                    const long long o = (long long)i * c_ldx;
                    f4 t;
                    t.x = x[0]; t.y = x[1];
                    *reinterpret_cast<f4*>(c_xo + o) = t;
                    st4(c_do + o, db);
                }
                if (!FINAL) {
                    const f2 hh = pack(ph.w, ph.w), ll = pack(pl.w, pl.w);
                    float rs = 0.f;
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        const f2 d = sub2(primal2<CP>(x[k], c[k], hh, ll, qc[k], qcl[k], ntc), x[k]);
                        csa[k] = add2(csa[k], d);
                        float d0, d1;
                        unpack(d, d0, d1);
                        dxa = fmaf(d0, d0, dxa);
                        dxa = fmaf(d1, d1, dxa);
                        rs += d0;                                 // row / column sums of X+ - X
                        rs += d1;
                    }
                    rsv[r] = rs;
                }
            }
        }
    };

    while (in_flight > 0) {
        // The oldest group's copies (wait_group counts the newer ones).
        if (in_flight > 2) cp_wait<2>();
        else if (in_flight == 2) cp_wait<1>();
        else cp_wait<0>();
        __syncwarp();
        if (c_left == 0) {
            c_tile = refs[st_c];
            open_consumer(c_tile);
        }
        float rsv[R];
        typedef std::true_type Y;
        typedef std::false_type N;
        if (!FINAL && c_count == R) {
            if (np == 0) group(Y(), std::integral_constant<int, 0>(), rsv);
            else if (np == 1) group(Y(), std::integral_constant<int, 1>(), rsv);
            else if (np == 2) group(Y(), std::integral_constant<int, 2>(), rsv);
            else group(Y(), std::integral_constant<int, 3>(), rsv);
        } else {
            group(N(), std::integral_constant<int, -1>(), rsv);
        }
        // The group's stage has been read: release it and refill the ring.
        __syncwarp();
        if (++st_c == ns) st_c = 0;
        --in_flight;
        refill();
        if (!FINAL) {
            const float tot = rows4_sum(rsv, lane);
            if ((lane & 7) == 0 && (lane >> 3) < c_count) c_rowpart[c_row + (lane >> 3) * c_step] = widen(tot);
            rows_in_batch += c_count;
            if (rows_in_batch >= FLUSH_ROWS) flush_sums();
        }
        c_left -= c_count;
        c_row += c_drow;
        c_count = min(R, c_left);
        if (c_left == 0) flush_tile();
    }
    pdl_release();
}

}  // namespace pdot
