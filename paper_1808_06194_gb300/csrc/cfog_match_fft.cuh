// K3 + K4 + K6: SSD template matching of control points by FP32 FFT
// correlation (Sec. III-G, Eq. 3-9) with argmin and sub-pixel fit (Sec. V-B).
//
// One CTA matches one CP.  For the template T (N x N x m, reference CFOG) and
// the search window S ((N+2r) x (N+2r) x m, sensed CFOG) Eq. 5 gives
//     S(v) = sum T^2 + sum_window ||D_sen||^2 - 2 sum_x T(x) S(x + v).
// Eq. 9 evaluates the correlation with a 3-D FFT over (x, y, channel); only
// channel lag 0 is a match, and the 3-D correlation at channel lag 0 equals
// the sum over channels of the 2-D correlations, so the channel FFT is not
// needed.  Per channel k the template block (real part) and its window
// (imaginary part) share one complex 2-D FFT; the two spectra are separated
// by Hermitian symmetry, and conj(T_k) S_k is accumulated (with a factor 4, taken
// out together with the -2 at the end); one inverse 2-D FFT then yields C(v) at
// every lag.  The middle term of Eq. 5 comes before the FFTs, from sums of
// ||D_sen||^2 - pivot: prefix sums of the rows, sliding sums down the columns.
// The FFT surface nominates the minimum; lags within 2e-5 of the energies behind
// it are re-scored directly (FP32 differences and sums, compensated block
// reduction), so the argmin is decided at the precision of the features.  The
// quadratic sub-pixel fit runs in FP64 on the 3 x 3 neighbourhood.
//
// Each FFT length is P = A * B: a decimation-in-frequency pass of radix A at
// stride B (then twiddles) and a pass of radix B on contiguous runs, each a
// register DFT (cfog_fft.cuh).  The spectrum stays in the two-digit reversed
// order (position a*B + b holds frequency a + A*b); the inverse runs the
// passes backwards, so no reordering pass exists.
//
// What bounds it: the shared-memory data path and the issue slots.  A plane
// element crosses shared memory three times (row pass 1 writes, row pass 2 and
// column pass 1 read and write, column pass 2 reads), about 19 wavefronts and
// 62 instructions per 32 elements, 0.82 SM cycles an element when the passes
// run alone on two CTAs of an SM (measured at P = 96; row pass 1 0.28, row
// pass 2 0.15, column pass 1 0.19, column pass 2 0.21).  Hence:
//   * a round's raw pixels reach their plane by 16-byte asynchronous copies,
//     and row pass 1 reads and overwrites them in place.  Before, it gathered
//     4-byte values from global memory in runs of B, most of the L1 wavefronts
//     of the kernel and half of its address arithmetic;
//   * column pass 2 holds a butterfly and its mirror, so the cross-spectrum is
//     formed in registers: the transformed plane is neither written nor read
//     again (a quarter of the shared-memory traffic), and no position table
//     exists;
//   * the state of a CP lives in shared memory, so that the passes have the
//     register file (128 registers, 16 warps per SM) to themselves: more warps
//     with fewer registers measured slower, and twiddles held in registers
//     spilled;
//   * the planes of several items are transformed side by side where they fit.
// Matcher of the batched step (1024 CPs, N 48..128, r 8..20, 2048^2 pair):
// 1.10 -> 0.91 ms; 4096 CPs of N 96, r 20: 6.8 -> 4.8 ms; 1000 CPs of N 96,
// r 16: 1.38 -> 0.91 ms.
#pragma once

#include "cfog_internal.cuh"
#include "cfog_fft.cuh"
#include "cfog_match_common.cuh"
#include "cfog_tc.cuh"
#include "cfog_plan.cuh"

#include <cfloat>
#include <climits>
#include <cmath>
#include <cstdint>

namespace cfog {
namespace {

// Kernel geometry: threads per CTA, CTAs per SM and the number of partial
// sums of the re-scoring.  The spectrum accumulators live in tensor memory
// (COLS columns per CTA).  No result depends on NT: every sum has an order of
// its own.  Kernel variants of one geometry differ only in the plans they may
// choose.
template <int NT_, int MINB_, int VT_>
struct Geometry {
    static constexpr int NT = NT_;
    static constexpr int MINB = MINB_;
    static constexpr int VT = VT_;
    static constexpr int COLS = fft_tmem_cols(MINB_);
};

// Tuned plans (the autotuner's choices) of the kernel variants that run this
// translation unit's geometry: entry [table][N][r] = (m << 16) | (plan code + 1),
// 0 = none (the cost model decides).
static __device__ int32_t g_plan_override[kPlanTables][kMaxFft + 1][kMaxRadius + 1];

// ------------------------------------------------------------ FFT passes --
// What every item of a control point shares.
struct CpView {
    JobView J;
    int ry0, rx0, sy0, sx0;   // template origin (reference), window origin (sensed)
    int N, r, m;
    float pivot;              // of the window's energy (box_sums)
    float scale;              // of the template's (row_fwd_s1)
};

// One (block, channel) item: where its window and template pixels lie.
struct Item {
    const float *s, *t;     // window and template origin, at or before it on a 4-pixel boundary
    int wh, ww, bh, bw;     // window and template block extents
    int sx, tx;             // first window and template column behind that boundary
};

__device__ __forceinline__ Item make_item(const CpView &c, const MatchPlan &p, int it) {
    const int blk = it / c.m, k = it - blk * c.m;
    const int iby = blk / p.x.nb, ibx = blk - iby * p.x.nb;
    const int by0 = iby * p.y.bs, bx0 = ibx * p.x.bs;
    Item q;
    q.bh = min(p.y.bs, c.N - by0);
    q.bw = min(p.x.bs, c.N - bx0);
    q.wh = q.bh + 2 * c.r;
    q.ww = q.bw + 2 * c.r;
    const int wx0 = c.sx0 + bx0, tx0 = c.rx0 + bx0;
    q.sx = wx0 & 3;
    q.tx = tx0 & 3;
    q.s = c.J.sen + (int64_t)k * c.J.sen_pp + (int64_t)(c.sy0 + by0) * c.J.sen_rp + (wx0 & ~3);
    q.t = c.J.ref + (int64_t)k * c.J.ref_pp + (int64_t)(c.ry0 + by0) * c.J.ref_rp + (tx0 & ~3);
    return q;
}

// Raw rows: row y of an item's plane first holds the item's raw pixels, the
// window row (raw_len(Px) floats, from the 4-pixel boundary at or before its
// first column) and behind it the template row, starting on a 16-byte boundary
// of the row and zero beyond their extents.
__device__ __forceinline__ float *raw_row(float2 *plane, int ld, int y) {
    return reinterpret_cast<float *>(plane + y * ld) + ((y & 1) << 1);   // ld is odd
}

// Asynchronous copy global -> shared of 16 or 4 bytes; the bytes past `valid`
// become zero and are not read.
template <int BYTES>
__device__ __forceinline__ void cp_async_fill(uint32_t dst, const float *src, int valid) {
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(valid) : "memory");
}

// Copy rows [0, rows) of raw pixels, columns [x0, x1) behind the boundary src
// points to, into the raw rows of a plane; the rest of len columns becomes
// zero.  A warp takes every (NT / 32)-th row, a lane the same BYTES of each,
// so a copy costs two additions and itself.
template <int NT, int BYTES>
__device__ __forceinline__ void stage_rows(float2 *plane, int ld, int off, const float *src, int64_t rp,
                                           int rows, int x0, int x1, int len) {
    constexpr int NW = NT / 32, F = BYTES / 4;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t dstep = (uint32_t)(NW * ld * 8);   // NW is even: the raw rows' offset stays
    const int64_t sstep = rp * NW;
    for (int x = lane * F; x < len; x += 32 * F) {
        const StageCopy c = stage_copy(F, x, x0, x1);
        uint32_t dst = smem_u32(raw_row(plane, ld, warp) + off + x);
        const float *s = src + warp * rp + c.col;
#pragma unroll 4
        for (int y = warp; y < rows; y += NW) {
            cp_async_fill<BYTES>(dst, s, c.bytes);
            dst += dstep;
            s += sstep;
        }
    }
}

// Start the copies of the raw pixels of n items into their planes: 16-byte
// copies where the volumes' alignment allows (vec), else 4-byte copies.  The
// caller waits for them and synchronises.  (One bulk copy per row, some 150
// short rows a plane, took the copy engine twice as long.)
template <int NT>
__device__ __forceinline__ void stage_items(const Item *items, int64_t srp, int64_t trp, float *planes,
                                            int pf, int ld, int len, int n, bool vec) {
    for (int g = 0; g < n; ++g) {
        const Item &q = items[g];
        float2 *plane = reinterpret_cast<float2 *>(planes + g * pf);
        if (vec) {
            stage_rows<NT, 16>(plane, ld, 0, q.s, srp, q.wh, q.sx, q.sx + q.ww, len);
            stage_rows<NT, 16>(plane, ld, len, q.t, trp, q.bh, q.tx, q.tx + q.bw, len);
        } else {
            stage_rows<NT, 4>(plane, ld, 0, q.s, srp, q.wh, q.sx, q.sx + q.ww, len);
            stage_rows<NT, 4>(plane, ld, len, q.t, trp, q.bh, q.tx, q.tx + q.bw, len);
        }
    }
}

// FFT lengths whose radices the first passes know at compile time (immediate
// offsets instead of address arithmetic per element); the others take the
// radix from the switch and the stride B at run time.
#define CFOG_FFT_LENGTHS(X)                                                                       \
    X(48, 8, 6) X(50, 10, 5) X(54, 9, 6) X(60, 10, 6) X(64, 8, 8) X(72, 9, 8) X(80, 10, 8)        \
    X(90, 10, 9) X(96, 12, 8) X(100, 10, 10) X(108, 12, 9) X(120, 12, 10) X(128, 16, 8)           \
    X(144, 12, 12) X(160, 16, 10) X(180, 15, 12)

// sum T^2 is a sum of integers, which does not depend on which thread took which
// row: lanes' shares of a row times a power of two that brings N^2 m times the largest
// T^2 of a sample to 2^40 or twice that (CFOG sums reach an eighth of it).  From 2^28 on
// the shares' rounding is below a float's, unless a few pixels that the sample took
// for typical outshine the rest (1e-7 then), and up to 2^20 shares of at most 2^42
// add up.  A sum outside [2^28, 2^42) is taken again by energy_direct.
constexpr int kEnergyExp = 40;
constexpr long long kEnergyMin = 1LL << 28;
constexpr float kEnergyMax = 4398046511104.f;      // 2^42

// Row pass 1 (radix A at stride B) on one plane, reading the raw pixels in
// place: template + i window.  A warp takes whole rows (32 / B of them, B
// lanes each), reads all of a row's pixels and then overwrites the row, so
// the pass needs no second buffer.  The rows of a warp lie D apart, with
// D * ld = B (mod 16): lane (k, j) then writes complex values at B k + j (mod
// 16) from a common base, consecutive banks (with consecutive rows instead,
// half of all shared-memory wavefronts were conflicts).  Rows outside the
// window or the template read `zero`; rows from the window's height up to Py
// are written as zeros.  BC: B if known at compile time, else 0.  Returns the
// lane's share of sum T^2 times `scale`.
template <int NT, int A, int BC>
__device__ __forceinline__ long long row_fwd_s1(float2 *plane, int ld, const float2 *tw, FastDiv divB,
                                            int D, int Py, int len, const Item &q, const float *zero,
                                            int warp0, float scale) {
    const int lane = threadIdx.x & 31;
    const int B = BC ? BC : divB.d;
    const int R = BC ? 32 / (BC ? BC : 1) : divB.div(32);
    const int k = BC ? lane / (BC ? BC : 1) : divB.div(lane), j = lane - k * B;
    const bool lane_ok = k < R;
    const int wh = q.wh, bh = q.bh;
    const int jt = lane_ok ? j : 0;
    const int so = q.sx + jt, to = len + q.tx + jt;
    const float2 *twj = tw + jt;
    long long tt = 0;
    // a warp's unit: unit q0 of the block of rows from y0.  Rows q0 + {0, D,
    // ..., (R-1) D} of R * D rows; for B = 8, whose half-warps hold two whole
    // rows each, rows 2 q0 + {0, 8, 1, 9} of 16 (less rounding up of Py)
    const bool b8 = B == 8;
    const int nq = b8 ? 4 : D, rows = b8 ? 16 : R * D;
    const int koff = b8 ? (k >> 1) + 8 * (k & 1) : k * D;
    for (int y0 = 0, q0 = warp0;; q0 += NT / 32) {
        while (q0 >= nq) {
            q0 -= nq;
            y0 += rows;
        }
        if (y0 >= Py) break;
        const int yf = y0 + (b8 ? 2 * q0 : q0), y = yf + koff;
        const bool ok = lane_ok && y < Py;
        float2 *o = plane + y * ld + j;
        if (yf >= wh) {   // the warp's rows all lie below the window
            if (ok) {
#pragma unroll
                for (int a = 0; a < A; ++a) o[a * B] = make_float2(0.f, 0.f);
            }
            continue;
        }
        float2 x[A];
        const float *raw = raw_row(plane, ld, y);
        const float *sp = lane_ok && y < wh ? raw + so : zero;
#pragma unroll
        for (int a = 0; a < A; ++a) x[a] = make_float2(0.f, sp[a * B]);
        if (yf < bh) {
            const float *tp = lane_ok && y < bh ? raw + to : zero;
#pragma unroll
            for (int a = 0; a < A; ++a) x[a].x = tp[a * B];
            float e = x[0].x * x[0].x;
#pragma unroll
            for (int a = 1; a < A; ++a) e = fmaf(x[a].x, x[a].x, e);
            tt += __float2ll_rn(fminf(e * scale, kEnergyMax));   // NaN: kEnergyMax
        }
        __syncwarp();
        rdft<A, false>(x);
#pragma unroll
        for (int a = 1; a < A; ++a) x[a] = c_mul(x[a], twj[a * B]);
        if (ok) {
#pragma unroll
            for (int a = 0; a < A; ++a) o[a * B] = x[a];
        }
    }
    return tt;
}

// Row pass 2 (radix B, contiguous runs) over rows [0, nrows) of n planes, rows fastest.
template <int NT, int Bv, bool INV>
__device__ __forceinline__ void row_s2(float *planes, int pf, int ld, int A, FastDiv divR, FastDiv divG) {
    // divR: rows of all planes, divG: rows of one
    const int total = divR.d * A;
    for (int b = threadIdx.x; b < total; b += NT) {
        const int a = divR.div(b), rr = b - a * divR.d;
        const int g = divG.div(rr), row = rr - g * divG.d;
        float2 *p = reinterpret_cast<float2 *>(planes + g * pf) + row * ld + a * Bv;
        float2 x[Bv];
#pragma unroll
        for (int u = 0; u < Bv; ++u) x[u] = p[u];
        rdft<Bv, INV>(x);
#pragma unroll
        for (int u = 0; u < Bv; ++u) p[u] = x[u];
    }
}

// Column pass 1 (radix A at stride B rows) over the columns of n planes,
// columns fastest: a warp's accesses are contiguous and its twiddles (almost)
// all the same.  divC: columns of all planes.
template <int NT, int A, int BC>
__device__ __forceinline__ void col_fwd_s1(float *planes, int pf, int ld, const float2 *tw, int Br,
                                           FastDiv divP, FastDiv divC) {
    const int B = BC ? BC : Br;
    const int total = divC.d * B, step = B * ld;
    for (int b = threadIdx.x; b < total; b += NT) {
        const int j = divC.div(b), f = b - j * divC.d;
        const int g = divP.div(f), c = f - g * divP.d;
        float2 *p = reinterpret_cast<float2 *>(planes + g * pf) + j * ld + c;
        const float2 *twj = tw + j;
        float2 x[A];
#pragma unroll
        for (int a = 0; a < A; ++a) x[a] = p[a * step];
        rdft<A, false>(x);
#pragma unroll
        for (int a = 1; a < A; ++a) x[a] = c_mul(x[a], twj[a * B]);
#pragma unroll
        for (int a = 0; a < A; ++a) p[a * step] = x[a];
    }
}

// Column pass 2 (radix B on contiguous rows) fused with the cross-spectrum.
// A thread transforms the butterfly of row digit a in the column of frequency
// fx and the one of -a in the column of -fx: together they hold every (f, -f)
// pair of that digit, from which the template's and the window's spectra
// separate, so the transformed plane is never written back and read again.
// The n items' products conj(T) S are summed in registers and added to the
// thread's accumulators in tensor memory (stored on the first round).
template <int NT, int Bv>
__device__ __forceinline__ void col_s2_accumulate(const float *planes, int pf, int ld, int Ay,
                                                  FastDiv divH, const unsigned *cols, int n,
                                                  uint32_t tm, bool first, float *dc_err) {
    constexpr int CH = Bv <= 8 ? 16 : 32;
    const int Hx = divH.d;
    const int total = Ay * Hx;
    // warps without an item of the last iteration leave
    for (int it0 = 0; it0 + (int)(threadIdx.x & ~31u) < total; it0 += NT, tm += CH) {
        const int it = it0 + threadIdx.x;
        const int a = it < total ? divH.div(it) : 0;
        const unsigned pk = it < total ? cols[it - a * Hx] : 0u;
        const int am = a ? Ay - a : 0;
        const int o1 = a * Bv * ld + (int)(pk & 0xffffu), o2 = am * Bv * ld + (int)(pk >> 16);
        float acc[CH];
#pragma unroll
        for (int b = 0; b < CH; ++b) acc[b] = 0.f;
        for (int g = 0; g < n; ++g) {
            const float2 *pl = reinterpret_cast<const float2 *>(planes + g * pf);
            const float2 *p1 = pl + o1, *p2 = pl + o2;
            float2 x1[Bv], x2[Bv];
#pragma unroll
            for (int u = 0; u < Bv; ++u) {
                x1[u] = p1[u * ld];
                x2[u] = p2[u * ld];
            }
            rdft<Bv, false>(x1);
            rdft<Bv, false>(x2);
            // 2 T = (z1.x + z2.x, z1.y - z2.y), 2 S = (z1.y + z2.y, z2.x - z1.x)
            auto add = [&](int b, const float2 &z1, const float2 &z2) {
                const float2 s = c_add(z1, z2), d = c_sub(z1, z2);
                acc[2 * b] = fmaf(s.x, s.y, fmaf(-d.x, d.y, acc[2 * b]));
                acc[2 * b + 1] = fmaf(-s.x, d.x, fmaf(-s.y, d.y, acc[2 * b + 1]));
            };
            if (a != 0) {
#pragma unroll
                for (int b = 0; b < Bv; ++b) add(b, x1[b], x2[Bv - 1 - b]);
            } else {
#pragma unroll
                for (int b = 0; b < Bv; ++b) add(b, x1[b], x2[(Bv - b) % Bv]);
            }
        }
        __syncwarp();
        if (!first) {
#pragma unroll
            for (int c = 0; c < CH; c += 16) {
                float v[16];
                tmem_ld16(tm + c, v);
                if (c == 0 && it == 0) {
                    // frequency 0, by far the largest: what its sum rounds off is kept
                    float sum, err;
                    two_sum(v[0], acc[0], sum, err);
                    *dc_err += err;
                }
#pragma unroll
                for (int u = 0; u < 16; ++u) acc[c + u] += v[u];
            }
        }
#pragma unroll
        for (int c = 0; c < CH; c += 16) tmem_st16(tm + c, acc + c);
    }
    tmem_wait_st();
}

// Inverse column pass 2 from the accumulators: the Hermitian pair of every
// butterfly is formed in registers, transformed and written to the plane.
// Frequency 0 goes to *dc instead: it adds the same to every lag, most of C,
// and the inverse of the rest rounds at the size of the rest.
template <int NT, int Bv>
__device__ __noinline__ void col_inv_s2(float2 *plane, int ld, int Ay, FastDiv divH,
                                        const unsigned *cols, uint32_t tm, float *dc) {
    constexpr int CH = Bv <= 8 ? 16 : 32;
    const int Hx = divH.d;
    const int total = Ay * Hx;
    for (int it0 = 0; it0 + (int)(threadIdx.x & ~31u) < total; it0 += NT, tm += CH) {
        const int it = it0 + threadIdx.x;
        float acc[CH];
#pragma unroll
        for (int c = 0; c < CH; c += 16) tmem_ld16(tm + c, acc + c);
        if (it == 0) {
            *dc = acc[0];
            acc[0] = 0.f;
        }
        const bool ok = it < total;
        const int a = ok ? divH.div(it) : 0;
        const unsigned pk = ok ? cols[it - a * Hx] : 0u;
        const int c1 = (int)(pk & 0xffffu), c2 = (int)(pk >> 16);
        const int am = a ? Ay - a : 0;
        float2 x1[Bv], x2[Bv];
#pragma unroll
        for (int b = 0; b < Bv; ++b) x1[b] = make_float2(acc[2 * b], acc[2 * b + 1]);
        if (a != 0) {
#pragma unroll
            for (int b = 0; b < Bv; ++b) x2[Bv - 1 - b] = make_float2(acc[2 * b], -acc[2 * b + 1]);
        } else {
#pragma unroll
            for (int b = 0; b < Bv; ++b) x2[(Bv - b) % Bv] = make_float2(acc[2 * b], -acc[2 * b + 1]);
        }
        rdft<Bv, true>(x1);
        rdft<Bv, true>(x2);
        float2 *p1 = plane + a * Bv * ld + c1, *p2 = plane + am * Bv * ld + c2;
        if (ok) {
#pragma unroll
            for (int u = 0; u < Bv; ++u) p1[u * ld] = x1[u];
            // a column that is its own mirror gets all its digits from x1
            if (c1 != c2) {
#pragma unroll
                for (int u = 0; u < Bv; ++u) p2[u * ld] = x2[u];
            }
        }
        __syncwarp();
    }
}

// Inverse column pass 1 (conjugate twiddles, then inverse radix A at stride B
// rows), columns fastest; only the rows of lags are written.
template <int NT, int A>
__device__ __noinline__ void col_inv_s1(float2 *plane, int ld, const float2 *tw, int B, FastDiv divP,
                                        int nout) {
    const int Px = divP.d;
    const int total = Px * B;
    for (int b = threadIdx.x; b < total; b += NT) {
        const int j = divP.div(b), c = b - j * Px;
        float2 *p = plane + j * ld + c;
        const int step = B * ld;
        float2 x[A];
#pragma unroll
        for (int a = 0; a < A; ++a) x[a] = p[a * step];
#pragma unroll
        for (int a = 1; a < A; ++a) x[a] = c_mul_conj(x[a], tw[a * B + j]);
        rdft<A, true>(x);
#pragma unroll
        for (int a = 0; a < A; ++a)
            if (j + a * B < nout) p[a * step] = x[a];
    }
}

// Inverse row pass 1 over the L rows of lags, j fastest, fused with the
// assembly of Eq. 5: surf holds the window energy's deviation from pivot N^2 (box
// sums of ||D_sen||^2 - pivot) and receives S = (sum T^2 + pivot N^2) - 2 C + deviation;
// base holds (sum T^2 + pivot N^2) - 2 C's share of frequency 0, as an exact two-part
// sum, and the product with the (two-part) scale is added to its high part in
// one rounding.
template <int NT, int A>
__device__ __noinline__ void row_inv_s1(const float2 *plane, int ld, const float2 *tw, FastDiv divB,
                                        int L, float2 scale, float2 base, float *surf) {
    const int B = divB.d;
    const int total = L * B;
    for (int b = threadIdx.x; b < total; b += NT) {
        const int row = divB.div(b), j = b - row * B;
        const float2 *p = plane + row * ld + j;
        float2 x[A];
#pragma unroll
        for (int a = 0; a < A; ++a) x[a] = p[a * B];
#pragma unroll
        for (int a = 1; a < A; ++a) x[a] = c_mul_conj(x[a], tw[a * B + j]);
        rdft<A, true>(x);
#pragma unroll
        for (int a = 0; a < A; ++a) {
            const int col = j + a * B;
            if (col < L) {
                float *s = surf + row * L + col;
                *s = fmaf(x[a].x, scale.x, base.x) + (fmaf(x[a].x, scale.y, base.y) + *s);
            }
        }
    }
}

#define CFOG_RADIX_SWITCH(R, CALL)                    \
    switch (R) {                                      \
        case 2: { constexpr int RR = 2; CALL; } break;  \
        case 3: { constexpr int RR = 3; CALL; } break;  \
        case 4: { constexpr int RR = 4; CALL; } break;  \
        case 5: { constexpr int RR = 5; CALL; } break;  \
        case 6: { constexpr int RR = 6; CALL; } break;  \
        case 8: { constexpr int RR = 8; CALL; } break;  \
        case 9: { constexpr int RR = 9; CALL; } break;  \
        case 10: { constexpr int RR = 10; CALL; } break; \
        case 12: { constexpr int RR = 12; CALL; } break; \
        case 15: { constexpr int RR = 15; CALL; } break; \
        default: { constexpr int RR = 16; CALL; } break; \
    }
// second-stage radices, 1 included
#define CFOG_RADIX_SWITCH1(R, CALL)                   \
    if ((R) == 1) { constexpr int RR = 1; CALL; } else CFOG_RADIX_SWITCH(R, CALL)

// exp(-2 pi i k / P) with the argument reduced to one quadrant, so that
// sincospif sees an exactly scaled value in [0, 1/4)
__device__ __forceinline__ float2 twiddle(int k, int P) {
    const int q = (4 * k) / P;
    const int rem = 4 * k - q * P;
    float s, c;
    sincospif(0.5f * ((float)rem / (float)P), &s, &c);
    float cs, sn;
    switch (q & 3) {
        case 0: cs = c; sn = s; break;
        case 1: cs = -s; sn = c; break;
        case 2: cs = -c; sn = -s; break;
        default: cs = s; sn = -c; break;
    }
    return make_float2(cs, -sn);
}

constexpr int kBoxChunks = 5;   // 160 columns: the usual windows in one go

// Pivot of the box sums and scale of sum T^2, from a sample of 32 pixels of the
// window and of the template, one per lane (a row and a column each).  Every warp
// takes the same sample: no barrier, and nothing depends on the CTA's threads.
//
// Pivot: the sample's largest ||D_sen||^2, rounded to eight significant bits, if
// three quarters of the sample reach half of it, else 0.  CFOG vectors have the same
// norm wherever the image has structure (1 unless eps weighs in), so there the
// summands ||D_sen||^2 - pivot are rounding-sized and the sums keep the digits that
// pivot N^2 would push out.  Where norms vary a pivot costs digits instead.  Eight
// bits make pivot N^2 an exact float.  Rms error of the box sums, N 128, r 20, of the
// energies, with pivots of 0, 1 and by the rule (emulated in FP32): unit norm 2e-8, 0,
// 0; norm 0.03 1.6e-7, 9e-5, 1e-11; 40 % of the window flat 7e-9, 4e-8, 7e-9; 98 % flat
// 4e-8, 5e-8, 4e-8.
//
// Scale: the power of two that brings N^2 times m times the sample's largest T^2, of
// a channel per lane (N^2 if that is 0), to 2^kEnergyExp or twice that.
__device__ __forceinline__ float2 sample_norms(const CpView &c) {
    const int lane = threadIdx.x & 31, col = (13 * lane + 5) & 31;
    const int N = c.N, W = c.N + 2 * c.r;
    const float s = __ldg(c.J.sen_sq + (int64_t)(c.sy0 + (lane * W + W / 2) / 32) * c.J.sen_rp +
                          (c.sx0 + (col * W + W / 2) / 32));
    const float t = __ldg(c.J.ref + (int64_t)(lane % c.m) * c.J.ref_pp +
                          (int64_t)(c.ry0 + (lane * N + N / 2) / 32) * c.J.ref_rp + (c.rx0 + (col * N + N / 2) / 32));
    const float v = fmaxf(s, 0.f), t2 = fmaxf(t * t, 0.f);   // NaN: 0
    const float top = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
    const float t_top = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(t2)));
    const bool use = __popc(__ballot_sync(0xffffffffu, v >= 0.5f * top)) >= 24 && top > 1e-30f && top < 1e30f;
    const float est = (t_top > 0.f ? t_top * (float)c.m : 1.f) * ((float)N * (float)N);
    const int ex = min(max((int)(__float_as_uint(est) >> 23) - 127, kEnergyExp - 120), kEnergyExp + 120);
    return make_float2(use ? __uint_as_float((__float_as_uint(top) + 0x8000u) & 0xffff0000u) : 0.f,
                       __uint_as_float((unsigned)(127 + kEnergyExp - ex) << 23));
}

// sum T^2 in two parts, read from the volume again.  Eight warps take the rows of
// every channel in turn, four rows' loads at a time.
__device__ __noinline__ float2 energy_direct(const CpView &c, float2 *red) {
    const int tid = threadIdx.x, lane = tid & 31, N = c.N;
    float hi = 0.f, lo = 0.f;
    for (int k = 0; k < c.m && tid < 256; ++k) {
        const float *tp = c.J.ref + (int64_t)k * c.J.ref_pp + (int64_t)c.ry0 * c.J.ref_rp + c.rx0;
        for (int y = tid >> 5; y < N; y += 32)
            for (int x = lane; x < N; x += 32) {
                float v[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) v[u] = y + 8 * u < N ? __ldg(tp + (int64_t)(y + 8 * u) * c.J.ref_rp + x) : 0.f;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    float err;
                    two_sum(hi, v[u] * v[u], hi, err);
                    lo += err;
                }
            }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float oh = __shfl_xor_sync(0xffffffffu, hi, o), ol = __shfl_xor_sync(0xffffffffu, lo, o);
        float sum, err;
        two_sum(hi, oh, sum, err);
        hi = sum;
        lo = (lo + ol) + err;
    }
    if ((tid & 31) == 0 && tid < 256) red[tid >> 5] = make_float2(hi, lo);
    __syncthreads();
    hi = red[0].x;
    lo = red[0].y;
    for (int w = 1; w < 8; ++w) {
        float sum, err;
        two_sum(hi, red[w].x, sum, err);
        hi = sum;
        lo = (lo + red[w].y) + err;
    }
    float2 r;
    two_sum(hi, lo, r.x, r.y);
    return r;
}

// Box sums of ||D_sen||^2 - pivot over the N x N template window at every lag
// (the second term of Eq. 5 less pivot N^2).  Rows: a warp takes four rows at a
// time, a warp prefix sum each straight from global memory, whose differences
// at distance N are the row sums.  Columns: up to 256 / L threads per lag
// column, each sliding over a segment of the row lags.
template <int NT>
__device__ __noinline__ void box_sums(CpView &c, float *scratch, float *out) {
    const float2 norms = sample_norms(c);
    const float pivot = norms.x;
    if (threadIdx.x == 0) {
        c.pivot = pivot;
        c.scale = norms.y;
    }
    const int N = c.N, W = N + 2 * c.r, L = 2 * c.r + 1, Lp = L | 1;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int NW = NT / 32;
    float *rows = scratch;                             // [W][Lp]
    float *pre = scratch + W * Lp + warp * kBoxRows * (W + 1);   // the rows' prefix sums
    for (int y0 = kBoxRows * warp; y0 < W; y0 += kBoxRows * NW) {
        const float *q[kBoxRows];
        float carry[kBoxRows];
#pragma unroll
        for (int i = 0; i < kBoxRows; ++i) {
            q[i] = c.J.sen_sq + (int64_t)(c.sy0 + min(y0 + i, W - 1)) * c.J.sen_rp + c.sx0;
            carry[i] = 0.f;
        }
        // kBoxChunks x 32 pixels of every row are in flight before the first is used
        for (int x0 = 0; x0 < W; x0 += 32 * kBoxChunks) {
            float v[kBoxRows][kBoxChunks];
#pragma unroll
            for (int ch = 0; ch < kBoxChunks; ++ch)
#pragma unroll
                for (int i = 0; i < kBoxRows; ++i) {
                    const int x = x0 + 32 * ch + lane;
                    v[i][ch] = x < W ? __ldg(q[i] + x) - pivot : 0.f;
                }
#pragma unroll
            for (int ch = 0; ch < kBoxChunks; ++ch) {
                if (x0 + 32 * ch >= W) break;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1)
#pragma unroll
                    for (int i = 0; i < kBoxRows; ++i) {
                        const float a = __shfl_up_sync(0xffffffffu, v[i][ch], o);
                        if (lane >= o) v[i][ch] += a;
                    }
                const int x = x0 + 32 * ch + lane;
#pragma unroll
                for (int i = 0; i < kBoxRows; ++i) {
                    const float p = v[i][ch] + carry[i];
                    carry[i] = __shfl_sync(0xffffffffu, p, 31);
                    if (x < W) pre[i * (W + 1) + x + 1] = p;
                }
            }
        }
        if (lane < kBoxRows) pre[lane * (W + 1)] = 0.f;
        __syncwarp();
#pragma unroll
        for (int i = 0; i < kBoxRows; ++i)
            if (y0 + i < W)
                for (int l = lane; l < L; l += 32)
                    rows[(y0 + i) * Lp + l] = pre[i * (W + 1) + l + N] - pre[i * (W + 1) + l];
        __syncwarp();
    }
    __syncthreads();
    const int nseg = max(1, 256 / L);   // fixed: the sums' order does not depend on NT
    const int ls = (L + nseg - 1) / nseg;
    for (int it = tid; it < L * nseg; it += NT) {
        const int lx = it % L, l0 = (it / L) * ls, l1 = min(L, l0 + ls);
        if (l0 >= l1) continue;
        const float *col = rows + lx;
        float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
        int y = 0;
#pragma unroll 4
        for (; y + 3 < N; y += 4) {
            a0 += col[(l0 + y) * Lp];
            a1 += col[(l0 + y + 1) * Lp];
            a2 += col[(l0 + y + 2) * Lp];
            a3 += col[(l0 + y + 3) * Lp];
        }
        for (; y < N; ++y) a0 += col[(l0 + y) * Lp];
        float acc = (a0 + a1) + (a2 + a3);
        out[l0 * L + lx] = acc;
        for (int ly = l0 + 1; ly < l1; ++ly) {
            acc += col[(ly + N - 1) * Lp] - col[(ly - 1) * Lp];
            out[ly * L + lx] = acc;
        }
    }
}

// The best kMaxCand of n scores by (value, index), the first of them given: arg-min
// rounds, each behind the last.  For windows with more lags in the band than the
// buffer holds (flat or periodic ones), where timing decides which entered it.
template <int NT>
__device__ __noinline__ void best_lags(const float *surf, int n, float v0, int i0, float *red_f, int *red_i,
                                       int *idx) {
    if (threadIdx.x == 0) idx[0] = i0;
    for (int c = 1; c < kMaxCand; ++c) {
        float v = INFINITY;
        int at = INT_MAX;
        for (int i = threadIdx.x; i < n; i += NT) {
            const float sv = surf[i];
            if ((sv > v0 || (sv == v0 && i > i0)) && (sv < v || (sv == v && i < at))) {
                v = sv;
                at = i;
            }
        }
        block_argmin<NT>(v, at, red_f, red_i, v0, i0);
        if (threadIdx.x == 0) idx[c] = i0;
    }
}

// position of frequency f after the forward passes of one axis
__device__ __forceinline__ int freq_pos(int f, const FftDim &d) { return (f % d.A) * d.B + f / d.A; }

// ------------------------------------------------------------------ kernel --
template <class V>
struct CoreShared {
    float red_f[V::NT / 32];
    int red_i[V::NT / 32];
    unsigned long long red_u[V::NT / 32];
    long long red_l[V::NT / 32];
    float2 red_cn[kMaxCand][V::VT / 32];
    int cand_n;
    int cand_idx[kCandBuf];
    float cand_val[kCandBuf];
    float cand_ssd[kMaxCand];
    int64_t cand_off[kMaxCand];
    unsigned cols[kMaxFft / 2 + 1];   // half of the columns and their mirrors: positions, packed
    int next;
    uint32_t tmem;
    Item item[2][V::NT > kFftThreads ? 2 * kMaxPlanes : kMaxPlanes]; // this round's items and the next one's
    CpView cv;                // the CP and its plan: kept here, not in registers, so that
    MatchPlan plan;           // the passes have the register file to themselves
    float dc;                 // accumulated frequency 0 ...
    float dc_err;             // ... and what its sum rounded off
    float band;               // width of the nomination band
    float2 base;              // what S has at every lag
    float zero[kMaxFft];      // a row of zeros
};

// sum T^2, in two parts, from the threads' integer sums; then the nomination band
// and, from tid 0, the part of S that is the same at every lag but frequency 0.
template <class V>
__device__ __noinline__ void energies(CoreShared<V> &sh, long long part, const float *surf) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    part = warp_sum(part);
    if (lane == 0) sh.red_l[warp] = part;
    __syncthreads();
    long long sum = sh.red_l[0];
#pragma unroll
    for (int w = 1; w < V::NT / 32; ++w) sum += sh.red_l[w];
    const float inv = __uint_as_float((254u << 23) - __float_as_uint(sh.cv.scale));   // 1 / scale
    const float hi = (float)sum;
    float2 tt = make_float2(hi * inv, (float)(sum - (long long)hi) * inv);
    if (sum < kEnergyMin || sum >= (long long)kEnergyMax) tt = energy_direct(sh.cv, &sh.red_cn[0][0]);
    if (threadIdx.x == 0) {
        const float N = (float)sh.cv.N, rest = sh.cv.pivot * (N * N);   // exact
        // the band is relative to the energies that the scores are the difference of:
        // the template's and the largest of the windows at the corner and middle lags
        const int L = 2 * sh.cv.r + 1;
        const float dev = fmaxf(fmaxf(fmaxf(surf[0], surf[L - 1]), fmaxf(surf[L * L - L], surf[L * L - 1])), surf[L * L / 2]);
        sh.band = kRescoreRel * (tt.x + fmaxf(rest + dev, 0.f));
        float energy, err;
        two_sum(tt.x, rest, energy, err);
        sh.base = make_float2(energy, err + tt.y);
    }
}

// The plan of class (N, r, m): the tuned plan when the table holds one and it
// fits the launch's shared memory; otherwise the cost model's, every thread
// costing one plan code and the CTA taking the least (cost, code).
template <class V>
__device__ __forceinline__ bool choose_plan(const MatchArgs &A, int N, int r, MatchPlan *plan,
                                            CoreShared<V> &sh) {
    static_assert(V::NT >= kPlanCodes, "one thread per plan code");
    const int tid = threadIdx.x;
    const PlanLimits &lim = A.lim;
    if (A.plan_table >= 0) {
        const int e = g_plan_override[A.plan_table][N][r];
        if (e != 0 && (e >> 16) == A.m &&
            plan_for_code(N, r, A.m, (e & 0xffff) - 1, lim, plan) >= 0 &&
            plan_smem_bytes(*plan, N, r, V::NT, plan->G) <= A.smem_bytes)
            return true;
    }
    const long long c = tid < kPlanCodes ? plan_for_code(N, r, A.m, tid, lim, plan) : -1;
    unsigned long long key = c < 0 ? ~0ull : ((unsigned long long)c << 8) | (unsigned)tid;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long k = __shfl_xor_sync(0xffffffffu, key, o);
        key = k < key ? k : key;
    }
    if ((tid & 31) == 0) sh.red_u[tid >> 5] = key;
    __syncthreads();
    key = sh.red_u[0];
#pragma unroll
    for (int w = 1; w < V::NT / 32; ++w) key = sh.red_u[w] < key ? sh.red_u[w] : key;
    if (key == ~0ull) return false;
    plan_for_code(N, r, A.m, (int)(key & 0xff), lim, plan);
    return true;
}

// Match control point `cp` with the whole CTA.  Every branch that returns
// early is uniform across the CTA. 
template <class V>
__device__ __forceinline__ void match_one(const MatchArgs &A, const int cp, CoreShared<V> &sh,
                                          unsigned char *smem_raw) {
    constexpr int NT = V::NT;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const JobView Jv = job_view(A, cp);
    const int N = A.tmpl[cp], r = A.radius[cp];
    const int px = A.cps[cp].x, py = A.cps[cp].y;
    const int qx = A.prior ? A.prior[cp].x : 0, qy = A.prior ? A.prior[cp].y : 0;
    const int m = A.m;
    const int Lside = 2 * r + 1;

    cfog_match_result res;
    res.dx = qx;
    res.dy = qy;
    res.sub_dx = (float)qx;
    res.sub_dy = (float)qy;
    res.ssd = INFINITY;
    res.status = CFOG_CP_OOB;

    const int t0 = N / 2;
    const int ry0 = py - t0, rx0 = px - t0;                 // template origin in ref
    const int sy0 = py + qy - t0 - r, sx0 = px + qx - t0 - r; // window origin in sen
    // a CP outside the launch bounds would need more shared memory than the
    // launch has: it is reported out of bounds and never touches the buffers
    const bool inside = Jv.ok && N >= 1 && r >= 0 && N <= A.tmpl_max && r <= A.radius_max &&
                        ry0 >= 0 && rx0 >= 0 && ry0 + N <= Jv.ref_h && rx0 + N <= Jv.ref_w &&
                        sy0 >= 0 && sx0 >= 0 && sy0 + N + 2 * r <= Jv.sen_h &&
                        sx0 + N + 2 * r <= Jv.sen_w;
    if (!inside) {
        if (tid == 0) A.out[cp] = res;
        return;
    }
    {
        MatchPlan p;
        const bool found = choose_plan<V>(A, N, r, &p, sh);
        if (!found) {
            if (tid == 0) A.out[cp] = res;
            return;
        }
        if (tid == 0) {
            sh.cv.J = Jv;
            sh.cv.ry0 = ry0;
            sh.cv.rx0 = rx0;
            sh.cv.sy0 = sy0;
            sh.cv.sx0 = sx0;
            sh.cv.N = N;
            sh.cv.r = r;
            sh.cv.m = m;
            sh.plan = p;
            sh.dc_err = 0.f;
        }
    }
    __syncthreads();
    const CpView &cv = sh.cv;
    const JobView &J = cv.J;
    const MatchPlan &plan = sh.plan;
    const FftDim &DY = plan.y;
    const FftDim &DX = plan.x;
    const int Py = DY.P, Px = DX.P, ld = plan.ld;
    const int pf = plane_floats(Py, ld);

    float *planes = reinterpret_cast<float *>(smem_raw);
    float2 *plane0 = reinterpret_cast<float2 *>(smem_raw);
    // A round transforms G items; with twice the threads and room for twice the
    // planes it transforms two rounds' items at once (summed as two rounds).
    const int G = plan.G;
    const bool twice = V::NT > kFftThreads && plan_smem_bytes(plan, N, r, NT, 2 * G) <= A.smem_bytes;
    const int per_round = twice ? 2 * G : G;
    float2 *twx = reinterpret_cast<float2 *>(planes + plan_region(plan, N, r, NT, per_round));
    float2 *twy = twx + Px;
    float *surf = reinterpret_cast<float *>(twy + Py);   // [Lside^2]

    if (tid < min(per_round, DY.nb * DX.nb * m)) sh.item[0][tid] = make_item(cv, plan, tid);
    box_sums<NT>(sh.cv, planes, surf);
    // twiddles exp(-2 pi i a j / P) at a * B + j: lanes of consecutive j read
    // consecutive values
    const FastDiv divBx(DX.B);
    {
        const FastDiv divBy(DY.B);
        if (tid < Px) {
            const int a = divBx.div(tid);
            twx[tid] = twiddle(a * (tid - a * DX.B), Px);
        }
        if (tid < Py) {
            const int a = divBy.div(tid);
            twy[tid] = twiddle(a * (tid - a * DY.B), Py);
        }
    }
    // the columns with position <= their mirror's, in ascending position
    {
        const int ax = divBx.div(tid), f = ax + DX.A * (tid - ax * DX.B);
        const int mir = tid < Px ? (f ? freq_pos(Px - f, DX) : 0) : 0;
        const bool half = tid < Px && tid <= mir;
        const unsigned b = __ballot_sync(0xffffffffu, half);
        if (lane == 0) sh.red_i[warp] = __popc(b);
        __syncthreads();   // also: box sums done with the planes, twiddles written
        int at = __popc(b & ((1u << lane) - 1u));
        for (int w = 0; w < warp; ++w) at += sh.red_i[w];
        if (half) sh.cols[at] = (unsigned)tid | ((unsigned)mir << 16);
    }

    // 16-byte copies need 16-byte aligned rows
    const bool vec = ((J.sen_rp | J.sen_pp | J.ref_rp | J.ref_pp) & 3) == 0 &&
                     ((reinterpret_cast<uintptr_t>(J.sen) | reinterpret_cast<uintptr_t>(J.ref)) & 15) == 0;
    const uint32_t tm = sh.tmem + ((uint32_t)(warp & 3) * 32u << 16) +
                        (uint32_t)(warp >> 2) * (uint32_t)(V::COLS / (NT / 128));
    long long tt_part = 0;   // sum T^2, per thread, times cv.scale
    const int items = DY.nb * DX.nb * m;
    const int nrows = DY.bs + 2 * r;
    const int len = raw_len(Px);
    const FastDiv divP(Px), divH(Px / 2 + 1), divG(nrows);
    // row spacing of the first pass: D * ld = B (mod 16) has a solution, ld being odd
    // (any will do for B = 16, one row per half-warp)
    int rowD = 1;
    while (DX.B < 16 && ((rowD * ld - DX.B) & 15)) ++rowD;
    FastDiv divR(nrows * per_round), divC(Px * per_round);
    for (int i0 = 0, par = 0; i0 < items; i0 += per_round, par ^= 1) {
        const int left = items - i0 - per_round;
        const int n = min(per_round, items - i0);
        const Item *it = sh.item[par];
        stage_items<NT>(it, J.sen_rp, J.ref_rp, planes, pf, ld, len, n, vec);
        // while the copies run: the next round's items
        if (tid >= 32 && tid - 32 < min(per_round, left))
            sh.item[par ^ 1][tid - 32] = make_item(cv, plan, i0 + n + tid - 32);
        if (left < 0) {   // a last round with fewer planes
            divR = FastDiv(nrows * n);
            divC = FastDiv(Px * n);
        }
        cp_async_wait_all();
        __syncthreads();
        // forward 2-D FFT of (template + i window), then the cross-spectrum
        for (int g = 0; g < n; ++g) {
            float2 *pl = reinterpret_cast<float2 *>(planes + g * pf);
            const int w0 = (warp + g * 3) & (NT / 32 - 1);   // spread the planes' last rows over the warps
#define CFOG_S1(P_, A_, B_)                                                                         \
    case P_: tt_part += row_fwd_s1<NT, A_, B_>(pl, ld, twx, divBx, rowD, Py, len, it[g], sh.zero, w0, cv.scale); break;
            switch (Px) {
                CFOG_FFT_LENGTHS(CFOG_S1)
                default:
                    CFOG_RADIX_SWITCH(DX.A, (tt_part += row_fwd_s1<NT, RR, 0>(pl, ld, twx, divBx, rowD, Py, len, it[g], sh.zero, w0, cv.scale)));
            }
        }
        __syncthreads();
        if (DX.B > 1) {
            CFOG_RADIX_SWITCH(DX.B, (row_s2<NT, RR, false>(planes, pf, ld, DX.A, divR, divG)));
            __syncthreads();
        }
#define CFOG_C1(P_, A_, B_) \
    case P_: col_fwd_s1<NT, A_, B_>(planes, pf, ld, twy, B_, divP, divC); break;
        switch (Py) {
            CFOG_FFT_LENGTHS(CFOG_C1)
            default:
                CFOG_RADIX_SWITCH(DY.A, (col_fwd_s1<NT, RR, 0>(planes, pf, ld, twy, DY.B, divP, divC)));
        }
        __syncthreads();
        for (int g = 0; g < n; g += G)
            CFOG_RADIX_SWITCH1(DY.B, (col_s2_accumulate<NT, RR>(planes + g * pf, pf, ld, DY.A, divH, sh.cols, min(G, n - g), tm, i0 + g == 0, &sh.dc_err)));
        __syncthreads();
    }

    energies<V>(sh, tt_part, surf);

    // the inverse passes backwards, then S(v) in surf
    CFOG_RADIX_SWITCH1(DY.B, (col_inv_s2<NT, RR>(plane0, ld, DY.A, divH, sh.cols, tm, &sh.dc)));
    __syncthreads();
    CFOG_RADIX_SWITCH(DY.A, (col_inv_s1<NT, RR>(plane0, ld, twy, DY.B, divP, Lside)));
    __syncthreads();
    if (DX.B > 1) {
        CFOG_RADIX_SWITCH(DX.B, (row_s2<NT, RR, true>(planes, pf, ld, DX.A, FastDiv(Lside), FastDiv(Lside))));
        __syncthreads();
    }
    {
        // the accumulated products carry a factor 4, Eq. 5 a factor -2
        const float area = (float)Py * (float)Px;
        float2 scale, base;
        scale.x = -0.5f / area;
        scale.y = fmaf(-scale.x, area, -0.5f) / area;
        const float dc = sh.dc, c0 = dc * scale.x;
        float err;
        two_sum(sh.base.x, c0, base.x, err);
        base.y = sh.base.y + err + fmaf(dc, scale.x, -c0) + fmaf(dc, scale.y, sh.dc_err * scale.x);
        CFOG_RADIX_SWITCH(DX.A, (row_inv_s1<NT, RR>(plane0, ld, twx, divBx, Lside, scale, base, surf)));
    }
    __syncthreads();
    const int L2 = Lside * Lside;
    float bv = INFINITY;
    int bi = INT_MAX;
    for (int i = tid; i < L2; i += NT) {
        const float sv = surf[i];
        if (sv < bv || (sv == bv && i < bi)) {
            bv = sv;
            bi = i;
        }
    }
    if (tid == 0) sh.cand_n = 0;
    float smin;
    int imin;
    block_argmin<NT>(bv, bi, sh.red_f, sh.red_i, smin, imin);
    // NaN or infinite features leave no lag to choose (imin may be no lag at all)
    const bool found = isfinite(smin);

    // lags inside the nomination band are re-scored directly
    const float band = sh.band;
    for (int i = tid; i < L2; i += NT) {
        const float sv = surf[i];
        if (found && sv <= smin + band) {
            const int slot = atomicAdd(&sh.cand_n, 1);
            if (slot < kCandBuf) {
                sh.cand_idx[slot] = i;
                sh.cand_val[slot] = sv;
            }
        }
    }
    __syncthreads();
    int ncand = sh.cand_n;
    if (ncand > kCandBuf) {
        best_lags<NT>(surf, L2, smin, imin, sh.red_f, sh.red_i, sh.cand_idx);
        ncand = kMaxCand;
    } else if (tid == 0) {
        // order by (FFT value, index) and keep the best kMaxCand
        for (int a = 1; a < ncand; ++a) {
            const int ii = sh.cand_idx[a];
            const float vv = sh.cand_val[a];
            int b = a - 1;
            while (b >= 0 && (sh.cand_val[b] > vv || (sh.cand_val[b] == vv && sh.cand_idx[b] > ii))) {
                sh.cand_idx[b + 1] = sh.cand_idx[b];
                sh.cand_val[b + 1] = sh.cand_val[b];
                --b;
            }
            sh.cand_idx[b + 1] = ii;
            sh.cand_val[b + 1] = vv;
        }
    }
    __syncthreads();
    ncand = min(ncand, kMaxCand);
    int win = imin;
    float win_ssd = smin;
    if (ncand > 1) {
        // one pass over the template per group of up to four candidates: each
        // template value is read once per group and compared with the window
        // value at every candidate lag of the group.  Eight elements per thread
        // are loaded before any is used, so the loads overlap; each thread
        // still visits its elements in the order e = tid, tid + NT, ...
        const int NN = N * N;
        if (tid < ncand) {
            const int li = sh.cand_idx[tid];
            const int vy = li / Lside - r, vx = li - (li / Lside) * Lside - r;
            sh.cand_off[tid] = (int64_t)vy * J.sen_rp + vx;
        }
        __syncthreads();
        // the sums run over VT partial sums, element e into partial sum e % VT;
        // a thread holds VT / NT of them (at least one) and visits its elements in order
        constexpr int H = V::VT > NT ? V::VT / NT : 1;
        constexpr int RT = V::VT < NT ? V::VT : NT;   // threads that take part
        float acc[H][kMaxCand];
#pragma unroll
        for (int h = 0; h < H; ++h)
#pragma unroll
            for (int c = 0; c < kMaxCand; ++c) acc[h][c] = 0.f;
        const FastDiv divN(N);
        constexpr int U = 8;
        if (tid < RT && ncand == 2) {
            // the usual near tie, two lags: sixteen elements per thread in
            // flight per round (the features were read long ago and mostly
            // come from DRAM), same element order, so the same sums
            constexpr int U2 = 16;
            const int64_t o0 = sh.cand_off[0], o1 = sh.cand_off[1];
            for (int k = 0; k < m; ++k) {
                const float *tp = J.ref + (int64_t)k * J.ref_pp + (int64_t)ry0 * J.ref_rp + rx0;
                const float *wp = J.sen + (int64_t)k * J.sen_pp + (int64_t)(sy0 + r) * J.sen_rp + (sx0 + r);
                for (int e0 = tid; e0 < NN; e0 += U2 * RT) {
                    float ta[U2], w0[U2], w1[U2];
#pragma unroll
                    for (int u = 0; u < U2; ++u) {
                        const int e = e0 + u * RT;
                        const bool ok = e < NN;
                        const int y = divN.div(e), x = e - y * N;
                        const float *wq = wp + (int64_t)y * J.sen_rp + x;
                        ta[u] = ok ? __ldg(tp + (int64_t)y * J.ref_rp + x) : 0.f;
                        w0[u] = ok ? __ldg(wq + o0) : 0.f;
                        w1[u] = ok ? __ldg(wq + o1) : 0.f;
                    }
#pragma unroll
                    for (int u = 0; u < U2; ++u) {
                        const float d0 = ta[u] - w0[u], d1 = ta[u] - w1[u];
                        acc[u % H][0] = fmaf(d0, d0, acc[u % H][0]);
                        acc[u % H][1] = fmaf(d1, d1, acc[u % H][1]);
                    }
                }
            }
        }
#pragma unroll
        for (int cg = 0; cg < kMaxCand; cg += 4) {
            if (cg >= ncand || ncand == 2 || tid >= RT) break;
            const int nc = min(4, ncand - cg);
            int64_t off4[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) off4[c] = sh.cand_off[cg + (c < nc ? c : 0)];
            for (int k = 0; k < m; ++k) {
                const float *tp = J.ref + (int64_t)k * J.ref_pp + (int64_t)ry0 * J.ref_rp + rx0;
                const float *wp = J.sen + (int64_t)k * J.sen_pp + (int64_t)(sy0 + r) * J.sen_rp + (sx0 + r);
                for (int e0 = tid; e0 < NN; e0 += U * RT) {
                    float ta[U], wb[U][4];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const int e = e0 + u * RT;
                        const bool ok = e < NN;
                        const int y = divN.div(e), x = e - y * N;
                        ta[u] = ok ? __ldg(tp + (int64_t)y * J.ref_rp + x) : 0.f;
                        const float *wq = wp + (int64_t)y * J.sen_rp + x;
#pragma unroll
                        for (int c = 0; c < 4; ++c) wb[u][c] = ok && c < nc ? __ldg(wq + off4[c]) : 0.f;
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u) {
#pragma unroll
                        for (int c = 0; c < 4; ++c) {
                            const float d = ta[u] - wb[u][c];
                            acc[u % H][cg + c] = fmaf(d, d, acc[u % H][cg + c]);
                        }
                    }
                }
            }
        }
        block_sum_comp_n<V::VT, RT, kMaxCand>(acc, ncand, sh.red_cn, sh.cand_ssd);
        __syncthreads();
        if (tid == 0) {
            int bc = 0;
            for (int c = 1; c < ncand; ++c)
                if (sh.cand_ssd[c] < sh.cand_ssd[bc] ||
                    (sh.cand_ssd[c] == sh.cand_ssd[bc] && sh.cand_idx[c] < sh.cand_idx[bc]))
                    bc = c;
            sh.red_i[0] = sh.cand_idx[bc];
            sh.red_f[0] = sh.cand_ssd[bc];
        }
        __syncthreads();
        win = sh.red_i[0];
        win_ssd = sh.red_f[0];
        __syncthreads();
    }

    if (A.surface) {
        const int Lmax = A.surf_side;
        float *dst = A.surface + (int64_t)cp * Lmax * Lmax;
        const int off = (Lmax - Lside) / 2;
        const FastDiv divL(Lside);
        for (int i = tid; i < L2; i += NT) {
            const int ly = divL.div(i), lx = i - ly * Lside;
            dst[(ly + off) * Lmax + (lx + off)] = surf[i];
        }
    }

    if (tid == 0 && !found) {
        res.status = CFOG_CP_NONFINITE;
        A.out[cp] = res;
    } else if (tid == 0) {
        const int vy = win / Lside - r, vx = win - (win / Lside) * Lside - r;
        res.dx = qx + vx;
        res.dy = qy + vy;
        res.ssd = win_ssd;
        double ox = 0.0, oy = 0.0;
        if (vx == -r || vx == r || vy == -r || vy == r) {
            res.status = CFOG_CP_EDGE_PEAK;
        } else {
            double f[9];
            for (int j = -1; j <= 1; ++j)
                for (int i = -1; i <= 1; ++i)
                    f[(j + 1) * 3 + (i + 1)] = (double)surf[(vy + r + j) * Lside + (vx + r + i)];
            subpixel_fit(f, ox, oy);
            res.status = CFOG_CP_OK;
        }
        res.sub_dx = (float)((double)res.dx + ox);
        res.sub_dy = (float)((double)res.dy + oy);
        A.out[cp] = res;
    }
}

// Set up and release what a CTA holds for all its CPs: the accumulators'
// tensor memory and the row of zeros.
template <class V>
__device__ __forceinline__ void cta_begin(CoreShared<V> &sh) {
    if (threadIdx.x < 32) {
        tmem_alloc(&sh.tmem, V::COLS);
        tmem_relinquish();
    }
    for (int i = threadIdx.x; i < kMaxFft; i += V::NT) sh.zero[i] = 0.f;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
}
template <class V>
__device__ __forceinline__ void cta_end(CoreShared<V> &sh) {
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x < 32) tmem_dealloc(sh.tmem, V::COLS);
}

// One CTA per CP in CP order (order == nullptr), or persistent CTAs draining
// a queue of CPs: slot i of the queue is CP order[i]; the next slot is taken
// with one atomic on `counter` (no waiting).
template <class V>
__global__ void __launch_bounds__(V::NT, V::MINB)
match_fft_kernel(const MatchArgs A, int *__restrict__ counter, const int *__restrict__ order) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ CoreShared<V> sh;
    // beside the planes' share of an SM (PlanLimits::smem_cap) and the reserved 1 KB
    static_assert(sizeof(sh) <= (V::MINB >= 3 ? 4032 : V::MINB == 2 ? 4096 : 5120), "static shared memory");
    cta_begin<V>(sh);
    for (;;) {
        int i = blockIdx.x;
        if (order) {
            if (threadIdx.x == 0) sh.next = atomicAdd(counter, 1);
            __syncthreads();
            i = sh.next;
            __syncthreads();
            if (i >= A.n) break;
            i = order[i];
        }
        match_one<V>(A, i, sh, smem_raw);
        if (!order) break;
        __syncthreads();
    }
    cta_end<V>(sh);
}

template <class V>
cfog_status launch_fft(const MatchArgs &a, int *counter, const int *order, int grid, int smem,
                       cudaStream_t s) {
    match_fft_kernel<V><<<grid, V::NT, smem, s>>>(a, counter, order);
    return check_launch("cfog_match: launch");
}

inline cfog_status write_plan_table(int table, size_t offset, const int32_t *src, size_t n) {
    const size_t base = (size_t)table * (kMaxFft + 1) * (kMaxRadius + 1) + offset;
    return check_cuda(cudaMemcpyToSymbol(g_plan_override, src, n * sizeof(int32_t), base * sizeof(int32_t)),
                      "cfog_match: plan table write");
}

// The kernel of one geometry as the host code sees it.
template <class V>
MatchKernel make_kernel() {
    return MatchKernel{reinterpret_cast<const void *>(match_fft_kernel<V>), V::NT, V::COLS, launch_fft<V>, write_plan_table};
}

}  // namespace
}  // namespace cfog
