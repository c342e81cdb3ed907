// FFT plan of one control point class (N, r): how the template is cut into
// blocks and which 2-D FFT size correlates each block with its search window.
//
// Sec. III-G computes the SSD surface of Eq. 3 through FFT correlation
// (Eq. 8-9).  The correlation is linear in the template, so the template may
// be cut into nb_y x nb_x blocks: each block of size b_y x b_x is correlated
// with its own (b_y + 2r) x (b_x + 2r) window and the cross-spectra of all
// blocks and channels are summed before one inverse FFT.  A P_y x P_x FFT
// with P >= b + 2r gives every lag in [-r, r] without circular wrap.  Every
// FFT length is a product P = A * B of two register radices, A, B in
// {2,3,4,5,6,8,9,10,12,15,16} (B = 1 allowed): two shared-memory passes per
// axis.  The plan depends only on (N, r, m) and the kernel variant's limits,
// so a CP's result never depends on its batch.  The search is exact integer
// arithmetic: host and device agree.
#pragma once

#include <cstdint>

namespace cfog {

constexpr int kMaxFft = 256;           // longest supported FFT side
constexpr int kMaxPlaneElems = 16384;  // largest P_y * P_x of any kernel variant
constexpr int kNbMax = 4;              // blocks per axis searched
constexpr int kPTries = 4;             // FFT lengths tried per axis
constexpr int kMaxPlanes = 4;          // planes transformed side by side
constexpr int kBoxRows = 4;            // window rows a warp takes at a time in the box sums

struct FftDim {
    int nb;   // number of template blocks along this axis
    int bs;   // block size ceil(N / nb); the last block may be shorter
    int P;    // FFT length, even
    int A;    // stage-1 radix (stride B), A >= B
    int B;    // stage-2 radix (contiguous); 1 = single stage
};

struct MatchPlan {
    FftDim y, x;
    int ld;   // row pitch of a plane, in complex values (odd)
    int G;    // planes transformed side by side: (block, channel) items per round
};

constexpr bool is_radix(int R) {
    return R == 2 || R == 3 || R == 4 || R == 5 || R == 6 || R == 8 || R == 9 || R == 10 ||
           R == 12 || R == 15 || R == 16;
}

// Split of every even length P <= kMaxFft into A * B (register radices, B may
// be 1, A >= B), as balanced as possible, and the smallest splittable length
// >= P.  The larger radix comes first: the last column pass holds two
// butterflies of radix B and their accumulators in registers.  Built at
// compile time; the host and the device read the same table.
struct SmoothTable {
    unsigned char A[kMaxFft + 1];
    unsigned char B[kMaxFft + 1];
    unsigned short next[kMaxFft + 2];   // 0: none up to kMaxFft
    constexpr SmoothTable() : A(), B(), next() {
        for (int P = 0; P <= kMaxFft; ++P) {
            A[P] = 0;
            B[P] = 0;
            if (P < 2 || (P & 1)) continue;
            int bestA = 0, bestB = 0, bestd = 1 << 30;
            for (int a = 2; a <= 16; ++a) {
                if (!is_radix(a) || P % a) continue;
                const int b = P / a;
                if (b > a || (b != 1 && !is_radix(b))) continue;
                const int d = a - b;
                if (d < bestd) {
                    bestd = d;
                    bestA = a;
                    bestB = b;
                }
            }
            A[P] = (unsigned char)bestA;
            B[P] = (unsigned char)bestB;
        }
        next[kMaxFft + 1] = 0;
        for (int P = kMaxFft; P >= 0; --P) next[P] = A[P] ? (unsigned short)P : next[P + 1];
    }
};

constexpr SmoothTable kSmoothHost{};
static __constant__ const SmoothTable kSmoothDev = SmoothTable{};

__host__ __device__ inline const SmoothTable &smooth_table() {
#ifdef __CUDA_ARCH__
    return kSmoothDev;
#else
    return kSmoothHost;
#endif
}

__host__ __device__ inline int ceil_log2(int v) {
    int c = 0;
    while ((1 << c) < v) ++c;
    return c;
}

// What a kernel variant gives a plan.
struct PlanLimits {
    int maxe;       // bound of P_y * P_x
    int smem_cap;   // dynamic shared memory of one CTA at the variant's CTAs per SM
    int tm_cols;    // tensor-memory columns per thread for the accumulators
    int threads;    // threads per CTA
};

// Floats of a staged row of raw pixels for an FFT of Px columns: 16-byte
// copies start at the 4-pixel boundary at or before its first column.
__host__ __device__ inline int raw_len(int Px) { return (Px + 3 + 3) & ~3; }

// Where a staging copy of F floats (4: 16 bytes, 1: 4 bytes) for column x of a
// raw row takes its bytes: a lane copies columns [x, x + F) behind the 4-pixel
// boundary, of which those in [x0, x1) are wanted.
struct StageCopy {
    int col;     // first source column behind the boundary
    int bytes;   // bytes read from there; the rest of the copy becomes zero
};
__host__ __device__ inline StageCopy stage_copy(int F, int x, int x0, int x1) {
    if (F == 4) {
        const int n = x1 - x < 4 ? x1 - x : 4;
        // a copy that reads nothing still names an address, which has to be
        // aligned to the copy's size and inside the row: the boundary itself
        return n > 0 ? StageCopy{x, 4 * n} : StageCopy{0, 0};
    }
    return x >= x0 && x < x1 ? StageCopy{x, 4} : StageCopy{x0, 0};
}

// Row pitch of a plane in complex values: odd, so that threads walking down a
// column of complex values hit distinct banks, and wide enough that a row's
// raw window and template pixels (from a 16-byte boundary of the row) fit into
// the row they are transformed in.
__host__ __device__ inline int plane_pitch(int Px) { return raw_len(Px) + 1; }

// Floats per plane (a multiple of 4: every plane starts on a 16-byte boundary).
__host__ __device__ inline int plane_floats(int Py, int ld) { return (2 * Py * ld + 3) & ~3; }

// Scratch floats of the box sums: row sums at an odd pitch and kBoxRows prefix rows per warp.
__host__ __device__ inline int box_floats(int N, int r, int threads) {
    const int W = N + 2 * r, L = 2 * r + 1;
    return W * (L | 1) + (threads / 32) * kBoxRows * (W + 1);
}

// Tensor-memory columns one thread needs for the accumulators: 2 B floats of
// every column butterfly pair it owns, in chunks of 16 columns.
__host__ __device__ inline int accum_chunk(int By) { return By <= 8 ? 16 : 32; }
__host__ __device__ inline int accum_cols(const FftDim &y, const FftDim &x, int threads) {
    const int pairs = y.A * (x.P / 2 + 1);
    return (pairs + threads - 1) / threads * accum_chunk(y.B);
}

// Floats before the twiddles: n planes, or the box-sum scratch.
__host__ __device__ inline int plan_region(const MatchPlan &p, int N, int r, int threads, int n) {
    const int planes = n * plane_floats(p.y.P, p.ld), box = (box_floats(N, r, threads) + 1) & ~1;
    return planes > box ? planes : box;
}

// Dynamic shared memory of the FFT matcher for a plan with n planes: the planes,
// the twiddles of both axes and the (2r+1)^2 scores.
__host__ __device__ inline int plan_smem_bytes(const MatchPlan &p, int N, int r, int threads, int n) {
    return 4 * (plan_region(p, N, r, threads, n) + 2 * (p.y.P + p.x.P) + (2 * r + 1) * (2 * r + 1));
}

// Integer cost of one length-P pass over a plane: each stage is a
// shared-memory round trip (100) plus arithmetic ~ log2 of its radix.
__host__ __device__ inline int fft_len_cost(int A, int B) {
    return 100 + 12 * ceil_log2(A) + (B > 1 ? 100 + 12 * ceil_log2(B) : 0);
}

// A plan named by a code: bits 4..7 the split index l (nby = l / kNbMax + 1,
// nbx = l % kNbMax + 1), bits 2..3 and 0..1 which of the first kPTries
// splittable lengths >= b + 2r the y and x axes take.  Returns its cost (or
// -1 when the code names no feasible plan) and fills *out.  The cost model's
// plan is the code of least cost, ties to the smaller code; the autotuner
// times codes and records the fastest per class.  A plane that leaves room
// for one CTA per SM only costs twice as much: it makes every CP of the launch
// run that way.  Of the 16384-element planes it costs a twelfth more only from
// radius kWideRadius on: classes of N 57 (r 32: 37) and more have no other plane
// there but of twice the elements, so a launch with such bounds runs one CTA per SM
// anyway, and smaller planes mostly transform more for nothing (1000 CPs, a charge of
// a quarter and of a twelfth: N 78, r 26 1.67 and 1.58 ms, N 76, r 27 1.76 and 1.58,
// N 176, r 26 5.65 and 5.18; N 99, r 26, whose small planes are 7 % dearer, 2.31 with
// them and 2.34 without; the double charge: N 128, r 32 5.3 ms, now 3.0).  Below it the
// double charge pays (1000 CPs of N 128, r 24: 2.5 ms, without 3.0), though not for few
// CPs, whose launches run one CTA per SM in any case (49 of N 72, r 23: 0.20 ms, with
// the larger plane 0.155): a CP's plan does not depend on its launch.
constexpr int kWideRadius = 26;
constexpr int kPlanCodes = kNbMax * kNbMax * kPTries * kPTries;

__host__ __device__ inline long long plan_for_code(int N, int r, int m, int code,
                                                   const PlanLimits &lim, MatchPlan *out) {
    if (code < 0 || code >= kPlanCodes) return -1;
    const int l = code >> 4, ty = (code >> 2) & 3, tx = code & 3;
    const int nby = l / kNbMax + 1, nbx = l % kNbMax + 1;
    const int bsy = (N + nby - 1) / nby, bsx = (N + nbx - 1) / nbx;
    if ((nby - 1) * bsy >= N || (nbx - 1) * bsx >= N) return -1;
    const int needy = bsy + 2 * r, needx = bsx + 2 * r;
    if (needy > kMaxFft || needx > kMaxFft) return -1;
    const SmoothTable &t = smooth_table();
    int Py = t.next[needy];
    for (int i = 0; i < ty && Py != 0; ++i) Py = t.next[Py + 1];
    int Px = t.next[needx];
    for (int i = 0; i < tx && Px != 0; ++i) Px = t.next[Px + 1];
    if (Py == 0 || Px == 0 || Py * Px > lim.maxe) return -1;
    const int Ay = t.A[Py], By = t.B[Py], Ax = t.A[Px], Bx = t.B[Px];
    out->y = FftDim{nby, bsy, Py, Ay, By};
    out->x = FftDim{nbx, bsx, Px, Ax, Bx};
    if (accum_cols(out->y, out->x, lim.threads) > lim.tm_cols) return -1;
    out->ld = plane_pitch(Px);
    out->G = 1;
    const int items = nby * nbx * m;
    const int fixed = plan_smem_bytes(*out, N, r, lim.threads, 1);
    const int plane = 4 * plane_floats(Py, out->ld);
    if (fixed <= lim.smem_cap) {
        // as many planes as fit, spread evenly over the rounds
        const int room = (lim.smem_cap - 4 * (2 * (Py + Px) + (2 * r + 1) * (2 * r + 1))) / plane;
        int g = room < items ? room : items;
        g = g < kMaxPlanes ? g : kMaxPlanes;
        const int rounds = (items + g - 1) / g;
        out->G = (items + rounds - 1) / rounds;
    }
    const long long per = (long long)Py * Px * (fft_len_cost(Ay, By) + fft_len_cost(Ax, Bx));
    const long long cost = per * (long long)(items + 1);
    if (fixed <= lim.smem_cap) return cost;
    return r >= kWideRadius && lim.maxe == kMaxPlaneElems ? cost + cost / 12 : 2 * cost;
}

// The code of least (cost, code).  A launch searches every class within its bounds
// once (688k codes for N up to 128 and r up to 20): a code's cost without the charge
// for its shared memory comes from two short tables, and one that the best so far
// beats at that is not worked out.
__host__ inline bool make_plan_host(int N, int r, int m, const PlanLimits &lim, MatchPlan *out) {
    static_assert(kNbMax == 4 && kPTries == 4, "the digits of a code");
    const SmoothTable &t = smooth_table();
    int P[kNbMax][kPTries], len[kNbMax][kPTries];   // lengths of nb blocks (0: none) and their cost
    for (int n = 0; n < kNbMax; ++n) {
        const int bs = (N + n) / (n + 1), need = bs + 2 * r;
        int at = n * bs < N && need <= kMaxFft ? t.next[need] : 0;
        for (int i = 0; i < kPTries; ++i) {
            P[n][i] = at;
            len[n][i] = at ? fft_len_cost(t.A[at], t.B[at]) : 0;
            at = at ? t.next[at + 1] : 0;
        }
    }
    long long best = -1;
    for (int code = 0; code < kPlanCodes; ++code) {
        const int ny = code >> 4 >> 2, nx = code >> 4 & 3, ty = code >> 2 & 3, tx = code & 3;
        const int area = P[ny][ty] * P[nx][tx];
        if (area == 0 || area > lim.maxe) continue;
        const long long floor_cost = (long long)area * (len[ny][ty] + len[nx][tx]) * ((ny + 1) * (nx + 1) * m + 1);
        if (best >= 0 && floor_cost >= best) continue;
        MatchPlan p;
        const long long c = plan_for_code(N, r, m, code, lim, &p);
        if (c >= 0 && (best < 0 || c < best)) {
            best = c;
            *out = p;
        }
    }
    return best >= 0;
}

}  // namespace cfog
