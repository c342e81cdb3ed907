// K2: block-based Harris feature-point detection (Sec. IV).
//
// One CTA per grid cell.  A warp marches down a strip of the cell's chip:
// every lane owns NC adjacent columns (the strip and a halo of four columns
// on each side), forms the structure-tensor products of the [-1,0,1]
// gradients of each new image row, takes its neighbours' by shuffles, filters
// them horizontally (9 taps, sigma 1.5) and adds the result to the nine output
// rows the image row belongs to, whose partial sums it holds in registers
// (the row loop is unrolled by nine, so that they never move).  The finished
// row's det - 0.04 tr^2 enters the lane's list of the k best; k rounds of a
// block-wide arg-max then pick the chip's k best (ties: smaller y, then
// smaller x).  Every sum runs over its taps in ascending order.
//
// What bounds it: the issue slots (65 % used at 8192^2, 16 warps per SM) and the
// image rows' latency (2.1 of 5.8 stall cycles per issue).  145 thread instructions
// per pixel, 54 of them the FMA of the two filters; strips of 56 columns over a
// 197-column cell and eight extra rows per segment add 1.3 and 1.1 times.  The FMA
// pipe is 39 % busy, DRAM at 5 % of the copy rate: nothing but the image row crosses
// memory.  The tiled form before it read every filter tap from shared memory (60
// loads per pixel, 33 % of the issue slots arithmetic).  8192^2 u16 pixels, 41 x 41
// cells: 1.20 -> 0.40 ms; 2048^2 f32, 32 x 32 cells: 67 -> 42 us; the same with
// eight points a cell 1.48 -> 0.67 ms and 97 -> 91 us.
#include "cfog_internal.cuh"

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdint>
#include <type_traits>

namespace cfog {
namespace {

constexpr int HR = 4;             // Gaussian radius
constexpr int HK = 2 * HR + 1;    // taps
constexpr int HWARPS = 8;         // warps per CTA at most
constexpr int KMAX = 8;
constexpr float KAPPA = 0.04f;

struct HarrisTaps {
    float w[2 * HR + 1];
};

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

// A pixel of the chip: its response and its position (y << 16) | x in the chip.
struct Cand {
    float v;
    int pos;
};
constexpr int kNoPos = INT_MAX;

// a ranks before b: larger response, then smaller y, then smaller x
__device__ __forceinline__ bool better(const Cand &a, const Cand &b) {
    return a.v > b.v || (a.v == b.v && a.pos < b.pos);
}

__device__ __forceinline__ void cell_chip(int h, int w, int gx, int gy, int chip, int margin, int gj,
                                          int gi, int &y0, int &y1, int &x0, int &x1) {
    const long long ih = h - 2 * margin, iw = w - 2 * margin;
    const int cy0 = margin + (int)(gj * ih / gy), cy1 = margin + (int)((gj + 1) * ih / gy);
    const int cx0 = margin + (int)(gi * iw / gx), cx1 = margin + (int)((gi + 1) * iw / gx);
    if (chip > 0) {
        const int cy = (cy0 + cy1) / 2, cx = (cx0 + cx1) / 2;
        const int a = cy - chip / 2, b = cx - chip / 2;
        y0 = max(a, cy0);
        y1 = min(a + chip, cy1);
        x0 = max(b, cx0);
        x1 = min(b + chip, cx1);
    } else {
        y0 = cy0;
        y1 = cy1;
        x0 = cx0;
        x1 = cx1;
    }
}

// A lane's image row segment: columns c0 - 1 .. c0 + NC.
template <int NC>
struct Seg {
    float v[NC + 2];
};

template <typename TIn, int NC>
__device__ __forceinline__ Seg<NC> load_seg(const TIn *__restrict__ row, int c0) {
    Seg<NC> s;
#pragma unroll
    for (int k = 0; k < NC + 2; ++k) s.v[k] = static_cast<float>(__ldg(row + (c0 - 1 + k)));
    return s;
}

// The k-th largest of the lanes' values v (k <= 32), the same for all lanes.
__device__ __forceinline__ float kth_best(float v, int k) {
    float m = v;
    for (int s = 0; s < k; ++s) {
        m = v;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        const unsigned eq = __ballot_sync(0xffffffffu, v == m);
        if ((threadIdx.x & 31) == __ffs(eq) - 1) v = -INFINITY;
    }
    return m;
}

// March over image rows yb - 4 .. ye + 3 of the strip whose lane owns columns
// c0 .. c0 + NC - 1, and enter the responses of rows [yb, ye), columns
// [sx, sx1) into the lane's list.  INSIDE: no row, column or neighbour leaves
// the image, and each image row is loaded once, two rows ahead; otherwise
// every gradient is formed at the clamped pixel.
template <typename TIn, int NC, int KL, bool INSIDE>
__device__ __forceinline__ void march(const TIn *__restrict__ img, int h, int w, int64_t pitch, int yb,
                                      int ye, int c0, int sx, int sx1, int y0, int x0,
                                      int k, const HarrisTaps &taps, Cand *best) {
    // The k-th largest of the lanes' best so far: what is smaller cannot be among
    // the chip's k best.  It keeps most pixels out of long lists, which are
    // costly to insert into, and is renewed every nine rows.
    float thr = -INFINITY;
    float acc[3][HK][NC];   // partial sums of nine output rows
    const int j0 = yb - HR, j1 = ye + HR;
    const TIn *next = img + (int64_t)(j0 + 2) * pitch;   // INSIDE: the row two below the current one
    Seg<NC> up, cur, dn;
    if constexpr (INSIDE) {
        up = load_seg<TIn, NC>(next - 3 * pitch, c0);
        cur = load_seg<TIn, NC>(next - 2 * pitch, c0);
        dn = load_seg<TIn, NC>(next - pitch, c0);
    }
    for (int jb = j0; jb < j1; jb += HK) {
        if constexpr (INSIDE) {
            // the next nine rows on their way to L2, one lane per 32-byte sector:
            // from DRAM a row takes longer than the step it is loaded ahead
            constexpr int SEC = 32 / (int)sizeof(TIn), POS = 32 * NC / SEC;
            for (int e = threadIdx.x & 31; e < HK * POS; e += 32) {
                const int y = jb + HK + 1 + e / POS;
                if (y <= j1)
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(img + (int64_t)y * pitch + (sx - HR + e % POS * SEC)));
            }
        }
#pragma unroll
        for (int ph = 0; ph < HK; ++ph) {
            const int j = jb + ph;
            if (j >= j1) break;
            float p[3][NC];
            if constexpr (INSIDE) {
#pragma unroll
                for (int i = 0; i < NC; ++i) {
                    const float gxv = cur.v[i + 2] - cur.v[i];
                    const float gyv = dn.v[i + 1] - up.v[i + 1];
                    p[0][i] = gxv * gxv;
                    p[1][i] = gyv * gyv;
                    p[2][i] = gxv * gyv;
                }
                up = cur;
                cur = dn;
                if (j + 1 < j1) dn = load_seg<TIn, NC>(next, c0);
                next += pitch;
            } else {
                const int cy = clampi(j, 0, h - 1);
                const TIn *rc = img + (int64_t)cy * pitch;
                const TIn *ru = img + (int64_t)max(cy - 1, 0) * pitch, *rd = img + (int64_t)min(cy + 1, h - 1) * pitch;
#pragma unroll
                for (int i = 0; i < NC; ++i) {
                    const int cx = clampi(c0 + i, 0, w - 1);
                    const float gxv = static_cast<float>(__ldg(rc + min(cx + 1, w - 1))) -
                                      static_cast<float>(__ldg(rc + max(cx - 1, 0)));
                    const float gyv = static_cast<float>(__ldg(rd + cx)) - static_cast<float>(__ldg(ru + cx));
                    p[0][i] = gxv * gxv;
                    p[1][i] = gyv * gyv;
                    p[2][i] = gxv * gyv;
                }
            }
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                // columns -4 .. NC + 3 of the lane: its own and the neighbours'
                float v[NC + 2 * HR], hp[NC];
#pragma unroll
                for (int u = 0; u < NC + 2 * HR; ++u) {
                    const int off = u - HR;                   // column relative to c0
                    const int dl = (off + 4 * NC) / NC - 4;   // the lane that owns it, relative
                    const int ci = off - dl * NC;
                    v[u] = dl == 0 ? p[q][ci]
                         : dl < 0  ? __shfl_up_sync(0xffffffffu, p[q][ci], -dl)
                                   : __shfl_down_sync(0xffffffffu, p[q][ci], dl);
                }
#pragma unroll
                for (int i = 0; i < NC; ++i) {
                    float s = 0.f;
#pragma unroll
                    for (int t = 0; t < HK; ++t) s = fmaf(taps.w[t], v[i + t], s);
                    hp[i] = s;
                }
                // row j is tap t of output row j + HR - t, whose sums lie in slot
                // (ph + HR - t) mod 9; tap 8 completes output row j - HR
#pragma unroll
                for (int t = 0; t < HK; ++t) {
                    const int slot = (ph + HR - t + 2 * HK) % HK;
#pragma unroll
                    for (int i = 0; i < NC; ++i)
                        acc[q][slot][i] = fmaf(taps.w[t], hp[i], t ? acc[q][slot][i] : 0.f);
                }
            }
            const int y = j - HR;
            if (y < yb) continue;
            constexpr int kLast = HR - (HK - 1) + 2 * HK;
            const int slot = (ph + kLast) % HK;
#pragma unroll
            for (int i = 0; i < NC; ++i) {
                const float a = acc[0][slot][i], b = acc[1][slot][i], cc = acc[2][slot][i];
                const float tr = a + b;
                const float resp = (a * b - cc * cc) - KAPPA * tr * tr;
                const int x = c0 + i;
                if (resp > best[KL - 1].v && resp >= thr && x >= sx && x < sx1) {
                    // insert into the sorted list; a lane's pixels come in ascending
                    // order, so equal responses stay behind the earlier ones
                    Cand cnd{resp, ((y - y0) << 16) | (x - x0)};
#pragma unroll
                    for (int s = 0; s < KL; ++s) {
                        if (cnd.v > best[s].v) {
                            const Cand t = best[s];
                            best[s] = cnd;
                            cnd = t;
                        }
                    }
                }
            }
        }
        if constexpr (KL > 1) thr = kth_best(best[0].v, k);
    }
}

// k: how many points a cell reports; KL >= k: length of a lane's list.
template <typename TIn, int NC, int KL>
__global__ void __launch_bounds__(32 * HWARPS, NC == 2 ? 2 : 1)
harris_march_kernel(const TIn *__restrict__ img, int h, int w, int64_t pitch, int grid_x, int grid_y,
                    int k, int chip, int margin, int strips, int seg_rows,
                    cfog_point *__restrict__ out, const HarrisTaps taps) {
    constexpr int SW = 32 * NC - 2 * HR;   // output columns of a strip
    __shared__ Cand wbest[HWARPS];
    __shared__ int wowner[HWARPS];
    __shared__ int winner;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nwarps = blockDim.x >> 5;
    const int gi = blockIdx.x, gj = blockIdx.y;
    int y0, y1, x0, x1;
    cell_chip(h, w, grid_x, grid_y, chip, margin, gj, gi, y0, y1, x0, x1);

    Cand best[KL];
#pragma unroll
    for (int s = 0; s < KL; ++s) best[s] = Cand{-INFINITY, kNoPos};

    const int seg = warp / strips, sx = x0 + (warp - seg * strips) * SW;
    const int yb = y0 + seg * seg_rows, ye = min(yb + seg_rows, y1);
    const int sx1 = min(sx + SW, x1);
    if (yb < ye && sx < sx1) {
        const int c0 = sx - HR + NC * lane;   // the lane's first column
        if (sx - HR - 1 >= 0 && sx - HR + 32 * NC <= w - 1 && yb - HR - 1 >= 0 && ye + HR <= h - 1)
            march<TIn, NC, KL, true>(img, h, w, pitch, yb, ye, c0, sx, sx1, y0, x0, k, taps, best);
        else
            march<TIn, NC, KL, false>(img, h, w, pitch, yb, ye, c0, sx, sx1, y0, x0, k, taps, best);
    }

    // k rounds of block arg-max; the owner of each winner pops it
    int ptr = 0;
    for (int s = 0; s < k; ++s) {
        Cand c = Cand{-INFINITY, kNoPos};
#pragma unroll
        for (int u = 0; u < KL; ++u)
            if (u == ptr) c = best[u];
        int owner = tid;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            Cand o;
            o.v = __shfl_down_sync(0xffffffffu, c.v, off);
            o.pos = __shfl_down_sync(0xffffffffu, c.pos, off);
            const int oo = __shfl_down_sync(0xffffffffu, owner, off);
            if (better(o, c)) {
                c = o;
                owner = oo;
            }
        }
        if (lane == 0) {
            wbest[warp] = c;
            wowner[warp] = owner;
        }
        __syncthreads();
        if (tid == 0) {
            Cand b = wbest[0];
            int bo = wowner[0];
            for (int u = 1; u < nwarps; ++u)
                if (better(wbest[u], b)) {
                    b = wbest[u];
                    bo = wowner[u];
                }
            const int idx = ((gj * grid_x) + gi) * k + s;
            if (b.pos == kNoPos) {
                out[idx] = cfog_point{-1, -1};
                winner = -1;
            } else {
                out[idx] = cfog_point{x0 + (b.pos & 0xffff), y0 + (b.pos >> 16)};
                winner = bo;
            }
        }
        __syncthreads();
        if (winner == tid) ++ptr;
        __syncthreads();
    }
}

// Launch for chips of at most ch x cw pixels.
template <typename TIn, int KL>
cfog_status launch_harris(const cfog_image *img, int grid_x, int grid_y, int k, int chip, int margin,
                          int ch, int cw, cfog_point *out, const HarrisTaps &taps, cudaStream_t st) {
    // Columns per lane: whichever covers the chip's width with fewer lanes
    // (57 columns: one strip of 88 rather than two of 56; 197: four of 56).
    // Long lists leave registers for two.
    const int s2 = (cw + 55) / 56, s3 = (cw + 87) / 88;
    const bool three = KL == 1 && 3 * s3 < 2 * s2;
    const int strips = three ? s3 : s2;
    // Row segments: each repeats eight rows, so only as many as give the chip
    // some 16 warps per SM, and none shorter than 16 rows.
    const long long want = 16LL * sm_count();
    long long segs = (want + (long long)grid_x * grid_y * strips - 1) / ((long long)grid_x * grid_y * strips);
    segs = std::min<long long>(segs, std::min(HWARPS / strips, (ch + 15) / 16));
    segs = std::max<long long>(segs, std::min(HWARPS / strips, (ch + 127) / 128));
    segs = std::max<long long>(segs, 1);
    const int seg_rows = (int)((ch + segs - 1) / segs);
    const dim3 grid(grid_x, grid_y);
    const int threads = 32 * strips * (int)segs;
    const TIn *data = static_cast<const TIn *>(img->data);
    if (three)
        harris_march_kernel<TIn, KL == 1 ? 3 : 2, KL><<<grid, threads, 0, st>>>(
            data, img->h, img->w, img->pitch, grid_x, grid_y, k, chip, margin, strips, seg_rows, out, taps);
    else
        harris_march_kernel<TIn, 2, KL><<<grid, threads, 0, st>>>(
            data, img->h, img->w, img->pitch, grid_x, grid_y, k, chip, margin, strips, seg_rows, out, taps);
    return check_launch("cfog_detect_cps: launch");
}

}  // namespace
}  // namespace cfog

extern "C" cfog_status cfog_detect_cps(const cfog_image *img, int32_t grid_x, int32_t grid_y,
                                       int32_t k, int32_t chip, int32_t margin, cfog_point *out_dev,
                                       void *stream) {
    CFOG_TRACE("cfog_detect_cps");
    using namespace cfog;
    CFOG_REQUIRE(img && img->data && out_dev, "cfog_detect_cps: null pointer");
    CFOG_REQUIRE(img->h > 0 && img->w > 0 && img->pitch >= img->w, "cfog_detect_cps: bad image");
    CFOG_REQUIRE(img->dtype == CFOG_DTYPE_F32 || img->dtype == CFOG_DTYPE_U16,
                 "cfog_detect_cps: unknown dtype %d", img->dtype);
    CFOG_REQUIRE(grid_x >= 1 && grid_y >= 1 && grid_x <= 65535 && grid_y <= 65535,
                 "cfog_detect_cps: bad grid %dx%d", grid_x, grid_y);
    CFOG_REQUIRE(k >= 1 && k <= KMAX, "cfog_detect_cps: k = %d outside [1, %d]", k, KMAX);
    CFOG_REQUIRE(margin >= 0 && 2 * margin < img->h && 2 * margin < img->w,
                 "cfog_detect_cps: margin %d leaves no interior", margin);
    const int ih = img->h - 2 * margin, iw = img->w - 2 * margin;
    CFOG_REQUIRE(grid_y <= ih && grid_x <= iw, "cfog_detect_cps: more cells than pixels");
    const int cell_h = (ih + grid_y - 1) / grid_y, cell_w = (iw + grid_x - 1) / grid_x;
    const int ch = chip > 0 ? (chip < cell_h ? chip : cell_h) : cell_h;
    const int cw = chip > 0 ? (chip < cell_w ? chip : cell_w) : cell_w;
    CFOG_REQUIRE(ch <= 256 && cw <= 256, "cfog_detect_cps: chip %dx%d exceeds 256x256", ch, cw);

    HarrisTaps taps{};
    const double sigma = 1.5;
    double sum = 0.0, tt[2 * HR + 1];
    for (int t = -HR; t <= HR; ++t) {
        tt[t + HR] = std::exp(-(double)(t * t) / (2.0 * sigma * sigma));
        sum += tt[t + HR];
    }
    for (int t = 0; t <= 2 * HR; ++t) taps.w[t] = (float)(tt[t] / sum);

    cudaStream_t st = as_stream(stream);
    const bool f32 = img->dtype == CFOG_DTYPE_F32;
    auto run = [&](auto kl) {
        constexpr int KL = decltype(kl)::value;
        return f32 ? launch_harris<float, KL>(img, grid_x, grid_y, k, chip, margin, ch, cw, out_dev, taps, st)
                   : launch_harris<uint16_t, KL>(img, grid_x, grid_y, k, chip, margin, ch, cw, out_dev, taps, st);
    };
    return k == 1  ? run(std::integral_constant<int, 1>{})
           : k <= 4 ? run(std::integral_constant<int, 4>{})
                    : run(std::integral_constant<int, KMAX>{});
}
