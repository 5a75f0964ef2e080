// body_resample.cuh -- the three image-rearranging bodies of Sec. 4.1:
// bilinear x2 upsampling, 3x3/s2/p1 max pooling and 3x3/s1/p1 im2col.
//
// All three are HBM-bound.  The vector paths give each warp a strip of rows
// of one plane: lane l holds input columns 4l..4l+3 of a 128-column band as
// one 128-bit load, the one-column halo comes from the neighbouring lane by
// shuffle, rows slide through registers so each input row is loaded once per
// strip, the next rows are loaded before the current one is used, and
// outputs leave as 128-bit (or 64-bit) streaming stores.  Rows that are not
// 16-byte multiples, and unaligned tensors, take the flat path (FlatRows
// below) with the same arithmetic.
#pragma once
#include "hf_device.cuh"

namespace hf {

// (plane, strip) of a warp's ring work items -- items it, it + step, ...
// with it = plane * ns + strip -- advanced without divisions.
struct ItemCursor {
    unsigned p, s;
    __device__ void init(int64_t it, unsigned ns)
    {
        p = (unsigned)(it / ns);
        s = (unsigned)(it - (int64_t)p * ns);
    }
    __device__ void step(unsigned dq, unsigned dr, unsigned ns)   // step = dq * ns + dr
    {
        s += dr;
        p += dq;
        if (s >= ns) s -= ns, ++p;
    }
};

// ------------------------------------------------------------------------
// The flat path, for rows of any length.  The rows of all planes are one
// sequence; a work item is R consecutive rows, whatever planes they belong
// to, and its pixels i = 0 .. R*W-1 go to lanes in memory order, so a row of
// 7 or 75 values leaves no lane idle and neighbours are at constant offsets
// (-W-1 .. W+1) from a pixel.  An item's input rows with their halo are one
// contiguous range: with a ring they arrive as one bulk copy, its ends
// rounded out to 16 bytes (the tensor's last values, past its last multiple
// of four, are patched in with plain loads); without one the lanes load them
// from global memory.  Only the division of a pixel's index by the row
// length remains, a multiply and a shift (indices stay below 1024).
//
// The bound is HBM at full occupancy and issue in a fused block of few warps:
// 32 pixels of upsample move 640 bytes, for which an SM has about 108 issue
// slots, and take about 100.  It replaces paths of
// one thread per output with two 64-bit divisions each.  On one GB300, before
// -> with it: upsample 8x64x75x75 + max pool 8x64x147x147 fused 287 -> 26.6
// us, im2col 8x64x112x112 alone 309 -> 46.0 us (5.6 TB/s), batch-norm
// 64x512x7x7 + im2col 32x256x14x14 fused 243 -> 22.3 us (18.6 with the
// statistics' deeper loads).
struct FlatRows {
    unsigned W, H, R;    // values per row, rows per plane, rows per item
    unsigned rows;       // rows of all planes
    unsigned mw, mh;     // ceil(2^20 / W), ceil(2^21 / H)
    static constexpr unsigned kMaxValues = 1014;   // values of an item (i * (W - 1) < 2^20)

    // rmax: rows an item may have; warps: of the grid; R is a multiple of
    // `multiple`.  Items are as large as rmax and as even as the number of
    // warps allows.
    __device__ void init(unsigned w, unsigned h, unsigned rows_, unsigned rmax, unsigned warps, unsigned multiple)
    {
        W = w;
        H = h;
        rows = rows_;
        const unsigned each = (rows + warps - 1) / warps;      // rows per warp
        const unsigned turns = (each + rmax - 1) / rmax;       // items per warp
        R = (each + turns - 1) / turns;
        R = min((R + multiple - 1) / multiple * multiple, rmax);
        mw = ((1u << 20) + W - 1) / W;
        mh = ((1u << 21) + H - 1) / H;
    }
    __device__ unsigned items() const { return (rows + R - 1) / R; }
    // row of pixel i of an item; plane (counted from the item's first) of
    // row t of that plane's run of rows, t < H + R
    __device__ unsigned row_of(unsigned i) const { return R == 1 ? 0u : (i * mw) >> 20; }
    __device__ unsigned plane_of(unsigned t) const { return H <= 1024 ? (t * mh) >> 21 : (t >= H ? 1u : 0u); }
};

// Plane p and row r in it of the first row of a warp's items it, it + step,
// ..., advanced without divisions: in items of few pixels, as max pool's two
// rows of 74, those were a fifth of the instructions (upsample 8x64x75x75 +
// max pool 8x64x147x147 28.4 -> 26.6 us; im2col, bound by its stores, gained
// nothing and divides).
struct FlatCursor {
    unsigned p, r, dp, dr;
    __device__ void init(const FlatRows &f, int64_t it, int64_t step)
    {
        const uint64_t row = it < (int64_t)f.items() ? (uint64_t)it * f.R : 0, d = (uint64_t)step * f.R;
        p = (unsigned)(row / f.H);
        r = (unsigned)(row - (uint64_t)p * f.H);
        dp = (unsigned)(d / f.H);   // beyond 32 bits only where no second item exists
        dr = (unsigned)(d - d / f.H * f.H);
    }
    __device__ void step(unsigned H)
    {
        p += dp;
        r += dr;
        if (r >= H) r -= H, ++p;
    }
};

// Reads of an item's values at offsets from its first pixel: from the stage,
// where every offset within the halo is inside the stage (values outside
// the tensor are never used), or from global memory where `ok`.
struct FlatStage {
    const float *p;
    __device__ float operator()(int off, bool) const { return p[off]; }
};
struct FlatGlobal {
    const float *p;
    __device__ float operator()(int off, bool ok) const { return ok ? __ldg(p + off) : 0.f; }
};

// The stage layout of values [lo, hi) of x (lo may be negative, hi past the
// end): stage float k holds value base + k, base = lo rounded down to a
// multiple of four.  Lane 0 copies what lies in [0, total / 4 * 4).
struct FlatCopy {
    int64_t base, src, end;   // first value of the stage, values copied [src, end)
    __device__ FlatCopy(int64_t lo, int64_t hi, int64_t total)
    {
        base = lo & ~(int64_t)3;
        src = base > 0 ? base : 0;
        const int64_t up = (hi + 3) & ~(int64_t)3, most = total & ~(int64_t)3;
        end = up < most ? up : most;
    }
    __device__ void fill(const WarpRing &r, int st, const float *x) const
    {
        const unsigned bytes = end > src ? (unsigned)(end - src) * 4u : 0u;
        r.expect(st, bytes);
        if (bytes) r.copy(st, (unsigned)(src - base) * 4u, x + src, bytes);
    }
    // all lanes, once the stage has landed: the tensor's last values
    __device__ void patch(unsigned char *stage, const float *x, int64_t hi, int64_t total, int lane) const
    {
        const int64_t last = total & ~(int64_t)3;
        const int64_t upto = hi < total ? hi : total;
        if (upto > last) {
            const int64_t first = last > base ? last : base;
            if (first + lane < upto) reinterpret_cast<float *>(stage)[first + lane - base] = __ldg(x + first + lane);
            __syncwarp();
        }
    }
};
// The range of the flat path's 32-bit rows, offsets and warp counts.
__device__ __forceinline__ bool flat_range(int64_t rows, int64_t W, const Ctx &cx)
{
    return rows < ((int64_t)1 << 31) && W < ((int64_t)1 << 29) && (int64_t)cx.grid * (cx.nthreads >> 5) < ((int64_t)1 << 31);
}
// Whether the flat path without a ring keeps enough warps busy: an item is at
// least one row, so a tensor has `rows` items at most, and below one for every
// `per` warps a thread per output is faster however long the rows are (one row
// of 1000003 values on one warp: 6160 / 3770 / 19600 us for upsample / max
// pool / im2col, a thread per output 25.6 / 5.1 / 43.3).  The lines are where
// a warp's 32 outputs in turn (0.20 / 0.24 / 0.63 us) cost what the threads'
// shares do (1.0 / 0.5 / 0.56 us an output).
__device__ __forceinline__ bool enough_rows(int64_t rows, const Ctx &cx, int per)
{
    return rows * per >= (int64_t)cx.grid * (cx.nthreads >> 5);
}
// Floats of a stage that an item's halo and the rounding take: base is up to
// three below lo, the copy's end up to three past hi.
constexpr unsigned kFlatPad = 8;

// ------------------------------------------------------------------------
// Bilinear x2, half-pixel centres.  Along one axis of length L, output 2i
// blends input i-1 and i with weights 1/4, 3/4 (output 0 is input 0) and
// output 2i+1 blends i and i+1 with 3/4, 1/4 (output 2L-1 is input L-1).
// Each blend is one fused multiply-add of an exactly scaled quarter, so it
// is correctly rounded; rows are blended horizontally first, then
// vertically, the order of the two-level formula.
struct BodyUpsample {
    using Args = hf_upsample2x_args;
    static constexpr int kId = HF_BODY_UPSAMPLE2X;
    static constexpr int kRows = 8;    // input rows per warp strip
    static constexpr int kBarriers = 0;
    // ring path: a stage holds the 6 input rows of an item and its two halo
    // rows (rows of up to 128 floats)
    static constexpr int kRingRows = 6;
    static constexpr bool kRingItem = true;
    static constexpr unsigned kRingMinBytes = 4096;   // the stage: one item

    // Which path: 16-byte rows of 64 values or more go to strips of whole
    // rows (four columns a lane), the others to the flat path.  Strips leave
    // lanes idle below 128 columns: 2^23 values in images of W = 8 / 16 /
    // 32 / 40 / 56 / 64 columns took 181 / 83 / 49 / 41 / 35 / 33 us alone,
    // the flat path 37 / 35 / 34 / 36 / 35 / 35 (112: 37 and 35).  In a narrow
    // interval the flat path's cost does not depend on W and a strip's falls
    // with it: 2^22 values with one warp an SM, W = 32 / 40 / 48 / 56 / 60 / 64 /
    // 96 / 112, strips 156 / 116 / 94 / 86 / 76 / 72 / 48 / 43 us, flat 65 to 70.
    // Rows of 129 to 252 columns are too long for a strip's stage, but two
    // rows with their halo still fit a flat item's: 57 us on registers, 51
    // flat (W = 224, four warps an SM; 39 and 37 us at full occupancy).
    // Longer ones keep the register path (W = 400: 39 us, 47 flat).
    // Small tensors of other rows cannot repay the flat path's start (a dozen
    // divisions and the ring): up to kFewOutputs outputs per thread go to a
    // thread each (60 rows of 75 columns 2.8 us, flat 3.9; 2000 rows 7.2 and
    // 5.2).
    static constexpr int kStripCols = 64;
    static constexpr int kFewOutputs = 1;
    static __host__ __device__ bool rows16(const Args &a)
    {
        return (a.W & 3) == 0 && aligned16(a.x) && aligned16(a.y);
    }
    static __host__ __device__ bool small(const Args &a, int64_t threads)   // of the grid
    {
        return !rows16(a) && 4 * (int64_t)a.P * a.H * a.W <= kFewOutputs * threads;
    }
    static __host__ __device__ bool strips(const Args &a)
    {
        return rows16(a) && a.W >= kStripCols && (a.W <= 128 || 4u * a.W + kFlatPad > kRingMinBytes / 4);
    }
    // a strip's rows (W <= 128) or a flat item's arrive as one bulk copy
    static __host__ bool uses_ring(const Args &a)
    {
        if ((int64_t)a.P * a.H * a.W <= 0) return false;
        return strips(a) ? a.W <= 128 : aligned16(a.x) && 3u * a.W + kFlatPad <= kRingMinBytes / 4;
    }
    // the flat path without one is up to three times slower, strips are not
    static __host__ bool needs_ring(const Args &a) { return !rows16(a) || a.W < kStripCols; }
    static __host__ double ring_work(const Args &a) { return 20.0 * a.P * a.H * a.W; }

    static __host__ size_t workspace_bytes(const Args &) { return 0; }
    static __host__ size_t smem_bytes(int, const Args &) { return 0; }
    static __host__ hf_status validate(const Args &a)
    {
        if (a.P < 0 || a.H < 0 || a.W < 0) return HF_ERR_INVALID;
        if ((int64_t)a.P * a.H * a.W == 0) return HF_OK;
        if (!a.x || !a.y) return HF_ERR_INVALID;
        if ((int64_t)a.P * a.H * a.W * 4 >= (int64_t)1 << 40) return HF_ERR_INVALID;
        return HF_OK;
    }

    static __device__ __forceinline__ float blend(float near, float far)
    {
        return __fmaf_rn(0.75f, near, __fmul_rn(0.25f, far));
    }

    struct Raw {
        float4 q;
        float left, right;   // halo columns fetched only at band edges
    };

    static __device__ __forceinline__ Raw load_row(const float *row, int c0, int W, bool act)
    {
        Raw r;
        r.q = act ? ldg4(row + c0) : make_float4(0.f, 0.f, 0.f, 0.f);
        const int lane = lane_id();
        r.left = 0.f;
        r.right = 0.f;
        if (act && lane == 0 && c0 > 0) r.left = __ldg(row + c0 - 1);
        if (act && lane == 31 && c0 + 4 < W) r.right = __ldg(row + c0 + 4);
        return r;
    }

    // Horizontal pass of one row: out[0..7] = outputs 2c0 .. 2c0+7.
    static __device__ __forceinline__ void hpass(const Raw &r, int c0, int W, float h[8])
    {
        const int lane = lane_id();
        float L = __shfl_up_sync(0xffffffffu, r.q.w, 1);
        float R = __shfl_down_sync(0xffffffffu, r.q.x, 1);
        if (lane == 0) L = r.left;
        if (lane == 31) R = r.right;
        const float C[4] = {r.q.x, r.q.y, r.q.z, r.q.w};
        const float Lf[4] = {L, r.q.x, r.q.y, r.q.z};
        const float Rt[4] = {r.q.y, r.q.z, r.q.w, R};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int col = c0 + i;
            h[2 * i] = col == 0 ? C[i] : blend(C[i], Lf[i]);
            h[2 * i + 1] = col == W - 1 ? C[i] : blend(C[i], Rt[i]);
        }
    }

    static __device__ void run_vec(const Args &a, const Ctx &cx)
    {
        const int H = a.H, W = a.W, Wo = 2 * W;
        const int nb = (W + 127) / 128;
        const int ns = (H + kRows - 1) / kRows;
        const int64_t items = (int64_t)a.P * ns * nb;
        const int nw = cx.nthreads >> 5;
        const int lane = lane_id();
        for (int64_t it = (int64_t)cx.block * nw + (cx.tid >> 5); it < items;
             it += (int64_t)cx.grid * nw) {
            const int b = (int)(it % nb);
            const int64_t ps = it / nb;
            const int s = (int)(ps % ns);
            const int64_t p = ps / ns;
            const int c0 = b * 128 + 4 * lane;
            const bool act = c0 < W;
            const float *xp = a.x + p * H * W;
            float *yp = a.y + p * (int64_t)(2 * H) * Wo;
            const int r0 = s * kRows;
            const int r1 = min(r0 + kRows, H);
            float hp[8], hc[8], hn[8];
            Raw rn = load_row(xp + (int64_t)min(r0 + 1, H - 1) * W, c0, W, act);
            if (r0 > 0) {
                Raw rp = load_row(xp + (int64_t)(r0 - 1) * W, c0, W, act);
                hpass(rp, c0, W, hp);
            }
            {
                Raw rc = load_row(xp + (int64_t)r0 * W, c0, W, act);
                hpass(rc, c0, W, hc);
            }
#pragma unroll 2
            for (int r = r0; r < r1; ++r) {
                // prefetch row r+2 while row r+1 is blended
                Raw rf = load_row(xp + (int64_t)min(r + 2, H - 1) * W, c0, W, act);
                hpass(rn, c0, W, hn);
                float e[8], o[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    e[i] = r == 0 ? hc[i] : blend(hc[i], hp[i]);
                    o[i] = r == H - 1 ? hc[i] : blend(hc[i], hn[i]);
                }
                if (act) {
                    float *ye = yp + (int64_t)(2 * r) * Wo + 2 * c0;
                    stcs4(ye, make_float4(e[0], e[1], e[2], e[3]));
                    stcs4(ye + 4, make_float4(e[4], e[5], e[6], e[7]));
                    float *yo = ye + Wo;
                    stcs4(yo, make_float4(o[0], o[1], o[2], o[3]));
                    stcs4(yo + 4, make_float4(o[4], o[5], o[6], o[7]));
                }
#pragma unroll
                for (int i = 0; i < 8; ++i) hp[i] = hc[i], hc[i] = hn[i];
                rn = rf;
            }
        }
    }

    // Ring path.  Work item = (plane, strip of R = 6 input rows); the strip
    // and its halo rows, [max(r0-1, 0), min(r0+R+1, H)), are contiguous and
    // arrive in one bulk copy in a stage of the warp's ring while the next
    // items' copies are in flight.  Lane l takes input columns 4l..4l+3 of
    // each row from shared memory (the halo columns from lanes l-1 and l+1
    // by shuffle; a band is the whole row, so lane 0's left and the last
    // lane's right column are outside the image and never blended) and
    // slides the horizontal passes of rows r-1, r, r+1 down the strip; each
    // output is the register path's blend of the same values, so the two
    // paths give the same bits.
    static __device__ bool run_ring(const Args &a, const Ctx &cx)
    {
        constexpr int R = kRingRows;
        const int H = a.H, W = a.W, Wo = 2 * W;
        const unsigned row_bytes = 4u * (unsigned)W;
        if (cx.ring_stage < (R + 2) * row_bytes || (int64_t)a.P * H >= ((int64_t)1 << 32)) return false;
        const unsigned ns = (unsigned)((H + R - 1) / R);
        const int64_t items = (int64_t)a.P * ns;
        WarpRing r;
        r.init(cx, 0);
        const int nw = cx.nthreads >> 5;
        const int64_t gw = (int64_t)cx.block * nw + (cx.tid >> 5), GW = (int64_t)cx.grid * nw;
        const unsigned dq = (unsigned)(GW / ns), dr = (unsigned)(GW % ns);
        const int lane = lane_id();
        const int c0 = 4 * lane;
        const bool act = c0 < W;
        ItemCursor fc, uc;   // the fill cursor runs S items ahead of the use cursor
        fc.init(gw, ns);
        uc = fc;
        ring_stream(
            r, gw, GW, items,
            [&](int st, int64_t) {
                const int r0 = (int)fc.s * R;
                const int ylo = max(r0 - 1, 0), yhi = min(r0 + R + 1, H);
                const unsigned bytes = (unsigned)(yhi - ylo) * row_bytes;   // rows are 16-byte multiples
                r.expect(st, bytes);
                r.copy(st, 0, a.x + ((uint64_t)fc.p * (unsigned)H + (unsigned)ylo) * W, bytes);
                fc.step(dq, dr, ns);
            },
            [&](const unsigned char *stage, int64_t) {
                const int r0 = (int)uc.s * R, r1 = min(r0 + R, H);
                const int ylo = max(r0 - 1, 0), yhi = min(r0 + R + 1, H);
                const unsigned char *base = stage + (act ? 4 * c0 : 0);
                auto hrow = [&](int y, float h[8]) {
                    y = min(max(y, ylo), yhi - 1);   // rows outside are never blended
                    Raw q;
                    q.q = *reinterpret_cast<const float4 *>(base + (unsigned)(y - ylo) * row_bytes);
                    q.left = 0.f;
                    q.right = 0.f;
                    hpass(q, c0, W, h);
                };
                float *yp = a.y + ((int64_t)uc.p * (2 * H) + 2 * r0) * Wo + 2 * c0;
                float hp[8], hc[8], hn[8];
                hrow(r0 - 1, hp);
                hrow(r0, hc);
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    const int rr = r0 + i;
                    hrow(rr + 1, hn);
                    if (rr < r1) {
                        float e[8], o[8];
#pragma unroll
                        for (int k = 0; k < 8; ++k) {
                            e[k] = rr == 0 ? hc[k] : blend(hc[k], hp[k]);
                            o[k] = rr == H - 1 ? hc[k] : blend(hc[k], hn[k]);
                        }
                        if (act) {
                            float *ye = yp + (int64_t)(2 * i) * Wo;
                            stcs4(ye, make_float4(e[0], e[1], e[2], e[3]));
                            stcs4(ye + 4, make_float4(e[4], e[5], e[6], e[7]));
                            stcs4(ye + Wo, make_float4(o[0], o[1], o[2], o[3]));
                            stcs4(ye + Wo + 4, make_float4(o[4], o[5], o[6], o[7]));
                        }
                    }
#pragma unroll
                    for (int k = 0; k < 8; ++k) hp[k] = hc[k], hc[k] = hn[k];
                }
                uc.step(dq, dr, ns);
            });
        r.finish();
        return true;
    }

    // One item of the flat path: pixel i gives the outputs (2r, 2r+1) x
    // (2c, 2c+1); in memory they start at 4*i - 2*c from the item's first.
    template <class Get>
    static __device__ __forceinline__ void flat_item(const Args &a, const FlatRows &f, unsigned g0, unsigned r0,
                                                     unsigned n, const Get &get)
    {
        const int W = (int)f.W;
        float *y0 = a.y + 4 * (int64_t)g0 * W;
        const bool y8 = (reinterpret_cast<uintptr_t>(a.y) & 7u) == 0;
#pragma unroll 2
        for (unsigned i = lane_id(); i < n; i += 32) {
            const unsigned lr = f.row_of(i), c = i - lr * f.W, t = r0 + lr;
            const unsigned r = t - f.plane_of(t) * f.H;
            const bool le = c == 0, re = c == f.W - 1, te = r == 0, be = r == f.H - 1;
            auto hrow = [&](int off, bool ok, float &h0, float &h1) {
                const float C = get(off, ok), L = get(off - 1, ok && !le), R = get(off + 1, ok && !re);
                h0 = le ? C : blend(C, L);
                h1 = re ? C : blend(C, R);
            };
            float u0, u1, c0, c1, d0, d1;
            hrow((int)i - W, !te, u0, u1);
            hrow((int)i, true, c0, c1);
            hrow((int)i + W, !be, d0, d1);
            const float2 e = make_float2(te ? c0 : blend(c0, u0), te ? c1 : blend(c1, u1));
            const float2 o = make_float2(be ? c0 : blend(c0, d0), be ? c1 : blend(c1, d1));
            float *ye = y0 + (4 * (int64_t)i - 2 * c), *yo = ye + 2 * W;
            if (y8) {
                stcs2(ye, e);
                stcs2(yo, o);
            } else {
                __stcs(ye, e.x);
                __stcs(ye + 1, e.y);
                __stcs(yo, o.x);
                __stcs(yo + 1, o.y);
            }
        }
    }

    static __device__ bool flat_ring(const Args &a, const Ctx &cx)
    {
        const int64_t rows = (int64_t)a.P * a.H, total = rows * a.W;
        const int nw = cx.nthreads >> 5;
        const int64_t gw = (int64_t)cx.block * nw + (cx.tid >> 5), GW = (int64_t)cx.grid * nw;
        const unsigned W = (unsigned)a.W, slots = min(cx.ring_stage, 4096u) / 4;
        if (!aligned16(a.x) || 3 * W + kFlatPad > slots || !WarpRing::available(cx, 0)) return false;
        FlatRows f;
        f.init(W, a.H, (unsigned)rows, min((slots - kFlatPad) / W - 2, FlatRows::kMaxValues / W), (unsigned)GW, 1);
        WarpRing r;
        r.init(cx, 0);
        FlatCursor uc;
        uc.init(f, gw, GW);
        auto copy = [&](int64_t it) {
            const int64_t g0 = it * f.R;
            return FlatCopy((g0 - 1) * W - 1, (min(g0 + (int64_t)f.R, rows) + 1) * W + 1, total);
        };
        ring_stream(
            r, gw, GW, f.items(), [&](int st, int64_t it) { copy(it).fill(r, st, a.x); },
            [&](unsigned char *stage, int64_t it) {
                const int64_t g0 = it * f.R, g1 = min(g0 + (int64_t)f.R, rows);
                const FlatCopy k = copy(it);
                k.patch(stage, a.x, (g1 + 1) * W + 1, total, r.lane);
                flat_item(a, f, (unsigned)g0, uc.r, (unsigned)(g1 - g0) * W,
                          FlatStage{reinterpret_cast<const float *>(stage) + (g0 * W - k.base)});
                uc.step(f.H);
            });
        r.finish();
        return true;
    }

    // The same items without a ring.
    static __device__ void flat_global(const Args &a, const Ctx &cx)
    {
        const int64_t rows = (int64_t)a.P * a.H;
        const int nw = cx.nthreads >> 5;
        const int64_t gw = (int64_t)cx.block * nw + (cx.tid >> 5), GW = (int64_t)cx.grid * nw;
        const unsigned W = (unsigned)a.W;
        FlatRows f;
        f.init(W, a.H, (unsigned)rows, max(1u, FlatRows::kMaxValues / W), (unsigned)GW, 1);
        for (int64_t it = gw; it < f.items(); it += GW) {
            const int64_t g0 = it * f.R, g1 = min(g0 + (int64_t)f.R, rows);
            flat_item(a, f, (unsigned)g0, (unsigned)g0 % f.H, (unsigned)(g1 - g0) * W, FlatGlobal{a.x + g0 * W});
        }
    }

    // One thread per output: few outputs, few long rows, and tensors of 2^31
    // rows or more.
    static __device__ void run_scalar(const Args &a, const Ctx &cx)
    {
        const int H = a.H, W = a.W, Ho = 2 * H, Wo = 2 * W;
        const int64_t total = (int64_t)a.P * Ho * Wo;
        for (int64_t i = (int64_t)cx.block * cx.nthreads + cx.tid; i < total;
             i += (int64_t)cx.grid * cx.nthreads) {
            const int ox = (int)(i % Wo);
            const int oy = (int)((i / Wo) % Ho);
            const int64_t p = i / ((int64_t)Wo * Ho);
            const float *xp = a.x + p * H * W;
            auto hrow = [&](int y) {
                const int c = ox >> 1;
                const float C = __ldg(xp + (int64_t)y * W + c);
                if (ox & 1)
                    return c == W - 1 ? C : blend(C, __ldg(xp + (int64_t)y * W + c + 1));
                return c == 0 ? C : blend(C, __ldg(xp + (int64_t)y * W + c - 1));
            };
            const int r = oy >> 1;
            const float hc = hrow(r);
            float v;
            if (oy & 1)
                v = r == H - 1 ? hc : blend(hc, hrow(r + 1));
            else
                v = r == 0 ? hc : blend(hc, hrow(r - 1));
            a.y[i] = v;
        }
    }

    // SMALL: with the rule on small tensors (a kernel launched alone is chosen
    // by it before the launch).
    template <bool SMALL, int>
    static __device__ __forceinline__ void run_as(const Args &a, const Ctx &cx)
    {
        if ((int64_t)a.P * a.H * a.W == 0) return;
        const bool flat = flat_range((int64_t)a.P * a.H, a.W, cx) &&
                          !(SMALL && small(a, (int64_t)cx.grid * cx.nthreads));
        if (strips(a)) {
            if (a.W <= 128 && WarpRing::available(cx, 0) && run_ring(a, cx)) return;
        } else if (flat && flat_ring(a, cx)) {
            return;
        }
        if (a.W >= kStripCols && rows16(a)) run_vec(a, cx);
        else if (flat && enough_rows((int64_t)a.P * a.H, cx, 12)) flat_global(a, cx);
        else run_scalar(a, cx);
    }
};

// The body without the flat path, launched alone where that is not the better
// one: strips of 16-byte rows, else one thread per output.  A kernel of its
// own, because beside the flat path the compiler's strips take up to 10 % and
// more registers.
struct BodyUpsamplePlain {
    using Of = BodyUpsample;
    using Args = Of::Args;
    static constexpr int kId = Of::kId;
    static __host__ bool pick(const Args &a, int, int64_t threads) { return Of::strips(a) || Of::small(a, threads); }
    static __host__ bool uses_ring(const Args &a)
    {
        return (int64_t)a.P * a.H * a.W > 0 && Of::rows16(a) && a.W <= 128;
    }
    static __device__ void run(const Args &a, const Ctx &cx)
    {
        if ((int64_t)a.P * a.H * a.W == 0) return;
        if (Of::rows16(a)) {
            if (a.W <= 128 && WarpRing::available(cx, 0) && Of::run_ring(a, cx)) return;
            Of::run_vec(a, cx);
        } else {
            Of::run_scalar(a, cx);
        }
    }
};

// ------------------------------------------------------------------------
// 3x3 max pooling, stride 2, padding 1 (padding never wins).
struct BodyMaxpool {
    using Args = hf_maxpool3s2_args;
    static constexpr int kId = HF_BODY_MAXPOOL3S2;
    static constexpr int kRows = 8;    // output rows per warp strip
    static constexpr int kBarriers = 0;
    // ring path: a stage must hold the 9 input rows of a strip of 4 output
    // rows (rows of up to 128 floats)
    static constexpr bool kRingItem = true;
    static constexpr unsigned kRingMinBytes = 4096;   // the stage: one item

    // Which path: 16-byte rows of 64 values or more go to strips of whole
    // rows (four columns a lane), the others to the flat path.  Strips leave
    // lanes idle below 128 columns: 2^23 values in images of W = 8 / 16 /
    // 32 / 40 / 56 / 64 columns took 74 / 43 / 28 / 25 / 22 / 21 us alone,
    // the flat path 22 / 22 / 21 / 22 / 22 / 21 (at W = 112 strips 18, flat 21).
    // With one warp an SM (2^22 values, W = 32 / 48 / 56 / 60 / 64) strips took
    // 66 / 46 / 40 / 39 / 34 us, flat 31 / 32 / 29 / 31 / 33.  Between, where a warp has
    // but a few items, the flat path's larger ones are less even: from 48
    // columns on, 1 to 12 rows a warp go to strips, from 60 on 1 to 32 (24 warps
    // an SM, 37000 rows of 56 outputs, 10 a warp, 7.6 us, flat 9.6; 16 warps,
    // 35000 rows of 60, 14 a warp, 7.2 and 8.2; 58 a warp 12.1 and 10.6; less
    // than one a warp 4.4 and 3.1).
    // Small tensors of other rows cannot repay the flat path's start (a dozen
    // divisions and the ring): up to two outputs per thread go to a thread each
    // (2000 rows of 38 outputs 3.2 us, flat 5.5), eight where no ring holds three
    // rows (27 a thread 26 us, flat 16).
    static constexpr int kStripCols = 64;
    static __host__ __device__ bool small(const Args &a, int64_t threads)   // of the grid
    {
        const int64_t rows = (int64_t)a.P * ((a.H - 1) / 2 + 1), warps = threads / 32;
        return rows16(a) ? a.W >= 48 && rows > warps && rows <= (a.W >= 60 ? 32 : 12) * warps
                         : rows * ((a.W - 1) / 2 + 1) <= (ring_rows(a) ? 2 : 8) * threads;
    }
    static __host__ __device__ bool rows16(const Args &a)
    {
        return (a.W & 3) == 0 && aligned16(a.x) && aligned16(a.y);
    }
    static __host__ __device__ bool strips(const Args &a) { return rows16(a) && a.W >= kStripCols; }
    // a strip's rows (W <= 128) or a flat item's arrive as one bulk copy
    static __host__ bool uses_ring(const Args &a)
    {
        if ((int64_t)a.P * a.H * a.W <= 0) return false;
        return strips(a) ? a.W <= 128 && a.H >= 2 : ring_rows(a);
    }
    static __host__ bool needs_ring(const Args &a) { return !strips(a); }   // as in BodyUpsample
    static __host__ double ring_work(const Args &a) { return 5.0 * a.P * a.H * a.W; }
    // three rows and the rounding fit a stage: what a flat item needs
    static __host__ __device__ bool ring_rows(const Args &a)
    {
        return aligned16(a.x) && 3u * a.W + kFlatPad <= kRingMinBytes / 4;
    }

    static __host__ size_t workspace_bytes(const Args &) { return 0; }
    static __host__ size_t smem_bytes(int, const Args &) { return 0; }
    static __host__ hf_status validate(const Args &a)
    {
        if (a.P < 0 || a.H < 0 || a.W < 0) return HF_ERR_INVALID;
        if ((int64_t)a.P * a.H * a.W == 0) return HF_OK;
        if (!a.x || !a.y) return HF_ERR_INVALID;
        if ((int64_t)a.P * a.H * a.W >= (int64_t)1 << 40) return HF_ERR_INVALID;
        return HF_OK;
    }

    static __device__ __forceinline__ float mx(float u, float v) { return v > u ? v : u; }

    struct Raw {
        float4 q;
        float left;
    };
    static __device__ __forceinline__ Raw load_row(const float *row, int c0, bool act, bool valid)
    {
        const float ninf = -__int_as_float(0x7f800000);
        Raw r;
        r.q = (act && valid) ? ldg4(row + c0) : make_float4(ninf, ninf, ninf, ninf);
        r.left = ninf;
        if (act && valid && lane_id() == 0 && c0 > 0) r.left = __ldg(row + c0 - 1);
        return r;
    }
    // Horizontal 3-wide maxima centred on input columns c0 and c0+2.
    static __device__ __forceinline__ float2 hmax(const Raw &r)
    {
        float L = __shfl_up_sync(0xffffffffu, r.q.w, 1);
        if (lane_id() == 0) L = r.left;
        return make_float2(mx(mx(L, r.q.x), r.q.y), mx(mx(r.q.y, r.q.z), r.q.w));
    }

    static __device__ void run_vec(const Args &a, const Ctx &cx)
    {
        const int H = a.H, W = a.W, Ho = (H - 1) / 2 + 1, Wo = (W - 1) / 2 + 1;
        const int nb = (W + 127) / 128;
        const int ns = (Ho + kRows - 1) / kRows;
        const int64_t items = (int64_t)a.P * ns * nb;
        const int nw = cx.nthreads >> 5;
        const int lane = lane_id();
        for (int64_t it = (int64_t)cx.block * nw + (cx.tid >> 5); it < items;
             it += (int64_t)cx.grid * nw) {
            const int b = (int)(it % nb);
            const int64_t ps = it / nb;
            const int s = (int)(ps % ns);
            const int64_t p = ps / ns;
            const int c0 = b * 128 + 4 * lane;
            const bool act = c0 < W;
            const float *xp = a.x + p * H * W;
            float *yp = a.y + p * (int64_t)Ho * Wo;
            const int o0 = s * kRows, o1 = min(o0 + kRows, Ho);
            // carried: horizontal maxima of input row 2*oy - 1
            float2 top = hmax(load_row(xp + (int64_t)(2 * o0 - 1) * W, c0, act, o0 > 0));
            Raw ra = load_row(xp + (int64_t)(2 * o0) * W, c0, act, 2 * o0 < H);
            Raw rb = load_row(xp + (int64_t)(2 * o0 + 1) * W, c0, act, 2 * o0 + 1 < H);
#pragma unroll 2
            for (int oy = o0; oy < o1; ++oy) {
                const int n0 = 2 * oy + 2, n1 = 2 * oy + 3;
                Raw na = load_row(xp + (int64_t)n0 * W, c0, act, oy + 1 < o1 && n0 < H);
                Raw nbr = load_row(xp + (int64_t)n1 * W, c0, act, oy + 1 < o1 && n1 < H);
                const float2 m0 = hmax(ra), m1 = hmax(rb);
                const float2 v = make_float2(mx(mx(top.x, m0.x), m1.x), mx(mx(top.y, m0.y), m1.y));
                if (act) stcs2(yp + (int64_t)oy * Wo + (c0 >> 1), v);
                top = m1;
                ra = na;
                rb = nbr;
            }
        }
    }

    // Ring path.  Work item = (plane, strip of R = 4 output rows); its
    // input rows [max(2*o0-1, 0), min(2*o1, H)) are contiguous and arrive
    // in one bulk copy in a stage of the warp's ring, the next items' copies
    // in flight meanwhile.  Lane l takes input columns 4l..4l+3 (output
    // columns 2l, 2l+1) of each of the strip's nine rows from shared memory
    // (nine independent loads); the left halo column comes from lane l-1 by
    // shuffle.  No loads are held in registers, so bytes in flight do not
    // depend on registers or warps.
    static constexpr int kRingRows = 4;   // output rows per ring work item

    static __device__ bool run_ring(const Args &a, const Ctx &cx)
    {
        constexpr int R = kRingRows, NR = 2 * R + 1;
        const int H = a.H, W = a.W, Ho = (H - 1) / 2 + 1, Wo = (W - 1) / 2 + 1;
        const unsigned row_bytes = 4u * (unsigned)W;
        if (cx.ring_stage < NR * row_bytes || (int64_t)a.P * H >= ((int64_t)1 << 32)) return false;
        const unsigned ns = (unsigned)((Ho + R - 1) / R);
        const int64_t items = (int64_t)a.P * ns;
        WarpRing r;
        r.init(cx, 0);
        const int nw = cx.nthreads >> 5;
        const int64_t gw = (int64_t)cx.block * nw + (cx.tid >> 5), GW = (int64_t)cx.grid * nw;
        const unsigned dq = (unsigned)(GW / ns), dr = (unsigned)(GW % ns);
        const int lane = lane_id();
        const int c0 = 4 * lane;
        const bool act = c0 < W;
        const float ninf = -__int_as_float(0x7f800000);
        ItemCursor fc, uc;   // the fill cursor runs S items ahead of the use cursor
        fc.init(gw, ns);
        uc = fc;
        ring_stream(
            r, gw, GW, items,
            [&](int st, int64_t) {
                const int o0 = (int)fc.s * R, o1 = min(o0 + R, Ho);
                const int ylo = max(2 * o0 - 1, 0), yhi = min(2 * o1, H);
                const unsigned first_row = fc.p * (unsigned)H + (unsigned)ylo;
                const unsigned bytes = (unsigned)(yhi - ylo) * row_bytes;   // rows are 16-byte multiples
                r.expect(st, bytes);
                r.copy(st, 0, a.x + (uint64_t)first_row * W, bytes);
                fc.step(dq, dr, ns);
            },
            [&](const unsigned char *stage, int64_t) {
                const int o0 = (int)uc.s * R, o1 = min(o0 + R, Ho);
                const int ylo = max(2 * o0 - 1, 0), yhi = min(2 * o1, H);
                // rows 2*o0-1 .. 2*o0+2R-1 at clamped (in-stage) offsets,
                // lanes past W reading column 0; row 2*o0-1 is padding in
                // the first strip and rows at or past H (odd H) in the last
                const unsigned char *base = stage + (act ? 4 * c0 : 0);
                float2 h[NR];
#pragma unroll
                for (int k = 0; k < NR; ++k) {
                    const int y = min(max(2 * o0 - 1 + k, ylo), yhi - 1);
                    const float4 q = *reinterpret_cast<const float4 *>(base + (unsigned)(y - ylo) * row_bytes);
                    float L = __shfl_up_sync(0xffffffffu, q.w, 1);
                    if (lane == 0) L = ninf;
                    h[k] = make_float2(mx(mx(L, q.x), q.y), mx(mx(q.y, q.z), q.w));
                }
                if (o0 == 0) h[0] = make_float2(ninf, ninf);
#pragma unroll
                for (int k = 1; k < NR; ++k)
                    if (2 * o0 - 1 + k >= yhi) h[k] = make_float2(ninf, ninf);
                float *yp = a.y + ((int64_t)uc.p * Ho + o0) * Wo + (c0 >> 1);
#pragma unroll
                for (int j = 0; j < R; ++j)
                    if (act && o0 + j < o1)
                        stcs2(yp + j * Wo, make_float2(mx(mx(h[2 * j].x, h[2 * j + 1].x), h[2 * j + 2].x),
                                                       mx(mx(h[2 * j].y, h[2 * j + 1].y), h[2 * j + 2].y)));
                uc.step(dq, dr, ns);
            });
        r.finish();
        return true;
    }

    // One item of the flat path: its pixels are output pixels (W and H of f
    // those of the output), get(0) is column 0 of the window centre of the
    // item's first row, which is row oy0 of its plane.  The order of the
    // maxima is the strips'; where W or an alignment rules strips out a NaN
    // never wins (`clean`), as in one running maximum over the window.
    template <class Get>
    static __device__ __forceinline__ void flat_item(const Args &a, const FlatRows &f, unsigned oy0, unsigned n,
                                                     float *y0, const Get &get)
    {
        const int W = a.W;
        const unsigned H = (unsigned)a.H;
        const bool clean = (a.W & 3) != 0 || !aligned16(a.x) || !aligned16(a.y);
        const float ninf = -__int_as_float(0x7f800000);
#pragma unroll 2
        for (unsigned i = lane_id(); i < n; i += 32) {
            const unsigned lr = f.row_of(i), ox = i - lr * f.W, t = oy0 + lr;
            const unsigned p = f.plane_of(t), oy = t - p * f.H;
            // input row 2*oy of plane p, counted from input row 2*oy0 of the
            // item's first plane
            const int cen = (int)(p * H + 2 * oy - 2 * oy0) * W + 2 * (int)ox;
            const bool te = oy == 0, be = 2 * oy + 1 >= H, le = ox == 0, re = 2 * (int)ox + 1 >= W;
            auto row3 = [&](int c, bool out) {
                float l = get(c - 1, !out && !le);
                const float x = get(c, !out);
                const float r = get(c + 1, !out && !re);
                if (le) l = ninf;
                if (clean) l = mx(ninf, l);
                const float h = mx(l, x);
                return out ? ninf : re ? h : mx(h, r);
            };
            const float h0 = row3(cen - W, te), h1 = row3(cen, false), h2 = row3(cen + W, be);
            __stcs(y0 + i, mx(mx(h0, h1), h2));
        }
    }

    static __device__ bool flat_ring(const Args &a, const Ctx &cx)
    {
        const int H = a.H;
        const unsigned W = (unsigned)a.W, Ho = (unsigned)(H - 1) / 2 + 1, Wo = (W - 1) / 2 + 1;
        const int64_t rows = (int64_t)a.P * Ho, total = (int64_t)a.P * H * W;
        const int nw = cx.nthreads >> 5;
        const int64_t gw = (int64_t)cx.block * nw + (cx.tid >> 5), GW = (int64_t)cx.grid * nw;
        const unsigned slots = min(cx.ring_stage, 4096u) / 4;
        if (!aligned16(a.x) || 3 * W + kFlatPad > slots || !WarpRing::available(cx, 0)) return false;
        FlatRows f;
        // R output rows need at most 2R + 1 input rows
        const unsigned rmax = ((slots - kFlatPad) / W - 1) / 2;
        f.init(Wo, Ho, (unsigned)rows, min(rmax, FlatRows::kMaxValues / Wo), (unsigned)GW, 1);
        WarpRing r;
        r.init(cx, 0);
        FlatCursor fc, uc;   // the fill cursor runs the ring's stages ahead
        fc.init(f, gw, GW);
        uc = fc;
        // input values of the item's output rows, halo included: n rows from
        // row c.r of plane c.p
        auto copy = [&](const FlatCursor &c, unsigned n, int64_t &hi) {
            const unsigned t = c.r + n - 1, pl = f.plane_of(t), oy1 = t - pl * Ho;
            const int64_t lo = ((int64_t)c.p * H + 2 * (int64_t)c.r - 1) * W - 1;
            hi = ((int64_t)(c.p + pl) * H + 2 * (int64_t)oy1 + 2) * W + 1;
            return FlatCopy(lo, hi, total);
        };
        int64_t hi;
        ring_stream(
            r, gw, GW, f.items(),
            [&](int st, int64_t it) {
                const unsigned q0 = (unsigned)it * f.R;
                copy(fc, min(f.R, f.rows - q0), hi).fill(r, st, a.x);
                fc.step(Ho);
            },
            [&](unsigned char *stage, int64_t it) {
                const unsigned q0 = (unsigned)it * f.R, n = min(f.R, f.rows - q0);
                const FlatCopy k = copy(uc, n, hi);
                k.patch(stage, a.x, hi, total, r.lane);
                const int64_t first = ((int64_t)uc.p * H + 2 * (int64_t)uc.r) * W;
                flat_item(a, f, uc.r, n * Wo, a.y + (int64_t)q0 * Wo,
                          FlatStage{reinterpret_cast<const float *>(stage) + (first - k.base)});
                uc.step(Ho);
            });
        r.finish();
        return true;
    }

    // The same items without a ring.
    static __device__ void flat_global(const Args &a, const Ctx &cx)
    {
        const int H = a.H;
        const unsigned Ho = (unsigned)(H - 1) / 2 + 1, Wo = (unsigned)(a.W - 1) / 2 + 1;
        const int64_t rows = (int64_t)a.P * Ho, W = a.W;
        const int nw = cx.nthreads >> 5;
        const int64_t gw = (int64_t)cx.block * nw + (cx.tid >> 5), GW = (int64_t)cx.grid * nw;
        FlatRows f;
        f.init(Wo, Ho, (unsigned)rows, max(1u, FlatRows::kMaxValues / Wo), (unsigned)GW, 1);
        for (int64_t it = gw; it < f.items(); it += GW) {
            const unsigned q0 = (unsigned)it * f.R, q1 = min(q0 + f.R, f.rows);
            const unsigned p0 = q0 / Ho, oy0 = q0 - p0 * Ho;
            flat_item(a, f, oy0, (q1 - q0) * Wo, a.y + (int64_t)q0 * Wo,
                      FlatGlobal{a.x + ((int64_t)p0 * H + 2 * (int64_t)oy0) * W});
        }
    }

    // One thread per output: few outputs, few long rows, and tensors of 2^31
    // rows or more.
    static __device__ void run_scalar(const Args &a, const Ctx &cx)
    {
        const int H = a.H, W = a.W, Ho = (H - 1) / 2 + 1, Wo = (W - 1) / 2 + 1;
        const int64_t total = (int64_t)a.P * Ho * Wo;
        const float ninf = -__int_as_float(0x7f800000);
        for (int64_t i = (int64_t)cx.block * cx.nthreads + cx.tid; i < total;
             i += (int64_t)cx.grid * cx.nthreads) {
            const int ox = (int)(i % Wo);
            const int oy = (int)((i / Wo) % Ho);
            const int64_t p = i / ((int64_t)Wo * Ho);
            const float *xp = a.x + p * H * W;
            float m = ninf;
            for (int ky = 0; ky < 3; ++ky) {
                const int iy = 2 * oy - 1 + ky;
                if (iy < 0 || iy >= H) continue;
                for (int kx = 0; kx < 3; ++kx) {
                    const int ix = 2 * ox - 1 + kx;
                    if (ix < 0 || ix >= W) continue;
                    m = mx(m, __ldg(xp + (int64_t)iy * W + ix));
                }
            }
            a.y[i] = m;
        }
    }

    // SMALL: with the rule on small tensors (a kernel launched alone is chosen
    // by it before the launch).
    template <bool SMALL, int>
    static __device__ __forceinline__ void run_as(const Args &a, const Ctx &cx)
    {
        if ((int64_t)a.P * a.H * a.W == 0) return;
        // not flat: also past 2^31 rows, where 16-byte rows keep the strips'
        // order of maxima, so that a NaN counts alike whatever the size
        const bool flat =
            flat_range((int64_t)a.P * a.H, a.W, cx) && !(SMALL && small(a, (int64_t)cx.grid * cx.nthreads));
        if (strips(a) || (!flat && rows16(a))) {
            if (a.W <= 128 && a.H >= 2 && WarpRing::available(cx, 0) && run_ring(a, cx)) return;
            run_vec(a, cx);
            return;
        }
        if (flat && flat_ring(a, cx)) return;
        // 16-byte rows are flat here, and stay so for the order of maxima
        if (flat && (rows16(a) || enough_rows((int64_t)a.P * ((a.H - 1) / 2 + 1), cx, 2))) flat_global(a, cx);
        else run_scalar(a, cx);
    }
};

// The body without the flat path, as BodyUpsamplePlain.
struct BodyMaxpoolPlain {
    using Of = BodyMaxpool;
    using Args = Of::Args;
    static constexpr int kId = Of::kId;
    static __host__ bool pick(const Args &a, int, int64_t threads) { return Of::strips(a) || Of::small(a, threads); }
    static __host__ bool uses_ring(const Args &a)
    {
        return (int64_t)a.P * a.H * a.W > 0 && Of::rows16(a) && a.W <= 128 && a.H >= 2;
    }
    static __device__ void run(const Args &a, const Ctx &cx)
    {
        if ((int64_t)a.P * a.H * a.W == 0) return;
        if (Of::rows16(a)) {
            if (a.W <= 128 && a.H >= 2 && WarpRing::available(cx, 0) && Of::run_ring(a, cx)) return;
            Of::run_vec(a, cx);
        } else {
            Of::run_scalar(a, cx);
        }
    }
};

// ------------------------------------------------------------------------
// im2col, 3x3 window, stride 1, padding 1: the flat path where three rows fit
// a ring's stage (or strips, below).  Without a ring, the vector path (W % 4
// == 0, W <= 64): a warp takes a chunk of rows of one (n, c) plane, each half-warp
// half of the chunk; lane holds 4 columns of three consecutive input rows
// and writes the nine shifted copies (ky, kx) of its columns for each row.
struct BodyIm2col {
    using Args = hf_im2col3_args;
    static constexpr int kId = HF_BODY_IM2COL3;
    static constexpr int kBarriers = 0;
    // ring path: a stage holds at least three rows (the flat path).  Strips
    // of whole 16-byte rows, a half-warp a row, take fewer instructions, which
    // narrow intervals are bound by: 2^22 values with one warp an SM, W = 48 / 56
    // / 60 / 64, 54 / 41 / 43 / 38 us, flat 51 / 46 / 49 / 50; two warps 29 / 23 /
    // 26 / 22 and 26 / 26 / 27 / 27; level from three on, and 1.2 to 4.7 times
    // slower at W = 40 .. 16.  So they take rows of kStripCols columns or more in
    // intervals of up to kStripThreads.  Beside the flat path they cost kernels
    // capped at 64 registers 100 bytes of spills and 5 to 11 % (histogram +
    // im2col; the 8-way launch on eight narrow intervals 552 us, 512 without),
    // so those are compiled without; and pairs have them in kernels of their own
    // for blocks with a narrow interval (batch-norm + im2col 64x64, 224 + 32
    // threads, 14.8 -> 13.1 us), which leaves the other blocks' code alone.
    static constexpr int kRingRows = 14;   // rows of a strip item
    static constexpr int kStripCols = 56, kStripThreads = 64;
    // Up to as many outputs per thread the flat path's start (a dozen
    // divisions and the ring) costs more than a thread per output: 60 rows of
    // 75 columns, 1 a thread, 3.3 us, flat 5.2; 600 of 30, 4 a thread, 4.1 and
    // 3.6; 300 of 112, 8 a thread, 5.6 and 3.9.
    static constexpr int kFewOutputs = 3;
    static __host__ __device__ bool rows16(const Args &a)
    {
        return (a.W & 3) == 0 && a.W <= 64 && aligned16(a.x) && aligned16(a.col);
    }
    static __host__ __device__ bool strips(const Args &a, int threads)   // of the interval
    {
        return threads <= kStripThreads && rows16(a) && a.W >= kStripCols;
    }
    static __host__ __device__ bool small(const Args &a, int64_t threads)   // of the grid
    {
        return !rows16(a) && 9 * (int64_t)a.N * a.C * a.H * a.W <= kFewOutputs * threads;
    }
    static constexpr bool kRingItem = true;
    static constexpr unsigned kRingMinBytes = 4096;   // the stage: one item
    static __host__ bool uses_ring(const Args &a)
    {
        return (int64_t)a.N * a.C * a.H * a.W > 0 && aligned16(a.x) && 3u * a.W + kFlatPad <= kRingMinBytes / 4;
    }
    static __host__ bool needs_ring(const Args &a) { return !rows16(a); }   // as in BodyUpsample
    static __host__ double ring_work(const Args &a) { return 40.0 * a.N * a.C * a.H * a.W; }

    static __host__ size_t workspace_bytes(const Args &) { return 0; }
    static __host__ size_t smem_bytes(int, const Args &) { return 0; }
    static __host__ hf_status validate(const Args &a)
    {
        if (a.N < 0 || a.C < 0 || a.H < 0 || a.W < 0) return HF_ERR_INVALID;
        if ((int64_t)a.N * a.C * a.H * a.W == 0) return HF_OK;
        if (!a.x || !a.col) return HF_ERR_INVALID;
        if ((int64_t)a.N * a.C * a.H * a.W * 9 >= (int64_t)1 << 40) return HF_ERR_INVALID;
        return HF_OK;
    }

    struct Row {
        float4 q;
        float L, R;   // columns c0-1 and c0+4 (0 outside the image)
    };

    static __device__ __forceinline__ float4 load(const float *xp, int iy, int H, int W, int c0,
                                                  bool act)
    {
        const bool ok = act && iy >= 0 && iy < H;
        return ok ? ldg4(xp + (int64_t)iy * W + c0) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    static __device__ __forceinline__ Row halo(float4 q, int c0, int W)
    {
        Row r;
        r.q = q;
        const int sub = lane_id() & 15;
        r.L = __shfl_up_sync(0xffffffffu, q.w, 1);
        r.R = __shfl_down_sync(0xffffffffu, q.x, 1);
        if (sub == 0) r.L = 0.f;
        if (c0 + 4 >= W) r.R = 0.f;
        return r;
    }

    // The three kx-shifted copies of one input row (rows ky*3 + 0..2).
    static __device__ __forceinline__ void emit(const Row &r, float *base, int64_t HW)
    {
        stcs4(base, make_float4(r.L, r.q.x, r.q.y, r.q.z));
        stcs4(base + HW, r.q);
        stcs4(base + 2 * HW, make_float4(r.q.y, r.q.z, r.q.w, r.R));
    }

    // Work items are (plane, chunk of rows); each half-warp takes half of a
    // chunk.  A plane is cut into as many chunks as give the interval's
    // warps about three items each (whole planes when there are enough of
    // them): with one item per plane, 2048 planes kept only 2048 of a
    // GB300's 9728 warp slots busy.  Every chunk re-reads its two halo rows
    // (from L2 in practice).
    static __device__ void run_vec(const Args &a, const Ctx &cx)
    {
        const int H = a.H, W = a.W;
        const int64_t HW = (int64_t)H * W;
        const int64_t planes = (int64_t)a.N * a.C;
        const int nw = cx.nthreads >> 5;
        const int64_t nwt = (int64_t)cx.grid * nw;
        const int lane = lane_id();
        const int half = lane >> 4;
        const int c0 = 4 * (lane & 15);
        const bool act = c0 < W;
        const int want = (int)min((3 * nwt + planes - 1) / planes, (int64_t)(H + 1) / 2);
        const int hh = ((H + max(want, 1) - 1) / max(want, 1) + 1) / 2;   // rows per half-warp
        const int nchunk = (H + 2 * hh - 1) / (2 * hh);
        const int64_t items = planes * nchunk;
        for (int64_t it = (int64_t)cx.block * nw + (cx.tid >> 5); it < items; it += nwt) {
            const int64_t pl = it / nchunk;
            const int ch = (int)(it - pl * nchunk);
            const int64_t n = pl / a.C;
            const int c = (int)(pl - n * a.C);
            const float *xp = a.x + pl * HW;
            float *cp = a.col + (n * a.C * 9 + (int64_t)c * 9) * HW;
            const int oyb = ch * 2 * hh + half * hh;
            const int oye = min(oyb + hh, H);
            Row up = halo(load(xp, oyb - 1, H, W, c0, act), c0, W);
            Row mid = halo(load(xp, oyb, H, W, c0, act), c0, W);
            float4 nq = load(xp, oyb + 1, H, W, c0, act);
#pragma unroll 2
            for (int i = 0; i < hh; ++i) {
                const int oy = oyb + i;
                const bool valid = act && oy < oye;
                float4 fq = load(xp, oy + 2, H, W, c0, act && oy + 1 < oye);
                Row dn = halo(nq, c0, W);
                if (valid) {
                    float *base = cp + (int64_t)oy * W + c0;
                    emit(up, base, HW);
                    emit(mid, base + 3 * HW, HW);
                    emit(dn, base + 6 * HW, HW);
                }
                up = mid;
                mid = dn;
                nq = fq;
            }
        }
    }

    // Ring path.  Work item = (plane, chunk of R = 14 rows); the chunk and
    // its halo rows, [max(r0-1, 0), min(r0+R+1, H)), are contiguous and
    // arrive in one bulk copy in a stage of the warp's ring.  As in the
    // register path each half-warp takes half of the chunk and lane l of a
    // half the columns 4l..4l+3, sliding three rows (from shared memory,
    // zero outside the image) and writing the nine shifted copies per row.
    static __device__ bool run_ring(const Args &a, const Ctx &cx)
    {
        constexpr int R = kRingRows, RH = R / 2;
        const int H = a.H, W = a.W;
        const int64_t HW = (int64_t)H * W;
        const unsigned row_bytes = 4u * (unsigned)W;
        const int64_t planes = (int64_t)a.N * a.C;
        if (cx.ring_stage < (R + 2) * row_bytes || planes * H >= ((int64_t)1 << 32)) return false;
        const unsigned ns = (unsigned)((H + R - 1) / R);
        const int64_t items = planes * ns;
        WarpRing r;
        r.init(cx, 0);
        const int nw = cx.nthreads >> 5;
        const int64_t gw = (int64_t)cx.block * nw + (cx.tid >> 5), GW = (int64_t)cx.grid * nw;
        const unsigned dq = (unsigned)(GW / ns), dr = (unsigned)(GW % ns);
        const int lane = lane_id();
        const int half = lane >> 4;
        const int c0 = 4 * (lane & 15);
        const bool act = c0 < W;
        const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
        ItemCursor fc, uc;   // the fill cursor runs S items ahead of the use cursor
        fc.init(gw, ns);
        uc = fc;
        ring_stream(
            r, gw, GW, items,
            [&](int st, int64_t) {
                const int r0 = (int)fc.s * R;
                const int ylo = max(r0 - 1, 0), yhi = min(r0 + R + 1, H);
                const unsigned bytes = (unsigned)(yhi - ylo) * row_bytes;   // rows are 16-byte multiples
                r.expect(st, bytes);
                r.copy(st, 0, a.x + ((uint64_t)fc.p * (unsigned)H + (unsigned)ylo) * W, bytes);
                fc.step(dq, dr, ns);
            },
            [&](const unsigned char *stage, int64_t) {
                const int r0 = (int)uc.s * R;
                const int ylo = max(r0 - 1, 0), yhi = min(r0 + R + 1, H);
                const unsigned char *base = stage + (act ? 4 * c0 : 0);
                auto ld = [&](int y) {
                    const int yc = min(max(y, ylo), yhi - 1);   // an in-stage row
                    const float4 q = *reinterpret_cast<const float4 *>(base + (unsigned)(yc - ylo) * row_bytes);
                    return (act && y >= 0 && y < H) ? q : zero;
                };
                const unsigned n = uc.p / (unsigned)a.C, c = uc.p - n * (unsigned)a.C;
                float *cp = a.col + ((int64_t)n * a.C * 9 + (int64_t)c * 9) * HW;
                const int oyb = r0 + half * RH, oye = min(oyb + RH, H);
                Row up = halo(ld(oyb - 1), c0, W);
                Row mid = halo(ld(oyb), c0, W);
#pragma unroll
                for (int i = 0; i < RH; ++i) {
                    const int oy = oyb + i;
                    Row dn = halo(ld(oy + 1), c0, W);
                    if (act && oy < oye) {
                        float *o = cp + (int64_t)oy * W + c0;
                        emit(up, o, HW);
                        emit(mid, o + 3 * HW, HW);
                        emit(dn, o + 6 * HW, HW);
                    }
                    up = mid;
                    mid = dn;
                }
                uc.step(dq, dr, ns);
            });
        r.finish();
        return true;
    }

    // One item of the flat path, VEC consecutive pixels per lane.  Shifted
    // copy k of pixel i lies at k*HW + i of its plane's output, so a warp's
    // stores are contiguous for any W; VEC == 4 (planes of 16-byte
    // multiples, items that start on one) makes them 128-bit and reads
    // three times six values for four pixels -- in one 128-bit and two
    // 32-bit loads where the rows are 16-byte multiples too.
    template <int VEC, class Get>
    static __device__ __forceinline__ void flat_item(const Args &a, const FlatRows &f, unsigned g0, unsigned n,
                                                     const Get &get)
    {
        const int W = (int)f.W;
        const int64_t HW = (int64_t)f.H * W;
        const unsigned p0 = g0 / f.H, r0 = g0 - p0 * f.H;
        // output of the item's first pixel, copy 0, if its plane went on
        float *o0 = a.col + ((int64_t)p0 * 9 * HW + (int64_t)r0 * W);
        if constexpr (VEC == 4)
            if ((W & 3) == 0) {   // the four pixels are of one row
                for (unsigned i = 4 * lane_id(); i < n; i += 128) {
                    const unsigned lr = f.row_of(i), t = r0 + lr, p = f.plane_of(t);
                    const unsigned c = i - lr * f.W, r = t - p * f.H;
                    const bool le = c == 0, re = c + 4 == f.W;
                    float *o = o0 + ((int64_t)p * 8 * HW + i);
#pragma unroll
                    for (int ky = 0; ky < 3; ++ky) {
                        const float *q = get.p + ((int)i + (ky - 1) * W);
                        float4 m = *reinterpret_cast<const float4 *>(q);
                        float L = q[-1], R = q[4];
                        if ((ky == 0 && r == 0) || (ky == 2 && r == f.H - 1)) m = make_float4(0.f, 0.f, 0.f, 0.f), L = R = 0.f;
                        if (le) L = 0.f;
                        if (re) R = 0.f;
                        emit(Row{m, L, R}, o + 3 * ky * HW, HW);
                    }
                }
                return;
            }
        for (unsigned i = VEC * lane_id(); i < n; i += 32 * VEC) {
            const unsigned lr = f.row_of(i), t = r0 + lr;
            const unsigned p = f.plane_of(t);
            unsigned c = i - lr * f.W, r = t - p * f.H;
            bool le[VEC], re[VEC], te[VEC], be[VEC];
#pragma unroll
            for (int v = 0; v < VEC; ++v) {
                le[v] = c == 0;
                re[v] = c == f.W - 1;
                te[v] = r == 0;
                be[v] = r == f.H - 1;
                if (++c == f.W) c = 0, ++r;   // planes end on multiples of VEC
            }
            float *o = o0 + ((int64_t)p * 8 * HW + i);
            // not unrolled: unrolled it took eight registers more in the
            // fused kernels, which cost them blocks of 640 threads
#pragma unroll 1
            for (int ky = 0; ky < 3; ++ky) {
                const int off = (int)i + (ky - 1) * W;
                float q[VEC + 2], w[3][VEC];
#pragma unroll
                for (int v = 0; v < VEC + 2; ++v) {
                    // the value at off + v - 1 is read by pixel v - 1 + {1, 0, -1}
                    // (for global loads: by one that is inside)
                    bool ok = false;
#pragma unroll
                    for (int kx = 0; kx < 3; ++kx) {
                        const int px = v - kx;
                        if (px < 0 || px >= VEC) continue;
                        const bool out = (ky == 0 && te[px]) || (ky == 2 && be[px]) || (kx == 0 && le[px]) ||
                                         (kx == 2 && re[px]);
                        ok = ok || !out;
                    }
                    q[v] = get(off + v - 1, ok);
                }
#pragma unroll
                for (int v = 0; v < VEC; ++v) {
                    const bool out = (ky == 0 && te[v]) || (ky == 2 && be[v]);
                    w[0][v] = out || le[v] ? 0.f : q[v];
                    w[1][v] = out ? 0.f : q[v + 1];
                    w[2][v] = out || re[v] ? 0.f : q[v + 2];
                }
#pragma unroll
                for (int kx = 0; kx < 3; ++kx) {
                    float *d = o + (3 * ky + kx) * HW;
                    if (VEC == 4) stcs4(d, make_float4(w[kx][0], w[kx][1 % VEC], w[kx][2 % VEC], w[kx][3 % VEC]));
                    else __stcs(d, w[kx][0]);
                }
            }
        }
    }

    template <int VEC>
    static __device__ __forceinline__ bool flat_ring(const Args &a, const Ctx &cx)
    {
        const int64_t rows = (int64_t)a.N * a.C * a.H, total = rows * a.W;
        const int nw = cx.nthreads >> 5;
        const int64_t gw = (int64_t)cx.block * nw + (cx.tid >> 5), GW = (int64_t)cx.grid * nw;
        const unsigned W = (unsigned)a.W, slots = min(cx.ring_stage, 4096u) / 4;
        // items of whole 16-byte multiples
        const unsigned mult = VEC == 1 || (W & 3) == 0 ? 1u : (W & 1) ? 4u : 2u;
        if (!aligned16(a.x) || (mult + 2) * W + kFlatPad > slots || !WarpRing::available(cx, 0)) return false;
        unsigned rmax = min((slots - kFlatPad) / W - 2, FlatRows::kMaxValues / W);
        rmax -= rmax % mult;
        FlatRows f;
        f.init(W, a.H, (unsigned)rows, rmax, (unsigned)GW, mult);
        WarpRing r;
        r.init(cx, 0);
        auto copy = [&](int64_t it) {
            const int64_t g0 = it * f.R;
            return FlatCopy((g0 - 1) * W - 1, (min(g0 + (int64_t)f.R, rows) + 1) * W + 1, total);
        };
        ring_stream(
            r, gw, GW, f.items(), [&](int st, int64_t it) { copy(it).fill(r, st, a.x); },
            [&](unsigned char *stage, int64_t it) {
                const int64_t g0 = it * f.R, g1 = min(g0 + (int64_t)f.R, rows);
                const FlatCopy k = copy(it);
                k.patch(stage, a.x, (g1 + 1) * W + 1, total, r.lane);
                flat_item<VEC>(a, f, (unsigned)g0, (unsigned)(g1 - g0) * W,
                               FlatStage{reinterpret_cast<const float *>(stage) + (g0 * W - k.base)});
            });
        r.finish();
        return true;
    }

    // The same items, one pixel per lane, without a ring.
    static __device__ void flat_global(const Args &a, const Ctx &cx)
    {
        const int64_t rows = (int64_t)a.N * a.C * a.H;
        const int nw = cx.nthreads >> 5;
        const int64_t gw = (int64_t)cx.block * nw + (cx.tid >> 5), GW = (int64_t)cx.grid * nw;
        const unsigned W = (unsigned)a.W;
        FlatRows f;
        f.init(W, a.H, (unsigned)rows, max(1u, FlatRows::kMaxValues / W), (unsigned)GW, 1);
        for (int64_t it = gw; it < f.items(); it += GW) {
            const int64_t g0 = it * f.R, g1 = min(g0 + (int64_t)f.R, rows);
            flat_item<1>(a, f, (unsigned)g0, (unsigned)(g1 - g0) * W, FlatGlobal{a.x + g0 * W});
        }
    }

    // One thread per output: few outputs, few long rows, and tensors of 2^31
    // rows or more.
    static __device__ void run_scalar(const Args &a, const Ctx &cx)
    {
        const int H = a.H, W = a.W;
        const int64_t HW = (int64_t)H * W;
        const int64_t total = (int64_t)a.N * a.C * 9 * HW;
        for (int64_t i = (int64_t)cx.block * cx.nthreads + cx.tid; i < total;
             i += (int64_t)cx.grid * cx.nthreads) {
            const int64_t pix = i % HW;
            const int64_t row = i / HW;            // n*C*9 + c*9 + ky*3 + kx
            const int k = (int)(row % 9);
            const int64_t plane = row / 9;         // n*C + c
            const int oy = (int)(pix / W), ox = (int)(pix % W);
            const int iy = oy + k / 3 - 1, ix = ox + k % 3 - 1;
            float v = 0.f;
            if (iy >= 0 && iy < H && ix >= 0 && ix < W) v = __ldg(a.x + plane * HW + (int64_t)iy * W + ix);
            a.col[i] = v;
        }
    }

    // SMALL: with the rule on small tensors; NARROW: with strips in intervals of
    // up to so many threads (a kernel launched alone is chosen by both before
    // the launch; N-way kernels keep them to one warp: with two the 8-way
    // launch on eight narrow intervals took 534 us, 528 with one).
    template <bool SMALL, int NARROW>
    static __device__ __forceinline__ void run_as(const Args &a, const Ctx &cx)
    {
        if ((int64_t)a.N * a.C * a.H * a.W == 0) return;
        const bool flat = flat_range((int64_t)a.N * a.C * a.H, a.W, cx) &&
                          !(SMALL && small(a, (int64_t)cx.grid * cx.nthreads));
        if (NARROW && cx.nthreads <= NARROW && strips(a, cx.nthreads) && WarpRing::available(cx, 0) &&
            run_ring(a, cx))
            return;
        if (flat) {
            const bool v4 = a.W >= 4 && ((int64_t)a.H * a.W & 3) == 0 && aligned16(a.col);
            if (v4 && flat_ring<4>(a, cx)) return;
            if (flat_ring<1>(a, cx)) return;
        }
        if (rows16(a)) run_vec(a, cx);
        else if (flat && enough_rows((int64_t)a.N * a.C * a.H, cx, 8)) flat_global(a, cx);
        else run_scalar(a, cx);
    }
};

// The body without the flat path, as BodyUpsamplePlain.
struct BodyIm2colPlain {
    using Of = BodyIm2col;
    using Args = Of::Args;
    static constexpr int kId = Of::kId;
    static __host__ bool pick(const Args &a, int block, int64_t threads)
    {
        return Of::strips(a, block) || Of::small(a, threads);
    }
    static __host__ bool uses_ring(const Args &a) { return (int64_t)a.N * a.C * a.H * a.W > 0 && Of::rows16(a); }
    static __device__ void run(const Args &a, const Ctx &cx)
    {
        if ((int64_t)a.N * a.C * a.H * a.W == 0) return;
        if (Of::rows16(a)) {
            if (WarpRing::available(cx, 0) && Of::run_ring(a, cx)) return;
            Of::run_vec(a, cx);
        } else {
            Of::run_scalar(a, cx);
        }
    }
};

} // namespace hf
