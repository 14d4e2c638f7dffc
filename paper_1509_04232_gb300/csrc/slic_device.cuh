// Device functions shared by the segmentation kernels: the padded centre
// record, Eq. (1) on paired FP32 instructions, the fixed-point rounding of the
// member sums, the seed positions and the connectivity rule. Every kernel that
// evaluates one of these uses the same operations in the same order, which is
// what makes single-frame and batched results bit-identical.
#pragma once

#include "slic_internal.cuh"

#include <cstdint>

namespace slicgb {
namespace {

constexpr unsigned kFull = 0xFFFFFFFFu;

// Cells off the grid have a sentinel centre, kSentinel in every coordinate, so
// that the candidate loops need no bounds checks. It has to lose to every centre
// of the grid: a pixel that chose it would count in a cell that does not exist.
// A centre that the caller gives may be anything, NaN included, so its record
// holds it within +-kFarCentre (NaN: -kFarCentre), and the weight of the spatial
// distance is at most kMaxWeight: every D is then finite, and the sentinels'
// ten times any other. (Outputs keep the values that the caller gave.)
constexpr float kSentinel = 1e18f, kFarCentre = 1e17f;
__device__ __forceinline__ float near_centre(float v) { return fminf(fmaxf(v, -kFarCentre), kFarCentre); }

// One record of the padded centre table: each field twice (see kCtabRec).
__device__ __forceinline__ void write_ctab(float *t, const float *c) {
    float4 *t4 = reinterpret_cast<float4 *>(t);
    t4[0] = make_float4(c[0], c[0], c[1], c[1]);
    t4[1] = make_float4(c[2], c[2], c[3], c[3]);
    t4[2] = make_float4(c[4], c[4], c[5], 0.0f);
}
// The record of a centre that may be the caller's.
__device__ __forceinline__ void write_ctab_near(float *t, const float *c) {
    float n[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) n[i] = i < 5 ? near_centre(c[i]) : c[i];
    write_ctab(t, n);
}

// Candidate tags 0..8 (scan position in the 3x3 window) for the keys
// (D & ~15) | t, read from the constant bank: the key is then one logical
// operation whose other constant, the mask, is its immediate. With the tag
// as a literal too, the pipelined pass executed 7 more instructions per
// pixel (ncu instruction counts; same results).
__constant__ unsigned c_tags[9] = {0, 1, 2, 3, 4, 5, 6, 7, 8};

__device__ __forceinline__ float fsqrt_approx(float x) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ void init_centre_position(int k, int W, int H, int S, int ns_c, float &xk, float &yk,
                                                     int &px, int &py) {
    const int c = k % ns_c, r = k / ns_c;
    const int x_first = c * S, x_last = min((c + 1) * S, W) - 1;
    const int y_first = r * S, y_last = min((r + 1) * S, H) - 1;
    // (first + last) / 2 is exact in float for any image below 2^23 pixels wide.
    xk = 0.5f * (float)(x_first + x_last);
    yk = 0.5f * (float)(y_first + y_last);
    px = (x_first + x_last) >> 1;  // floor of the midpoint
    py = (y_first + y_last) >> 1;
}

// Seed perturbation (Sec. 2, the original SLIC's first step): the pixel of
// lowest gradient G = |I(x+1,y) - I(x-1,y)|^2 + |I(x,y+1) - I(x,y-1)|^2
// (features, neighbours clamped into the image) among the 3x3 pixels around
// the seed pixel (px, py). The seed pixel is the first candidate; a later
// one (dy outer, dx inner, in-image only) wins only with a strictly lower G.
// fetch(x, y, f) gives the features of an in-image pixel. Returns whether the
// seed moved, with the chosen pixel and its features.
template <typename Fetch>
__device__ __forceinline__ bool perturb_seed(const Fetch &fetch, int W, int H, int px, int py, int &bx, int &by,
                                             float (&fb)[3]) {
    float f[5][5][3];  // features of the 5x5 block around (px, py), clamped; corners unused
#pragma unroll
    for (int j = 0; j < 5; ++j) {
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            if ((i == 0 || i == 4) && (j == 0 || j == 4)) continue;
            fetch(min(max(px - 2 + i, 0), W - 1), min(max(py - 2 + j, 0), H - 1), f[j][i]);
        }
    }
    auto grad = [&](int i, int j) {
        float g = 0.0f;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float gx = f[j][i + 1][c] - f[j][i - 1][c], gy = f[j + 1][i][c] - f[j - 1][i][c];
            g += gx * gx + gy * gy;
        }
        return g;
    };
    float best = grad(2, 2);
    int bi = 2, bj = 2;
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy) {
#pragma unroll
        for (int dx = -1; dx <= 1; ++dx) {
            if ((dx == 0 && dy == 0) || px + dx < 0 || px + dx >= W || py + dy < 0 || py + dy >= H) continue;
            const float g = grad(2 + dx, 2 + dy);
            if (g < best) {
                best = g;
                bi = 2 + dx;
                bj = 2 + dy;
            }
        }
    }
    bx = px + bi - 2;
    by = py + bj - 2;
#pragma unroll
    for (int c = 0; c < 3; ++c) fb[c] = f[bj][bi][c];
    return bi != 2 || bj != 2;
}

// Paired FP32 arithmetic: a 64-bit operand holds two floats (low, high);
// each element is rounded exactly as the scalar instruction would be.
__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ unsigned long long sub2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// min of two non-negative floats (a NaN operand loses), IEEE (no flush).
__device__ __forceinline__ float fmin_nan(float a, float b) {
    float r;
    asm("min.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}
// The same over three operands (one instruction on sm_100 and later).
__device__ __forceinline__ float fmin3_nan(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// round(x * fs) (nearest, ties to even) for two values with one paired
// fused multiply-add on the FMA pipe, as a biased word: with M = 1.5 * 2^23,
// x * fs + M lies in [2^23, 2^24) where the float spacing is 1, so the one
// rounding of the fused multiply-add is the rounding to an integer, and the
// float's bits are that integer + kFixBias (the bits of M). Exact for
// |x * fs| < 2^22 (features below 128 at the 2^15 colour scale, 8-bit values
// at scale 1), and equal to __float2int_rn(x * fs) + kFixBias there since fs
// is a power of two. Sums of such words taken mod 2^32, minus count *
// kFixBias, are the sums of the rounded values, exactly, whenever those fit
// in 31 bits: at most 2^22 per value, and at most 256 values (a 16x16 block or
// unit, a pair of a tile's private copies) go into one word, 2^30 in all.
constexpr unsigned kFixBias = 0x4B400000u;
__device__ __forceinline__ void fix_round2_biased(float x0, float x1, float fs, unsigned &r0, unsigned &r1) {
    const unsigned long long m = fma2(pack2(x0, x1), pack2(fs, fs), pack2(12582912.0f, 12582912.0f));
    float m0, m1;
    unpack2(m, m0, m1);
    r0 = __float_as_uint(m0);
    r1 = __float_as_uint(m1);
}

// Eq. (1) for two pixels (colour pairs l, a, b; column pair x) against one
// centre record: d_lab = sqrt(dl^2 + da^2 + db^2), d_xy = sqrt(dx^2 + dy^2),
// D = (m/S) d_xy + d_lab, as the two pixels' keys (D & ~15) | t.
__device__ __forceinline__ void eval_keys(const ulonglong2 &la, const ulonglong2 &bx, unsigned long long ddy2,
                                          unsigned long long ww, unsigned long long l, unsigned long long a,
                                          unsigned long long b, unsigned long long x, unsigned t, float &k0,
                                          float &k1) {
    const unsigned long long dl = sub2(la.x, l), da = sub2(la.y, a), db = sub2(bx.x, b);
    const unsigned long long s = fma2(dl, dl, fma2(da, da, mul2(db, db)));
    const unsigned long long dx = sub2(bx.y, x);
    const unsigned long long q = fma2(dx, dx, ddy2);
    float s0, s1, q0, q1;
    unpack2(s, s0, s1);
    unpack2(q, q0, q1);
    const unsigned long long D = fma2(ww, pack2(fsqrt_approx(q0), fsqrt_approx(q1)),
                                      pack2(fsqrt_approx(s0), fsqrt_approx(s1)));
    float d0, d1;
    unpack2(D, d0, d1);
    k0 = __uint_as_float((__float_as_uint(d0) & ~15u) | t);
    k1 = __uint_as_float((__float_as_uint(d1) & ~15u) | t);
}

// Geometry of the fused connectivity kernels (see conn_strip).
constexpr int kConnOut = 120;   // output columns per strip
constexpr int kConnSeg = 32;    // output rows per segment (64: 8 x 1080p keep 45 % of the chip's
                                // warps busy, 59 us against 52; 2 frames 47 against 27 us)

__device__ __forceinline__ int32_t conn_col_sentinel(int x, int W, int32_t v) {
    return x < 0 ? -1 : (x >= W ? -3 : v);
}

// NC: the labels were written by an earlier launch (read-only loads); else by
// other CTAs of this launch (L2 loads).
template <bool NC, typename T>
__device__ __forceinline__ T conn_ld(const T *p) {
    return NC ? __ldg(p) : __ldcg(p);
}

template <bool NC>
__device__ __forceinline__ int4 conn_load_row(const int32_t *in, int W, int H, int y, int x0, bool vec) {
    if (y < 0) return make_int4(-2, -2, -2, -2);
    if (y >= H) return make_int4(-4, -4, -4, -4);
    const int32_t *row = in + (size_t)y * W;
    if (vec && x0 >= 0 && x0 + 3 < W) return conn_ld<NC>(reinterpret_cast<const int4 *>(row + x0));
    int4 v;
    v.x = (x0 >= 0 && x0 < W) ? conn_ld<NC>(row + x0) : conn_col_sentinel(x0, W, 0);
    v.y = (x0 + 1 >= 0 && x0 + 1 < W) ? conn_ld<NC>(row + x0 + 1) : conn_col_sentinel(x0 + 1, W, 0);
    v.z = (x0 + 2 >= 0 && x0 + 2 < W) ? conn_ld<NC>(row + x0 + 2) : conn_col_sentinel(x0 + 2, W, 0);
    v.w = (x0 + 3 >= 0 && x0 + 3 < W) ? conn_ld<NC>(row + x0 + 3) : conn_col_sentinel(x0 + 3, W, 0);
    return v;
}

// Sentinels back into a first-pass row (its values outside the image are
// meaningless): the whole row when y is outside, else the lane's columns
// outside (edge lanes only).
__device__ __forceinline__ int4 conn_mask_row(int4 v, int W, int H, int y, int x0, bool edge_lane) {
    if (y < 0) return make_int4(-2, -2, -2, -2);
    if (y >= H) return make_int4(-4, -4, -4, -4);
    if (edge_lane) {
        v.x = conn_col_sentinel(x0, W, v.x);
        v.y = conn_col_sentinel(x0 + 1, W, v.y);
        v.z = conn_col_sentinel(x0 + 2, W, v.z);
        v.w = conn_col_sentinel(x0 + 3, W, v.w);
    }
    return v;
}

// The rule for a pixel none of whose neighbours (left, up, right, down;
// sentinels for missing ones) carries its label: the neighbours' majority,
// the first in that order among the largest counts. With at most four
// values, the left one wins whenever it matches another; else the upper one
// when it matches the right or lower one; else the right one when it matches
// the lower one; else all are distinct and the first valid one wins. No
// valid neighbour at all keeps the label.
__device__ __forceinline__ int32_t conn_majority(int32_t own, int32_t l, int32_t u, int32_t r, int32_t d) {
    const bool el = l == u || l == r || l == d, eu = u == r || u == d, er = r == d;
    const int32_t fv = l >= 0 ? l : (u >= 0 ? u : (r >= 0 ? r : d));
    const int32_t res = el ? l : (eu ? u : (er ? r : fv));
    return res >= 0 ? res : own;
}
// The same where all four neighbours are labels (no sentinel): the first
// valid one is the left one, and the result is always a label.
__device__ __forceinline__ int32_t conn_majority_inner(int32_t l, int32_t u, int32_t r, int32_t d) {
    const bool el = l == u || l == r || l == d, eu = u == r || u == d, er = r == d;
    return el ? l : (eu ? u : (er ? r : l));
}

// Where two rows (or their neighbours) differ: zero where equal.
__device__ __forceinline__ int4 conn_diff(const int4 &a, const int4 &b) {
    return make_int4(a.x ^ b.x, a.y ^ b.y, a.z ^ b.z, a.w ^ b.w);
}

// One pass of the majority rule at row y for the lane's 4 pixels, from the
// rows above, at and below y (left/right neighbours across lanes) and the
// differences of the row to the one above (vu) and to the one below (vd). A
// pixel keeps its label when a neighbour shares it (the common case), that is
// when the smallest of its four differences is zero; the majority is evaluated
// only when some pixel of the warp needs it. A difference serves both of its
// pixels, across rows too: 2.25 per pixel where four comparisons per pixel made
// the kernel issue-bound (57.5 instructions per pixel). INNER: every neighbour
// the warp's results depend on is inside the image.
template <bool INNER>
__device__ __forceinline__ int4 conn_rule4(const int4 &up, const int4 &c, const int4 &dn, const int4 &vu,
                                           const int4 &vd) {
    const int32_t left = __shfl_up_sync(0xffffffffu, c.w, 1), right = __shfl_down_sync(0xffffffffu, c.x, 1);
    const unsigned h0 = left ^ c.x, h1 = c.x ^ c.y, h2 = c.y ^ c.z, h3 = c.z ^ c.w, h4 = c.w ^ right;
    const unsigned m0 = min(__vimin3_u32(h0, h1, vu.x), (unsigned)vd.x),
                   m1 = min(__vimin3_u32(h1, h2, vu.y), (unsigned)vd.y),
                   m2 = min(__vimin3_u32(h2, h3, vu.z), (unsigned)vd.z),
                   m3 = min(__vimin3_u32(h3, h4, vu.w), (unsigned)vd.w);
    int4 r = c;
    if (__any_sync(0xffffffffu, (m0 | m1 | m2 | m3) != 0u)) {
        auto rule = [](int32_t own, int32_t l, int32_t u, int32_t rt, int32_t d) {
            return INNER ? conn_majority_inner(l, u, rt, d) : conn_majority(own, l, u, rt, d);
        };
        if (m0) r.x = rule(c.x, left, up.x, c.y, dn.x);
        if (m1) r.y = rule(c.y, c.x, up.y, c.z, dn.y);
        if (m2) r.z = rule(c.z, c.y, up.z, c.w, dn.z);
        if (m3) r.w = rule(c.w, c.z, up.w, right, dn.w);
    }
    return r;
}

// Both connectivity passes fused, streaming down vertical strips. A warp
// holds 128 columns [sx - 4, sx + 124) of one strip (lane l: columns
// sx - 4 + 4l .. +3) and walks down a segment of rows with a rolling window
// of input rows and first-pass rows in registers (horizontal neighbours by
// shuffles): input row q + 2 gives the first pass at row q + 1, which gives
// the second pass at row q. Lanes 1..30 write columns [sx, sx + 120); the
// two outer lanes only supply neighbours. Every pixel sees exactly the
// inputs of the two separate passes, so the result equals theirs.
//
// Positions outside the image hold negative sentinels, one per side (left
// -1, above -2, right -3, below -4): a sentinel never equals a label or
// another side's sentinel, which is all the rule needs to skip missing
// neighbours.
template <bool NC>
__device__ __forceinline__ void conn_strip(const int32_t *in, int32_t *labels, int W, int H, int sx, int ry0, int ry1,
                                           bool labels_vec, int lane) {
    const int x0 = sx - 4 + 4 * lane;
    const bool vec = (W & 3) == 0;
    const bool edge_lane = x0 < 0 || x0 + 3 >= W;
    // Input rows q .. q + 2 (q + 3 in flight) and first-pass rows q - 1, q.
    int4 a_m2 = conn_load_row<NC>(in, W, H, ry0 - 2, x0, vec), a_m1 = conn_load_row<NC>(in, W, H, ry0 - 1, x0, vec);
    int4 a0 = conn_load_row<NC>(in, W, H, ry0, x0, vec), a1 = conn_load_row<NC>(in, W, H, ry0 + 1, x0, vec);
    int4 a2 = conn_load_row<NC>(in, W, H, ry0 + 2, x0, vec);
    const int4 va = conn_diff(a_m1, a0);
    int4 v01 = conn_diff(a0, a1);  // of input rows q and q + 1
    int4 l_m1 = conn_mask_row(conn_rule4<false>(a_m2, a_m1, a0, conn_diff(a_m2, a_m1), va), W, H, ry0 - 1, x0,
                              edge_lane);
    int4 l0 = conn_mask_row(conn_rule4<false>(a_m1, a0, a1, va, v01), W, H, ry0, x0, edge_lane);
    int4 w0 = conn_diff(l_m1, l0);  // of first-pass rows q - 1 and q
    // Columns sx - 4 .. sx + 123 all inside the image: no lane holds a
    // sentinel column, so rows 1 .. H - 3 take the rule without them.
    const bool inner_cols = sx >= 4 && sx + 124 <= W;
    const bool writer = lane >= 1 && lane <= 30;
    const bool out_vec = vec && labels_vec && x0 >= 0 && x0 + 3 < W;
    for (int q = ry0; q < ry1; ++q) {
        const int4 a3 = conn_load_row<NC>(in, W, H, q + 3, x0, vec);  // one row ahead of its use
        const int4 v12 = conn_diff(a1, a2);
        int4 l1, w1, o;
        if (inner_cols && q >= 1 && q + 2 < H) {
            // input rows q .. q + 2 and first-pass rows q - 1 .. q + 1
            // are all inside the image
            l1 = conn_rule4<true>(a0, a1, a2, v01, v12);
            w1 = conn_diff(l0, l1);
            o = conn_rule4<true>(l_m1, l0, l1, w0, w1);
        } else {
            l1 = conn_mask_row(conn_rule4<false>(a0, a1, a2, v01, v12), W, H, q + 1, x0, edge_lane);
            w1 = conn_diff(l0, l1);
            o = conn_rule4<false>(l_m1, l0, l1, w0, w1);
        }
        v01 = v12;
        w0 = w1;
        if (writer) {
            int32_t *out = labels + (size_t)q * W;
            if (out_vec) {
                *reinterpret_cast<int4 *>(out + x0) = o;
            } else {
                const int32_t ov[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (x0 + j >= 0 && x0 + j < W) out[x0 + j] = ov[j];
            }
        }
        l_m1 = l0;
        l0 = l1;
        a0 = a1;
        a1 = a2;
        a2 = a3;
    }
}

// The same for R rows, ry0 .. ry0 + R - 1 (labels of this launch), with every
// input row loaded before the first is used: conn_strip waits one L2 latency
// per row.
template <int R>
__device__ __forceinline__ void conn_block(const int32_t *in, int32_t *labels, int W, int H, int sx, int ry0,
                                           bool labels_vec, int lane) {
    const int x0 = sx - 4 + 4 * lane;
    const bool vec = (W & 3) == 0, edge_lane = x0 < 0 || x0 + 3 >= W;
    int4 a[R + 4], l[R + 2];
#pragma unroll
    for (int j = 0; j < R + 4; ++j) a[j] = conn_load_row<false>(in, W, H, ry0 - 2 + j, x0, vec);
    const bool inner = sx >= 4 && sx + 124 <= W && ry0 >= 2 && ry0 + R + 2 <= H;  // no sentinel anywhere
#pragma unroll
    for (int j = 0; j < R + 2; ++j)
        l[j] = inner ? conn_rule4<true>(a[j], a[j + 1], a[j + 2], conn_diff(a[j], a[j + 1]), conn_diff(a[j + 1], a[j + 2]))
                     : conn_mask_row(conn_rule4<false>(a[j], a[j + 1], a[j + 2], conn_diff(a[j], a[j + 1]),
                                                       conn_diff(a[j + 1], a[j + 2])),
                                     W, H, ry0 - 1 + j, x0, edge_lane);
    const bool writer = lane >= 1 && lane <= 30;
    const bool out_vec = vec && labels_vec && x0 >= 0 && x0 + 3 < W;
#pragma unroll
    for (int j = 0; j < R; ++j) {
        const int4 wu = conn_diff(l[j], l[j + 1]), wd = conn_diff(l[j + 1], l[j + 2]);
        const int4 o = inner ? conn_rule4<true>(l[j], l[j + 1], l[j + 2], wu, wd)
                             : conn_rule4<false>(l[j], l[j + 1], l[j + 2], wu, wd);
        if (writer && ry0 + j < H) {
            int32_t *out = labels + (size_t)(ry0 + j) * W;
            if (out_vec) {
                *reinterpret_cast<int4 *>(out + x0) = o;
            } else {
                const int32_t ov[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (x0 + q >= 0 && x0 + q < W) out[x0 + q] = ov[q];
            }
        }
    }
}

}  // namespace
}  // namespace slicgb
