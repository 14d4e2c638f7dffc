// One frame in one launch: the whole segmentation of a frame whose features
// fit in the chip's shared memory.
//
// A cooperative launch of one CTA per SM. Every CTA owns a run of work units
// (a unit is a rectangle of at most 16 x 16 pixels inside one grid cell, so
// all its pixels share their nine candidate centres), converts their pixels
// once and keeps the features in shared memory for every pass. A pass is:
// centres of the CTA's cell window from the previous pass's member sums (the
// centre update, done redundantly by the CTAs that need a centre, so it takes
// no launch and no barrier of its own), Eq. (1) for every pixel, member sums
// into global memory, grid barrier. The last pass writes labels; with the
// local connectivity rule one more barrier separates them from its two
// passes. The launch replaces 2 * iterations + 4 launches whose gaps, feature
// traffic and partly filled last waves took most of a single frame's time:
// 320x240, 10 iterations, 119 -> 47 us; 1920x1080, 5 iterations, 193 -> 107 us.
// A small frame is bound by the latency of a pass, 3.5 us at 320x240: centres
// 1.2, evaluation 0.9, barrier 1.4 (clock stamps). A large one is bound by
// instruction issue (46 % of the cycles) and by the drain of its sums before the
// barrier: 13.8 us per pass at 1920x1080, S = 16, of which centres 1.3,
// evaluation 9.4, barrier 3.1.
//
// Results are those of the launch-per-stage path, bit for bit: the same
// operations on the same values, and exact integer sums.
#include "slic_device.cuh"

#include <algorithm>
#include <type_traits>

namespace slicgb {

__device__ float g_lut_frame[256];  // sRGB byte -> linear (this file's copy)

namespace {

constexpr int kFrThreads = 512;
constexpr int kFrWarps = kFrThreads / 32;
// A warp's bins: word q (3 colours, packed x / y / count) of candidate t in
// copy c at q * 40 + t * 4 + c. Lanes use copy lane % 4: neighbouring lanes
// mostly pick the same candidate, and with one copy an atomic instruction
// took 8 passes over shared memory (ncu), a quarter of the launch.
constexpr int kFrBinWords = 160;
constexpr int kFrMaxSmem = 227 * 1024;

// A unit's first pixel and extent (wl x hl pixels, clipped to its cell and the
// image), its cell k and the window records of its nine candidates (their
// index times 3, a record being 3 x 16 bytes).
struct __align__(16) FrUnit {
    int k, x0, y0;
    short wl, hl;
    unsigned short rec[9], pad[7];
};

__device__ __forceinline__ int ld_acquire(const int *p) {
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// NP: pixel pairs per lane of a unit (up to 32 * NP pairs); XS: 8 pairs per
// unit row, so a lane's pairs share their columns.
template <int NP, bool XS>
__global__ void __launch_bounds__(kFrThreads, 1) k_frame(const __grid_constant__ ResidentFrame a) {
    extern __shared__ __align__(16) unsigned char fr_smem[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int G = gridDim.x, c = blockIdx.x;
    const int W = a.W, H = a.H, S = a.S, ns_c = a.ns_c, K = a.K, upc = a.ncx * a.ncy;
    const int u0 = (int)((long long)a.units * c / G), u1 = (int)((long long)a.units * (c + 1) / G), nu = u1 - u0;
    // Cells of this CTA's units: k0 .. k1; it owns (clears, reports) the
    // cells whose first unit it has: ko0 .. ko1 - 1. Its window: three runs
    // of `win` cells, from k0 - 1 less, at and plus one grid row, then a
    // sentinel record for candidates off the grid.
    const int k0 = u0 / upc, nk = nu > 0 ? (u1 - 1) / upc - k0 + 1 : 0;
    const int ko0 = (u0 + upc - 1) / upc, ko1 = (u1 + upc - 1) / upc;
    const int win = a.win, sent = 3 * win;
    float4 *const f_la = reinterpret_cast<float4 *>(fr_smem);  // [unit][NP][32] (l0, l1, a0, a1) of a pair
    float2 *const f_b = reinterpret_cast<float2 *>(f_la + (size_t)a.max_units * NP * 32);
    float *const ctab = reinterpret_cast<float *>(f_b + (size_t)a.max_units * NP * 32);
    FrUnit *const units = reinterpret_cast<FrUnit *>(ctab + (size_t)(sent + 1) * kCtabRec);
    unsigned *const bins = reinterpret_cast<unsigned *>(units + a.max_units) + warp * kFrBinWords;
    float *const lut = reinterpret_cast<float *>(bins - warp * kFrBinWords + kFrWarps * kFrBinWords);

    // Grid barrier in two halves: every CTA arrives once per barrier; the
    // counter is zero at launch (launch_resident clears it).
    int barriers = 0;
    auto arrive = [&]() {
        __syncthreads();
        if (tid == kFrThreads - 32) {  // (the other warps go on meanwhile)
            __threadfence();
            atomicAdd(a.ctrl, 1);
        }
        ++barriers;
    };
    auto wait = [&]() -> bool {
        bool ok = true;
        if (tid == 0) {
            const int target = barriers * G;
            unsigned n = 0;
            while (ld_acquire(a.ctrl) < target && ++n < a.polls) {
            }
            ok = n < a.polls;
            if (!ok) atomicOr(a.err, 4);
        }
        return __syncthreads_and(ok ? 1 : 0) != 0;
    };

    // Sums of passes 0 and 1 cleared (three sets rotate: one filled, one
    // read, one cleared), the stopping test's state reset.
    const size_t set_words = (size_t)K * 6;
    for (int i = tid; i < (ko1 - ko0) * 6; i += kFrThreads) {
        a.acc[(size_t)ko0 * 6 + i] = 0;
        a.acc[set_words + (size_t)ko0 * 6 + i] = 0;
    }
    if (c == 0 && tid == 0) {
        for (int i = 0; i < 3 * kResidLanes; ++i) (&a.cstate->resid[0][0])[i] = 0;
        a.cstate->done = 0;
        a.cstate->iters = 0;
    }
    arrive();

    for (int i = tid; i < 256; i += kFrThreads) lut[i] = g_lut_frame[i];
    for (int i = lane; i < kFrBinWords; i += 32) bins[i] = 0u;
    // The units.
    for (int ul = tid; ul < nu; ul += kFrThreads) {
        const int u = u0 + ul, k = u / upc, sub = u - k * upc, sy = sub / a.ncx, sx = sub - sy * a.ncx;
        const int cy = k / ns_c, cx = k - cy * ns_c;
        FrUnit n;
        n.k = k;
        n.x0 = cx * S + sx * a.cw;
        n.y0 = cy * S + sy * a.uh;
        n.wl = (short)max(0, min(min(a.cw, (cx + 1) * S - n.x0), W - n.x0));
        n.hl = (short)max(0, min(min(a.uh, (cy + 1) * S - n.y0), H - n.y0));
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            const int dy = t / 3 - 1, dx = t % 3 - 1;
            const bool in = cy + dy >= 0 && cy + dy < a.ns_r && cx + dx >= 0 && cx + dx < ns_c;
            n.rec[t] = (unsigned short)(3 * (in ? (dy + 1) * win + k - k0 + 1 + dx : sent));
        }
        units[ul] = n;
    }
    __syncthreads();
    // Initial centres of the window.
    for (int e = tid; e <= sent; e += kFrThreads) {
        const int seg = e / win, j = e - seg * win, k = k0 + (seg - 1) * ns_c - 1 + j;
        float rec[6] = {kSentinel, kSentinel, kSentinel, kSentinel, kSentinel, 0.0f};
        if (e < sent && j < nk + 2 && k >= 0 && k < K) {
            if (a.init) {
#pragma unroll
                for (int i = 0; i < 6; ++i) {
                    const float v = a.init[(size_t)k * 6 + i];
                    rec[i] = i < 5 ? near_centre(v) : v;
                }
            } else {
                int px, py;
                init_centre_position(k, W, H, S, ns_c, rec[3], rec[4], px, py);
                float fv[3];
                bool moved = false;
                auto fetch = [&](int x, int y, float (&o)[3]) {
                    const uint8_t *q = a.rgb + ((size_t)y * W + x) * a.C;
                    convert_pixel(a.conv, q[0], q[1], q[2], lut, o[0], o[1], o[2]);
                };
                if (a.perturb) {
                    int bx, by;
                    moved = perturb_seed(fetch, W, H, px, py, bx, by, fv);
                    if (moved) {
                        rec[3] = (float)bx;
                        rec[4] = (float)by;
                    }
                } else {
                    fetch(px, py, fv);
                }
                rec[0] = fv[0];
                rec[1] = fv[1];
                rec[2] = fv[2];
            }
        }
        write_ctab(ctab + (size_t)e * kCtabRec, rec);
    }

    // This lane's pairs within a unit.
    int prow[NP], pcol[NP];
#pragma unroll
    for (int i = 0; i < NP; ++i) {
        if (XS) {
            prow[i] = (lane >> 3) + 4 * i;
            pcol[i] = 2 * (lane & 7);
        } else {
            const int p = lane + 32 * i;
            prow[i] = p / a.ppr;
            pcol[i] = 2 * (p - prow[i] * a.ppr);
        }
    }
    // Features of the CTA's units, once (pixels outside a unit: black).
    for (int ul = warp; ul < nu; ul += kFrWarps) {
        const FrUnit &n = units[ul];
        unsigned px[NP][2];  // (r, g, b) bytes of the pairs; all loads first
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const bool in0 = prow[i] < n.hl && pcol[i] < n.wl, in1 = in0 && pcol[i] + 1 < n.wl;
            const uint8_t *q = a.rgb + ((size_t)(n.y0 + prow[i]) * W + n.x0 + pcol[i]) * a.C;
            px[i][0] = px[i][1] = 0u;
            if (a.C == 4 && ((uintptr_t)a.rgb & 3) == 0) {
                if (in0) px[i][0] = __ldg(reinterpret_cast<const unsigned *>(q));
                if (in1) px[i][1] = __ldg(reinterpret_cast<const unsigned *>(q) + 1);
            } else if (a.C == 3 && in1 && ((uintptr_t)q & 1) == 0) {
                const unsigned short *h = reinterpret_cast<const unsigned short *>(q);
                const unsigned h0 = __ldg(h), h1 = __ldg(h + 1), h2 = __ldg(h + 2);
                px[i][0] = h0 | (h1 << 16);
                px[i][1] = (h1 >> 8) | (h2 << 8);
            } else {
                if (in0) px[i][0] = __ldg(q) | ((unsigned)__ldg(q + 1) << 8) | ((unsigned)__ldg(q + 2) << 16);
                if (in1)
                    px[i][1] = __ldg(q + a.C) | ((unsigned)__ldg(q + a.C + 1) << 8) |
                               ((unsigned)__ldg(q + a.C + 2) << 16);
            }
        }
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            float f[2][3];
#pragma unroll
            for (int j = 0; j < 2; ++j)
                convert_pixel(a.conv, px[i][j] & 255u, (px[i][j] >> 8) & 255u, (px[i][j] >> 16) & 255u, lut, f[j][0],
                              f[j][1], f[j][2]);
            f_la[((size_t)ul * NP + i) * 32 + lane] = make_float4(f[0][0], f[1][0], f[0][1], f[1][1]);
            f_b[((size_t)ul * NP + i) * 32 + lane] = make_float2(f[0][2], f[1][2]);
        }
    }

    bool ok = wait();  // (also: the window's centres are complete)
    const float fs = a.fix_scale, fix_inv = 1.0f / a.fix_scale;
    const unsigned long long ww = pack2(a.w, a.w);

    for (int pass = 0; ok && pass <= a.iterations; ++pass) {
        if (pass > 0) {
            // Update `pass` from the sums of pass - 1, after the stopping
            // test (see conv_stop): a stopped frame goes to its last pass.
            if (a.eps > 0.0f && pass >= 2) {
                long long e = 0;
#pragma unroll
                for (int i = 0; i < kResidLanes; ++i) e += __ldcg(&a.cstate->resid[(pass - 1) % 3][i]);
                if ((double)e < (double)a.eps * (double)kResidScale * (double)K) {
                    if (c == 0 && tid == 0) a.cstate->done = 1;
                    pass = a.iterations;
                    goto evaluate;
                }
            }
            const long long *src = a.acc + (size_t)((pass - 1) % 3) * set_words;
            long long *clr = a.acc + (size_t)((pass + 1) % 3) * set_words;
            for (int e0 = 0; e0 < sent; e0 += kFrThreads) {  // (the same trip count on every lane)
                const int e = e0 + tid, seg = e / win, j = e - seg * win, k = k0 + (seg - 1) * ns_c - 1 + j;
                float move = 0.0f;
                if (e < sent && j < nk + 2 && k >= 0 && k < K) {
                    const longlong2 *s = reinterpret_cast<const longlong2 *>(src + (size_t)k * 6);
                    const longlong2 s01 = __ldcg(s), s23 = __ldcg(s + 1), s45 = __ldcg(s + 2);
                    float *rec = ctab + (size_t)e * kCtabRec;
                    const bool own = seg == 1 && k >= ko0 && k < ko1;
                    if (s45.y > 0) {  // as update_centre
                        const float fn = (float)s45.y;
                        float n[6];
                        n[0] = __fdiv_rn((float)s01.x * fix_inv, fn);
                        n[1] = __fdiv_rn((float)s01.y * fix_inv, fn);
                        n[2] = __fdiv_rn((float)s23.x * fix_inv, fn);
                        n[3] = __fdiv_rn((float)s23.y, fn);
                        n[4] = __fdiv_rn((float)s45.x, fn);
                        n[5] = fn;
                        if (own) move = fabsf(n[3] - rec[6]) + fabsf(n[4] - rec[8]);
                        write_ctab(rec, n);
                    } else {
                        rec[10] = 0.0f;
                    }
                    if (own) {
                        longlong2 *z = reinterpret_cast<longlong2 *>(clr + (size_t)k * 6);
                        z[0] = make_longlong2(0, 0);
                        z[1] = make_longlong2(0, 0);
                        z[2] = make_longlong2(0, 0);
                    }
                }
                if (a.eps > 0.0f) {
                    long long v = (long long)__float2ll_rn(move * kResidScale);
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFull, v, o);
                    if (lane == 0 && v != 0)
                        atomicAdd(reinterpret_cast<unsigned long long *>(
                                      &a.cstate->resid[pass % 3][(c * kFrWarps + warp) % kResidLanes]),
                                  (unsigned long long)v);
                }
            }
            if (c == 0 && tid == 0) {
                if (a.eps > 0.0f)
                    for (int i = 0; i < kResidLanes; ++i) a.cstate->resid[(pass + 1) % 3][i] = 0;
                a.cstate->iters = pass;
            }
            __syncthreads();
        }
    evaluate:
        const bool last = pass == a.iterations;
        unsigned long long *const acc =
            reinterpret_cast<unsigned long long *>(a.acc) + (size_t)(pass % 3) * set_words;
        // M pairs per lane of unit ul, from pair i0 (all NP of them, or one half).
        auto evaluate_unit = [&](auto pairs, int ul, int i0) {
            constexpr int M = decltype(pairs)::value;
            const FrUnit n = units[ul];
            if (n.wl <= 0 || n.hl <= 0) return;  // (the warp's)
            int row[M], col[M];
#pragma unroll
            for (int i = 0; i < M; ++i) {
                if (M == NP) {
                    row[i] = prow[i];
                    col[i] = pcol[i];
                } else if (XS) {
                    row[i] = (lane >> 3) + 4 * (i0 + i);
                    col[i] = 2 * (lane & 7);
                } else {
                    const int p = lane + 32 * (i0 + i);
                    row[i] = p / a.ppr;
                    col[i] = 2 * (p - row[i] * a.ppr);
                }
            }
            const float4 *const u_la = f_la + ((size_t)ul * NP + i0) * 32 + lane;
            const float2 *const u_b = f_b + ((size_t)ul * NP + i0) * 32 + lane;
            unsigned long long l[M], aa[M], b[M], x[M];
            float fy[M];
#pragma unroll
            for (int i = 0; i < M; ++i) {
                const ulonglong2 la = *reinterpret_cast<const ulonglong2 *>(u_la + 32 * i);
                l[i] = la.x;
                aa[i] = la.y;
                b[i] = *reinterpret_cast<const unsigned long long *>(u_b + 32 * i);
                const float fx = (float)(n.x0 + col[i]);
                x[i] = pack2(fx, fx + 1.0f);
                fy[i] = (float)(n.y0 + row[i]);
            }
            // Eq. (1), candidates two at a time as in the pipelined kernel
            float bk[M][2];
#pragma unroll
            for (int i = 0; i < M; ++i) bk[i][0] = bk[i][1] = __int_as_float(0x7F800000);
#pragma unroll
            for (int t0 = 0; t0 < 9; t0 += 2) {
                const int nt = t0 < 8 ? 2 : 1;
                float kk[2][M][2];
#pragma unroll
                for (int q = 0; q < nt; ++q) {
                    const float *rp = ctab + 4 * n.rec[t0 + q];
                    const ulonglong2 la = *reinterpret_cast<const ulonglong2 *>(rp);
                    const ulonglong2 bx = *reinterpret_cast<const ulonglong2 *>(rp + 4);
                    const float yy = rp[8];
#pragma unroll
                    for (int i = 0; i < M; ++i) {
                        const float ddy = __fsub_rn(yy, fy[i]), ddy2 = __fmul_rn(ddy, ddy);
                        eval_keys(la, bx, pack2(ddy2, ddy2), ww, l[i], aa[i], b[i], XS ? x[0] : x[i], c_tags[t0 + q],
                                  kk[q][i][0], kk[q][i][1]);
                    }
                }
#pragma unroll
                for (int i = 0; i < M; ++i)
#pragma unroll
                    for (int j = 0; j < 2; ++j)
                        bk[i][j] = nt == 2 ? fmin3_nan(bk[i][j], kk[0][i][j], kk[1][i][j])
                                           : fmin_nan(bk[i][j], kk[0][i][j]);
            }
            int t[M][2];  // winning candidate, -1 outside the unit
#pragma unroll
            for (int i = 0; i < M; ++i)
#pragma unroll
                for (int j = 0; j < 2; ++j)
                    t[i][j] = row[i] < n.hl && col[i] + j < n.wl ? (int)(__float_as_uint(bk[i][j]) & 15u) : -1;
            if (last) {
                int32_t *const dst = a.connect ? a.lbl_tmp : a.labels;
#pragma unroll
                for (int i = 0; i < M; ++i) {
                    const size_t p = (size_t)(n.y0 + row[i]) * W + n.x0 + col[i];
                    int v[2];
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        const int q = (int)__umulhi((unsigned)t[i][j], 0x55555556u);  // t / 3
                        v[j] = n.k - ns_c - 1 + t[i][j] + q * (ns_c - 3);
                    }
                    if (t[i][1] >= 0 && ((p & 1) == 0) && a.labels_vec2) {
                        *reinterpret_cast<int2 *>(dst + p) = make_int2(v[0], v[1]);
                    } else {
                        if (t[i][0] >= 0) dst[p] = v[0];
                        if (t[i][1] >= 0) dst[p + 1] = v[1];
                    }
                }
            } else {
                // Member sums of the unit's nine candidates: pixels that stay
                // with their own cell (candidate 4, the most frequent by far)
                // add up in registers and then across the warp; the others go
                // to the warp's bins in shared memory. Colours are biased
                // words (fix_round2_biased); x and y count from the unit's
                // corner: 11 + 11 + 10 bits, enough for 256 pixels of a
                // 16 x 16 unit.
                unsigned o[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                for (int i = 0; i < M; ++i) {
                    unsigned v[2][4];
                    float f0, f1;
                    unpack2(l[i], f0, f1);
                    fix_round2_biased(f0, f1, fs, v[0][0], v[1][0]);
                    unpack2(aa[i], f0, f1);
                    fix_round2_biased(f0, f1, fs, v[0][1], v[1][1]);
                    unpack2(b[i], f0, f1);
                    fix_round2_biased(f0, f1, fs, v[0][2], v[1][2]);
                    v[0][3] = (unsigned)col[i] + ((unsigned)row[i] << 11) + (1u << 22);
                    v[1][3] = v[0][3] + 1u;
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        if (t[i][j] == 4) {
#pragma unroll
                            for (int q = 0; q < 4; ++q) o[q] += v[j][q];
                        } else if (t[i][j] >= 0) {
#pragma unroll
                            for (int q = 0; q < 4; ++q) atomicAdd(&bins[q * 40 + t[i][j] * 4 + (lane & 3)], v[j][q]);
                        }
                    }
                }
#pragma unroll
                for (int q = 0; q < 4; ++q) o[q] = __reduce_add_sync(kFull, o[q]);
                __syncwarp();
                // Lane 3 * t + part adds two of candidate t's six sums (one sum
                // per lane, whole records per instruction, was 8 % slower).
                if (lane < 27) {
                    const int q = lane / 3, part = lane - 3 * q;
                    auto word = [&](int w) {  // the four copies' sum (own: the warp's)
                        if (q == 4) return w == 0 ? o[0] : w == 1 ? o[1] : w == 2 ? o[2] : o[3];
                        const uint4 p = *reinterpret_cast<const uint4 *>(bins + w * 40 + q * 4);
                        return p.x + p.y + p.z + p.w;
                    };
                    const unsigned xyn = word(3), cnt = xyn >> 22;
                    if (cnt != 0) {
                        const unsigned bias = cnt * kFixBias;
                        long long v0, v1;
                        if (part == 0) {
                            v0 = (int)(word(0) - bias);
                            v1 = (int)(word(1) - bias);
                        } else if (part == 1) {
                            v0 = (int)(word(2) - bias);
                            v1 = (long long)(xyn & 0x7FFu) + (long long)cnt * n.x0;
                        } else {
                            v0 = (long long)((xyn >> 11) & 0x7FFu) + (long long)cnt * n.y0;
                            v1 = (long long)cnt;
                        }
                        unsigned long long *g = acc + (size_t)(n.k + (q / 3 - 1) * ns_c + q % 3 - 1) * 6 + 2 * part;
                        atomicAdd(g, (unsigned long long)v0);
                        atomicAdd(g + 1, (unsigned long long)v1);
                    }
                }
                __syncwarp();
                reinterpret_cast<uint4 *>(bins)[lane] = make_uint4(0u, 0u, 0u, 0u);
                if (lane < 8) reinterpret_cast<uint4 *>(bins)[32 + lane] = make_uint4(0u, 0u, 0u, 0u);
                __syncwarp();
            }
        };
        // Each warp takes an equal run of the units; where NP is even, of
        // half units: with 54 units (1920x1080, S = 16) on 16 warps whole
        // ones would leave ten warps idle for the fourth round.
        if (NP % 2 == 0) {
            constexpr int kHalf = NP % 2 == 0 ? NP / 2 : 1;
            int h = 2 * nu * warp / kFrWarps;
            const int h1 = 2 * nu * (warp + 1) / kFrWarps;
            if ((h & 1) && h < h1) {
                evaluate_unit(std::integral_constant<int, kHalf>(), h >> 1, kHalf);
                ++h;
            }
            for (; h + 1 < h1; h += 2) evaluate_unit(std::integral_constant<int, NP>(), h >> 1, 0);
            if (h < h1) evaluate_unit(std::integral_constant<int, kHalf>(), h >> 1, 0);
        } else {
            for (int ul = warp; ul < nu; ul += kFrWarps) evaluate_unit(std::integral_constant<int, NP>(), ul, 0);
        }
        if (!last) {
            arrive();
            ok = wait();
        }
    }
    if (ok) {
        // The centres the labels were assigned against.
        for (int i = tid; i < (ko1 - ko0) * 6; i += kFrThreads) {
            const int k = ko0 + i / 6, q = i % 6;
            float v = ctab[(size_t)(win + k - k0 + 1) * kCtabRec + 2 * q];
            if (fabsf(v) == kFarCentre && a.init) v = a.init[(size_t)k * 6 + q];  // (held there: as it was given)
            a.centres[(size_t)k * 6 + q] = v;
        }
        if (a.connect) {
            arrive();
            ok = wait();
            const int strips = (W + kConnOut - 1) / kConnOut, segs = (H + a.conn_rows - 1) / a.conn_rows;
            for (int u = warp * G + c; ok && u < strips * segs; u += G * kFrWarps) {
                const int seg = u / strips, sx = (u - seg * strips) * kConnOut, ry0 = seg * a.conn_rows;
                if (a.conn_rows == 1)
                    conn_block<1>(a.lbl_tmp, a.labels, W, H, sx, ry0, a.labels_vec != 0, lane);
                else if (a.conn_rows == 2)
                    conn_block<2>(a.lbl_tmp, a.labels, W, H, sx, ry0, a.labels_vec != 0, lane);
                else
                    conn_strip<false>(a.lbl_tmp, a.labels, W, H, sx, ry0, min(ry0 + a.conn_rows, H), a.labels_vec != 0,
                                      lane);
            }
        }
    }
}

template <int NP, bool XS>
cudaError_t launch_as(const ResidentFrame &a, int grid, size_t smem, cudaStream_t s) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(kFrThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_frame<NP, XS>, a);
}

template <int NP, bool XS>
cudaError_t configure_as() {
    return cudaFuncSetAttribute(k_frame<NP, XS>, cudaFuncAttributeMaxDynamicSharedMemorySize, kFrMaxSmem);
}

}  // namespace

cudaError_t upload_lut_frame(const float *lut256) {
    cudaError_t e = cudaMemcpyToSymbol(g_lut_frame, lut256, 256 * sizeof(float));
    if (e == cudaSuccess) e = configure_as<1, true>();
    if (e == cudaSuccess) e = configure_as<2, true>();
    if (e == cudaSuccess) e = configure_as<4, true>();
    if (e == cudaSuccess) e = configure_as<1, false>();
    if (e == cudaSuccess) e = configure_as<2, false>();
    if (e == cudaSuccess) e = configure_as<3, false>();
    if (e == cudaSuccess) e = configure_as<4, false>();
    return e;
}

// The split of a frame into units: a cell is cut into ncx x ncy rectangles
// of at most cw x uh pixels, cw and uh at most 16, NP pixel pairs per lane.
bool plan_resident(int W, int H, int S, int ns_c, int ns_r, int sms, size_t sums_bytes, ResidentPlan *plan) {
    plan->grid = 0;
    const long long K = (long long)ns_c * ns_r;
    // Below 7 x 7 pixels per cell fewer than half of a unit's lanes have work.
    // At S = 7 one launch still wins: 320x240, 10 iterations, 50 us against 124
    // with a launch per stage, 1280x720 152 against 236. So it does up to the
    // largest frames that fit: 1920x1200, S = 16, 203 against 358 us.
    if (S < 7 || sms < 1 || (size_t)K * 6 * sizeof(long long) * 3 > sums_bytes) return false;
    double best = 0.0;
    for (int np = 1; np <= 4; ++np) {
        ResidentPlan p{};
        p.ncx = (S + 15) / 16;
        p.cw = (S + p.ncx - 1) / p.ncx;
        p.ppr = (p.cw + 1) / 2;
        const int rows = std::min(std::min(32 * np / p.ppr, 16), S);
        p.ncy = (S + rows - 1) / rows;
        p.uh = (S + p.ncy - 1) / p.ncy;
        p.np = np;
        p.xs = p.ppr == 8 ? 1 : 0;
        if (np == 3 && p.xs) continue;  // 12 rows of 8 pairs: not built
        const long long upc = (long long)p.ncx * p.ncy, units = K * upc;
        if (units >= (1LL << 30)) continue;
        p.units = (int)units;
        p.grid = (int)std::min<long long>(sms, units);
        p.max_units = (int)((units + p.grid - 1) / p.grid);
        p.win = (upc == 1 ? p.max_units : (p.max_units - 1) / (int)upc + 2) + 2;
        p.smem = (size_t)p.max_units * (np * 32 * 24 + sizeof(FrUnit)) + (size_t)(3 * p.win + 1) * kCtabRec * 4 +
                 kFrWarps * kFrBinWords * 4 + 256 * 4;
        if (p.smem > (size_t)kFrMaxSmem || 3 * (3 * p.win) > 65535) continue;
        // Rounds of units per warp, each with its own fixed part (window
        // records, warp reductions, flush): about 0.6 of a pair's work.
        // Even np: half units (see k_frame), at half a pair's work more.
        const int halves = (2 * p.max_units + kFrWarps - 1) / kFrWarps, rounds = (p.max_units + kFrWarps - 1) / kFrWarps;
        const double cost = np % 2 ? rounds * (np + 0.6) : 0.5 * halves * np + 0.6 * (rounds + (halves & 1) * 0.5);
        if (plan->grid == 0 || cost < best) {
            best = cost;
            *plan = p;
        }
    }
    if (plan->grid == 0) return false;
    // Connectivity: one or two rows per warp while the chip has a warp for
    // each (a warp's latency is what counts: 320x240 takes 1.5 us this way,
    // 6.5 us with segments of 4 rows), else segments streamed row by row.
    const long long strips = (W + kConnOut - 1) / kConnOut, warps = (long long)plan->grid * kFrWarps;
    const long long rows = (strips * H + warps - 1) / warps;
    plan->conn_rows = rows <= 2 ? (int)rows : (int)std::max<long long>(4, std::min<long long>(kConnSeg, rows));
    return true;
}

cudaError_t launch_resident(ResidentFrame a, const ResidentPlan &p, cudaStream_t s) {
    a.units = p.units;
    a.max_units = p.max_units;
    a.win = p.win;
    a.cw = p.cw;
    a.uh = p.uh;
    a.ncx = p.ncx;
    a.ncy = p.ncy;
    a.ppr = p.ppr;
    a.conn_rows = p.conn_rows;
    // The barrier counter starts every launch at zero, whatever a launch that
    // was overlapped or that gave up has left in it (320x240, 10 iterations:
    // 47.7 us with the clear, 47.1 with a counter that the launch's last CTA
    // cleared).
    const cudaError_t e = cudaMemsetAsync(a.ctrl, 0, sizeof(int), s);
    if (e != cudaSuccess) return e;
    if (p.xs) {
        if (p.np == 1) return launch_as<1, true>(a, p.grid, p.smem, s);
        if (p.np == 2) return launch_as<2, true>(a, p.grid, p.smem, s);
        return launch_as<4, true>(a, p.grid, p.smem, s);
    }
    if (p.np == 1) return launch_as<1, false>(a, p.grid, p.smem, s);
    if (p.np == 2) return launch_as<2, false>(a, p.grid, p.smem, s);
    if (p.np == 3) return launch_as<3, false>(a, p.grid, p.smem, s);
    return launch_as<4, false>(a, p.grid, p.smem, s);
}

}  // namespace slicgb
