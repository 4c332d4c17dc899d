// raster.cu -- tile rasterizers (one thread block per tile of 256 pixels:
// 16x16, 32x8 or 8x32).
//
// Front-to-back alpha blending of Sec. III-D, Eq. (7): for each pixel, over
// the tile's depth-sorted Gaussians, alpha = min(0.99, o exp(p)) (Eqs. (10)-(12)),
// pairs with alpha < 1/255 are skipped, the loop stops (without adding) once
// the transmittance would fall below 1e-4, C += c alpha T, out = C + T bg.
//
// RoofGS mode (Sec. IV-B): the tile's [start, end) comes with the entries of a frame of
// runs (runs.cu); with sorted entries the block finds it in the sorted keys (warp-cooperative
// search). While a batch of records is staged in shared memory, each Gaussian's coefficients are folded (Eqs.
// (13)-(15)) -- -1/2 and log o absorbed, C1..C6 -- in TILE-LOCAL coordinates
// (pixel and mean shifted by the tile origin, so the FP32 terms stay small at
// 4K); every thread owns PPT vertically adjacent pixels (x, y) ... (x,
// y+PPT-1), two by default (the paper's dual-pixel scheme), one or four on
// request: the first exponent is the FMA chain of Eq. (16) on hoisted x^2, xy,
// y^2, x, y, each next one follows from Eq. (20) (two additions per extra
// row). Pairs with P < -ln 255 are skipped before any exponential (Eq. (23));
// alpha = min(0.99, exp^(P)) with the bit-level exponential of Eq. (24)
// (Eq. (25)). With 2 or 4 pixels per thread the timed kernel blends the thread's
// pixels in pairs with packed FP32x2 FMAs (the same roundings as one at a time). A
// warp whose pixels are all finished skips the batch (vote); the block leaves once
// every pixel is finished.
#include "rg_internal.cuh"

namespace rg {

// Eq. (24) evaluated in FP32: I = floor(P 2^23 log2 e + 2^23 (127 - sigma)).
// With w = fma(P, log2 e, 127 - sigma) in [64, 128) (P in [-ln 255, 0]),
// 2^23 * w is exactly the FP32 result of fma(P, 2^23 log2 e, 2^23 (127 - sigma))
// (scaling by 2^23 commutes with rounding) and is an integer multiple of 64, so
// I = 2^23 w = 2^29 + 64 * mantissa(w) = (bits(w) << 6) + 2^31 (mod 2^32):
// one FFMA and one integer shift-add instead of a float->int conversion.
__device__ __forceinline__ float fast_exp(float P)
{
    const float w = fmaf(P, 1.44269502f, 126.954323f);
    return __uint_as_float((__float_as_uint(w) << 6) + 0x80000000u);
}

__global__ void k_fast_exp_eval(const float* P, float* out, long long n)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = fast_exp(P[i]);
}

template <bool FAST, bool COUNT>
__device__ __forceinline__ void blend(float P, float r, float g, float b, float& T, float& c0, float& c1, float& c2,
                                      bool& done, unsigned& n_eval, unsigned& n_blend)
{
    if (COUNT && !done) {
        n_eval++;
        if (P >= -LN255F) n_blend++;
    }
    if (!done && P >= -LN255F) {
        const float e = FAST ? fast_exp(P) : expf(P);
        const float alpha = fminf(0.99f, e);
        const float Tn = fmaf(-T, alpha, T); // T (1 - alpha)
        if (Tn < 1e-4f) {
            done = true;
        } else {
            const float wgt = alpha * T;
            c0 = fmaf(r, wgt, c0);
            c1 = fmaf(g, wgt, c1);
            c2 = fmaf(b, wgt, c2);
            T = Tn;
        }
    }
}

// A thread's pixels blended in pairs with packed FP32x2 arithmetic (FFMA2 / FMUL2: one
// instruction for both pixels of a pair). Per pixel the operations and roundings of
// blend<FAST, false>, written with -alpha (the shift-add of Eq. (24) without its + 2^31
// is -exp^(P): that addition only sets the sign bit) and with the negated colours nr, ng,
// nb: T + T (-alpha) = T (1 - alpha) and c + (-r)(-alpha T) = c + r (alpha T) round to the
// same values. A pixel's state is its skip threshold thr: -ln 255 while it blends, +inf
// once finished; a pixel below its threshold takes -alpha = 0, which leaves its T and
// colour unchanged. One branch skips the Gaussian when no pixel of the thread needs it;
// the stop below 1e-4 (at most once in a pixel's life) is a branch around the common path
// (4K raster 0.558 -> 0.476 ms against selects on every pair and a finished flag beside
// the threshold test; 0.476 -> 0.453 ms with the branches taken once for all of the
// thread's pairs instead of once per pair).
template <bool FAST, int NH>
__device__ __forceinline__ void blend_pairs(const float (&P)[2 * NH], float2 nr, float2 ng, float2 nb,
                                                 float2 (&T)[NH], float2 (&cr)[NH], float2 (&cg)[NH],
                                                 float2 (&cb)[NH], float (&thr)[2 * NH])
{
    bool u[2 * NH];
    bool any = false;
#pragma unroll
    for (int i = 0; i < 2 * NH; i++) {
        u[i] = P[i] >= thr[i];
        any = any || u[i];
    }
    if (!any) return;
    float2 Tn[NH], nw[NH];
    bool stop = false;
#pragma unroll
    for (int h = 0; h < NH; h++) {
        float ea, eb; // -exp^(P), or -expf(P)
        if constexpr (FAST) {
            const float2 w = __ffma2_rn(make_float2(P[2 * h], P[2 * h + 1]), make_float2(1.44269502f, 1.44269502f),
                                        make_float2(126.954323f, 126.954323f));
            ea = __uint_as_float(__float_as_uint(w.x) << 6);
            eb = __uint_as_float(__float_as_uint(w.y) << 6);
        } else {
            ea = -expf(P[2 * h]);
            eb = -expf(P[2 * h + 1]);
        }
        const float2 na = make_float2(u[2 * h] ? fmaxf(-0.99f, ea) : 0.0f, u[2 * h + 1] ? fmaxf(-0.99f, eb) : 0.0f);
        Tn[h] = __ffma2_rn(T[h], na, T[h]);
        nw[h] = __fmul2_rn(na, T[h]); // -alpha T
        stop = stop || Tn[h].x < 1e-4f || Tn[h].y < 1e-4f;
    }
    if (stop) { // a pixel that would fall below 1e-4 adds nothing (weight 0, T kept) and finishes
#pragma unroll
        for (int h = 0; h < NH; h++) {
            if (Tn[h].x < 1e-4f) {
                nw[h].x = 0.0f;
                Tn[h].x = T[h].x;
                thr[2 * h] = __int_as_float(0x7f800000); // +inf: finished
            }
            if (Tn[h].y < 1e-4f) {
                nw[h].y = 0.0f;
                Tn[h].y = T[h].y;
                thr[2 * h + 1] = __int_as_float(0x7f800000);
            }
        }
    }
#pragma unroll
    for (int h = 0; h < NH; h++) {
        cr[h] = __ffma2_rn(nr, nw[h], cr[h]);
        cg[h] = __ffma2_rn(ng, nw[h], cg[h]);
        cb[h] = __ffma2_rn(nb, nw[h], cb[h]);
        T[h] = Tn[h];
    }
}

// The same blend for a thread with one pixel: the skip threshold as its state, the stop
// below 1e-4 a branch around the common path (bit-identical to blend<FAST, false>).
template <bool FAST>
__device__ __forceinline__ void blend_one(float P, float nr, float ng, float nb, float& T, float& cr, float& cg,
                                               float& cb, float& thr)
{
    if (!(P >= thr)) return;
    float e; // -exp^(P), or -expf(P)
    if constexpr (FAST) e = __uint_as_float(__float_as_uint(fmaf(P, 1.44269502f, 126.954323f)) << 6);
    else e = -expf(P);
    const float na = fmaxf(-0.99f, e); // -alpha
    float Tn = fmaf(T, na, T);
    float nw = na * T; // -alpha T
    if (Tn < 1e-4f) { // once in the pixel's life: adds nothing, T kept, finished
        nw = 0.0f;
        Tn = T;
        thr = __int_as_float(0x7f800000);
    }
    cr = fmaf(nr, nw, cr);
    cg = fmaf(ng, nw, cg);
    cb = fmaf(nb, nw, cb);
    T = Tn;
}

// The same blend without branches, for frames of few tiles, where the latency of each warp's own chain
// of records bounds the rasterizer and not the issue slots: with selects instead of the skip and stop
// branches the records' exponents overlap the blends before them. Bit-identical to the two above.
template <int NH>
__device__ __forceinline__ void blend_pairs_straight(const float (&P)[2 * NH], float2 nr, float2 ng, float2 nb,
                                                     float2 (&T)[NH], float2 (&cr)[NH], float2 (&cg)[NH],
                                                     float2 (&cb)[NH], float (&thr)[2 * NH])
{
    const float inf = __int_as_float(0x7f800000);
#pragma unroll
    for (int h = 0; h < NH; h++) {
        const float2 w = __ffma2_rn(make_float2(P[2 * h], P[2 * h + 1]), make_float2(1.44269502f, 1.44269502f),
                                    make_float2(126.954323f, 126.954323f));
        const float ea = __uint_as_float(__float_as_uint(w.x) << 6); // -exp^(P)
        const float eb = __uint_as_float(__float_as_uint(w.y) << 6);
        const float2 na = make_float2(P[2 * h] >= thr[2 * h] ? fmaxf(-0.99f, ea) : 0.0f,
                                      P[2 * h + 1] >= thr[2 * h + 1] ? fmaxf(-0.99f, eb) : 0.0f);
        const float2 Tn = __ffma2_rn(T[h], na, T[h]);
        float2 nw = __fmul2_rn(na, T[h]); // -alpha T
        const bool sx = Tn.x < 1e-4f, sy = Tn.y < 1e-4f; // adds nothing, T kept, finished
        nw = make_float2(sx ? 0.0f : nw.x, sy ? 0.0f : nw.y);
        thr[2 * h] = sx ? inf : thr[2 * h];
        thr[2 * h + 1] = sy ? inf : thr[2 * h + 1];
        T[h] = make_float2(sx ? T[h].x : Tn.x, sy ? T[h].y : Tn.y);
        cr[h] = __ffma2_rn(nr, nw, cr[h]);
        cg[h] = __ffma2_rn(ng, nw, cg[h]);
        cb[h] = __ffma2_rn(nb, nw, cb[h]);
    }
}

// sums the per-thread work counters of a counting launch into the frame counters
__device__ __forceinline__ void flush_counts(Counters* c, unsigned n_eval, unsigned n_blend)
{
    unsigned long long e = n_eval, b = n_blend;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        e += __shfl_xor_sync(0xffffffffu, e, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&c->n_pairs, e);
        atomicAdd(&c->n_blends, b);
    }
}

// First index i in [0, n) with (keys[i] >> shift) >= t, n if none (keys sorted): a
// 33-ary search by one warp, each round 32 lanes probe and one ballot keeps the part
// that holds the boundary (six dependent loads for 68 M keys). Warp-uniform result.
// K: 32-bit keys or 16-bit tile ids.
template <typename K>
__device__ __forceinline__ unsigned warp_lower_bound(const K* __restrict__ keys, unsigned n, int shift, unsigned t)
{
    const int lane = threadIdx.x & 31;
    unsigned lo = 0, hi = n; // the answer lies in [lo, hi]
    while (hi - lo > 32) {
        const unsigned probe = lo + (unsigned)(((unsigned long long)(hi - lo) * (unsigned)(lane + 1)) / 33u);
        const bool less = (unsigned)((unsigned long long)__ldg(&keys[probe]) >> shift) < t;
        const int c = __popc(__ballot_sync(0xffffffffu, less)); // lanes 0..c-1 probe below the boundary
        const unsigned plo = __shfl_sync(0xffffffffu, probe, c > 0 ? c - 1 : 0);
        const unsigned phi = __shfl_sync(0xffffffffu, probe, c < 32 ? c : 31);
        if (c > 0) lo = plo + 1;
        if (c < 32) hi = phi;
    }
    const unsigned i = lo + (unsigned)lane;
    const bool less = i < hi && (unsigned)((unsigned long long)__ldg(&keys[i]) >> shift) < t;
    return lo + (unsigned)__popc(__ballot_sync(0xffffffffu, less));
}

// Limited frames (RunArgs::limit) have the first RUN_LIMIT entries of every tile in vals. A tile that is read
// further before its pixels are finished is left to a second launch (REST), before which its other entries are
// written: its pixels' T stand in the place of its first entries (negative: finished), their colours in the image.
// (With the further entries fetched by the tile's own block the code around the loop cost every tile 3 to 5 %.)
enum { WHOLE = 0, LIMITED = 1, REST = 2 };

// One tile of the RoofGS rasterizer (a block of 256 / PPT threads).
template <bool FAST, int PPT, bool COUNT, bool STRAIGHT = false, int MODE = WHOLE>
__device__ __forceinline__ void raster_tile(const RasterArgs& a, const int tile)
{
    constexpr int NT = 256 / PPT; // threads per tile of 256 pixels (16 x 16, 32 x 8 or 8 x 32)
    constexpr int NH = (PPT + 1) / 2; // pixel pairs of a thread (one pixel of the last pair unused at PPT 1)
    __shared__ float4 s_c0[NT];       // C1, C2, C3, C4
    __shared__ float4 s_c1[NT];       // C5, C6, -b, -b (1 pixel per thread: C5, C6, -r, -g)
    // -r, -r, -g, -g (pairs for the packed blend; 1 pixel per thread: -b in .x)
    __shared__ float4 s_cn[PPT == 1 ? 1 : NT];
    __shared__ float s_cb[PPT == 1 ? NT : 1];
    const int tx = tile % a.tiles_x, ty = tile / a.tiles_x;
    const int x0 = tx * a.cam.tw, y0 = ty * a.cam.th;
    const int t = threadIdx.x;
    // the thread's pixels: (x, y), (x, y+1), ..., (x, y+PPT-1)
    const int lx = t & (a.cam.tw - 1);
    const int ly = (t >> a.cam.tw_log2) * PPT;
    const int px = x0 + lx, py = y0 + ly;
    const int W = a.cam.W, H = a.cam.H;
    bool done[PPT];
    // the packed pair blend keeps a pixel's state as its skip threshold instead: -ln 255 while it
    // blends, +inf once finished (one compare per pixel and Gaussian instead of two tests)
    constexpr bool PAIRS = !COUNT && PPT >= 2;
    constexpr bool ONE = !COUNT && PPT == 1;
    float thr[PPT];
    // transmittance and colour of pixel i in component i & 1 of pair i / 2
    float2 T2[NH], R2[NH], G2[NH], B2[NH];
#pragma unroll
    for (int h = 0; h < NH; h++) {
        T2[h] = make_float2(1.0f, 1.0f);
        R2[h] = G2[h] = B2[h] = make_float2(0.0f, 0.0f);
    }
#pragma unroll
    for (int i = 0; i < PPT; i++) {
        done[i] = !(px < W && py + i < H);
        thr[i] = done[i] ? __int_as_float(0x7f800000) : -LN255F;
    }
    // hoisted pixel terms (tile-local)
    const float x = (float)lx, y = (float)ly;
    const float xx = x * x, xy = x * y, yy = y * y, y2p1 = 2.0f * y + 1.0f;
    unsigned n_eval = 0, n_blend = 0;
    uint2 range;
    if (MODE == WHOLE && (a.skeys || a.skeys16)) { // warps 0 and 1 search the first entries of tiles `tile` and `tile + 1`
        __shared__ unsigned s_bound[2];
        const int warp = t >> 5;
        if (warp < 2) {
            const unsigned n = a.ctr->n_entries;
            const unsigned key = (unsigned)tile;
            const unsigned b = a.skeys16 ? warp_lower_bound(a.skeys16, n, 0, key + (unsigned)warp)
                                         : warp_lower_bound(a.skeys, n, a.tile_shift, key + (unsigned)warp);
            if ((t & 31) == 0) s_bound[warp] = b;
        }
        __syncthreads();
        range = s_bound[1] > s_bound[0] ? make_uint2(s_bound[0], s_bound[1]) : make_uint2(0u, 0u);
        if (t == 0) a.ranges_out[tile] = range;
    } else {
        range = a.ranges[tile];
    }
    // the record of entry j, and whether it is fetched while the batch before it is blended (eight
    // registers; two pixels per thread: 256 tiles 22.4 -> 20.4 us, 1080p 126 -> 123 us; four pixels, 4K:
    // 391 -> 396 us, not done)
    constexpr int UNROLL = PPT == 4 ? 2 : (STRAIGHT ? 8 : 4);
    constexpr bool AHEAD = PPT == 2 && !COUNT && MODE != REST;
    float4 q0 = make_float4(0.0f, 0.0f, 0.0f, 0.0f), q1 = q0;
    unsigned first = range.x, end = range.y; // entries blended next
    if (MODE != WHOLE) {
        const unsigned limit = a.row_limit[ty];
        if (range.y - range.x > limit) end = range.x + limit;
    }
    auto fetch = [&](unsigned j) {
        if (j < end) {
            unsigned id = a.vals[j];
            if (id >= (unsigned long long)a.n) id = 0; // only after a failed (timed-out) sort
            q0 = __ldg(&a.rec[2 * id]);
            q1 = __ldg(&a.rec[2 * id + 1]);
        }
    };
    auto finished = [&](bool& all_done) { // every pixel of the thread, of the block
        all_done = true;
#pragma unroll
        for (int i = 0; i < PPT; i++)
            all_done = all_done && ((PAIRS || ONE) ? thr[i] == __int_as_float(0x7f800000) : done[i]);
        return __syncthreads_count(!all_done) == 0;
    };
    bool all_done = false;
    if constexpr (MODE == REST) { // the pixels as the first kernel left them
        first = end;
        end = range.y;
#pragma unroll
        for (int i = 0; i < PPT; i++) {
            const float Ti = __uint_as_float(a.vals[range.x + (unsigned)(i * NT + t)]);
            thr[i] = Ti < 0.0f ? __int_as_float(0x7f800000) : -LN255F;
            ((i & 1) ? T2[i >> 1].y : T2[i >> 1].x) = fabsf(Ti);
            if (px < W && py + i < H) {
                const size_t plane = (size_t)W * H, o = (size_t)(py + i) * W + px;
                ((i & 1) ? R2[i >> 1].y : R2[i >> 1].x) = a.out[o];
                ((i & 1) ? G2[i >> 1].y : G2[i >> 1].x) = a.out[plane + o];
                ((i & 1) ? B2[i >> 1].y : B2[i >> 1].x) = a.out[2 * plane + o];
            }
        }
    }
    if (AHEAD) fetch(first + t);
    for (unsigned start = first; start < end; start += NT) {
        if (finished(all_done)) break;
        const unsigned j = start + t;
        if (!AHEAD) fetch(j);
        if (j < end) {
            const float u = q0.x - (float)x0, v = q0.y - (float)y0;
            const float ca = q0.z, cbq = q0.w, cc = q1.x, logo = q1.y;
            // Eq. (15): folded coefficients
            const float C1 = -0.5f * ca, C2 = -0.5f * cbq, C3 = -0.5f * cc;
            const float C4 = fmaf(ca, u, 0.5f * cbq * v);
            const float C5 = fmaf(cc, v, 0.5f * cbq * u);
            const float C0 = fmaf(ca * u, u, fmaf(cbq * u, v, cc * v * v)); // Eq. (14)
            const float C6 = fmaf(-0.5f, C0, logo);
            const unsigned rg = __float_as_uint(q1.z), bb = __float_as_uint(q1.w);
            const float fr = __half2float(__ushort_as_half((unsigned short)(rg & 0xffffu)));
            const float fg = __half2float(__ushort_as_half((unsigned short)(rg >> 16)));
            const float fb = __half2float(__ushort_as_half((unsigned short)(bb & 0xffffu)));
            s_c0[t] = make_float4(C1, C2, C3, C4);
            if constexpr (PPT == 1) {
                s_c1[t] = make_float4(C5, C6, -fr, -fg);
                s_cb[t] = -fb;
            } else {
                s_c1[t] = make_float4(C5, C6, -fb, -fb);
                s_cn[t] = make_float4(-fr, -fr, -fg, -fg);
            }
        }
        __syncthreads();
        if (AHEAD) fetch(j + NT);
        const int cnt = min((unsigned)NT, end - start);
        if (!__all_sync(0xffffffffu, all_done)) {
#pragma unroll(UNROLL) // records per iteration, 4K raster: 4 pixels 0.564 -> 0.558 ms (2), 2 pixels 0.549 -> 0.540 ms and 1 pixel 1.059 -> 0.900 ms (4)
            for (int k = 0; k < cnt; k++) {
                const float4 c0 = s_c0[k];
                const float4 c1 = s_c1[k];
                // negated colours, from the pairs' layout or the one-pixel layout
                float nr, ng, nb;
                float4 cn = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if constexpr (PPT == 1) {
                    nr = c1.z;
                    ng = c1.w;
                    nb = s_cb[k];
                } else {
                    cn = s_cn[k];
                    nr = cn.x;
                    ng = cn.z;
                    nb = c1.z;
                }
                // Eq. (16): P(x, y) = C1 x^2 + C2 xy + C3 y^2 + C4 x + C5 y + C6
                float P[PPT];
                P[0] = fmaf(c0.x, xx, fmaf(c0.y, xy, fmaf(c0.z, yy, fmaf(c0.w, x, fmaf(c1.x, y, c1.y)))));
                if (PPT >= 2) {
                    // Eq. (20): P(x, y+1) = P(x, y) + C2 x + C3 (2y + 1) + C5; the step to the next
                    // row grows by 2 C3 per row
                    float d = fmaf(c0.y, x, fmaf(c0.z, y2p1, c1.x));
#pragma unroll
                    for (int i = 1; i < PPT; i++) {
                        if (i > 1) d = fmaf(2.0f, c0.z, d);
                        P[i] = P[i - 1] + d;
                    }
                }
                if constexpr (PAIRS && STRAIGHT) {
                    blend_pairs_straight<NH>(P, make_float2(cn.x, cn.y), make_float2(cn.z, cn.w), make_float2(c1.z, c1.w),
                                             T2, R2, G2, B2, thr);
                } else if constexpr (PAIRS) {
                    blend_pairs<FAST, NH>(P, make_float2(cn.x, cn.y), make_float2(cn.z, cn.w), make_float2(c1.z, c1.w),
                                         T2, R2, G2, B2, thr);
                } else if constexpr (ONE) {
                    blend_one<FAST>(P[0], nr, ng, nb, T2[0].x, R2[0].x, G2[0].x, B2[0].x, thr[0]);
                } else {
#pragma unroll
                    for (int i = 0; i < PPT; i++) {
                        float& Ti = (i & 1) ? T2[i >> 1].y : T2[i >> 1].x;
                        float& Ri = (i & 1) ? R2[i >> 1].y : R2[i >> 1].x;
                        float& Gi = (i & 1) ? G2[i >> 1].y : G2[i >> 1].x;
                        float& Bi = (i & 1) ? B2[i >> 1].y : B2[i >> 1].x;
                        blend<FAST, COUNT>(P[i], -nr, -ng, -nb, Ti, Ri, Gi, Bi, done[i], n_eval, n_blend);
                    }
                }
            }
        }
    }
    const bool rest = MODE == LIMITED && end < a.ranges[tile].y && !finished(all_done); // (loaded again: no register meanwhile)
    if constexpr (MODE == LIMITED) {
        if (rest) {
            if (t == 0) {
                a.rest_list[atomicAdd(a.rest_count, 1u)] = (unsigned)tile;
                a.rest_flag[tile] = 1u;
            }
#pragma unroll
            for (int i = 0; i < PPT; i++) {
                const float Ti = (i & 1) ? T2[i >> 1].y : T2[i >> 1].x;
                a.vals_out[a.ranges[tile].x + (unsigned)(i * NT + t)] =
                    __float_as_uint(thr[i] == __int_as_float(0x7f800000) ? -Ti : Ti);
            }
        }
    }
    if (COUNT) flush_counts(a.count, n_eval, n_blend);
    const size_t plane = (size_t)W * H;
#pragma unroll
    for (int i = 0; i < PPT; i++) {
        if (px < W && py + i < H) {
            const size_t o = (size_t)(py + i) * W + px;
            const float Ti = (i & 1) ? T2[i >> 1].y : T2[i >> 1].x;
            const float r = (i & 1) ? R2[i >> 1].y : R2[i >> 1].x, g = (i & 1) ? G2[i >> 1].y : G2[i >> 1].x,
                        b = (i & 1) ? B2[i >> 1].y : B2[i >> 1].x;
            a.out[o] = rest ? r : r + Ti * a.cam.bg[0];
            a.out[plane + o] = rest ? g : g + Ti * a.cam.bg[1];
            a.out[2 * plane + o] = rest ? b : b + Ti * a.cam.bg[2];
        }
    }
}

template <bool FAST, int PPT, bool COUNT, bool STRAIGHT = false, int MODE = WHOLE>
__global__ void __launch_bounds__(256 / PPT) k_raster_roofgs(RasterArgs a)
{
    grid_dependency_wait();
    raster_tile<FAST, PPT, COUNT, STRAIGHT, MODE>(a, (int)ordered_tile(a.order, blockIdx.x));
}

// the tiles that a LIMITED launch left unfinished
template <bool FAST, int PPT>
__global__ void __launch_bounds__(256 / PPT) k_raster_roofgs_rest(RasterArgs a)
{
    grid_dependency_wait();
    const unsigned n = *a.rest_count;
    for (unsigned b = blockIdx.x; b < n; b += gridDim.x) {
        raster_tile<FAST, PPT, false, false, REST>(a, (int)a.rest_list[b]);
        __syncthreads(); // the staged records are written again
    }
}
// blocks of such a launch (its list is in about the order of the first one, the longest tiles first)
static unsigned rest_blocks(int ppt) { return (unsigned)(4 * ppt * device_sm_count()); }

// Every view of a batch in one persistent launch: each block takes (view, tile) items
// from one work counter (views in order, tiles in order) until all are done, and
// rasterizes the tile with that view's arguments (kernel parameter space).
template <bool FAST, int PPT>
__global__ void __launch_bounds__(256 / PPT) k_raster_views(const __grid_constant__ RasterViews m)
{
    __shared__ unsigned s_g;
    grid_dependency_wait();
    const unsigned total = m.tile_prefix[m.n_views];
    while (true) {
        if (threadIdx.x == 0) s_g = atomicAdd(m.claim, 1u);
        __syncthreads();
        const unsigned g = s_g;
        if (g >= total) break;
        int v = 0;
        while (v + 1 < m.n_views && m.tile_prefix[v + 1] <= g) v++;
        raster_tile<FAST, PPT, false>(m.views[v], (int)(g - m.tile_prefix[v]));
        __syncthreads(); // every thread has read s_g before it is claimed again
    }
}

template <bool FAST, int PPT>
static void raster_views_launch(const RasterViews& m, cudaStream_t s)
{
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_raster_views<FAST, PPT>, 256 / PPT, 0);
    const unsigned total = m.tile_prefix[m.n_views];
    unsigned grid = (unsigned)((per_sm > 0 ? per_sm : 1) * device_sm_count());
    if (grid > total) grid = total;
    if (grid) launch_dependent(k_raster_views<FAST, PPT>, dim3(grid), dim3(256 / PPT), 0, s, m);
}

void launch_raster_views(const RasterViews& m, int fast_exp, int ppt, cudaStream_t s)
{
    if (fast_exp) {
        if (ppt == 1) raster_views_launch<true, 1>(m, s);
        else if (ppt == 4) raster_views_launch<true, 4>(m, s);
        else raster_views_launch<true, 2>(m, s);
    } else {
        if (ppt == 1) raster_views_launch<false, 1>(m, s);
        else if (ppt == 4) raster_views_launch<false, 4>(m, s);
        else raster_views_launch<false, 2>(m, s);
    }
}

template <bool COUNT>
static void raster_roofgs_variant(const RasterArgs& a, const RunArgs* runs, cudaStream_t s)
{
    const unsigned tiles = (unsigned)(a.tiles_x * a.tiles_y);
    if constexpr (!COUNT) {
        if (a.limit != RUN_ALL) {
            auto launch = [&](auto kernel, auto rest, unsigned ppt) {
                launch_dependent(kernel, dim3(tiles), dim3(256 / ppt), 0, s, a);
                launch_runs_rest(*runs, s);
                launch_dependent(rest, dim3(rest_blocks((int)ppt)), dim3(256 / ppt), 0, s, a);
            };
            if (a.fast_exp) {
                if (a.ppt == 1) launch(k_raster_roofgs<true, 1, false, false, LIMITED>, k_raster_roofgs_rest<true, 1>, 1);
                else if (a.ppt == 4) launch(k_raster_roofgs<true, 4, false, false, LIMITED>, k_raster_roofgs_rest<true, 4>, 4);
                else launch(k_raster_roofgs<true, 2, false, false, LIMITED>, k_raster_roofgs_rest<true, 2>, 2);
            } else {
                if (a.ppt == 1) launch(k_raster_roofgs<false, 1, false, false, LIMITED>, k_raster_roofgs_rest<false, 1>, 1);
                else if (a.ppt == 4) launch(k_raster_roofgs<false, 4, false, false, LIMITED>, k_raster_roofgs_rest<false, 4>, 4);
                else launch(k_raster_roofgs<false, 2, false, false, LIMITED>, k_raster_roofgs_rest<false, 2>, 2);
            }
            return;
        }
    }
    // two pixels per thread and at most 20 tiles per SM: the blend without branches. 256 tiles, 10 k Gaussians
    // 32.5 -> 20.2 us; 256 to 2,451 tiles, 30 k / 400 k Gaussians 20-35 % / 0-10 % less; 3,600 tiles and more fill
    // the issue slots, and branches win (82 against 98 us, 1080p 124 against 150), as with four pixels per thread
    // at any size once pixels finish early (256 tiles, 400 k: 1,043 against 1,120)
    if (a.fast_exp && !COUNT && a.ppt == 2 && tiles <= 20u * (unsigned)device_sm_count()) {
        launch_dependent(k_raster_roofgs<true, 2, false, true>, dim3(tiles), dim3(128), 0, s, a);
    } else if (a.fast_exp) {
        if (a.ppt == 1) launch_dependent(k_raster_roofgs<true, 1, COUNT>, dim3(tiles), dim3(256), 0, s, a);
        else if (a.ppt == 4) launch_dependent(k_raster_roofgs<true, 4, COUNT>, dim3(tiles), dim3(64), 0, s, a);
        else launch_dependent(k_raster_roofgs<true, 2, COUNT>, dim3(tiles), dim3(128), 0, s, a);
    } else {
        if (a.ppt == 1) launch_dependent(k_raster_roofgs<false, 1, COUNT>, dim3(tiles), dim3(256), 0, s, a);
        else if (a.ppt == 4) launch_dependent(k_raster_roofgs<false, 4, COUNT>, dim3(tiles), dim3(64), 0, s, a);
        else launch_dependent(k_raster_roofgs<false, 2, COUNT>, dim3(tiles), dim3(128), 0, s, a);
    }
}

void launch_raster_roofgs(const RasterArgs& a, const RunArgs* runs, cudaStream_t s)
{
    if (a.count) raster_roofgs_variant<true>(a, runs, s);
    else raster_roofgs_variant<false>(a, runs, s);
}

// Plain 3DGS rasterizer: expf, the exponent of Eq. (10) in the completed-square form of
// exact_power() from the double-float mean, shifted to the tile origin when a record is staged
// (u.hi - x0 is exact). k_raster_exact_count, one pixel per thread, runs when the work counters are
// asked for; k_raster_exact is the timed kernel. Both evaluate the same operations with the same
// roundings per pixel, so their images are bit-identical.
constexpr int E_THREADS = 256;

__global__ void __launch_bounds__(E_THREADS) k_raster_exact_count(RasterArgs a)
{
    __shared__ float4 s_m[E_THREADS];
    __shared__ float4 s_q[E_THREADS];
    __shared__ float4 s_rgb[E_THREADS];
    grid_dependency_wait();
    if (a.count->n_entries_total > (unsigned long long)a.cap) return; // the caller grows the workspace and renders again
    const int tile = blockIdx.x;
    const int tx = tile % a.tiles_x, ty = tile / a.tiles_x;
    const int x0 = tx * a.cam.tw, y0 = ty * a.cam.th;
    const int lxi = threadIdx.x & (a.cam.tw - 1), lyi = threadIdx.x >> a.cam.tw_log2;
    const int px = x0 + lxi, py = y0 + lyi;
    const int W = a.cam.W, H = a.cam.H;
    const bool inside = px < W && py < H;
    bool done = !inside;
    const float lx = (float)lxi, ly = (float)lyi;
    float T = 1.0f, c0 = 0.f, c1 = 0.f, c2 = 0.f;
    unsigned n_eval = 0, n_blend = 0;
    const uint2 range = a.ranges[tile];
    for (unsigned start = range.x; start < range.y; start += E_THREADS) {
        if (__syncthreads_count(!done) == 0) break;
        const unsigned j = start + threadIdx.x;
        if (j < range.y) {
            unsigned id = a.vals[j];
            if (id >= (unsigned long long)a.n) id = 0; // only after a failed (timed-out) sort
            const float4* const rec = a.erec + 3 * (size_t)id;
            const float4 m = __ldg(rec);
            s_m[threadIdx.x] = make_float4(m.x - (float)x0, m.y, m.z - (float)y0, m.w);
            s_q[threadIdx.x] = __ldg(rec + 1);
            s_rgb[threadIdx.x] = __ldg(rec + 2);
        }
        __syncthreads();
        const int cnt = min((unsigned)E_THREADS, range.y - start);
        for (int k = 0; !done && k < cnt; k++) {
            const float4 q = s_q[k];
            const float power = exact_power(s_m[k], q, lx, ly); // Eq. (10), <= 0
            n_eval++;
            const float alpha = fminf(0.99f, q.w * expf(power)); // Eqs. (11)-(12)
            if (alpha < 1.0f / 255.0f) continue;
            n_blend++;
            const float Tn = T * (1.0f - alpha);
            if (Tn < 1e-4f) {
                done = true;
                continue;
            }
            const float4 c = s_rgb[k];
            const float wgt = alpha * T;
            c0 = fmaf(c.x, wgt, c0);
            c1 = fmaf(c.y, wgt, c1);
            c2 = fmaf(c.z, wgt, c2);
            T = Tn;
        }
    }
    flush_counts(a.count, n_eval, n_blend);
    if (inside) {
        const size_t plane = (size_t)W * H, o = (size_t)py * W + px;
        a.out[o] = fmaf(T, a.cam.bg[0], c0);
        a.out[plane + o] = fmaf(T, a.cam.bg[1], c1);
        a.out[2 * plane + o] = fmaf(T, a.cam.bg[2], c2);
    }
}

// One block of 256 / PPT threads per tile, PPT (2 or 4) vertically adjacent pixels per thread, blended in
// pairs with packed FP32x2 arithmetic. Most pairs of a tile's list lie below 1/255 in most pixels: the
// exponent alone decides those (exact_skip_below, staged with the record), and only a thread with a
// pixel at or above it evaluates expf and the exact test. Bound by issue slots (2.7 instructions per
// cycle at 1080p, the last wave of heavy tiles aside): 4K, 3 M Gaussians 950 -> 730 us against one
// pixel per thread with expf on every pair, 1080p, 500 k 300 -> 240 us.
// Records are staged with the operands of the packed instructions doubled.
template <int PPT, int MODE>
__device__ __forceinline__ void exact_tile(const RasterArgs& a, const int tile)
{
    constexpr int NT = 256 / PPT, NH = PPT / 2;
    __shared__ float4 s_a[NT]; // u - x0, skip threshold, opacity
    __shared__ float4 s_b[NT]; // -(v.hi - y0) twice, -v.lo twice
    __shared__ float4 s_c[NT]; // -c twice, -u.lo twice
    __shared__ float4 s_d[NT]; // quad.x twice, quad.z twice
    __shared__ float4 s_rg[NT]; // r, r, g, g
    __shared__ float2 s_bb[NT]; // b, b
    const int t = threadIdx.x;
    const int tx = tile % a.tiles_x, ty = tile / a.tiles_x;
    const int x0 = tx * a.cam.tw, y0 = ty * a.cam.th;
    const int lxi = t & (a.cam.tw - 1), lyi = (t >> a.cam.tw_log2) * PPT;
    const int px = x0 + lxi, py = y0 + lyi;
    const int W = a.cam.W, H = a.cam.H;
    const float INF = __int_as_float(0x7f800000);
    const float lx = (float)lxi;
    float2 ly[NH], T[NH], R[NH], G[NH], B[NH];
    float lim[PPT]; // -inf while the pixel blends, +inf once finished
#pragma unroll
    for (int h = 0; h < NH; h++) {
        ly[h] = make_float2((float)(lyi + 2 * h), (float)(lyi + 2 * h + 1));
        T[h] = make_float2(1.0f, 1.0f);
        R[h] = G[h] = B[h] = make_float2(0.0f, 0.0f);
    }
#pragma unroll
    for (int i = 0; i < PPT; i++) lim[i] = px < W && py + i < H ? -INF : INF;
    const uint2 range = a.ranges[tile];
    // the record of entry j, and whether it is fetched while the batch before it is blended (few tiles:
    // 672 tiles 49.8 -> 47.0 us; four pixels per thread at 4K 676 -> 701 us, not done)
    constexpr bool AHEAD = PPT == 2 && MODE != REST;
    float4 m = make_float4(0.0f, 0.0f, 0.0f, 0.0f), q = m, c = m;
    unsigned first = range.x, end = range.y; // entries blended next
    if (MODE != WHOLE) {
        const unsigned limit = a.row_limit[ty];
        if (range.y - range.x > limit) end = range.x + limit;
    }
    auto fetch = [&](unsigned j) {
        if (j < end) {
            unsigned id = a.vals[j];
            if (id >= (unsigned long long)a.n) id = 0; // only after a failed (timed-out) sort
            const float4* const rec = a.erec + 3 * (size_t)id;
            m = __ldg(rec);
            q = __ldg(rec + 1);
            c = __ldg(rec + 2);
        }
    };
    auto finished = [&](bool& all_done) { // every pixel of the thread, of the block
        all_done = true;
#pragma unroll
        for (int i = 0; i < PPT; i++) all_done = all_done && lim[i] == INF;
        return __syncthreads_count(!all_done) == 0;
    };
    bool all_done = false;
    if constexpr (MODE == REST) { // the pixels as the first kernel left them
        first = end;
        end = range.y;
#pragma unroll
        for (int i = 0; i < PPT; i++) {
            const float Ti = __uint_as_float(a.vals[range.x + (unsigned)(i * NT + t)]);
            lim[i] = Ti < 0.0f ? INF : -INF;
            (i & 1 ? T[i / 2].y : T[i / 2].x) = fabsf(Ti);
            if (px < W && py + i < H) {
                const size_t plane = (size_t)W * H, o = (size_t)(py + i) * W + px;
                (i & 1 ? R[i / 2].y : R[i / 2].x) = a.out[o];
                (i & 1 ? G[i / 2].y : G[i / 2].x) = a.out[plane + o];
                (i & 1 ? B[i / 2].y : B[i / 2].x) = a.out[2 * plane + o];
            }
        }
    }
    if (AHEAD) fetch(first + t);
    for (unsigned start = first; start < end; start += NT) {
        if (finished(all_done)) break;
        const unsigned j = start + t;
        if (!AHEAD) fetch(j);
        if (j < end) {
            const float mz = m.z - (float)y0;
            s_a[t] = make_float4(m.x - (float)x0, exact_skip_below(q.w), q.w, 0.0f);
            s_b[t] = make_float4(-mz, -mz, -m.w, -m.w);
            s_c[t] = make_float4(-q.y, -q.y, -m.y, -m.y);
            s_d[t] = make_float4(q.x, q.x, q.z, q.z);
            s_rg[t] = make_float4(c.x, c.x, c.y, c.y);
            s_bb[t] = make_float2(c.z, c.z);
        }
        __syncthreads();
        if (AHEAD) fetch(j + NT);
        const int cnt = min((unsigned)NT, end - start);
        if (__all_sync(0xffffffffu, all_done)) continue;
#pragma unroll 2
        for (int k = 0; k < cnt; k++) {
            const float4 va = s_a[k], vb = s_b[k], vc = s_c[k], vd = s_d[k];
            const float dx = __fsub_rn(lx, va.x);
            float P[PPT];
            bool u[PPT], any = false;
#pragma unroll
            for (int h = 0; h < NH; h++) { // exact_power() of the pair
                const float2 dy = __fadd2_rn(__fadd2_rn(ly[h], make_float2(vb.x, vb.y)), make_float2(vb.z, vb.w));
                const float2 tt = __fadd2_rn(__ffma2_rn(make_float2(vc.x, vc.y), dy, make_float2(dx, dx)),
                                             make_float2(vc.z, vc.w));
                const float2 p = __ffma2_rn(__fmul2_rn(make_float2(vd.x, vd.y), tt), tt,
                                            __fmul2_rn(__fmul2_rn(make_float2(vd.z, vd.w), dy), dy));
                P[2 * h] = p.x;
                P[2 * h + 1] = p.y;
                u[2 * h] = p.x >= va.y && p.x >= lim[2 * h];
                u[2 * h + 1] = p.y >= va.y && p.y >= lim[2 * h + 1];
                any = any || u[2 * h] || u[2 * h + 1];
            }
            if (!any) continue;
            float2 al[NH];
            any = false;
#pragma unroll
            for (int i = 0; i < PPT; i++) {
                const float e = fminf(0.99f, va.z * expf(P[i])); // Eqs. (11)-(12)
                u[i] = u[i] && !(e < 1.0f / 255.0f);
                (i & 1 ? al[i / 2].y : al[i / 2].x) = u[i] ? e : 0.0f;
                any = any || u[i];
            }
            if (!any) continue;
            float2 Tn[NH], w[NH];
            bool stop = false;
#pragma unroll
            for (int h = 0; h < NH; h++) { // alpha 0 leaves T and the colour as they are
                Tn[h] = __fmul2_rn(T[h], __fadd2_rn(make_float2(1.0f, 1.0f), make_float2(-al[h].x, -al[h].y)));
                w[h] = __fmul2_rn(al[h], T[h]);
                stop = stop || Tn[h].x < 1e-4f || Tn[h].y < 1e-4f;
            }
            if (stop) { // a pixel that would fall below 1e-4 adds nothing and finishes
#pragma unroll
                for (int h = 0; h < NH; h++) {
                    if (Tn[h].x < 1e-4f) {
                        w[h].x = 0.0f;
                        Tn[h].x = T[h].x;
                        lim[2 * h] = INF;
                    }
                    if (Tn[h].y < 1e-4f) {
                        w[h].y = 0.0f;
                        Tn[h].y = T[h].y;
                        lim[2 * h + 1] = INF;
                    }
                }
            }
            const float4 rg = s_rg[k];
            const float2 bb = s_bb[k];
#pragma unroll
            for (int h = 0; h < NH; h++) {
                R[h] = __ffma2_rn(make_float2(rg.x, rg.y), w[h], R[h]);
                G[h] = __ffma2_rn(make_float2(rg.z, rg.w), w[h], G[h]);
                B[h] = __ffma2_rn(bb, w[h], B[h]);
                T[h] = Tn[h];
            }
        }
    }
    const bool rest = MODE == LIMITED && end < a.ranges[tile].y && !finished(all_done); // (loaded again: no register meanwhile)
    if constexpr (MODE == LIMITED) {
        if (rest) {
            if (t == 0) {
                a.rest_list[atomicAdd(a.rest_count, 1u)] = (unsigned)tile;
                a.rest_flag[tile] = 1u;
            }
#pragma unroll
            for (int i = 0; i < PPT; i++) {
                const float Ti = i & 1 ? T[i / 2].y : T[i / 2].x;
                a.vals_out[a.ranges[tile].x + (unsigned)(i * NT + t)] = __float_as_uint(lim[i] == INF ? -Ti : Ti);
            }
        }
    }
    const size_t plane = (size_t)W * H;
#pragma unroll
    for (int i = 0; i < PPT; i++) {
        if (px < W && py + i < H) {
            const size_t o = (size_t)(py + i) * W + px;
            const float Ti = i & 1 ? T[i / 2].y : T[i / 2].x;
            const float r = i & 1 ? R[i / 2].y : R[i / 2].x, g = i & 1 ? G[i / 2].y : G[i / 2].x,
                        b = i & 1 ? B[i / 2].y : B[i / 2].x;
            a.out[o] = rest ? r : fmaf(Ti, a.cam.bg[0], r);
            a.out[plane + o] = rest ? g : fmaf(Ti, a.cam.bg[1], g);
            a.out[2 * plane + o] = rest ? b : fmaf(Ti, a.cam.bg[2], b);
        }
    }
}

template <int PPT, int MODE>
__global__ void __launch_bounds__(256 / PPT) k_raster_exact(RasterArgs a)
{
    grid_dependency_wait();
    if constexpr (MODE == REST) {
        const unsigned n = *a.rest_count;
        for (unsigned b = blockIdx.x; b < n; b += gridDim.x) {
            exact_tile<PPT, MODE>(a, (int)a.rest_list[b]);
            __syncthreads(); // the staged records are written again
        }
    } else {
        exact_tile<PPT, MODE>(a, (int)ordered_tile(a.order, blockIdx.x));
    }
}

// Four pixels per thread where the tiles fill the GPU more than once (16 blocks of 64 threads per SM
// are resident); below that a tile's own chain of pairs bounds the frame, and four warps per tile get
// through it faster than two. Per pass, two / four pixels per thread: 672 tiles (499x333) 106 / 113 us,
// 8,160 (1080p) 477 / 445 us, 32,400 (4K) 1988 / 1876 us.
void launch_raster_exact(const RasterArgs& a, const RunArgs* runs, cudaStream_t s)
{
    const unsigned tiles = (unsigned)(a.tiles_x * a.tiles_y);
    if (a.count) launch_dependent(k_raster_exact_count, dim3(tiles), dim3(E_THREADS), 0, s, a);
    else if (a.limit != RUN_ALL) { // only with many tiles
        launch_dependent(k_raster_exact<4, LIMITED>, dim3(tiles), dim3(64), 0, s, a);
        launch_runs_rest(*runs, s);
        launch_dependent(k_raster_exact<4, REST>, dim3(rest_blocks(4)), dim3(64), 0, s, a);
    } else if (tiles <= 16u * (unsigned)device_sm_count()) {
        launch_dependent(k_raster_exact<2, WHOLE>, dim3(tiles), dim3(128), 0, s, a);
    } else {
        launch_dependent(k_raster_exact<4, WHOLE>, dim3(tiles), dim3(64), 0, s, a);
    }
}

void launch_fast_exp_eval(const float* P, float* out, long long n, cudaStream_t s)
{
    if (n <= 0) return;
    k_fast_exp_eval<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(P, out, n);
}

} // namespace rg
