// backward.cu -- gradients of the exact-mode (plain 3DGS) render.
//
// Not part of the paper (which only renders); it differentiates the forward of
// Sec. III-D: C = sum_i c_i alpha_i T_i + T_final bg, alpha_i = min(0.99, o_i exp(p_i))
// (Eqs. (7), (10)-(12)), T_{i+1} = T_i (1 - alpha_i).
//
//  * k_raster_backward: one block per tile, two or four pixels per thread. Each pixel first
//    replays its front-to-back blend to find its final transmittance and last blended pair
//    (transmittance is recomputed, never stored), then walks the same pairs back to
//    front: T_i = T_{i+1} / (1 - alpha_i), S (G . colour behind pair i, G = dL/dpixel) grows by
//    (G . c_i) alpha_i T_i, and
//        dL/dc_i = G alpha_i T_i,   dL/dalpha_i = (G . c_i) T_i - S / (1 - alpha_i).
//    Through the exponent p = -1/2 (A t^2 + dy^2 / Sigma'_yy), t = dx - c dy, A = Sigma'_yy / det, the
//    Gaussian's image-space gradients follow from the sums of dL/dp times t, dy, t^2, t dy and dy^2
//    (no cancellation for thin Gaussians): these five, d(opacity) and d(rgb) are added over a
//    thread's pixels and the warp before they go to memory.
//  * k_preprocess_backward: one thread per Gaussian, the chain rule through the
//    conic (inverse of Sigma'), Sigma' = (J W M)(J W M)^T + 0.3 I with M = R(q) diag(s),
//    the perspective Jacobian J (tangent clamp included), the projected mean and the
//    view-dependent SH colour (coefficients and view direction).
#include "rg_internal.cuh"

namespace rg {

// Sum over the warp of nine values per lane, in 14 shuffles instead of 45: at each of the first three
// steps a lane keeps the half of the eight values that its lane bit selects. Value j ends in lanes
// 4 j .. 4 j + 3, the ninth in every lane.
__device__ __forceinline__ float warp_sum9(const float (&v)[9], float& ninth)
{
    const int lane = threadIdx.x & 31;
    float a[4], b[2];
#pragma unroll
    for (int j = 0; j < 4; j++) {
        const bool up = lane & 16;
        a[j] = (up ? v[j + 4] : v[j]) + __shfl_xor_sync(0xffffffffu, up ? v[j] : v[j + 4], 16);
    }
#pragma unroll
    for (int j = 0; j < 2; j++) {
        const bool up = lane & 8;
        b[j] = (up ? a[j + 2] : a[j]) + __shfl_xor_sync(0xffffffffu, up ? a[j] : a[j + 2], 8);
    }
    const bool up = lane & 4;
    float c = (up ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, up ? b[0] : b[1], 4);
    c += __shfl_xor_sync(0xffffffffu, c, 2);
    c += __shfl_xor_sync(0xffffffffu, c, 1);
    ninth = v[8];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ninth += __shfl_xor_sync(0xffffffffu, ninth, o);
    return c;
}

// exact_power() of a pair of vertically adjacent pixels with packed FP32x2 arithmetic (the same
// operations and roundings), and the offsets it is formed from: dy = y - v, t = (x - u) - c dy.
// The record's operands are staged doubled: b = -(v.hi - y0) twice, -v.lo twice; c = -c twice, -u.lo
// twice; d = quad.x twice, quad.z twice.
__device__ __forceinline__ float2 power_pair(float dx, float2 ly, const float4& b, const float4& c, const float4& d,
                                             float2& t, float2& dy)
{
    dy = __fadd2_rn(__fadd2_rn(ly, make_float2(b.x, b.y)), make_float2(b.z, b.w));
    t = __fadd2_rn(__ffma2_rn(make_float2(c.x, c.y), dy, make_float2(dx, dx)), make_float2(c.z, c.w));
    return __ffma2_rn(__fmul2_rn(make_float2(d.x, d.y), t), t, __fmul2_rn(__fmul2_rn(make_float2(d.z, d.w), dy), dy));
}

// Bound by issue slots (2.6 instructions per cycle; the last wave of heavy tiles takes a sixth of the
// time). With one pixel per thread a warp summed nine values over its lanes in 45 shuffles and nine
// atomics for each of its eight warps and every pair, reached or not: 1250 us at 1080p with 500 k Gaussians,
// now 760 us (two warps per tile, 14 shuffles, one atomic instruction of nine lanes).
// SINGLY: pixel by pixel, for a large or non-finite dL/dimage (k_backward_begin).
template <int PPT, bool SINGLY>
__device__ __forceinline__ void backward_tile(const BackwardArgs& a, const int tile)
{
    constexpr int NT = 256 / PPT, NH = PPT / 2;
    __shared__ float4 s_a[NT]; // u - x0, skip threshold, opacity, Gaussian
    __shared__ float4 s_b[NT], s_c[NT], s_d[NT]; // as power_pair() takes them
    __shared__ float4 s_rgb[NT];
    __shared__ int s_last;
    const int th = threadIdx.x, lane = th & 31;
    const int tx = tile % a.tiles_x, ty = tile / a.tiles_x;
    const int x0 = tx * a.cam.tw, y0 = ty * a.cam.th;
    const int lxi = th & (a.cam.tw - 1), lyi = (th >> a.cam.tw_log2) * PPT;
    const int px = x0 + lxi, py = y0 + lyi;
    const int W = a.cam.W, H = a.cam.H;
    const float lx = (float)lxi;
    const uint2 range = a.ranges[tile];
    if (th == 0) s_last = -1;
    // the record of entry j; blended: the block's last blended entry (colours are staged too), -1 in the replay
    auto stage = [&](unsigned j, int blended) {
        unsigned id = a.vals[j];
        if (id >= (unsigned long long)a.n) id = 0;
        const float4* const rec = a.erec + 3 * (size_t)id;
        const float4 m = __ldg(rec), q = __ldg(rec + 1);
        unsigned g = 0;
        if (blended >= 0) {
            const float4 c = __ldg(rec + 2);
            s_rgb[th] = c;
            g = a.order ? a.order[id] : id;
            if (c.w != 0.0f && (int)j <= blended) // its exponent is undefined: of its gradients only the colour's is a number
                for (int k = 0; k < 6; k++) atomicAdd(a.gbuf + (size_t)g * GBUF + k, __int_as_float(0x7fffffff));
        }
        const float mz = m.z - (float)y0;
        s_a[th] = make_float4(m.x - (float)x0, exact_skip_below(q.w), q.w, __uint_as_float(g));
        s_b[th] = make_float4(-mz, -mz, -m.w, -m.w);
        s_c[th] = make_float4(-q.y, -q.y, -m.y, -m.y);
        s_d[th] = make_float4(q.x, q.x, q.z, q.z);
    };

    // 1) forward replay: final transmittance and the last blended pair of each pixel
    const float INF = __int_as_float(0x7f800000);
    float2 ly[NH], T[NH];
    float lim[PPT]; // -inf while the pixel blends, +inf once finished
    int last[PPT];
#pragma unroll
    for (int h = 0; h < NH; h++) {
        ly[h] = make_float2((float)(lyi + 2 * h), (float)(lyi + 2 * h + 1));
        T[h] = make_float2(1.0f, 1.0f);
    }
#pragma unroll
    for (int i = 0; i < PPT; i++) {
        lim[i] = px < W && py + i < H ? -INF : INF;
        last[i] = -1;
    }
    for (unsigned start = range.x; start < range.y; start += NT) {
        bool all_done = true;
#pragma unroll
        for (int i = 0; i < PPT; i++) all_done = all_done && lim[i] == INF;
        if (__syncthreads_count(!all_done) == 0) break;
        if (start + th < range.y) stage(start + th, -1);
        __syncthreads();
        const int cnt = min((unsigned)NT, range.y - start);
        if (__all_sync(0xffffffffu, all_done)) continue;
#pragma unroll 2
        for (int k = 0; k < cnt; k++) {
            const float4 va = s_a[k];
            const float dx = __fsub_rn(lx, va.x);
            float P[PPT];
            bool u[PPT], any = false;
#pragma unroll
            for (int h = 0; h < NH; h++) {
                float2 t, dy;
                const float2 p = power_pair(dx, ly[h], s_b[k], s_c[k], s_d[k], t, dy);
                P[2 * h] = p.x;
                P[2 * h + 1] = p.y;
            }
#pragma unroll
            for (int i = 0; i < PPT; i++) {
                u[i] = P[i] >= va.y && P[i] >= lim[i];
                any = any || u[i];
            }
            if (!any) continue;
#pragma unroll
            for (int i = 0; i < PPT; i++) {
                float& Ti = i & 1 ? T[i / 2].y : T[i / 2].x;
                const float alpha = fminf(0.99f, va.z * expf(P[i]));
                u[i] = u[i] && !(alpha < 1.0f / 255.0f);
                const float Tn = __fmul_rn(Ti, __fsub_rn(1.0f, alpha));
                const bool stop = Tn < 1e-4f;
                if (u[i] && stop) lim[i] = INF;
                if (u[i] && !stop) {
                    Ti = Tn;
                    last[i] = (int)(start + k);
                }
            }
        }
    }
    __syncthreads();
    int top = -1;
#pragma unroll
    for (int i = 0; i < PPT; i++) top = max(top, last[i]);
    top = __reduce_max_sync(0xffffffffu, top);
    if (lane == 0 && top >= 0) atomicMax(&s_last, top);
    float2 G[NH][3], S[NH];
#pragma unroll
    for (int h = 0; h < NH; h++) {
        const size_t plane = (size_t)W * H, o = (size_t)(py + 2 * h) * W + px;
        const bool in0 = px < W && py + 2 * h < H, in1 = px < W && py + 2 * h + 1 < H;
#pragma unroll
        for (int c = 0; c < 3; c++)
            G[h][c] = make_float2(in0 ? a.dL_dimg[c * plane + o] : 0.0f, in1 ? a.dL_dimg[c * plane + o + W] : 0.0f);
        S[h].x = (G[h][0].x * a.cam.bg[0] + G[h][1].x * a.cam.bg[1] + G[h][2].x * a.cam.bg[2]) * T[h].x;
        S[h].y = (G[h][0].y * a.cam.bg[0] + G[h][1].y * a.cam.bg[1] + G[h][2].y * a.cam.bg[2]) * T[h].y;
    }
    __syncthreads();
    const int block_last = s_last;
    if (block_last < 0) return;

    // 2) back to front over the same pairs
    float2 R[NH][3]; // SINGLY: the colour behind the pair
    if constexpr (SINGLY)
#pragma unroll
        for (int h = 0; h < NH; h++)
#pragma unroll
            for (int c = 0; c < 3; c++) R[h][c] = make_float2(a.cam.bg[c] * T[h].x, a.cam.bg[c] * T[h].y);
    const unsigned first_batch = range.x + (((unsigned)block_last - range.x) / NT) * NT;
    for (long long start = first_batch; start >= (long long)range.x; start -= NT) {
        __syncthreads();
        if ((unsigned)start + th < range.y) stage((unsigned)start + th, block_last);
        __syncthreads();
        const int cnt = (int)min((long long)NT, (long long)top + 1 - start); // the warp's last pair
        for (int k = cnt - 1; k >= 0; k--) {
            const int jj = (int)start + k;
            const float4 va = s_a[k];
            const float dx = __fsub_rn(lx, va.x);
            float2 P[NH], t[NH], dy[NH];
            bool u[PPT], any = false;
#pragma unroll
            for (int h = 0; h < NH; h++) {
                P[h] = power_pair(dx, ly[h], s_b[k], s_c[k], s_d[k], t[h], dy[h]);
                u[2 * h] = P[h].x >= va.y && jj <= last[2 * h];
                u[2 * h + 1] = P[h].y >= va.y && jj <= last[2 * h + 1];
                any = any || u[2 * h] || u[2 * h + 1];
            }
            if (!__any_sync(0xffffffffu, any)) continue;
            float v[9];
#pragma unroll
            for (int g = 0; g < 9; g++) v[g] = 0.0f;
            if constexpr (SINGLY) {
                const float4 c = s_rgb[k];
                const float rgb[3] = {c.x, c.y, c.z};
#pragma unroll
                for (int i = 0; i < PPT; i++) {
                    auto of = [&](float2& x) -> float& { return i & 1 ? x.y : x.x; };
                    const int h = i / 2;
                    const float e = expf(of(P[h])), oe = va.z * e, alpha = fminf(0.99f, oe);
                    if (!u[i] || alpha < 1.0f / 255.0f) continue;
                    const float inv = __frcp_rn(1.0f - alpha);
                    const float Ti = of(T[h]) *= inv, w = alpha * Ti;
                    float dal = 0.0f;
#pragma unroll
                    for (int g = 0; g < 3; g++) {
                        dal += of(G[h][g]) * (rgb[g] * Ti - of(R[h][g]) * inv);
                        of(R[h][g]) += rgb[g] * w;
                        v[6 + g] += of(G[h][g]) * w;
                    }
                    if (oe > 0.99f) continue; // clamped
                    const float dp = dal * alpha, ti = of(t[h]), dyi = of(dy[h]);
                    v[0] += dp * ti;
                    v[1] += dp * dyi;
                    v[2] += dp * ti * ti;
                    v[3] += dp * ti * dyi;
                    v[4] += dp * dyi * dyi;
                    v[5] += dal * e;
                }
            } else if (any) {
                const float4 c = s_rgb[k];
#pragma unroll
                for (int h = 0; h < NH; h++) {
                    // alpha of the pair's pixels (0 where the pixel skips it: T and S stay), and what
                    // multiplies dL/dalpha in dL/dp and dL/do (0 where alpha is clamped)
                    float al[2], ap[2], eo[2], inv[2];
#pragma unroll
                    for (int i = 0; i < 2; i++) {
                        const float e = expf(i ? P[h].y : P[h].x), oe = va.z * e, alpha = fminf(0.99f, oe);
                        const bool use = u[2 * h + i] && !(alpha < 1.0f / 255.0f);
                        al[i] = use ? alpha : 0.0f;
                        ap[i] = oe > 0.99f ? 0.0f : al[i];
                        eo[i] = use && !(oe > 0.99f) ? e : 0.0f;
                        inv[i] = __frcp_rn(1.0f - al[i]);
                    }
                    const float2 vi = make_float2(inv[0], inv[1]);
                    T[h] = __fmul2_rn(T[h], vi); // in front of the pair
                    const float2 w = __fmul2_rn(make_float2(al[0], al[1]), T[h]);
                    const float2 gc = __ffma2_rn(G[h][2], make_float2(c.z, c.z),
                                                 __ffma2_rn(G[h][1], make_float2(c.y, c.y),
                                                            __fmul2_rn(G[h][0], make_float2(c.x, c.x))));
                    const float2 si = __fmul2_rn(S[h], vi);
                    const float2 dal = __ffma2_rn(gc, T[h], make_float2(-si.x, -si.y));
                    S[h] = __ffma2_rn(gc, w, S[h]);
                    const float2 dp = __fmul2_rn(dal, make_float2(ap[0], ap[1]));
                    const float2 dt = __fmul2_rn(dp, t[h]), dd = __fmul2_rn(dp, dy[h]);
                    v[0] += dt.x + dt.y;
                    v[1] += dd.x + dd.y;
                    v[2] += fmaf(dt.x, t[h].x, dt.y * t[h].y);
                    v[3] += fmaf(dt.x, dy[h].x, dt.y * dy[h].y);
                    v[4] += fmaf(dd.x, dy[h].x, dd.y * dy[h].y);
                    v[5] += fmaf(dal.x, eo[0], dal.y * eo[1]);
#pragma unroll
                    for (int g = 0; g < 3; g++) v[6 + g] += fmaf(G[h][g].x, w.x, G[h][g].y * w.y);
                }
            }
            float ninth;
            const float sum = warp_sum9(v, ninth);
            // lanes 0, 4, .. 28 add the first eight sums, lane 1 the ninth: neighbouring words
            float* const out = a.gbuf + (size_t)__float_as_uint(va.w) * GBUF;
            if ((lane & 3) == 0) atomicAdd(out + (lane >> 2), sum);
            else if (lane == 1) atomicAdd(out + 8, ninth);
        }
    }
}

template <int PPT>
__global__ void __launch_bounds__(256 / PPT) k_raster_backward(BackwardArgs a)
{
    grid_dependency_wait();
    if (*a.singly) return;
    backward_tile<PPT, false>(a, (int)ordered_tile(a.tile_order, blockIdx.x));
}

// Its work in a frame of such a dL/dimage. (A choice within one kernel takes 92 registers instead of 72: 1080p 987 -> 1,028 us.)
__global__ void __launch_bounds__(128) k_raster_backward_singly(BackwardArgs a)
{
    grid_dependency_wait();
    if (!*a.singly) return;
    const unsigned tiles = (unsigned)(a.tiles_x * a.tiles_y);
    for (unsigned b = blockIdx.x; b < tiles; b += gridDim.x) {
        backward_tile<2, true>(a, (int)ordered_tile(a.tile_order, b));
        __syncthreads(); // the staged records are written again
    }
}

// Clears the sums, and sees whether the pairs' sums will do: they take the pixel that skips a Gaussian with weight 0, which is
// nothing only while every factor is finite. |G| and |G . bg| up to about 1e30 are enough (colours lie in [0, 1], the weights
// add up to at most 1, 1 / (1 - alpha) is at most 100).
__global__ void __launch_bounds__(256) k_backward_begin(BackwardArgs a, float limit)
{
    grid_dependency_wait();
    const long long stride = (long long)gridDim.x * 256, i0 = (long long)blockIdx.x * 256 + threadIdx.x;
    float4* const sums = reinterpret_cast<float4*>(a.gbuf);
#pragma unroll 4
    for (long long i = i0; i < a.n * (GBUF / 4); i += stride) sums[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    const long long values = 3ll * a.cam.W * a.cam.H;
    bool large = false;
#pragma unroll 4
    for (long long i = i0; i < values; i += stride) large |= !(fabsf(a.dL_dimg[i]) <= limit);
    if (large) *a.singly = 1u;
}

// gradient of the real SH basis (polynomial form; the tangential projection of the
// view direction removes the normal component)
__device__ __forceinline__ void sh_basis_grad(float x, float y, float z, float gx[16], float gy[16], float gz[16])
{
    const float k1 = 0.4886025119029199f, k2a = 1.0925484305920792f, k20 = 0.31539156525252005f;
    const float k22 = 0.5462742152960396f, k33 = 0.5900435899266435f, k32 = 2.890611442640554f;
    const float k31 = 0.4570457994644658f, k30 = 0.3731763325901154f, k32b = 1.445305721320277f;
#pragma unroll
    for (int k = 0; k < 16; k++) gx[k] = gy[k] = gz[k] = 0.f;
    gy[1] = k1;
    gz[2] = k1;
    gx[3] = k1;
    gx[4] = k2a * y; gy[4] = k2a * x;
    gy[5] = k2a * z; gz[5] = k2a * y;
    gz[6] = 6.f * k20 * z;
    gx[7] = k2a * z; gz[7] = k2a * x;
    gx[8] = 2.f * k22 * x; gy[8] = -2.f * k22 * y;
    gx[9] = 6.f * k33 * x * y; gy[9] = 3.f * k33 * (x * x - y * y);
    gx[10] = k32 * y * z; gy[10] = k32 * x * z; gz[10] = k32 * x * y;
    gy[11] = k31 * (5.f * z * z - 1.f); gz[11] = 10.f * k31 * y * z;
    gz[12] = k30 * (15.f * z * z - 3.f);
    gx[13] = k31 * (5.f * z * z - 1.f); gz[13] = 10.f * k31 * x * z;
    gx[14] = 2.f * k32b * x * z; gy[14] = -2.f * k32b * y * z; gz[14] = k32b * (x * x - y * y);
    gx[15] = 3.f * k33 * (x * x - y * y); gy[15] = -6.f * k33 * x * y;
}

// A block's SH rows travel through shared memory both ways, so that the 192-byte rows are read and
// written coalesced (row pitch 49: no bank conflicts); each thread reading and writing its own rows
// moved a sector per word. 500 k Gaussians: 340 -> 51 us (0.26 GB: 0.75 of the measured HBM rate).
constexpr int PB_THREADS = 128, PB_PITCH = 49;

__global__ void __launch_bounds__(PB_THREADS) k_preprocess_backward(BackwardArgs a)
{
    __shared__ float s_sh[PB_THREADS * PB_PITCH];
    grid_dependency_wait();
    const long long base = (long long)blockIdx.x * PB_THREADS;
    const long long i = base + threadIdx.x;
    const int rows = (int)min((long long)PB_THREADS, a.n - base);
    const float* const shp = a.sh + 48 * base;
    for (int j = threadIdx.x; j < rows * 12; j += PB_THREADS) {
        const float4 f = __ldg(reinterpret_cast<const float4*>(shp) + j);
        float* const d = &s_sh[(j / 12) * PB_PITCH + 4 * (j % 12)];
        d[0] = f.x;
        d[1] = f.y;
        d[2] = f.z;
        d[3] = f.w;
    }
    __syncthreads();
    float dm[3] = {0.f, 0.f, 0.f}, ds[3] = {0.f, 0.f, 0.f}, dq[4] = {0.f, 0.f, 0.f, 0.f}, dop = 0.f;
    float* const sh = &s_sh[threadIdx.x * PB_PITCH]; // the Gaussian's SH, then its gradient
    if (i < a.n && a.touched[i] == 0) { // emitted no entry: no pixel depends on it
#pragma unroll
        for (int k = 0; k < 48; k++) sh[k] = 0.f;
    } else if (i < a.n) {
        const float4* const gp = reinterpret_cast<const float4*>(a.gbuf + (size_t)GBUF * i);
        const float4 g0 = gp[0], g1 = gp[1];
        const float gb = a.gbuf[(size_t)GBUF * i + 8];
        dop = g1.y;
        const CamDev& c = a.cam;
        const float mx = a.means[3 * i], my = a.means[3 * i + 1], mz = a.means[3 * i + 2];
        const float s[3] = {a.scales[3 * i], a.scales[3 * i + 1], a.scales[3 * i + 2]};
        const float4 q4 = *reinterpret_cast<const float4*>(a.quats + 4 * i);
        const float qr[4] = {q4.x, q4.y, q4.z, q4.w};
        float p[3];
#pragma unroll
        for (int r = 0; r < 3; r++) p[r] = c.R[3 * r] * mx + c.R[3 * r + 1] * my + c.R[3 * r + 2] * mz + c.t[r];
        const float qnorm = sqrtf(qr[0] * qr[0] + qr[1] * qr[1] + qr[2] * qr[2] + qr[3] * qr[3]);
        const float w = qr[0] / qnorm, x = qr[1] / qnorm, y = qr[2] / qnorm, z = qr[3] / qnorm;
        float Q[9];
        Q[0] = 1.f - 2.f * (y * y + z * z); Q[1] = 2.f * (x * y - w * z);     Q[2] = 2.f * (x * z + w * y);
        Q[3] = 2.f * (x * y + w * z);     Q[4] = 1.f - 2.f * (x * x + z * z); Q[5] = 2.f * (y * z - w * x);
        Q[6] = 2.f * (x * z - w * y);     Q[7] = 2.f * (y * z + w * x);     Q[8] = 1.f - 2.f * (x * x + y * y);
        float M[9];
#pragma unroll
        for (int r = 0; r < 3; r++)
#pragma unroll
            for (int k = 0; k < 3; k++) M[3 * r + k] = Q[3 * r + k] * s[k];
        const float iz = 1.0f / p[2];
        const float xz = p[0] * iz, yz = p[1] * iz;
        const bool inx = xz > -c.limx && xz < c.limx, iny = yz > -c.limy && yz < c.limy;
        const float cxz = fminf(c.limx, fmaxf(-c.limx, xz)), cyz = fminf(c.limy, fmaxf(-c.limy, yz));
        const float J00 = c.fx * iz, J02 = -c.fx * cxz * iz, J11 = c.fy * iz, J12 = -c.fy * cyz * iz;
        float A2[6];
#pragma unroll
        for (int k = 0; k < 3; k++) {
            A2[k] = J00 * c.R[k] + J02 * c.R[6 + k];
            A2[3 + k] = J11 * c.R[3 + k] + J12 * c.R[6 + k];
        }
        float U[6];
#pragma unroll
        for (int r = 0; r < 2; r++)
#pragma unroll
            for (int k = 0; k < 3; k++)
                U[3 * r + k] = A2[3 * r] * M[k] + A2[3 * r + 1] * M[3 + k] + A2[3 * r + 2] * M[6 + k];
        const float sa = U[0] * U[0] + U[1] * U[1] + U[2] * U[2] + 0.3f;
        const float sc = U[3] * U[3] + U[4] * U[4] + U[5] * U[5] + 0.3f;
        const float sb = U[0] * U[3] + U[1] * U[4] + U[2] * U[5];
        // det Sigma' by the Lagrange identity |U0 x U1|^2 + 0.3 (|U0|^2 + |U1|^2) + 0.09, as the
        // forward computes it (sa sc - sb^2 cancels for thin Gaussians)
        const float x0 = U[1] * U[5] - U[2] * U[4], x1 = U[2] * U[3] - U[0] * U[5], x2 = U[0] * U[4] - U[1] * U[3];
        const float det = x0 * x0 + x1 * x1 + x2 * x2 + 0.3f * (sa + sc - 0.6f) + 0.09f;
        // K d = (A t, dy / Sigma'_yy - c A t) for a pixel offset d: dL/d(u, v) = sum dL/dp K d and
        // dL/dSigma' = 1/2 sum dL/dp (K d)(K d)^T
        const float A = sc / det, cc = sb / sc, isc = 1.0f / sc, cA = cc * A;
        const float g_u = A * g0.x, g_v = isc * g0.y - cA * g0.x;
        const float tt = g0.z, ty = g0.w, yy = g1.x;
        const float H00 = 0.5f * A * A * tt, H01 = 0.5f * (A * isc * ty - A * cA * tt);
        const float H11 = 0.5f * (isc * isc * yy - 2.0f * cA * isc * ty + cA * cA * tt);
        // dL/dU = 2 H U
        float dU[6];
#pragma unroll
        for (int k = 0; k < 3; k++) {
            dU[k] = 2.f * (H00 * U[k] + H01 * U[3 + k]);
            dU[3 + k] = 2.f * (H01 * U[k] + H11 * U[3 + k]);
        }
        // U = A2 M: dA2 = dU M^T, dM = A2^T dU
        float dA2[6], dM[9];
#pragma unroll
        for (int r = 0; r < 2; r++)
#pragma unroll
            for (int k = 0; k < 3; k++)
                dA2[3 * r + k] = dU[3 * r] * M[3 * k] + dU[3 * r + 1] * M[3 * k + 1] + dU[3 * r + 2] * M[3 * k + 2];
#pragma unroll
        for (int r = 0; r < 3; r++)
#pragma unroll
            for (int k = 0; k < 3; k++) dM[3 * r + k] = A2[r] * dU[k] + A2[3 + r] * dU[3 + k];
        // M = Q diag(s)
        float dQ[9];
#pragma unroll
        for (int k = 0; k < 3; k++) ds[k] = dM[k] * Q[k] + dM[3 + k] * Q[3 + k] + dM[6 + k] * Q[6 + k];
#pragma unroll
        for (int r = 0; r < 3; r++)
#pragma unroll
            for (int k = 0; k < 3; k++) dQ[3 * r + k] = dM[3 * r + k] * s[k];
        // rotation of the unit quaternion (w, x, y, z)
        float dqn[4];
        dqn[0] = 2.f * (-z * dQ[1] + y * dQ[2] + z * dQ[3] - x * dQ[5] - y * dQ[6] + x * dQ[7]);
        dqn[1] = 2.f * (y * dQ[1] + z * dQ[2] + y * dQ[3] - 2.f * x * dQ[4] - w * dQ[5] + z * dQ[6] + w * dQ[7] -
                        2.f * x * dQ[8]);
        dqn[2] = 2.f * (-2.f * y * dQ[0] + x * dQ[1] + w * dQ[2] + x * dQ[3] + z * dQ[5] - w * dQ[6] + z * dQ[7] -
                        2.f * y * dQ[8]);
        dqn[3] = 2.f * (-2.f * z * dQ[0] - w * dQ[1] + x * dQ[2] + w * dQ[3] - 2.f * z * dQ[4] + y * dQ[5] + x * dQ[6] +
                        y * dQ[7]);
        const float qn[4] = {w, x, y, z};
        const float dotq = qn[0] * dqn[0] + qn[1] * dqn[1] + qn[2] * dqn[2] + qn[3] * dqn[3];
#pragma unroll
        for (int k = 0; k < 4; k++) dq[k] = (dqn[k] - qn[k] * dotq) / qnorm;
        // A2 = J W: dJ = dA2 W^T (only the four non-zero entries of J)
        const float dJ00 = dA2[0] * c.R[0] + dA2[1] * c.R[1] + dA2[2] * c.R[2];
        const float dJ02 = dA2[0] * c.R[6] + dA2[1] * c.R[7] + dA2[2] * c.R[8];
        const float dJ11 = dA2[3] * c.R[3] + dA2[4] * c.R[4] + dA2[5] * c.R[5];
        const float dJ12 = dA2[3] * c.R[6] + dA2[4] * c.R[7] + dA2[5] * c.R[8];
        float dp[3];
        const float iz2 = iz * iz;
        dp[0] = g_u * c.fx * iz + (inx ? dJ02 * (-c.fx * iz2) : 0.f);
        dp[1] = g_v * c.fy * iz + (iny ? dJ12 * (-c.fy * iz2) : 0.f);
        dp[2] = -g_u * c.fx * p[0] * iz2 - g_v * c.fy * p[1] * iz2 - dJ00 * c.fx * iz2 - dJ11 * c.fy * iz2 +
                dJ02 * (inx ? 2.f * c.fx * p[0] * iz2 * iz : c.fx * cxz * iz2) +
                dJ12 * (iny ? 2.f * c.fy * p[1] * iz2 * iz : c.fy * cyz * iz2);
#pragma unroll
        for (int k = 0; k < 3; k++) dm[k] = c.R[k] * dp[0] + c.R[3 + k] * dp[1] + c.R[6 + k] * dp[2];
        // colour = clamp(sum_k Y_k(d) SH_k + 0.5)
        const float vx = mx - c.campos[0], vy = my - c.campos[1], vz = mz - c.campos[2];
        const float vn = sqrtf(vx * vx + vy * vy + vz * vz);
        const float dx = vx / vn, dy = vy / vn, dz = vz / vn;
        const int nk = (a.sh_degree + 1) * (a.sh_degree + 1);
        float Y[16];
        sh_basis(dx, dy, dz, Y);
        const float gch[3] = {g1.z, g1.w, gb};
        float gc[3]; // dL/dcolour, 0 for a clamped channel
#pragma unroll
        for (int ch = 0; ch < 3; ch++) {
            float raw = 0.5f;
#pragma unroll
            for (int k = 0; k < 16; k++)
                if (k < nk) raw += Y[k] * sh[3 * k + ch];
            gc[ch] = raw > 0.0f && raw < 1.0f ? gch[ch] : 0.0f;
        }
        float gx[16], gy[16], gz[16], gd[3] = {0.f, 0.f, 0.f};
        sh_basis_grad(dx, dy, dz, gx, gy, gz);
#pragma unroll
        for (int k = 0; k < 16; k++) {
            float e = 0.0f;
#pragma unroll
            for (int ch = 0; ch < 3; ch++) {
                if (k < nk) e += gc[ch] * sh[3 * k + ch];
                sh[3 * k + ch] = k < nk ? Y[k] * gc[ch] : 0.0f;
            }
            gd[0] += e * gx[k];
            gd[1] += e * gy[k];
            gd[2] += e * gz[k];
        }
        const float dd = gd[0] * dx + gd[1] * dy + gd[2] * dz; // tangential part / |v|
        dm[0] += (gd[0] - dd * dx) / vn;
        dm[1] += (gd[1] - dd * dy) / vn;
        dm[2] += (gd[2] - dd * dz) / vn;
    }
    if (i < a.n) {
#pragma unroll
        for (int k = 0; k < 3; k++) {
            a.dmeans[3 * i + k] = dm[k];
            a.dscales[3 * i + k] = ds[k];
        }
#pragma unroll
        for (int k = 0; k < 4; k++) a.dquats[4 * i + k] = dq[k];
        a.dopac[i] = dop;
    }
    __syncthreads();
    float* const out = a.dsh + 48 * base;
    for (int j = threadIdx.x; j < rows * 48; j += PB_THREADS) out[j] = s_sh[(j / 48) * PB_PITCH + j % 48];
}

void launch_raster_backward(const BackwardArgs& a, cudaStream_t s)
{
    const unsigned tiles = (unsigned)(a.tiles_x * a.tiles_y);
    float bg = 1.0f;
    for (int c = 0; c < 3; c++) bg = fmaxf(bg, fabsf(a.cam.bg[c]));
    const long long work = a.n * (GBUF / 4) + 3ll * a.cam.W * a.cam.H, blocks = (work + 1023) / 1024, all = 8ll * device_sm_count();
    launch_dependent(k_backward_begin, dim3((unsigned)(blocks < all ? blocks : all)), dim3(256), 0, s, a, 1e30f / bg);
    // the forward's rule (launch_raster_exact): a small image's tiles (475 at 400x304) want more warps per tile (two / four
    // pixels per thread: autograd step 1.94 / 2.00 ms), 1080p fewer sums over warps (1.04 / 1.01 ms)
    if (tiles <= 16u * (unsigned)device_sm_count()) launch_dependent(k_raster_backward<2>, dim3(tiles), dim3(128), 0, s, a);
    else launch_dependent(k_raster_backward<4>, dim3(tiles), dim3(64), 0, s, a);
    const unsigned most = 8u * (unsigned)device_sm_count();
    launch_dependent(k_raster_backward_singly, dim3(tiles < most ? tiles : most), dim3(128), 0, s, a);
}

void launch_preprocess_backward(const BackwardArgs& a, cudaStream_t s)
{
    if (a.n <= 0) return;
    launch_dependent(k_preprocess_backward, dim3((unsigned)((a.n + PB_THREADS - 1) / PB_THREADS)), dim3(PB_THREADS), 0, s, a);
}

} // namespace rg
