// frontend.cu -- front ends of the renderer and the scene conversion kernels.
//
//  * k_frontend_fused: the RoofGS fused preprocess + duplicate + key kernel
//    (Sec. IV-A.3): one thread per Gaussian (taken in quantized-depth order
//    when the Gaussians were sorted by depth first) projects, culls, decodes
//    INT8 SH (Eq. (8)) and FP16 geometry (Sec. IV-A.1), computes the snug box
//    and the 32-bit tile|quantized-depth key (Sec. IV-A.2, Eq. (9)); the warps
//    then walk the Gaussians' tile rows in parallel (lane k takes the k-th
//    row), keep per row only the tiles the ellipse reaches, and count entries;
//    the block allocates its entries with one shared-memory prefix sum and one
//    device-wide slot (decoupled look-back, ordered by block, so equal keys stay
//    in Gaussian order) and writes the (key or 16-bit tile id, value) array
//    cooperatively: consecutive lanes write consecutive entries (coalesced), whichever
//    Gaussian and row they belong to. Only the raster record and the key-value
//    array go to global memory, besides the digit counts of the entry sort
//    (each tile row is a run of consecutive tile ids; counted per block in
//    shared memory, added to one of a few global copies).
//  * k_frontend_runs: the renderer's default where it applies: the fused kernel's
//    per-Gaussian work, but each tile row of a Gaussian leaves as one run of tile columns;
//    runs.cu writes the entries from those runs, in their final place.
//  * k_depth_keys: quantized depth and index of every Gaussian, the input of
//    the per-Gaussian depth sort, and the digit counts of that sort.
//  * k_exact_depth_keys, k_exact_runs: the plain 3DGS front end over tile-row runs, in
//    the order of the float depth; k_exact_preprocess -> k_exact_scan ->
//    k_exact_duplicate: the same entries one by one with 64-bit keys of 32-bit tile id |
//    32-bit float depth (Sec. II-A), for tile grids too large for runs.
//  * scene conversion: finite-value check, per-(degree, channel) max |SH|,
//    and the compact attribute encoder.
#include <atomic>

#include "rg_internal.cuh"

namespace rg {

__device__ __forceinline__ float h_lo(unsigned w) { return __half2float(__ushort_as_half((unsigned short)(w & 0xffffu))); }
__device__ __forceinline__ float h_hi(unsigned w) { return __half2float(__ushort_as_half((unsigned short)(w >> 16))); }

// signed INT8 code j (0..47) of a 48-byte code block held in 12 words
__device__ __forceinline__ float sh_code(const unsigned (&w)[12], int j)
{
    return (float)(((int)(w[j >> 2] << (24 - 8 * (j & 3)))) >> 24);
}

__device__ __forceinline__ int sh_band(int k) { return k == 0 ? 0 : (k < 4 ? 1 : (k < 9 ? 2 : 3)); }

// two FP32 values rounded to FP16 (round to nearest even), packed low | high << 16
__device__ __forceinline__ unsigned pack_h2(float lo, float hi)
{
    return (unsigned)__half_as_ushort(__float2half_rn(lo)) | ((unsigned)__half_as_ushort(__float2half_rn(hi)) << 16);
}

// ---------------------------------------------------------------------------
// Fused front end (RoofGS)
// ---------------------------------------------------------------------------
#ifndef RG_FE_THREADS
#define RG_FE_THREADS 256
#endif
constexpr int FE_THREADS = RG_FE_THREADS;
constexpr int FE_WARPS = FE_THREADS / 32;
constexpr int RADIX_FE = 256;

// Adds the digits of the w consecutive tiles t0 .. t0 + w - 1 to the block's
// digit counts: pass 0 digit t & 255 (difference array: +1 where a run of digits
// starts, -1 after it ends, full cycles of 256 added to every digit via entry 0),
// pass 1 digit t >> 8 (t < 2^16).
__device__ __forceinline__ void count_tile_digits(unsigned* s_d0, unsigned* s_h1, int passes, unsigned t0, unsigned w)
{
    const unsigned full = w >> 8, r = w & 255u;
    if (full) atomicAdd(&s_d0[0], full);
    if (r) {
        const unsigned d = t0 & 255u, e = d + r;
        atomicAdd(&s_d0[d], 1u);
        if (e < 256u) {
            atomicSub(&s_d0[e], 1u);
        } else if (e > 256u) { // the run wraps past digit 255
            atomicAdd(&s_d0[0], 1u);
            atomicSub(&s_d0[e - 256u], 1u);
        }
    }
    if (passes > 1) {
        const unsigned t1 = t0 + w - 1u, h0 = t0 >> 8, h1 = t1 >> 8;
        if (h0 == h1) {
            atomicAdd(&s_h1[h0], w);
        } else {
            atomicAdd(&s_h1[h0], ((h0 + 1u) << 8) - t0);
            for (unsigned h = h0 + 1u; h < h1; h++) atomicAdd(&s_h1[h], 256u);
            atomicAdd(&s_h1[h1], t1 - (h1 << 8) + 1u);
        }
    }
}

__device__ __forceinline__ unsigned warp_inclusive_scan(unsigned x, int lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// Gaussian i of the fused front ends: culling, projection, colour; its raster record goes to
// rec[at]. Returns whether it lies inside the depth interval and is not too transparent; rt has
// rows if its box is not empty.
__device__ __forceinline__ bool roofgs_project(const FrontendArgs& a, const long long i, const long long at, RowTest& rt,
                                               unsigned& qd)
{
    bool front = false;
    rt.ty0 = 0;
    rt.ty1 = -1; // no rows unless the box is non-empty
    qd = 0;
    if (i < a.n) {
        const float4 ga = __ldg(&a.geoA[i]); // mean, log o
        const float pz = view_z(a.cam, ga.x, ga.y, ga.z);
        // depth interval (Sec. IV-A.2) and opacity culling o >= 1/255
        front = pz > a.cam.zn && pz <= a.cam.zf && ga.w >= -LN255F;
        if (front) {
            const uint4 gb = __ldg(&a.geoB[i]);
            Binned b;
            if (project_bin(a.cam, ga.x, ga.y, ga.z, pz, h_lo(gb.x), h_hi(gb.x), h_lo(gb.y), h_hi(gb.y), h_lo(gb.z),
                            h_hi(gb.z), h_lo(gb.w), true, ga.w, b)) {
                rt = row_test(b);
                qd = quantize_depth(pz, a.cam.zn, a.lay);
                // conic in the paper's (a, b, c) of Eq. (10): b multiplies dx*dy
                const float inv = 1.0f / b.det;
                const float ca = b.sc * inv, cb = -2.0f * b.sb * inv, cc = b.sa * inv;
                // INT8 SH (Eq. (8)) decoded in registers, evaluated per band
                unsigned w[12];
                {
                    const uint4 p0 = __ldg(&a.shq[3 * i]); // one 48-byte block per Gaussian
                    const uint4 p1 = __ldg(&a.shq[3 * i + 1]);
                    const uint4 p2 = __ldg(&a.shq[3 * i + 2]);
                    w[0] = p0.x; w[1] = p0.y; w[2] = p0.z; w[3] = p0.w;
                    w[4] = p1.x; w[5] = p1.y; w[6] = p1.z; w[7] = p1.w;
                    w[8] = p2.x; w[9] = p2.y; w[10] = p2.z; w[11] = p2.w;
                }
                float dx, dy, dz;
                view_dir(a.cam, ga.x, ga.y, ga.z, dx, dy, dz);
                float Y[16];
                sh_basis(dx, dy, dz, Y);
                float acc[4][3];
#pragma unroll
                for (int d = 0; d < 4; d++) acc[d][0] = acc[d][1] = acc[d][2] = 0.0f;
#pragma unroll
                for (int k = 0; k < 16; k++)
#pragma unroll
                    for (int ch = 0; ch < 3; ch++)
                        acc[sh_band(k)][ch] = fmaf(Y[k], sh_code(w, 3 * k + ch), acc[sh_band(k)][ch]);
                const float g = a.per_gauss_scale ? h_hi(gb.w) : 1.0f;
                float rgb[3];
#pragma unroll
                for (int ch = 0; ch < 3; ch++) {
                    float sum = a.band_scale[ch] * acc[0][ch];
                    sum = fmaf(a.band_scale[3 + ch], acc[1][ch], sum);
                    sum = fmaf(a.band_scale[6 + ch], acc[2][ch], sum);
                    sum = fmaf(a.band_scale[9 + ch], acc[3][ch], sum);
                    rgb[ch] = clamp01(fmaf(g, sum, 0.5f));
                }
                a.rec[2 * at] = make_float4(b.u, b.v, ca, cb);
                a.rec[2 * at + 1] = make_float4(cc, ga.w, __uint_as_float(pack_h2(rgb[0], rgb[1])),
                                               __uint_as_float(pack_h2(rgb[2], 0.0f)));
            }
        }
    }
    return front;
}

// One block of the fused front end: virtual block vb (blocks of a view are numbered in
// the order they claimed work, so every predecessor of the ordered allocation is
// running or done) of the view described by a.
__device__ __forceinline__ void frontend_block(const FrontendArgs& a, const unsigned vb)
{
    __shared__ unsigned s_wsum[FE_WARPS];
    __shared__ RowTestS s_rt[FE_THREADS];   // per-row test of each thread's Gaussian
    __shared__ unsigned s_q[FE_THREADS];    // quantized depth, Eq. (9)
    __shared__ unsigned s_id[FE_THREADS];   // Gaussian index of each slot
    __shared__ unsigned s_cnt[FE_THREADS];  // entries of each slot's Gaussian
    __shared__ unsigned long long s_base;
    // digit counts of the block's entries for the entry sort (8-bit digits of the
    // tile id): pass 0 as a difference array over the digits (tile rows are runs of
    // consecutive tiles), pass 1 as plain counts
    __shared__ unsigned s_d0[RADIX_FE + 1], s_h1[RADIX_FE];

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (a.hist_passes)
        for (int j = tid; j < 2 * RADIX_FE + 1; j += FE_THREADS) (j <= RADIX_FE ? s_d0[j] : s_h1[j - RADIX_FE - 1]) = 0u;
    __syncthreads();
    const long long slot = (long long)vb * FE_THREADS + tid;
    // Gaussian of this slot: slots follow depth order when an order is given, so
    // the entries come out sorted by depth and only the tile bits remain to sort
    const long long i = slot < a.n ? (a.order ? (long long)a.order[slot] : slot) : a.n;

    RowTest rt;
    unsigned qd;
    const bool front = roofgs_project(a, i, i, rt, qd);
    s_rt[tid] = shared_row_test(rt);
    s_q[tid] = qd;
    s_id[tid] = (unsigned)i;
    __syncwarp();

    // Entries per Gaussian. The warp's Gaussians have rows_l tile rows each; the
    // warp walks all of its rows 32 at a time (lane k takes the k-th row of the
    // chunk, whichever Gaussian it belongs to) and adds each row's width to its
    // Gaussian's count with a shared-memory atomic (measured faster than a
    // segmented warp reduction: a chunk's rows belong to few Gaussians).
    const int rows_l = rt.ty1 - rt.ty0 + 1 > 0 ? rt.ty1 - rt.ty0 + 1 : 0;
    const unsigned rincl = warp_inclusive_scan((unsigned)rows_l, lane);
    const unsigned rexcl = rincl - (unsigned)rows_l;
    const unsigned wrows = __shfl_sync(0xffffffffu, rincl, 31);
    s_cnt[tid] = 0u;
    __syncwarp();
    for (unsigned r0 = 0; r0 < wrows; r0 += 32) {
        const unsigned k = r0 + (unsigned)lane;
        int owner = 0; // Gaussian (lane) of warp row k
#pragma unroll
        for (int step = 16; step > 0; step >>= 1)
            if (__shfl_sync(0xffffffffu, rincl, owner + step - 1) <= k) owner += step;
        const unsigned rl = k - __shfl_sync(0xffffffffu, rexcl, owner);
        unsigned w = 0;
        int txa, txb;
        const int ty = k < wrows ? s_rt[warp * 32 + owner].ty0 + (int)rl : 0;
        if (k < wrows && row_range(s_rt[warp * 32 + owner], ty, a.cam.tw_log2, a.cam.th, txa, txb))
            w = (unsigned)(txb - txa + 1);
        if (w) {
            atomicAdd(&s_cnt[warp * 32 + owner], w);
            if (a.hist_passes)
                count_tile_digits(s_d0, s_h1, a.hist_passes, (unsigned)ty * (unsigned)a.lay.tiles_x + (unsigned)txa, w);
        }
    }
    __syncwarp();
    const unsigned cnt = s_cnt[tid];
    // block-level prefix sum of the entry counts
    const unsigned x = warp_inclusive_scan(cnt, lane);
    if (lane == 31) s_wsum[warp] = x;
    const int nfront = __syncthreads_count(front);
    const int nvis = __syncthreads_count(cnt > 0);
    if (warp == 0) {
        unsigned ws = lane < FE_WARPS ? s_wsum[lane] : 0u;
        ws = warp_inclusive_scan(ws, lane);
        if (lane < FE_WARPS) s_wsum[lane] = ws; // inclusive warp totals
    }
    __syncthreads();
    const unsigned block_total = s_wsum[FE_WARPS - 1];

    // one device-wide allocation per block, ordered by block
    if (warp == 0) {
        const unsigned long long base =
            lookback_exclusive(a.status, vb, (unsigned long long)block_total, a.ctr, a.sticky, ERR_FE_LOOKBACK);
        if (lane == 0) {
            s_base = base;
            if (nvis) atomicAdd(&a.ctr->n_visible, (unsigned)nvis);
            if (nfront) atomicAdd(&a.ctr->n_front, (unsigned)nfront);
            const unsigned nblocks = (unsigned)((a.n + FE_THREADS - 1) / FE_THREADS);
            if (vb == nblocks - 1) {
                const unsigned long long total = base + block_total;
                a.ctr->n_entries_total = total;
                a.ctr->n_entries = (unsigned)(total < (unsigned long long)a.cap ? total : (unsigned long long)a.cap);
            }
            if (base + block_total > (unsigned long long)a.cap) {
                atomicOr(&a.ctr->overflow, 1u);
                atomicOr(&a.sticky->overflow, 1u);
            }
        }
    }
    __syncthreads();
    const unsigned long long base = s_base;

    // Emission: the warp's entries are contiguous and in (Gaussian, row, tile)
    // order, so the warp walks its rows again 32 at a time, scans the row
    // widths, and writes 32 consecutive entries per store instruction (lane e
    // finds the row of its entry with a 5-step search over the scan and takes
    // the row's first tile, depth and Gaussian from that lane).
    const int b_d = a.lay.b_d;
    const unsigned tiles_x = (unsigned)a.lay.tiles_x;
    unsigned long long out = base + (warp ? s_wsum[warp - 1] : 0u); // the warp's first entry
    for (unsigned r0 = 0; r0 < wrows; r0 += 32) {
        const unsigned k = r0 + (unsigned)lane;
        int owner = 0;
#pragma unroll
        for (int step = 16; step > 0; step >>= 1)
            if (__shfl_sync(0xffffffffu, rincl, owner + step - 1) <= k) owner += step;
        const unsigned rl = k - __shfl_sync(0xffffffffu, rexcl, owner);
        unsigned w = 0, tb = 0, q = 0, id = 0;
        if (k < wrows) {
            const RowTestS& G = s_rt[warp * 32 + owner];
            const int ty = G.ty0 + (int)rl;
            int txa, txb;
            if (row_range(G, ty, a.cam.tw_log2, a.cam.th, txa, txb)) {
                w = (unsigned)(txb - txa + 1);
                tb = (unsigned)ty * tiles_x + (unsigned)txa; // tile of the row's first entry
            }
            q = s_q[warp * 32 + owner];
            id = s_id[warp * 32 + owner];
        }
        const unsigned incl = warp_inclusive_scan(w, lane);
        const unsigned chunk = __shfl_sync(0xffffffffu, incl, 31);
        tb -= incl - w; // entry e of the chunk, if in this row, has tile tb + e (mod 2^32)
        // entries at or past the capacity are counted but not written
        const bool fits = out < (unsigned long long)a.cap;
        const unsigned room = fits ? (unsigned)((unsigned long long)a.cap - out) : 0u;
        const unsigned long long o = fits ? out : 0ull;
        unsigned* const kp = a.keys + o;
        unsigned short* const kp16 = a.keys16 ? a.keys16 + o : nullptr;
        unsigned* const vp = a.vals + o;
        for (unsigned e0 = 0; e0 < chunk; e0 += 32) {
            const unsigned e = e0 + (unsigned)lane;
            int pos = 0; // row (lane) of entry e
#pragma unroll
            for (int step = 16; step > 0; step >>= 1)
                if (__shfl_sync(0xffffffffu, incl, pos + step - 1) <= e) pos += step;
            const unsigned tile = __shfl_sync(0xffffffffu, tb, pos) + e;
            const unsigned qe = __shfl_sync(0xffffffffu, q, pos);
            const unsigned ide = __shfl_sync(0xffffffffu, id, pos);
            if (e < chunk && e < room) {
                if (a.keys16) kp16[e] = (unsigned short)tile;
                else kp[e] = (b_d >= 32) ? qe : ((tile << b_d) | qe);
                vp[e] = ide;
            }
        }
        out += chunk;
    }

    // The block's digit counts (complete since the barriers after the count
    // loop) go to one copy of the frame's histograms: the last warp turns the
    // difference array into counts, 8 digits per lane.
    if (a.hist_passes && warp == FE_WARPS - 1) {
        unsigned* const H = a.hist + (size_t)(vb % FE_HIST_COPIES) * (2 * RADIX_FE);
        unsigned c[8], run = 0;
#pragma unroll
        for (int j = 0; j < 8; j++) {
            run += s_d0[8 * lane + j];
            c[j] = run;
        }
        const unsigned incl = warp_inclusive_scan(run, lane);
        const unsigned before = incl - run;
#pragma unroll
        for (int j = 0; j < 8; j++)
            if (c[j] + before) atomicAdd(&H[8 * lane + j], c[j] + before);
        if (a.hist_passes > 1) {
#pragma unroll
            for (int j = 0; j < 8; j++) {
                const unsigned v = s_h1[8 * lane + j];
                if (v) atomicAdd(&H[RADIX_FE + 8 * lane + j], v);
            }
        }
    }
}

// Full occupancy (64 warps per SM, 32 registers): the kernel is latency-bound on
// its depth-ordered gathers and shuffles, and 8 blocks of 256 threads per SM
// measured 0.41 ms at 4K against 0.52 ms at 4 blocks per SM (61 registers)
__global__ void __launch_bounds__(FE_THREADS, 2048 / FE_THREADS) k_frontend_fused(FrontendArgs a)
{
    __shared__ unsigned s_vb;
    grid_dependency_wait();
    if (threadIdx.x == 0) s_vb = atomicAdd(&a.ctr->fe_block_ctr, 1u);
    __syncthreads();
    frontend_block(a, s_vb);
}

// Every view of a batch in one grid: a block claims the next of all views' blocks
// (views in order, each view's blocks in order) and runs it with that view's
// arguments, read from the kernel's parameter space.
__global__ void __launch_bounds__(FE_THREADS, 2048 / FE_THREADS)
    k_frontend_views(const __grid_constant__ FrontendViews m)
{
    __shared__ unsigned s_g;
    grid_dependency_wait();
    if (threadIdx.x == 0) s_g = atomicAdd(m.claim, 1u);
    __syncthreads();
    const unsigned g = s_g;
    int v = 0;
    while (v + 1 < m.n_views && m.block_prefix[v + 1] <= g) v++;
    frontend_block(m.views[v], g - m.block_prefix[v]);
}

void launch_frontend_views(const FrontendViews& m, cudaStream_t s)
{
    const unsigned blocks = m.block_prefix[m.n_views];
    if (blocks == 0) return;
    launch_dependent(k_frontend_views, dim3(blocks), dim3(FE_THREADS), 0, s, m);
}

// the depth key of Gaussian i: its quantized depth (Eq. (9)), or the bits of its float depth (positive
// floats order as their bits); a culled Gaussian comes last
__device__ __forceinline__ unsigned depth_key(const FrontendArgs& a, long long i)
{
    const float4 ga = __ldg(&a.geoA[i]);
    const float pz = view_z(a.cam, ga.x, ga.y, ga.z);
    const bool front = pz > a.cam.zn && pz <= a.cam.zf && ga.w >= -LN255F;
    return front ? quantize_depth(pz, a.cam.zn, a.lay) : a.lay.qmax;
}
__device__ __forceinline__ unsigned depth_key(const ExactArgs& a, long long i)
{
    const float pz = view_z(a.cam, a.means[3 * i], a.means[3 * i + 1], a.means[3 * i + 2]);
    return pz > a.cam.zn && pz <= a.cam.zf ? __float_as_uint(pz) : 0xffffffffu;
}

// Grid-stride over the Gaussians; each block also counts the 8-bit digits of its
// keys for the depth sort's passes in shared memory and adds them to `hist`
// ([passes][256], zeroed beforehand) once at the end. Few large blocks: every block's
// counts meet in the same 1,024 words (eight blocks of 256 threads per SM took 24.6 / 15.5 us for 3 M /
// 500 k Gaussians, two of 1,024 take 13.7 / 6.5).
constexpr int DK_THREADS = 1024;

static unsigned depth_key_blocks(long long n)
{
    const long long need = (n + DK_THREADS - 1) / DK_THREADS, most = 2ll * device_sm_count();
    return (unsigned)(need < 1 ? 1 : (need < most ? need : most));
}

__global__ void __launch_bounds__(DK_THREADS) k_depth_keys(FrontendArgs a, unsigned* keys, unsigned* vals, Counters* ctr,
                                                    unsigned* hist, int passes, unsigned* status0,
                                                    long long status_words)
{
    __shared__ unsigned s_h[4][256];
    grid_dependency_wait();
    for (int j = threadIdx.x; j < 4 * 256; j += DK_THREADS) (&s_h[0][0])[j] = 0u;
    // the look-back status of the depth sort's first pass (no histogram kernel runs before it)
    for (long long j = (long long)blockIdx.x * DK_THREADS + threadIdx.x; j < status_words; j += (long long)gridDim.x * DK_THREADS)
        status0[j] = 0u;
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x == 0) ctr->n_entries = (unsigned)a.n;
#pragma unroll 4
    for (long long i = (long long)blockIdx.x * DK_THREADS + threadIdx.x; i < a.n; i += (long long)gridDim.x * DK_THREADS) {
        const unsigned q = depth_key(a, i);
        keys[i] = q;
        vals[i] = (unsigned)i;
        for (int p = 0; p < passes; p++) atomicAdd(&s_h[p][(q >> (8 * p)) & 255u], 1u);
    }
    __syncthreads();
    for (int j = threadIdx.x; j < passes * 256; j += DK_THREADS) {
        const unsigned c = (&s_h[0][0])[j];
        if (c) atomicAdd(&hist[j], c);
    }
}

void launch_depth_keys(const FrontendArgs& a, unsigned* keys, unsigned* vals, Counters* ctr, unsigned* hist,
                       int passes, unsigned* status0, cudaStream_t s)
{
    launch_dependent(k_depth_keys, dim3(depth_key_blocks(a.n)), dim3(DK_THREADS), 0, s, a, keys, vals, ctr, hist, passes, status0,
                     sort_status_words(4, a.n));
}

int frontend_block_threads() { return FE_THREADS; }

void launch_frontend_fused(const FrontendArgs& a, cudaStream_t s)
{
    if (a.n <= 0) return;
    const unsigned blocks = (unsigned)((a.n + FE_THREADS - 1) / FE_THREADS);
    launch_dependent(k_frontend_fused, dim3(blocks), dim3(FE_THREADS), 0, s, a);
}

// ---------------------------------------------------------------------------
// Front end of a frame of tile-row runs (at most RUN_MAX_GRID x RUN_MAX_GRID tiles)
// ---------------------------------------------------------------------------
// The fused kernel allocates every block's entries in order and writes them one by one, and the
// sort then moves them twice. Here a block writes one 4-byte run per tile row of a Gaussian, its
// runs grouped by tile row and in slot order within a row, at a place that need not be ordered;
// runs.cu gathers them by tile row and writes each entry once, in its final place.
// Records and values are indexed by slot (depth order), so a block's records go out together.
static_assert(FE_THREADS == RUN_SLOTS, "one slot per thread");
constexpr int RUN_CACHE = 256;  // tile rows of a warp kept from the counting walk to the placing one

// dynamic shared memory of a front-end block, per tile row
struct RunRowSmem {
    unsigned mask[FE_WARPS]; // which slots have a run in the row (one word per warp)
    unsigned ents;           // their entries
    unsigned first;          // first run of the row in the block's list
    unsigned char before[8]; // runs of the earlier warps (at most 7 x 32)
};
static_assert(FE_WARPS == 8, "the earlier warps' runs fit a byte");

// Emits the runs of a block: every thread holds rows_l tile rows of its slot's Gaussian;
// range(owner thread, row, ty, txa, txb) gives the owner's row-th tile row and its tile columns
// (false: none). Returns the warp's mask of Gaussians with an entry. Every thread calls it.
// stage: FE_WARPS * RUN_CACHE words of shared memory that range reads but nothing else does: where
// the warps' rows were all kept, range is not called again and the runs go out through it. (Shared
// memory is scarce here: what it leaves of the L1 holds the depth-ordered gathers. With 8 KB of its
// own for the runs the kernel took 309 us at 4K.)
template <class F>
__device__ __forceinline__ unsigned emit_runs(const RunArgs& r, const unsigned vb, const int rows_l, unsigned* const stage,
                                              F range)
{
    extern __shared__ __align__(16) unsigned char run_smem[];
    RunRowSmem* const R = reinterpret_cast<RunRowSmem*>(run_smem);
    __shared__ unsigned s_cache[FE_WARPS][RUN_CACHE]; // owner | ty << 5 | first << 14 | last << 23
    constexpr unsigned NO_TILES = 1u << 14; // first 1, last 0: no run has it (every one of the 32 bits is used: a run of
                                            // lane 31 in the last tile of a 512 x 512 grid is ~0)
    __shared__ unsigned s_w[FE_WARPS];
    __shared__ unsigned s_base;
    static_assert(RUN_MAX_GRID <= 512, "nine bits for a tile row or column");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int j = tid; j < r.rows * (int)(sizeof(RunRowSmem) / 4); j += FE_THREADS) reinterpret_cast<unsigned*>(R)[j] = 0u;
    __syncthreads(); // also: the row tests of all slots are in shared memory
    const unsigned rincl = warp_inclusive_scan((unsigned)rows_l, lane);
    const unsigned rexcl = rincl - (unsigned)rows_l;
    const unsigned wrows = __shfl_sync(0xffffffffu, rincl, 31);
    // the warp's tile rows, 32 at a time: lane k takes the k-th, whichever Gaussian it belongs to
    auto tiles_of = [&](unsigned k) {
        int owner = 0; // Gaussian (lane) of warp row k
#pragma unroll
        for (int step = 16; step > 0; step >>= 1)
            if (__shfl_sync(0xffffffffu, rincl, owner + step - 1) <= k) owner += step;
        const unsigned rl = k - __shfl_sync(0xffffffffu, rexcl, owner);
        int ty, txa, txb;
        if (k < wrows && range(warp * 32 + owner, (int)rl, ty, txa, txb))
            return (unsigned)owner | ((unsigned)ty << 5) | ((unsigned)txa << 14) | ((unsigned)txb << 23);
        return NO_TILES;
    };
    unsigned vis = 0;
    for (unsigned r0 = 0; r0 < wrows; r0 += 32) {
        const unsigned v = tiles_of(r0 + (unsigned)lane);
        if (r0 + 32 <= RUN_CACHE) s_cache[warp][r0 + lane] = v;
        if (v != NO_TILES) {
            const unsigned owner = v & 31u, ty = (v >> 5) & 511u;
            atomicOr(&R[ty].mask[warp], 1u << owner);
            atomicAdd(&R[ty].ents, (v >> 23) - ((v >> 14) & 511u) + 1u);
            vis |= 1u << owner;
        }
    }
    const bool staged = __syncthreads_count(wrows > RUN_CACHE) == 0;
    unsigned total = 0;
    for (int g = 0; g < r.rows; g += FE_THREADS) {
        const int row = g + tid;
        unsigned n = 0, lo = 0, hi = 0;
        if (row < r.rows)
#pragma unroll
            for (int q = 0; q < FE_WARPS; q++) {
                if (q < 4) lo |= n << (8 * q);
                else hi |= n << (8 * (q - 4));
                n += (unsigned)__popc(R[row].mask[q]);
            }
        unsigned x = warp_inclusive_scan(n, lane);
        if (lane == 31) s_w[warp] = x;
        __syncthreads();
        unsigned all = 0;
#pragma unroll
        for (int q = 0; q < FE_WARPS; q++) {
            if (q < warp) x += s_w[q];
            all += s_w[q];
        }
        if (row < r.rows) {
            R[row].first = total + x - n;
            *reinterpret_cast<uint2*>(R[row].before) = make_uint2(lo, hi);
        }
        total += all;
        __syncthreads();
    }
    if (tid == 0) {
        // any free part of the run buffer; a block that finds none (only when the frame's entries
        // exceed the workspace too) leaves its runs out
        const unsigned long long at = atomicAdd(&r.ctr->n_runs, (unsigned long long)total);
        s_base = at + total <= (unsigned long long)r.run_cap ? (unsigned)at : 0xffffffffu;
    }
    __syncthreads();
    const unsigned base = s_base;
    const bool ok = base != 0xffffffffu;
    for (int row = tid; row < r.rows; row += FE_THREADS) {
        const unsigned n = (row + 1 < r.rows ? R[row + 1].first : total) - R[row].first;
        const size_t at = (size_t)row * r.blocks + vb;
        r.cnt[at] = R[row].ents | (ok ? n << RUN_CNT_SHIFT : 0u);
        if (r.tot && R[row].ents) atomicAdd(&r.tot[row], (unsigned long long)R[row].ents | ((unsigned long long)(ok ? n : 0u) << RUN_TOT_SHIFT));
        if (n) r.seg[at] = base + R[row].first;
    }
    if (ok) {
        for (unsigned r0 = 0; r0 < wrows; r0 += 32) {
            const unsigned v = r0 + 32 <= RUN_CACHE ? s_cache[warp][r0 + lane] : tiles_of(r0 + (unsigned)lane);
            if (v == NO_TILES) continue;
            const unsigned owner = v & 31u;
            const RunRowSmem& q = R[(v >> 5) & 511u];
            const unsigned pos = q.first + q.before[warp] + (unsigned)__popc(q.mask[warp] & ((1u << owner) - 1u));
            const unsigned w = run_pack((unsigned)warp * 32u + owner, (v >> 14) & 511u, v >> 23);
            if (staged) stage[pos] = w;
            else r.runs[base + pos] = w;
        }
        if (staged) {
            __syncthreads();
            for (unsigned j = (unsigned)tid; j < total; j += FE_THREADS) r.runs[base + j] = stage[j];
        }
    }
    return __reduce_or_sync(0xffffffffu, vis);
}

// the depth sort's error bits, which are the frame's too (one thread of the grid reads them)
__device__ __forceinline__ unsigned depth_error(const RunArgs& r)
{
    return blockIdx.x == 0 && threadIdx.x == 0 ? r.depth_ctr->error : 0u;
}

// Resident blocks per SM: 5 (48 registers). What shared memory leaves of the L1 holds the depth-ordered
// gathers, so more blocks cost more than they hide, above all with the per-row words of 8K: 4 / 5 / 6
// blocks 213 / 196 / 207 us at 4K, 105 / 101 / 130 us at 8K, 37 / 33 / 33 us at 1080p. The tile rows found
// by the counting walk are kept for the placing one (8 KB; 217 -> 201 us at 4K against walking twice).
__global__ void __launch_bounds__(FE_THREADS, 5) k_frontend_runs(FrontendArgs a, RunArgs r)
{
    __shared__ RowTestS s_rt[FE_THREADS];
    static_assert(sizeof(s_rt) >= FE_WARPS * RUN_CACHE * 4, "the runs are staged over the row tests");
    grid_dependency_wait();
    const int tid = threadIdx.x;
    const long long slot = (long long)blockIdx.x * FE_THREADS + tid;
    const long long i = slot < a.n ? (long long)a.order[slot] : a.n;
    const unsigned error = depth_error(r); // (loaded early, used late)
    RowTest rt;
    unsigned qd;
    const bool front = roofgs_project(a, i, slot, rt, qd);
    const int rows_l = rt.ty1 >= rt.ty0 ? rt.ty1 - rt.ty0 + 1 : 0;
    if (rows_l) s_rt[tid] = shared_row_test(rt);
    const unsigned vis = emit_runs(r, blockIdx.x, rows_l, reinterpret_cast<unsigned*>(s_rt), [&](int t, int k, int& ty, int& txa, int& txb) {
        const RowTestS& G = s_rt[t];
        ty = G.ty0 + k;
        return row_range(G, ty, a.cam.tw_log2, a.cam.th, txa, txb);
    });
    const int nfront = __syncthreads_count(front);
    const int nvis = __syncthreads_count((vis >> (tid & 31)) & 1u);
    if (tid == 0) {
        if (nvis) atomicAdd(&a.ctr->n_visible, (unsigned)nvis);
        if (nfront) atomicAdd(&a.ctr->n_front, (unsigned)nfront);
        if (error) atomicOr(&a.ctr->error, error);
    }
}

// the shared memory of the largest tile grids needs the opt-in (once per device and kernel; setting it
// twice does no harm)
template <typename K>
static void run_smem_opt_in(K kernel, std::atomic<bool> (&opted)[64])
{
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && opted[dev].load()) return;
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, RUN_MAX_GRID * (int)sizeof(RunRowSmem));
    if (dev >= 0 && dev < 64) opted[dev].store(true);
}

void launch_frontend_runs(const FrontendArgs& a, const RunArgs& r, cudaStream_t s)
{
    if (r.blocks == 0) return;
    static std::atomic<bool> opted[64];
    run_smem_opt_in(k_frontend_runs, opted);
    launch_dependent(k_frontend_runs, dim3(r.blocks), dim3(FE_THREADS), (size_t)r.rows * sizeof(RunRowSmem), s, a, r);
}

// ---------------------------------------------------------------------------
// Plain 3DGS front end (exact mode)
// ---------------------------------------------------------------------------
constexpr int EX_THREADS = 256;

// The raster record of a Gaussian binned as b: the exponent of Eq. (10) with the quadratic form
// completed in dx, -1/2 ((Sigma'_yy / det) (dx - c dy)^2 + dy^2 / Sigma'_yy), c = Sigma'_xy / Sigma'_yy
// (no cancellation for thin Gaussians), and the mean as double-floats (b's FP32 u, v only bin the
// Gaussian). Where the exponent is undefined, one of 0 and an alpha of 0.99 are written (the rasterizers compare exponents
// before they evaluate alpha): returns whether it is.
__device__ __forceinline__ bool exact_record(const ExactArgs& a, float opacity, const Binned& b, float mx, float my,
                                             float mz, float4& mean, float4& quad)
{
    quad = make_float4(-0.5f * __fdiv_rn(b.sc, b.det), __fdiv_rn(b.sb, b.sc), __fdiv_rn(-0.5f, b.sc), opacity);
    mean = project_mean_df(a.cam, mx, my, mz);
    if (!exact_undefined(mean)) return false;
    mean = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    quad = make_float4(0.0f, 0.0f, 0.0f, 1.0f);
    return true;
}

// Adds the terms of words 4 V0 .. 4 V1 - 1 of a Gaussian's degree-3 SH coefficients (FP32) to its colour
// c; word4(v) gives words 4 v .. 4 v + 3.
template <int V0, int V1, class F>
__device__ __forceinline__ void exact_colour(const float (&Y)[16], int sh_degree, float (&c)[3], F word4)
{
    const int nk = (sh_degree + 1) * (sh_degree + 1);
#pragma unroll
    for (int v4 = V0; v4 < V1; v4++) {
        const float4 f = word4(v4);
        const float e[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const int j = 4 * v4 + u;
            const int k = j / 3, ch = j % 3;
            if (k < nk) c[ch] = fmaf(Y[k], e[u], c[ch]);
        }
    }
}

// Front end in index order: the frames whose tile grid is too large for runs.
__global__ void __launch_bounds__(EX_THREADS) k_exact_preprocess(ExactArgs a)
{
    grid_dependency_wait();
    const long long i = (long long)blockIdx.x * EX_THREADS + threadIdx.x;
    if (i >= a.n) return;
    a.touched[i] = 0;
    const float mx = a.means[3 * i], my = a.means[3 * i + 1], mz = a.means[3 * i + 2];
    const float pz = view_z(a.cam, mx, my, mz);
    const bool front = pz > a.cam.zn && pz <= a.cam.zf;
    const unsigned fm = __ballot_sync(__activemask(), front);
    if (front && __popc(fm & ((1u << (threadIdx.x & 31)) - 1u)) == 0) atomicAdd(&a.ctr->n_front, (unsigned)__popc(fm));
    if (!front) return;
    const float4 q = *reinterpret_cast<const float4*>(&a.quats[4 * i]);
    Binned b;
    const bool vis = project_bin(a.cam, mx, my, mz, pz, q.x, q.y, q.z, q.w, a.scales[3 * i], a.scales[3 * i + 1],
                                 a.scales[3 * i + 2], false, 0.0f, b);
    const unsigned vm = __ballot_sync(__activemask(), vis);
    if (vis && __popc(vm & ((1u << (threadIdx.x & 31)) - 1u)) == 0) atomicAdd(&a.ctr->n_visible, (unsigned)__popc(vm));
    if (!vis) return;
    a.depth[i] = pz;
    a.rect[i] = make_int4(b.tx0, b.ty0, b.tx1, b.ty1);
    a.touched[i] = (unsigned)((b.tx1 - b.tx0 + 1) * (b.ty1 - b.ty0 + 1));
    const bool undefined = exact_record(a, a.opac[i], b, mx, my, mz, a.rec[3 * i], a.rec[3 * i + 1]);
    float dx, dy, dz, Y[16], c[3] = {0.5f, 0.5f, 0.5f};
    view_dir(a.cam, mx, my, mz, dx, dy, dz);
    sh_basis(dx, dy, dz, Y);
    const float4* const shp = reinterpret_cast<const float4*>(a.sh + 48 * i);
    exact_colour<0, 12>(Y, a.sh_degree, c, [&](int v) { return shp[v]; });
    a.rec[3 * i + 2] = make_float4(clamp01(c[0]), clamp01(c[1]), clamp01(c[2]), undefined ? 1.0f : 0.0f);
}

__global__ void __launch_bounds__(DK_THREADS) k_exact_depth_keys(ExactArgs a, unsigned* keys, unsigned* vals, Counters* ctr,
                                                          unsigned* hist, unsigned* status0, long long status_words)
{
    __shared__ unsigned s_h[4][256];
    grid_dependency_wait();
    for (int j = threadIdx.x; j < 4 * 256; j += DK_THREADS) (&s_h[0][0])[j] = 0u;
    for (long long j = (long long)blockIdx.x * DK_THREADS + threadIdx.x; j < status_words; j += (long long)gridDim.x * DK_THREADS)
        status0[j] = 0u;
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x == 0) ctr->n_entries = (unsigned)a.n;
#pragma unroll 4
    for (long long i = (long long)blockIdx.x * DK_THREADS + threadIdx.x; i < a.n; i += (long long)gridDim.x * DK_THREADS) {
        const unsigned k = depth_key(a, i);
        keys[i] = k;
        vals[i] = (unsigned)i;
#pragma unroll
        for (int p = 0; p < 4; p++) atomicAdd(&s_h[p][(k >> (8 * p)) & 255u], 1u);
    }
    __syncthreads();
    for (int j = threadIdx.x; j < 4 * 256; j += DK_THREADS) {
        const unsigned c = (&s_h[0][0])[j];
        if (c) atomicAdd(&hist[j], c);
    }
}

// Which tiles of a Gaussian's rectangle hold a pixel of alpha >= 1/255, from the rasterizer's own
// record: -p = kx^-1 t^2 + sz dy^2 (t = dx - c dy) has to be at most `level` = ln(255 o). The level is
// raised and the extents are widened by more than the FP32 rounding of this test and of
// exact_power(), so no pair that the rasterizer would blend is lost:
//  * exact_power() forms t from dx and c dy, each at most rx = sqrt(2 level Sigma'_xx) on the
//    contour, with a rounding of 2^-23 of each; p then moves by at most 2 sqrt(level / kx) times that, and
//    1 / kx = Sigma'_yy / (2 det) <= 1 / 0.6 by the dilation: 2.2e-6 rx. The level is raised by 0.01 + 1e-5 rx;
//  * the extents below carry a few roundings of |u| + rx (2^-23 each); they are widened by 1/16 + 1e-5 (|u| + rx).
// The pixels of a tile outside the rectangle's 3-sigma box count too, as the rasterizer evaluates them.
struct ExactRow {
    float u, v, level, kx, sz, c, ys, padx, pady;
    int tx0, tx1, ty0;
};

__device__ __forceinline__ ExactRow exact_row(const Binned& b, const float4& mean, const float4& quad, bool undefined,
                                              bool& any)
{
    ExactRow r;
    const float ext = sqrtf(12.0f * fmaxf(b.sa, b.sc)); // at least sqrt(2 level Sigma'_xx), level <= ln 255
    r.level = LN255F + logf(quad.w) + 0.01f + 1e-5f * ext;
    r.u = mean.x;
    r.v = mean.z;
    if (undefined) { // blends in every tile of the rectangle: NaN keeps them all
        r.u = r.v = __int_as_float(0x7fffffff);
        r.level = __int_as_float(0x7f800000);
    }
    any = r.level > 0.0f;
    r.kx = -1.0f / quad.x;
    r.sz = -quad.z;
    r.c = quad.y;
    r.ys = r.c * sqrtf(r.level / (r.sz * (r.kx * r.sz + r.c * r.c))); // dy of the right-most point
    r.padx = 0.0625f + 1e-5f * (fabsf(r.u) + ext);
    r.pady = 0.0625f + 1e-5f * (fabsf(r.v) + ext);
    r.tx0 = b.tx0;
    r.tx1 = b.tx1;
    r.ty0 = b.ty0;
    return r;
}

// the tiles [txa, txb] of tile row ty; false if none. Comparisons are written so that a NaN keeps tiles.
__device__ __forceinline__ bool exact_row_range(const ExactRow& g, int ty, const CamDev& cam, int& txa, int& txb)
{
    const float d0 = (float)(ty * cam.th) - g.v - g.pady, d1 = (float)(ty * cam.th + cam.th - 1) - g.v + g.pady;
    const float near = fmaxf(fmaxf(d0, -d1), 0.0f); // the band's least |dy|
    if (g.sz * near * near > g.level) return false;
    const float yr = fminf(fmaxf(g.ys, d0), d1), yl = fminf(fmaxf(-g.ys, d0), d1);
    const float xr = g.u + g.c * yr + sqrtf(fmaxf(g.level - g.sz * yr * yr, 0.0f) * g.kx) + g.padx;
    const float xl = g.u + g.c * yl - sqrtf(fmaxf(g.level - g.sz * yl * yl, 0.0f) * g.kx) - g.padx;
    const float a0 = fmaxf(ceilf(xl), 0.0f), a1 = fminf(floorf(xr), (float)(cam.W - 1)); // NaN: the whole row
    if (a0 > a1) return false;
    txa = max((int)a0 >> cam.tw_log2, g.tx0);
    txb = min((int)a1 >> cam.tw_log2, g.tx1);
    return txa <= txb;
}

// The front end of an exact frame of runs: one slot (Gaussian in depth order) per thread. Its record
// goes to its slot; the frame's entries are counted by the rectangles (plain 3DGS's entries), while the
// runs leave out the tiles where the Gaussian stays below 1/255 (about two thirds of the entries at
// 4K), which the rasterizer would skip pixel by pixel. Bound by its depth-ordered gathers (240 B per
// Gaussian), which fill the L1 pipe (0.78 of its wavefronts) before HBM: 418 us at 4K with 3 M Gaussians with
// every attribute array gathered by itself, 374 with the geometry in one 48-byte row (three or five
// blocks per SM: 434 / 374), 321 with the SH rows fetched asynchronously as below as well (three / five: 351 /
// 407). It replaced an index-ordered preprocessing of 265 us and pays for that many times: with
// the entries in depth order no 64-bit key is written or sorted, and the whole exact frame went from 13.3 to
// 2.1 ms (4K, 3 M), 1.40 to 0.50 ms (1080p, 500 k) by it.
__global__ void __launch_bounds__(FE_THREADS, 4) k_exact_runs(ExactArgs a, RunArgs r, int keep_all)
{
    // the warps' SH rows, half a row at a time; then the slots' row tests
    constexpr int SH_HALF = 24, SH_PITCH = 28; // words (the pitch: 16-byte reads without bank conflicts)
    __shared__ __align__(16) float s_sh[FE_WARPS][32 * SH_PITCH];
    ExactRow* const s_row = reinterpret_cast<ExactRow*>(s_sh);
    __shared__ unsigned long long s_sum[FE_WARPS];
    static_assert(sizeof(s_sh) >= FE_THREADS * sizeof(ExactRow) && sizeof(s_sh) >= FE_WARPS * RUN_CACHE * 4,
                  "the row tests, then the staged runs, lie over the SH rows");
    grid_dependency_wait();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long slot = (long long)blockIdx.x * FE_THREADS + tid;
    bool front = false, vis = false;
    int rows_l = 0;
    unsigned tiles = 0;
    const unsigned error = depth_error(r); // (loaded early, used late)
    const unsigned ordered = slot < a.n ? a.order[slot] : 0xffffffffu;
    const bool here = ordered < (unsigned long long)a.n; // (a slot that a timed-out depth sort left out holds anything)
    const unsigned i = here ? ordered : 0u;
    // The colour's SH rows (192 bytes each, in depth order anywhere in memory) come asynchronously, half a
    // row at a time, six lanes to a row; each thread reads its own from shared memory. A thread loading its
    // own row touched 32 lines with every instruction, which filled the L1 pipe.
    auto fetch = [&](unsigned rows, int half) {
#pragma unroll
        for (int it = 0; it < 6; it++) {
            const int q = it * 32 + lane, g = q / 6, part = q % 6;
            const unsigned j = __shfl_sync(0xffffffffu, i, g);
            if ((rows >> g) & 1u) {
                const unsigned dst = (unsigned)__cvta_generic_to_shared(&s_sh[warp][g * SH_PITCH + 4 * part]);
                const float* src = a.sh + 48 * (size_t)j + SH_HALF * half + 4 * part;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst), "l"(src) : "memory");
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    auto arrived = [&]() {
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        __syncwarp();
    };
    const float4 m = here ? __ldg(&a.geo[3 * (size_t)i]) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    const float pz = view_z(a.cam, m.x, m.y, m.z);
    front = here && pz > a.cam.zn && pz <= a.cam.zf;
    fetch(__ballot_sync(0xffffffffu, front), 0);
    Binned b;
    if (front) {
        const float4 q = __ldg(&a.geo[3 * (size_t)i + 1]), s = __ldg(&a.geo[3 * (size_t)i + 2]);
        vis = project_bin(a.cam, m.x, m.y, m.z, pz, q.x, q.y, q.z, q.w, s.x, s.y, s.z, false, 0.0f, b);
    }
    const unsigned seen = __ballot_sync(0xffffffffu, vis);
    const float4* const own = reinterpret_cast<const float4*>(&s_sh[warp][lane * SH_PITCH]);
    float Y[16], c[3] = {0.5f, 0.5f, 0.5f};
    float dx, dy, dz;
    view_dir(a.cam, m.x, m.y, m.z, dx, dy, dz);
    sh_basis(dx, dy, dz, Y);
    arrived();
    if (vis) exact_colour<0, 6>(Y, a.sh_degree, c, [&](int v) { return own[v]; });
    __syncwarp();
    fetch(seen, 1);
    ExactRow row;
    bool any = false, undefined = false;
    if (vis) {
        float4 mean, quad;
        undefined = exact_record(a, m.w, b, m.x, m.y, m.z, mean, quad);
        a.rec[3 * slot] = mean;
        a.rec[3 * slot + 1] = quad;
        a.rect[slot] = make_int4(b.tx0, b.ty0, b.tx1, b.ty1);
        tiles = (unsigned)((b.tx1 - b.tx0 + 1) * (b.ty1 - b.ty0 + 1));
        row = exact_row(b, mean, quad, undefined, any);
        if (any || keep_all) rows_l = b.ty1 - b.ty0 + 1;
    }
    if (here) a.touched[i] = tiles;
    arrived();
    if (vis) {
        exact_colour<6, 12>(Y, a.sh_degree, c, [&](int v) { return own[v - 6]; });
        a.rec[3 * slot + 2] = make_float4(clamp01(c[0]), clamp01(c[1]), clamp01(c[2]), undefined ? 1.0f : 0.0f);
    }
    __syncthreads(); // the row tests lie over the SH rows of other warps
    if (rows_l) s_row[tid] = row;
    emit_runs(r, blockIdx.x, rows_l, reinterpret_cast<unsigned*>(s_row), [&](int t, int k, int& ty, int& txa, int& txb) {
        const ExactRow& G = s_row[t];
        ty = G.ty0 + k;
        if (keep_all) {
            txa = G.tx0;
            txb = G.tx1;
            return true;
        }
        return exact_row_range(G, ty, a.cam, txa, txb);
    });
    unsigned long long sum = tiles;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) s_sum[warp] = sum;
    const int nfront = __syncthreads_count(front);
    const int nvis = __syncthreads_count(vis);
    if (tid == 0) {
        if (nvis) atomicAdd(&a.ctr->n_visible, (unsigned)nvis);
        if (nfront) atomicAdd(&a.ctr->n_front, (unsigned)nfront);
        if (error) atomicOr(&a.ctr->error, error);
        sum = 0;
        for (int q = 0; q < FE_WARPS; q++) sum += s_sum[q];
        if (sum) atomicAdd(&a.ctr->n_entries_total, sum);
    }
}

void launch_exact_depth_keys(const ExactArgs& a, unsigned* keys, unsigned* vals, Counters* ctr, unsigned* hist,
                             unsigned* status0, cudaStream_t s)
{
    launch_dependent(k_exact_depth_keys, dim3(depth_key_blocks(a.n)), dim3(DK_THREADS), 0, s, a, keys, vals, ctr, hist, status0,
                     sort_status_words(4, a.n));
}

void launch_exact_runs(const ExactArgs& a, const RunArgs& r, bool keep_all, cudaStream_t s)
{
    if (r.blocks == 0) return;
    static std::atomic<bool> opted[64];
    run_smem_opt_in(k_exact_runs, opted);
    launch_dependent(k_exact_runs, dim3(r.blocks), dim3(FE_THREADS), (size_t)r.rows * sizeof(RunRowSmem), s, a, r,
                     keep_all ? 1 : 0);
}

constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = EX_THREADS * SCAN_ITEMS;

// Exclusive scan of the tile counts (single pass, decoupled look-back).
__global__ void __launch_bounds__(EX_THREADS) k_exact_scan(ExactArgs a)
{
    __shared__ unsigned s_vb;
    __shared__ unsigned long long s_wsum[EX_THREADS / 32];
    grid_dependency_wait();
    __shared__ unsigned long long s_base;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) s_vb = atomicAdd(&a.ctr->fe_block_ctr, 1u);
    __syncthreads();
    const unsigned vb = s_vb;
    const long long start = (long long)vb * SCAN_TILE + (long long)tid * SCAN_ITEMS;
    unsigned v[SCAN_ITEMS];
    unsigned long long sum = 0;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; k++) {
        v[k] = (start + k < a.n) ? a.touched[start + k] : 0u;
        sum += v[k];
    }
    unsigned long long x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_wsum[warp] = x;
    __syncthreads();
    if (warp == 0) {
        unsigned long long ws = lane < EX_THREADS / 32 ? s_wsum[lane] : 0ull;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, ws, o);
            if (lane >= o) ws += y;
        }
        if (lane < EX_THREADS / 32) s_wsum[lane] = ws;
    }
    __syncthreads();
    const unsigned long long block_total = s_wsum[EX_THREADS / 32 - 1];
    if (warp == 0) {
        const unsigned long long base = lookback_exclusive(a.status, vb, block_total, a.ctr, a.sticky, ERR_SCAN_LOOKBACK);
        if (lane == 0) {
            s_base = base;
            const unsigned nblocks = (unsigned)((a.n + SCAN_TILE - 1) / SCAN_TILE);
            if (vb == nblocks - 1) {
                const unsigned long long total = base + block_total;
                a.ctr->n_entries_total = total;
                a.ctr->n_entries = (unsigned)(total < (unsigned long long)a.cap ? total : (unsigned long long)a.cap);
                if (total > (unsigned long long)a.cap) {
                    atomicOr(&a.ctr->overflow, 1u);
                    atomicOr(&a.sticky->overflow, 1u);
                }
            }
        }
    }
    __syncthreads();
    unsigned long long run = s_base + (x - sum) + (warp ? s_wsum[warp - 1] : 0ull);
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; k++) {
        if (start + k < a.n) a.offsets[start + k] = (unsigned)(run > 0xffffffffull ? 0xffffffffull : run);
        run += v[k];
    }
}

// Duplicate (plain 3DGS, Sec. II-A): one (64-bit key, value) entry per tile of each
// Gaussian's rectangle, at the Gaussian's exclusive-scan offset. The entries of a
// warp's 32 consecutive Gaussians are contiguous and in (Gaussian, row, tile) order,
// so the warp walks their tile rows 32 at a time (lane k takes the k-th row) and
// writes 32 consecutive entries per store instruction, as the fused front end does.
// It also counts the sort's digits: the four depth digits are the same for every
// entry of a Gaussian (one shared atomic each per Gaussian), the tile digits of a
// row are a run of consecutive tile ids (count_tile_digits); the block's counts go
// to one of FE_HIST_COPIES copies once, at the end of its grid-stride loop.
constexpr int DUP_HIST_STRIDE = 8; // passes per copy of the digit counts ([copy][8][256])

__global__ void __launch_bounds__(EX_THREADS) k_exact_duplicate(ExactArgs a)
{
    __shared__ unsigned s_hd[4][RADIX_FE];             // depth digits (key bits 0..31)
    __shared__ unsigned s_d0[RADIX_FE + 1], s_h1[RADIX_FE]; // tile digits (key bits 32..47)
    grid_dependency_wait();
    const int tid = threadIdx.x, lane = tid & 31;
    const bool count = a.hist != nullptr;
    if (count) {
        for (int j = tid; j < 4 * RADIX_FE; j += EX_THREADS) (&s_hd[0][0])[j] = 0u;
        for (int j = tid; j < 2 * RADIX_FE + 1; j += EX_THREADS) (j <= RADIX_FE ? s_d0[j] : s_h1[j - RADIX_FE - 1]) = 0u;
        __syncthreads();
    }
    const unsigned tiles_x = (unsigned)a.lay.tiles_x;
    for (long long base = (long long)blockIdx.x * EX_THREADS; base < a.n; base += (long long)gridDim.x * EX_THREADS) {
        const long long i = base + tid;
        unsigned cnt = 0, zb = 0, off = 0;
        int4 r = make_int4(0, 0, -1, -1);
        if (i < a.n) {
            cnt = a.touched[i];
            off = a.offsets[i];
            if (cnt) {
                r = a.rect[i];
                zb = __float_as_uint(a.depth[i]);
                if (count)
#pragma unroll
                    for (int p = 0; p < 4; p++) atomicAdd(&s_hd[p][(zb >> (8 * p)) & 255u], cnt);
            }
        }
        const int rows_l = cnt ? r.w - r.y + 1 : 0;
        const unsigned width = cnt ? (unsigned)(r.z - r.x + 1) : 0u;
        const unsigned rincl = warp_inclusive_scan((unsigned)rows_l, lane);
        const unsigned rexcl = rincl - (unsigned)rows_l;
        const unsigned wrows = __shfl_sync(0xffffffffu, rincl, 31);
        // the warp's first entry: the offset of its first Gaussian (lanes past n hold the total)
        unsigned long long out = __shfl_sync(0xffffffffu, off, 0);
        for (unsigned r0 = 0; r0 < wrows; r0 += 32) {
            const unsigned k = r0 + (unsigned)lane;
            int owner = 0; // lane (Gaussian) of warp row k
#pragma unroll
            for (int step = 16; step > 0; step >>= 1)
                if (__shfl_sync(0xffffffffu, rincl, owner + step - 1) <= k) owner += step;
            const unsigned rl = k - __shfl_sync(0xffffffffu, rexcl, owner);
            const unsigned ow = __shfl_sync(0xffffffffu, width, owner);
            const int oty = __shfl_sync(0xffffffffu, r.y, owner);
            const int otx = __shfl_sync(0xffffffffu, r.x, owner);
            const unsigned oz = __shfl_sync(0xffffffffu, zb, owner);
            unsigned w = 0, tb = 0;
            if (k < wrows) {
                w = ow;
                tb = (unsigned)(oty + (int)rl) * tiles_x + (unsigned)otx; // tile of the row's first entry
                if (count) count_tile_digits(s_d0, s_h1, a.tile_passes, tb, w);
            }
            const unsigned incl = warp_inclusive_scan(w, lane);
            const unsigned chunk = __shfl_sync(0xffffffffu, incl, 31);
            tb -= incl - w; // entry e of the chunk, if in this row, has tile tb + e
            for (unsigned e0 = 0; e0 < chunk; e0 += 32) {
                const unsigned e = e0 + (unsigned)lane;
                int pos = 0; // row (lane) of entry e
#pragma unroll
                for (int step = 16; step > 0; step >>= 1)
                    if (__shfl_sync(0xffffffffu, incl, pos + step - 1) <= e) pos += step;
                const unsigned tile = __shfl_sync(0xffffffffu, tb, pos) + e;
                const unsigned z = __shfl_sync(0xffffffffu, oz, pos);
                const unsigned gl = (unsigned)__shfl_sync(0xffffffffu, owner, pos);
                const unsigned long long dst = out + e;
                if (e < chunk && dst < (unsigned long long)a.cap) {
                    a.keys[dst] = ((unsigned long long)tile << 32) | z;
                    a.vals[dst] = (unsigned)(base + (long long)(tid & ~31) + gl);
                }
            }
            out += chunk;
        }
    }
    if (count) {
        __syncthreads();
        unsigned* const H = a.hist + (size_t)(blockIdx.x % FE_HIST_COPIES) * (DUP_HIST_STRIDE * RADIX_FE);
        for (int j = tid; j < 4 * RADIX_FE; j += EX_THREADS) {
            const unsigned c = (&s_hd[0][0])[j];
            if (c) atomicAdd(&H[j], c);
        }
        if (tid < 32) { // the tile digits: difference array -> counts, 8 digits per lane
            unsigned c[8], run = 0;
#pragma unroll
            for (int j = 0; j < 8; j++) {
                run += s_d0[8 * lane + j];
                c[j] = run;
            }
            const unsigned incl = warp_inclusive_scan(run, lane);
            const unsigned before = incl - run;
#pragma unroll
            for (int j = 0; j < 8; j++)
                if (c[j] + before) atomicAdd(&H[4 * RADIX_FE + 8 * lane + j], c[j] + before);
        }
        if (a.tile_passes > 1)
            for (int j = tid; j < RADIX_FE; j += EX_THREADS)
                if (s_h1[j]) atomicAdd(&H[5 * RADIX_FE + j], s_h1[j]);
    }
}

void launch_exact_preprocess(const ExactArgs& a, cudaStream_t s)
{
    if (a.n <= 0) return;
    launch_dependent(k_exact_preprocess, dim3((unsigned)((a.n + EX_THREADS - 1) / EX_THREADS)), dim3(EX_THREADS), 0, s, a);
}
void launch_exact_scan(const ExactArgs& a, cudaStream_t s)
{
    if (a.n <= 0) return;
    launch_dependent(k_exact_scan, dim3((unsigned)((a.n + SCAN_TILE - 1) / SCAN_TILE)), dim3(EX_THREADS), 0, s, a);
}
void launch_exact_duplicate(const ExactArgs& a, cudaStream_t s)
{
    if (a.n <= 0) return;
    const long long need = (a.n + EX_THREADS - 1) / EX_THREADS;
    const long long cap = 8ll * device_sm_count(); // grid-stride: digit counts flushed once per block
    launch_dependent(k_exact_duplicate, dim3((unsigned)(need < cap ? need : cap)), dim3(EX_THREADS), 0, s, a);
}

// ---------------------------------------------------------------------------
// Scene conversion (one-off at scene creation)
// ---------------------------------------------------------------------------
__global__ void k_check_attributes(const float* means, const float* scales, const float* quats, const float* opac,
                                   const float* sh, long long n, unsigned* flag)
{
    const long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long stride = (long long)gridDim.x * blockDim.x;
    bool bad = false, range = false;
    auto finite = [&](const float* p, long long count) {
        for (long long i = i0; i < count; i += stride) bad |= !isfinite(p[i]);
    };
    finite(means, 3 * n);
    finite(scales, 3 * n);
    finite(quats, 4 * n);
    finite(sh, 48 * n);
    for (long long i = i0; i < n; i += stride) {
        bad |= !isfinite(opac[i]);
        range |= !(opac[i] >= 0.0f && opac[i] <= 1.0f);
    }
    const unsigned f = __reduce_or_sync(0xffffffffu, (bad ? 1u : 0u) | (range ? 2u : 0u));
    if (f && (threadIdx.x & 31) == 0) atomicOr(flag, f);
}

void launch_check_attributes(const float* means, const float* scales, const float* quats, const float* opac,
                             const float* sh, long long n, unsigned* flag, cudaStream_t s)
{
    if (n <= 0) return;
    long long blocks = (48 * n + 255) / 256;
    if (blocks > 16ll * device_sm_count()) blocks = 16ll * device_sm_count();
    k_check_attributes<<<(unsigned)blocks, 256, 0, s>>>(means, scales, quats, opac, sh, n, flag);
}

__global__ void k_pack_geometry(const float* means, const float* scales, const float* quats, const float* opac,
                                long long n, float4* geo)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    geo[3 * i] = make_float4(means[3 * i], means[3 * i + 1], means[3 * i + 2], opac[i]);
    geo[3 * i + 1] = make_float4(quats[4 * i], quats[4 * i + 1], quats[4 * i + 2], quats[4 * i + 3]);
    geo[3 * i + 2] = make_float4(scales[3 * i], scales[3 * i + 1], scales[3 * i + 2], 0.0f);
}

void launch_pack_geometry(const float* means, const float* scales, const float* quats, const float* opac, long long n,
                          float4* geo, cudaStream_t s)
{
    if (n <= 0) return;
    k_pack_geometry<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(means, scales, quats, opac, n, geo);
}

// max |SH| per (degree, channel): float bits of non-negative values order like integers
__global__ void k_sh_absmax(const float* sh, long long n, unsigned* maxbits)
{
    __shared__ unsigned s_max[12];
    if (threadIdx.x < 12) s_max[threadIdx.x] = 0u;
    __syncthreads();
    unsigned local[12];
#pragma unroll
    for (int k = 0; k < 12; k++) local[k] = 0u;
    const long long total = n * 48;
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < total; j += (long long)gridDim.x * blockDim.x) {
        const int e = (int)(j % 48), k = e / 3, ch = e % 3;
        const unsigned bits = __float_as_uint(fabsf(sh[j]));
        const int slot = sh_band(k) * 3 + ch;
#pragma unroll
        for (int t = 0; t < 12; t++)
            if (t == slot) local[t] = max(local[t], bits);
    }
#pragma unroll
    for (int t = 0; t < 12; t++) atomicMax(&s_max[t], local[t]);
    __syncthreads();
    if (threadIdx.x < 12) atomicMax(&maxbits[threadIdx.x], s_max[threadIdx.x]);
}

void launch_sh_absmax(const float* sh, long long n, unsigned* maxbits, cudaStream_t s)
{
    if (n <= 0) return;
    long long blocks = (n * 48 + 255) / 256;
    if (blocks > 152 * 8) blocks = 152 * 8;
    k_sh_absmax<<<(unsigned)blocks, 256, 0, s>>>(sh, n, maxbits);
}

struct CompactParams {
    float band_scale[12];
    int per_gauss;
};

__global__ void k_compact(const float* means, const float* scales, const float* quats, const float* logo,
                          const float* sh, long long n, CompactParams p, float4* geoA, uint4* geoB, uint4* shq)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float* c = sh + 48 * i;
    float g = 1.0f;
    if (p.per_gauss) {
        float gm = 0.0f;
        for (int e = 0; e < 48; e++) {
            const float s = p.band_scale[sh_band(e / 3) * 3 + e % 3];
            const float den127 = __fmul_rn(127.0f, s);
            const float r = den127 > 0.0f ? __fdiv_rn(fabsf(c[e]), den127) : 0.0f;
            gm = fmaxf(gm, r);
        }
        g = __half2float(__float2half_rn(gm));
    }
    unsigned char codes[48];
    for (int e = 0; e < 48; e++) {
        const float s = p.band_scale[sh_band(e / 3) * 3 + e % 3];
        const float den = p.per_gauss ? __fmul_rn(g, s) : s;
        int q = 0;
        if (den > 0.0f) {
            q = __float2int_rn(__fdiv_rn(c[e], den));
            q = max(-127, min(127, q));
        }
        codes[e] = (unsigned char)(signed char)q;
    }
    for (int pl = 0; pl < 3; pl++) {
        unsigned w[4];
        for (int k = 0; k < 4; k++)
            w[k] = (unsigned)codes[16 * pl + 4 * k] | ((unsigned)codes[16 * pl + 4 * k + 1] << 8) |
                   ((unsigned)codes[16 * pl + 4 * k + 2] << 16) | ((unsigned)codes[16 * pl + 4 * k + 3] << 24);
        shq[3 * i + pl] = make_uint4(w[0], w[1], w[2], w[3]);
    }
    geoA[i] = make_float4(means[3 * i], means[3 * i + 1], means[3 * i + 2], logo[i]);
    geoB[i] = make_uint4(pack_h2(quats[4 * i], quats[4 * i + 1]), pack_h2(quats[4 * i + 2], quats[4 * i + 3]),
                         pack_h2(scales[3 * i], scales[3 * i + 1]), pack_h2(scales[3 * i + 2], g));
}

void launch_compact(const float* means, const float* scales, const float* quats, const float* logo, const float* sh,
                    long long n, const float* band_scale, int per_gauss, float4* geoA, uint4* geoB, uint4* shq,
                    cudaStream_t s)
{
    if (n <= 0) return;
    CompactParams p;
    for (int k = 0; k < 12; k++) p.band_scale[k] = band_scale[k];
    p.per_gauss = per_gauss;
    k_compact<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(means, scales, quats, logo, sh, n, p, geoA, geoB, shq);
}

} // namespace rg
