// runs.cu -- grouping of the frame's entries by tile from tile-row runs.
//
// A Gaussian's entries in one tile row are a run of consecutive tile columns, so the depth-ordered
// Gaussians are a list of runs about a fifth as long as the list of entries, and the entries never
// need to be written before they are in their final place. The front end (emit_runs, frontend.cu)
// leaves each block's runs grouped by tile row, in slot (depth) order within a row, and each (tile
// row, block) count; here
//  * k_run_rows: per tile row, cuts the row's blocks into chunks of at most CHUNK_RUNS runs;
//  * k_run_collect: per chunk, gathers the blocks' runs into one list per tile row and counts the
//    chunk's entries per tile column (a difference array: two shared atomics per run);
//  * k_run_offsets: per tile row, turns the chunks' column counts into the first slot of every
//    (chunk, column) and writes every tile's [start, end): the entries lie in tile-id order;
//  * k_run_expand: per chunk, writes the values (slots) of every column. For every 32 runs and
//    column one word says which of the 32 cover the column: a run toggles its bit at its first
//    column and after its last (two shared atomics), a prefix XOR over the columns fills it in. A
//    warp then takes a column: each lane holds 64 runs' bits, a scan of the bit counts places its
//    values, and the column's values go to consecutive addresses in run (depth) order.
// The order within a tile is that of the stable sort of the 32-bit (or 64-bit) keys, and no key is
// stored, counted or moved.
//
// What bounds it: each run is moved twice (4 B block-local, 8 B by row) and each value written once,
// so HBM is far from busy; k_run_expand, the longest, is bound by issue slots and the latency of its
// shared-memory reads (ncu: 1.8 instructions per cycle with three blocks of 256 threads per SM and a
// column at a time, 405 us at 4K with 3 M Gaussians; five blocks and two columns at a time 281 us).
// Kernel times (ncu) of the front end and the grouping, with every entry written, against the scatter by
// tile row with one radix pass it replaced: 4K, 3 M Gaussians 792 -> 591 us (front end 201, rows 14,
// collect 85, offsets 11, expand 281, in windows of 120 columns; limited frames: expand 175, see k_run_expand); 8K, 1 M, against the fused front end with
// three radix passes 1295 -> 541 us; 1080p,
// 500 k 93 -> 89 us; 256 x 256, 10 k 35 -> 26 us.
#include "rg_internal.cuh"

namespace rg {

constexpr int RUN_THREADS = 256;
constexpr int RUN_WARPS = RUN_THREADS / 32;
constexpr int CHUNK_RUNS = 2048;                // runs of a chunk at most: 64 per lane of a warp
constexpr int CHUNK_STEP = CHUNK_RUNS - RUN_SLOTS; // a chunk ends with the block that reaches this many
constexpr int CHUNK_BLOCKS = 1024;              // blocks of a chunk at most (sparse tile rows)
// tile columns expanded at a time: the most that five blocks per SM leave room for (45 KB each). k_run_offsets and k_run_expand with
// 112 / 120 / 128: 2048 x 1152 37.8 / 37.7 / 35.6 us, 2560 x 1440 46.9 / 47.6 / 46.5, 5120 x 2880 144.4 / 146.3 / 143.5, 4K 71.3 / 69.4 / 68.8,
// 1366 x 768 (86 columns) 25.9 / 25.9 / 25.8; 64 to 88 with five or six blocks took 1 to 3 % more at 4K
constexpr int COLS = 128;
constexpr int PITCH = CHUNK_RUNS / 32 + 2;      // words per column: 64 masks, padded (8-byte loads, no bank conflicts)

// chunks a tile row of a small frame has at most: its row r has chunks r * small_chunks(blocks) and up
__host__ __device__ __forceinline__ unsigned small_chunks(unsigned blocks)
{
    return blocks * (unsigned)RUN_SLOTS / CHUNK_STEP + 1;
}

unsigned run_chunk_cap(unsigned run_cap, int rows, unsigned blocks)
{
    if (blocks <= RUN_SMALL_BLOCKS) return (unsigned)rows * small_chunks(blocks);
    return run_cap / CHUNK_STEP + (unsigned)rows * (blocks / CHUNK_BLOCKS + 2);
}

template <typename T>
__device__ __forceinline__ T run_warp_scan(T x)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// inclusive scan over the block (every thread calls it); s_w: one word per warp; total = the sum
template <int WARPS, typename T>
__device__ __forceinline__ T run_block_scan(T v, T* s_w, T& total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const T x = run_warp_scan(v);
    if (lane == 31) s_w[warp] = x;
    __syncthreads();
    T before = 0, all = 0;
#pragma unroll
    for (int q = 0; q < WARPS; q++) {
        const T t = s_w[q];
        if (q < warp) before += t;
        all += t;
    }
    total = all;
    __syncthreads(); // s_w may be written again after the call
    return x + before;
}

// The chunk of a block with `run` runs of its row before it: a new chunk starts where the runs before
// a block reach the next multiple of CHUNK_STEP (the blocks of a chunk then hold at most CHUNK_STEP -
// 1 + RUN_SLOTS runs) and at every CHUNK_BLOCKS-th block. Where both happen at once an empty chunk
// lies between.
__device__ __forceinline__ unsigned chunk_of(unsigned run, unsigned block)
{
    return run / CHUNK_STEP + block / CHUNK_BLOCKS;
}

// An exact frame beyond its capacity keeps the tiles of the rectangles Gaussian by Gaussian in index order, row by row, as
// the entries that fit are the first ones plain 3DGS duplicates: the Gaussian with which they pass `cap`, and how many of its
// tiles fit. It is one of the `len` from lo on, `before` tiles lie before those. Every thread of the block calls it; s_w: one
// word per warp. A part of the Gaussians per warp, then the part that passes the capacity again, down to a warp's lanes.
template <int WARPS>
__device__ __noinline__ uint2 find_cut(const unsigned* touched, unsigned lo, unsigned len, unsigned long long before,
                                       unsigned long long cap, unsigned long long* s_w)
{
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    while (len > 32) {
        const unsigned part = (len + WARPS - 1) / WARPS, end = lo + len;
        const unsigned w0 = lo + warp * part, w1 = w0 + part < end ? w0 + part : end;
        unsigned long long sum = 0;
#pragma unroll 8
        for (unsigned i = w0 + lane; i < w1; i += 32) sum += touched[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if (lane == 0) s_w[warp] = sum;
        __syncthreads();
        unsigned k = 0;
        while (k + 1 < WARPS && before + s_w[k] <= cap) before += s_w[k++];
        __syncthreads();
        lo += k * part;
        len = lo < end ? (part < end - lo ? part : end - lo) : 0u;
    }
    const unsigned t = lane < len ? touched[lo + lane] : 0u;
    const unsigned long long upto = before + run_warp_scan((unsigned long long)t);
    const int first = __ffs((int)__ballot_sync(0xffffffffu, upto > cap)) - 1; // there is one
    const unsigned fits = (unsigned)(cap - (upto - t));
    return make_uint2(lo + (unsigned)(first < 0 ? 0 : first), __shfl_sync(0xffffffffu, fits, first < 0 ? 0 : first));
}

// find_cut over the blocks of k_run_rows: each adds up a part of the Gaussians, the last one to finish looks into the part that
// passes the capacity. (One block for all of 3 M Gaussians took 0.4 ms.)
template <int WARPS>
__device__ __noinline__ void cut_by_rows(const RunArgs& a, unsigned long long* s_w)
{
    __shared__ bool s_last;
    const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, n = (unsigned)a.n, rows = (unsigned)a.rows;
    const unsigned long long cap = (unsigned long long)a.cap;
    const unsigned part = (n + rows - 1u) / rows, lo = blockIdx.x * part;
    unsigned long long sum = 0;
#pragma unroll 8
    for (unsigned i = threadIdx.x; i < part; i += 32 * WARPS)
        if (lo + i < n) sum += a.touched[lo + i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) s_w[warp] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        sum = 0;
        for (int q = 0; q < WARPS; q++) sum += s_w[q];
        st_volatile_u64(&a.parts[blockIdx.x], sum);
        __threadfence();
        s_last = atomicAdd(&a.ctr->cut_ctr, 1u) == rows - 1u;
        __threadfence();
    }
    __syncthreads();
    if (!s_last) return;
    unsigned k = 0; // the part that passes the capacity
    unsigned long long before = 0;
    for (; k < rows; k += 32) {
        const unsigned long long t = k + lane < rows ? ld_volatile_u64(&a.parts[k + lane]) : 0ull;
        const unsigned long long upto = before + run_warp_scan(t);
        const unsigned over = __ballot_sync(0xffffffffu, upto > cap);
        if (over) {
            const int first = __ffs((int)over) - 1;
            before = __shfl_sync(0xffffffffu, upto - t, first);
            k += (unsigned)first;
            break;
        }
        before = __shfl_sync(0xffffffffu, upto, 31);
    }
    const unsigned from = k * part; // (there is one: k < rows and from < n)
    const uint2 cut = find_cut<WARPS>(a.touched, from, from < n ? (part < n - from ? part : n - from) : 0u, before, cap, s_w);
    if (threadIdx.x == 0) {
        a.ctr->cut = cut.x;
        a.ctr->cut_tiles = cut.y;
    }
}

// One block of 1024 threads per tile row: a scan of the blocks' counts, and the row's chunks.
__global__ void __launch_bounds__(1024, 2) k_run_rows(RunArgs a)
{
    constexpr int WARPS = 32;
    __shared__ unsigned s_r[WARPS];
    __shared__ unsigned long long s_e[WARPS];
    __shared__ unsigned s_chunk;
    grid_dependency_wait();
    const unsigned row = blockIdx.x, tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const unsigned long long boxes = a.box_total ? a.ctr->n_entries_total : 0ull; // (loaded early, used late)
    const unsigned* const cnt = a.cnt + (size_t)row * a.blocks;
    const unsigned per = (a.blocks + 32u * WARPS - 1u) / (32u * WARPS), b0 = tid * per;
    const unsigned b1 = b0 + per < a.blocks ? b0 + per : a.blocks;
    unsigned p = 0, last = 0; // runs of this thread's blocks, of its last block
    unsigned long long e = 0;
#pragma unroll 4
    for (unsigned b = b0; b < b1; b++) {
        const unsigned c = cnt[b];
        last = c >> RUN_CNT_SHIFT;
        p += last;
        e += c & RUN_CNT_ENTRIES;
    }
    const unsigned rx = run_warp_scan(p);
    const unsigned long long ex = run_warp_scan(e);
    if (lane == 31) {
        s_r[warp] = rx;
        s_e[warp] = ex;
    }
    __syncthreads();
    unsigned rbefore = 0, rtot = 0;
    unsigned long long ebefore = 0, etot = 0;
#pragma unroll
    for (int q = 0; q < WARPS; q++) {
        if (q < (int)warp) {
            rbefore += s_r[q];
            ebefore += s_e[q];
        }
        rtot += s_r[q];
        etot += s_e[q];
    }
    const unsigned rend = rbefore + rx; // runs up to the end of this thread's blocks
    if (b0 < b1 && b1 == a.blocks) {    // the thread of the row's last block
        const unsigned n = rtot ? chunk_of(rend - last, a.blocks - 1) + 1 : 0u;
        // where the row's runs and chunks lie does not matter, only that no two rows share a place
        const unsigned base = atomicAdd(&a.ctr->n_row_runs, rtot), chunk = atomicAdd(&a.ctr->n_chunks, n);
        if (!a.box_total && etot) atomicAdd(&a.ctr->n_entries_total, etot);
        a.row[row] = RunRow{chunk, n, base, rtot, etot};
        s_chunk = chunk;
    }
    __syncthreads();
    if (boxes > (unsigned long long)a.cap) cut_by_rows<WARPS>(a, s_e);
    if (!rtot || b0 >= b1) return;
    p = rend - p;
    e = ebefore + ex - e;
    int prev = -1; // chunk of the block before
    if (b0) prev = (int)chunk_of(p - (cnt[b0 - 1] >> RUN_CNT_SHIFT), b0 - 1);
    for (unsigned b = b0; b < b1; b++) {
        const unsigned c = cnt[b];
        a.pre[(size_t)row * a.blocks + b] = p;
        for (const int k = (int)chunk_of(p, b); prev < k;) {
            prev++;
            a.chunk[s_chunk + (unsigned)prev] = RunChunk{b, p, e};
        }
        p += c >> RUN_CNT_SHIFT;
        e += c & RUN_CNT_ENTRIES;
    }
}

// runs of chunk c of a row: [first block, end block), [first run, end run) of the row's list
__device__ __forceinline__ void chunk_bounds(const RunArgs& a, const RunRow& r, unsigned c, RunChunk& k, unsigned& bend,
                                             unsigned& rend)
{
    k = a.chunk[r.chunk + c];
    if (c + 1 < r.nchunks) {
        const RunChunk n = a.chunk[r.chunk + c + 1];
        bend = n.block;
        rend = n.run;
    } else {
        bend = a.blocks;
        rend = r.runs;
    }
}

struct alignas(16) CollectSmem {
    unsigned short own[CHUNK_RUNS];      // block (from the chunk's first) whose runs start at a run, 1-based; 0: none
    int d[RUN_MAX_GRID + 1];             // the columns' difference array
    unsigned from[CHUNK_BLOCKS];         // where run j of the chunk lies, if in the block: from + j
    int w[RUN_WARPS];
};

// The runs of chunk `chunk` of a tile row: front-end blocks [block, bend), runs [run, run + n) of the
// row. A thread takes eight consecutive runs; all its loads are in flight together. Which block a run
// lies in follows from a maximum scan over the blocks' first runs. clip: the frame has more entries
// than the workspace holds. It keeps those whose place in (tile row, slot, column) order lies below the
// capacity; `entry` entries of the frame lie before the chunk then. An exact frame keeps the tiles that come first in
// index order: cut.x, cut.y of find_cut.
__device__ __forceinline__ void collect_chunk(const RunArgs& a, const RunRow& r, unsigned row, unsigned chunk,
                                              unsigned block, unsigned bend, unsigned run, unsigned n, bool clip,
                                              unsigned long long entry, uint2 cut, CollectSmem& S)
{
    constexpr int PER = CHUNK_RUNS / RUN_THREADS;
    const unsigned tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const size_t at = (size_t)row * a.blocks;
    for (int j = (int)tid; j <= a.cols; j += RUN_THREADS) S.d[j] = 0;
    static_assert(CHUNK_RUNS * 2 == RUN_THREADS * 16, "16 bytes of own per thread");
    reinterpret_cast<uint4*>(S.own)[tid] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
#pragma unroll 4
    for (unsigned b = block + tid; b < bend; b += RUN_THREADS) {
        const unsigned first = a.pre[at + b] - run;
        if (a.cnt[at + b] >> RUN_CNT_SHIFT) {
            S.own[first] = (unsigned short)(b - block + 1);
            S.from[b - block] = a.seg[at + b] - first;
        }
    }
    __syncthreads();
    unsigned own[PER]; // block of each run, 1-based (a running maximum)
    {
        const uint4 q = reinterpret_cast<const uint4*>(S.own)[tid];
        const unsigned w[4] = {q.x, q.y, q.z, q.w};
        unsigned m = 0;
#pragma unroll
        for (int u = 0; u < PER; u++) {
            const unsigned o = u & 1 ? w[u >> 1] >> 16 : w[u >> 1] & 0xffffu;
            m = o > m ? o : m;
            own[u] = m;
        }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, m, o);
            if ((int)lane >= o) m = y > m ? y : m;
        }
        if (lane == 31) S.w[warp] = (int)m;
        unsigned before = __shfl_up_sync(0xffffffffu, m, 1);
        if (lane == 0) before = 0;
        __syncthreads();
        for (unsigned k = 0; k < warp; k++) before = (unsigned)S.w[k] > before ? (unsigned)S.w[k] : before;
#pragma unroll
        for (int u = 0; u < PER; u++) own[u] = before > own[u] ? before : own[u];
    }
    const unsigned j0 = PER * tid;
    unsigned v[PER];
#pragma unroll
    for (int u = 0; u < PER; u++) {
        const unsigned j = j0 + (unsigned)u;
        v[u] = j < n ? a.runs[S.from[own[u] - 1] + j] : 0u;
    }
    unsigned room = 0, kept = 0; // clip: entries that still fit before the thread's first run; entries of its runs
    if (clip && !a.box_total) { // (a walk over the runs before each run instead of this scan: frames of half the room 1,407 us at 4K, 275 at 1080p)
        int sum = 0, all;
#pragma unroll
        for (int u = 0; u < PER; u++)
            if (j0 + (unsigned)u < n) sum += (int)(run_last(v[u]) - run_first(v[u]) + 1u);
        __syncthreads(); // S.w is read above
        const unsigned before = (unsigned)(run_block_scan<RUN_WARPS>(sum, S.w, all) - sum);
        const unsigned long long cap = (unsigned long long)a.cap, p = entry + before;
        room = p < cap ? (unsigned)(cap - p) : 0u;
    }
    uint2* const list = a.list + r.base + run;
#pragma unroll
    for (int u = 0; u < PER; u++) {
        const unsigned j = j0 + (unsigned)u;
        if (j >= n) break;
        unsigned ta = run_first(v[u]), tb = run_last(v[u]);
        const unsigned b = block + own[u] - 1;
        if (clip && a.box_total) {
            const unsigned g = a.gauss[b * RUN_SLOTS + run_slot(v[u])];
            if (g >= cut.x) {
                int left = 0; // of the rectangle's tiles in the row, those kept
                if (g == cut.x) {
                    const int4 q = a.rect[b * RUN_SLOTS + run_slot(v[u])];
                    left = (int)cut.y - ((int)row - q.y) * (q.z - q.x + 1) + q.x;
                }
                if (left <= (int)ta) { // an empty run
                    ta = 1;
                    tb = 0;
                } else if ((int)tb >= left) {
                    tb = (unsigned)left - 1u;
                }
            }
        } else if (clip) {
            const unsigned width = tb - ta + 1u, fits = width < room ? width : room;
            tb = ta + fits - 1u;
            if (fits == 0u) { // an empty run
                ta = 1;
                tb = 0;
            }
            room -= fits;
        }
        list[j] = make_uint2(b * RUN_SLOTS + run_slot(v[u]), ta | (tb << 16));
        if (ta <= tb) {
            kept += tb - ta + 1u;
            atomicAdd(&S.d[ta], 1);
            atomicSub(&S.d[tb + 1], 1);
        }
    }
    __syncthreads();
    const int pitch = run_pitch(a.cols);
    int carry = 0;
    for (int g = 0; g < a.cols; g += RUN_THREADS) {
        const int col = g + (int)tid;
        int all;
        const int x = run_block_scan<RUN_WARPS>(col < a.cols ? S.d[col] : 0, S.w, all);
        if (col < a.cols) a.col[(size_t)chunk * pitch + col] = (unsigned)(carry + x);
        carry += all;
    }
    if (clip) {
        int all;
        run_block_scan<RUN_WARPS>((int)kept, S.w, all);
        if (tid == 0 && all) atomicAdd(&a.kept[row], (unsigned)all);
    }
}

// Grid (blocks per row, rows): block x of a row takes its chunks x, x + gridDim.x, ...
// (six blocks per SM: latency-bound; four, five, eight: 4K 98, 99, 103 us with k_run_rows, six 92)
__global__ void __launch_bounds__(RUN_THREADS, 6) k_run_collect(RunArgs a)
{
    __shared__ CollectSmem S;
    grid_dependency_wait();
    const unsigned row = blockIdx.y;
    const unsigned long long total = a.ctr->n_entries_total;
    const uint2 cut = make_uint2(a.ctr->cut, a.ctr->cut_tiles);
    const RunRow r = a.row[row];
    if (blockIdx.x >= r.nchunks) return;
    const bool clip = total > (unsigned long long)a.cap;
    unsigned long long start = 0;
    if (clip && !a.box_total)
        for (unsigned q = 0; q < row; q++) start += a.row[q].entries;
    for (unsigned c = blockIdx.x; c < r.nchunks; c += gridDim.x) {
        RunChunk k;
        unsigned bend, rend;
        chunk_bounds(a, r, c, k, bend, rend);
        if (rend > k.run)
            collect_chunk(a, r, row, r.chunk + c, k.block, bend, k.run, rend - k.run, clip, start + k.entry, cut, S);
        else // no run: no entries in any column
            for (int j = (int)threadIdx.x; j < a.cols; j += RUN_THREADS)
                a.col[(size_t)(r.chunk + c) * run_pitch(a.cols) + j] = 0u;
    }
}

// Small frames (at most RUN_SMALL_BLOCKS front-end blocks), which the number of dependent launches
// bounds: block x of a row takes chunk x, which it finds itself from the blocks' counts, and the
// front end summed the rows' totals; k_run_rows and k_run_offsets are not launched.
__global__ void __launch_bounds__(RUN_THREADS) k_run_collect_small(RunArgs a)
{
    __shared__ CollectSmem S;
    __shared__ unsigned s_w[RUN_WARPS], s_first, s_end, s_run, s_rend, s_chunks;
    __shared__ unsigned long long s_before, s_all;
    static_assert(RUN_SMALL_BLOCKS <= RUN_THREADS, "one thread per front-end block");
    grid_dependency_wait();
    const unsigned row = blockIdx.y, tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const unsigned long long boxes = a.box_total ? a.ctr->n_entries_total : 0ull;
    if (warp == RUN_WARPS - 1) { // totals of the earlier rows, and of the frame
        unsigned long long before = 0, all = 0;
        for (unsigned q = lane; (int)q < a.rows; q += 32) {
            const unsigned long long t = a.tot[q];
            before += q < row ? t : 0ull;
            all += t;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            before += __shfl_xor_sync(0xffffffffu, before, o);
            all += __shfl_xor_sync(0xffffffffu, all, o);
        }
        if (lane == 0) {
            s_before = before;
            s_all = all & RUN_TOT_ENTRIES;
        }
    }
    if (tid == 0) {
        s_first = s_run = 0xffffffffu;
        s_end = s_rend = 0u;
    }
    const unsigned rn = tid < a.blocks ? a.cnt[(size_t)row * a.blocks + tid] >> RUN_CNT_SHIFT : 0u;
    unsigned rtot;
    const unsigned p = run_block_scan<RUN_WARPS>(rn, s_w, rtot) - rn; // its barriers order the shared words above
    if (tid < a.blocks && chunk_of(p, 0) == blockIdx.x) {
        a.pre[(size_t)row * a.blocks + tid] = p;
        atomicMin(&s_first, tid);
        atomicMax(&s_end, tid + 1);
        atomicMin(&s_run, p);
        atomicMax(&s_rend, p + rn);
    }
    if (tid == a.blocks - 1) s_chunks = rtot ? chunk_of(p, 0) + 1 : 0u;
    __syncthreads();
    RunRow r{row * small_chunks(a.blocks), s_chunks, (unsigned)(s_before >> RUN_TOT_SHIFT), rtot,
             a.tot[row] & RUN_TOT_ENTRIES};
    if (tid == 0 && blockIdx.x == 0) {
        a.row[row] = r;
        if (row == 0 && !a.box_total) a.ctr->n_entries_total = s_all;
    }
    if (blockIdx.x >= r.nchunks) return;
    if (tid == s_first) a.chunk[r.chunk + blockIdx.x] = RunChunk{tid, p, 0ull};
    const bool clip = (a.box_total ? boxes : s_all) > (unsigned long long)a.cap;
    unsigned long long entry = s_before & RUN_TOT_ENTRIES;
    uint2 cut = make_uint2(0u, 0u);
    if (clip && a.box_total) {
        __shared__ unsigned long long s_cut[RUN_WARPS];
        cut = find_cut<RUN_WARPS>(a.touched, 0u, (unsigned)a.n, 0ull, (unsigned long long)a.cap, s_cut);
    } else if (clip) { // and the row's entries before the chunk
        unsigned all;
        run_block_scan<RUN_WARPS>(tid < s_first ? a.cnt[(size_t)row * a.blocks + tid] & RUN_CNT_ENTRIES : 0u, s_w, all);
        entry += all;
    }
    collect_chunk(a, r, row, r.chunk + blockIdx.x, s_first, s_end, s_run, s_rend - s_run, clip, entry, cut, S);
}


// A row of a limited frame is limited where RUN_LIMIT of its entries bring this optical depth to a pixel on average (a pixel
// is finished at ln 1e4 = 9.2, a tile when its last pixel is). Opacity alone does not tell: small Gaussians cover little of a
// tile. Us per RoofGS frame, all entries / limited everywhere / from a depth of 12 / of 24, at 4K: opacities around 0.5 (trained scenes),
// 3 M 1291 / 1046 / 1046 / 1047, all of them x 0.5 1468 / 1263 / 1263 / 1468, x 0.35 1599 / 1530 / 1615 / 1596, x 0.1 2238 / 2558 / 2239 /
// 2238; specks of opacity 0.5 in the middle 6 % of the image, 2 px: 6 M 1148 / 1438 / 1151 / 1147, 3 M 686 / 840 / 686 / 685, 4 px, 3 M
// 714 / 648 / 650 / 714; of opacity 0.9, 2 px, 6 M 1074 / 1097 / 1096 / 1073. 8: x 0.2 1997 against 1847. (Exact mode alike.) A rule
// with the depth's variance beside its mean (z of 2 and 3) chose no better.
constexpr float LIMIT_DEPTH = 12.0f;

// A frame beyond its capacity: the entries kept in the rows before `row`, and in all (called by one warp).
__device__ __forceinline__ void kept_before(const RunArgs& a, unsigned row, unsigned long long& before, unsigned long long& all)
{
    before = all = 0;
    for (unsigned q = threadIdx.x & 31u; (int)q < a.rows; q += 32) {
        const unsigned e = a.kept[q];
        before += q < row ? e : 0u;
        all += e;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        before += __shfl_xor_sync(0xffffffffu, before, o);
        all += __shfl_xor_sync(0xffffffffu, all, o);
    }
}

// What an entry of a Gaussian of opacity o and Sigma' = (sa, sb, sc) adds to the optical depth of its tile's pixels on average:
// the integral of -ln(1 - o exp(-d^T Sigma'^-1 d / 2)) is 2 pi sqrt(det Sigma') Li2(o), spread over the tiles of the box of
// alpha >= 1/255. (Li2(o) = o + o^2 / 4 + o^3 / 9 + ...: to 2 % by the cubic below.)
__device__ __forceinline__ float entry_depth(float o, float sa, float sc, float det, float tw, float th)
{
    const float t = 2.0f * (__logf(fmaxf(o, 1e-6f)) + LN255F);
    const float tiles = (__fdividef(2.0f * __fsqrt_rn(t * sa), tw) + 1.0f) * (__fdividef(2.0f * __fsqrt_rn(t * sc), th) + 1.0f);
    const float x = __fdividef(6.2831853f * __fsqrt_rn(det) * o * (1.0f + o * (0.2f + 0.4f * o * o)), tiles * 256.0f);
    return x >= 0.0f && x < 1e30f ? x : 0.0f; // (0 for what is no number)
}

// One block per tile row: OFF_SEGS segments of the row's chunks x OFF_COLS columns at a time.
constexpr int OFF_SEGS = 4, OFF_COLS = 256;

__global__ void __launch_bounds__(OFF_SEGS* OFF_COLS) k_run_offsets(RunArgs a)
{
    __shared__ unsigned s_sum[OFF_SEGS][OFF_COLS];
    __shared__ unsigned s_first[OFF_COLS];
    __shared__ unsigned s_w[OFF_COLS / 32];
    __shared__ unsigned s_start;
    __shared__ float2 s_depth[OFF_COLS / 32];
    grid_dependency_wait();
    const unsigned row = blockIdx.x, tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const unsigned long long cap = (unsigned long long)a.cap;
    const RunRow r = a.row[row];
    const int pitch = run_pitch(a.cols);
    const unsigned sg = tid / OFF_COLS, c = tid % OFF_COLS;
    const unsigned per = (r.nchunks + OFF_SEGS - 1) / OFF_SEGS;
    const unsigned k0 = sg * per, k1 = k0 + per < r.nchunks ? k0 + per : r.nchunks;
    if (warp == OFF_SEGS * OFF_COLS / 32 - 1) { // entries of the earlier tile rows; of the frame (row 0)
        unsigned long long before = 0, all = 0;
        for (unsigned k = lane; (int)k < a.rows; k += 32) {
            const unsigned long long e = a.row[k].entries;
            before += k < row ? e : 0ull;
            all += e;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            before += __shfl_xor_sync(0xffffffffu, before, o);
            all += __shfl_xor_sync(0xffffffffu, all, o);
        }
        const unsigned long long total = a.box_total ? a.ctr->n_entries_total : all;
        if (total > cap) kept_before(a, row, before, all);
        if (lane == 0) s_start = (unsigned)(before < cap ? before : cap);
        if (lane == 0 && row == 0) {
            a.ctr->n_entries = (unsigned)(total <= cap ? total : (a.box_total ? cap : all));
            if (total > cap) {
                atomicOr(&a.ctr->overflow, 1u);
                atomicOr(&a.sticky->overflow, 1u);
            }
        }
    }
    // A limited frame pays where pixels are finished early: the optical depth of the row's entries, from 256 runs spread over
    // its list, decides (one run per lane of eight warps: one warp for all of them took 10 us)
    if (a.limit != RUN_ALL && sg == OFF_SEGS / 2) {
        float sum = 0.0f, len = 0.0f;
        if (r.runs) {
            const uint2 q = __ldg(&a.list[r.base + (unsigned)((unsigned long long)r.runs * c / OFF_COLS)]);
            float o, sa, sc, det;
            if (a.box_total) {
                const float4 e = __ldg(&a.rec[3 * (size_t)q.x + 1]); // -Sigma'_yy / (2 det), Sigma'_xy / Sigma'_yy, -1 / (2 Sigma'_yy)
                o = e.w;
                sc = __fdividef(-0.5f, e.z);
                det = __fdividef(-0.5f * sc, e.x);
                sa = __fdividef(det, sc) + e.y * e.y * sc;
            } else {
                const float4 e = __ldg(&a.rec[2 * (size_t)q.x]), f = __ldg(&a.rec[2 * (size_t)q.x + 1]); // conic (a, b, c)
                o = __expf(f.y);
                det = __fdividef(1.0f, fmaf(e.z, f.x, -0.25f * e.w * e.w));
                sa = f.x * det;
                sc = e.z * det;
            }
            len = (float)((q.y >> 16) + 1u - (q.y & 0xffffu)); // (0 for a dropped run)
            sum = entry_depth(o, sa, sc, det, (float)a.tw, (float)a.th) * len;
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            sum += __shfl_xor_sync(0xffffffffu, sum, d);
            len += __shfl_xor_sync(0xffffffffu, len, d);
        }
        if (lane == 0) s_depth[c / 32] = make_float2(sum, len);
    }
    unsigned run = 0; // entries of the row's earlier columns
    for (int g = 0; g < a.cols; g += OFF_COLS) {
        const int col = g + (int)c;
        unsigned* const p = a.col + (size_t)r.chunk * pitch + col;
        unsigned sum = 0;
        if (col < a.cols)
#pragma unroll 8
            for (unsigned k = k0; k < k1; k++) sum += p[(size_t)k * pitch];
        s_sum[sg][c] = sum;
        __syncthreads();
        unsigned total = 0, incl = 0;
        if (sg == 0) {
#pragma unroll
            for (int q = 0; q < OFF_SEGS; q++) total += s_sum[q][c];
            incl = run_warp_scan(total);
            if (lane == 31) s_w[warp] = incl;
        }
        __syncthreads();
        unsigned row_all = 0;
#pragma unroll
        for (int q = 0; q < OFF_COLS / 32; q++) {
            if (sg == 0 && q < (int)warp) incl += s_w[q];
            row_all += s_w[q];
        }
        if (sg == 0) {
            const unsigned first = s_start + run + incl - total;
            s_first[c] = first;
            if (col < a.cols) {
                // entries past the capacity are not written
                const unsigned b = first < a.cap ? first : (unsigned)a.cap;
                const unsigned e = first + total < a.cap ? first + total : (unsigned)a.cap;
                a.ranges[(size_t)row * a.cols + col] = e > b ? make_uint2(b, e) : make_uint2(0u, 0u);
                if (a.rest_flag) a.rest_flag[(size_t)row * a.cols + col] = 0u;
            }
            if (a.order.list) add_tile(a.order, a.ctr->tiles, col < a.cols, row * (unsigned)a.cols + (unsigned)col, total);
        }
        __syncthreads();
        if (col < a.cols) {
            unsigned at = s_first[c];
            for (unsigned q = 0; q < sg; q++) at += s_sum[q][c];
#pragma unroll 8
            for (unsigned k = k0; k < k1; k++) {
                const unsigned n = p[(size_t)k * pitch];
                p[(size_t)k * pitch] = at;
                at += n;
            }
        }
        run += row_all;
        __syncthreads();
    }
    if (tid == 0 && a.limit != RUN_ALL) {
        float sum = 0.0f, len = 0.0f;
#pragma unroll
        for (int q = 0; q < OFF_COLS / 32; q++) {
            sum += s_depth[q].x;
            len += s_depth[q].y;
        }
        a.row_limit[row] = sum * (float)RUN_LIMIT >= LIMIT_DEPTH * len ? a.limit : RUN_ALL;
    }
}

constexpr int SUBS = CHUNK_RUNS / 32, SEGS = RUN_THREADS / SUBS, SEG_COLS = COLS / SEGS;
static_assert(SUBS == 64 && SEGS * SUBS == RUN_THREADS && SEG_COLS % 2 == 0, "a lane holds two words of 32 runs");

struct ExpandSmem {
    unsigned mask[COLS][PITCH];
    unsigned seg[SEGS][SUBS]; // (put_first may read the word before id) XOR of a segment of columns, then of the segments before it
    unsigned id[CHUNK_RUNS];
    unsigned first[RUN_MAX_GRID]; // first slot in vals of the chunk's entries of each column
    unsigned w[RUN_WARPS];
    unsigned start;
    unsigned need[3][2]; // bit b: columns 8 b .. 8 b + 7 have an entry to be written; of three chunks in turn
};
static_assert(RUN_MAX_GRID <= 64 * 8 && COLS % 8 == 0, "a bit for every eight columns, a window of whole bits");
static_assert(sizeof(ExpandSmem) <= 48 * 1024, "no opt-in to more shared memory");

// k_run_offsets for the chunk of one block of a small frame: the first slot of each of its columns
// (S.first), from the column counts of all chunks of the row; block 0 of a row writes the ranges.
__device__ __forceinline__ void small_offsets(const RunArgs& a, const RunRow& r, unsigned row, ExpandSmem& S)
{
    const unsigned tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const unsigned long long cap = (unsigned long long)a.cap;
    if (warp == RUN_WARPS - 1) {
        const unsigned long long total = a.ctr->n_entries_total;
        unsigned long long before = 0, all = 0;
        for (unsigned q = lane; q < row; q += 32) before += a.tot[q] & RUN_TOT_ENTRIES;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
        if (total > cap) kept_before(a, row, before, all);
        if (lane == 0) S.start = (unsigned)(before < cap ? before : cap);
        if (lane == 0 && blockIdx.x == 0 && row == 0) {
            a.ctr->n_entries = (unsigned)(total <= cap ? total : (a.box_total ? cap : all));
            if (total > cap) {
                atomicOr(&a.ctr->overflow, 1u);
                atomicOr(&a.sticky->overflow, 1u);
            }
        }
    }
    const int pitch = run_pitch(a.cols);
    unsigned run = 0; // entries of the row's earlier columns
    for (int g = 0; g < a.cols; g += RUN_THREADS) {
        const int col = g + (int)tid;
        unsigned total = 0, before = 0; // of the column, of the earlier chunks
        if (col < a.cols)
            for (unsigned k = 0; k < r.nchunks; k++) {
                const unsigned n = a.col[(size_t)(r.chunk + k) * pitch + col];
                before += k < blockIdx.x ? n : 0u;
                total += n;
            }
        unsigned all;
        const unsigned incl = run_block_scan<RUN_WARPS>(total, S.w, all);
        const unsigned first = S.start + run + incl - total;
        if (col < a.cols) {
            S.first[col] = first + before;
            if (blockIdx.x == 0) {
                const unsigned b = first < a.cap ? first : (unsigned)a.cap;
                const unsigned e = first + total < a.cap ? first + total : (unsigned)a.cap;
                a.ranges[(size_t)row * a.cols + col] = e > b ? make_uint2(b, e) : make_uint2(0u, 0u);
            }
        }
        if (blockIdx.x == 0 && a.order.list)
            add_tile(a.order, a.ctr->tiles, col < a.cols, row * (unsigned)a.cols + (unsigned)col, total);
        run += all;
    }
}

// Writes the first run of mask m (its highest bit) to vals[d] and drops it from m; nothing if m is 0 (d
// then runs on unused). Without a branch: about a fifth of the lanes have a run left, and a branch per
// column cost more than the idle lanes (88 -> 64 M warp instructions for 18 M entries).
__device__ __forceinline__ void put_first(unsigned& m, unsigned* vals, unsigned& d, const unsigned* id)
{
    unsigned j, rest;
    asm("bfind.shiftamt.u32 %0, %1;" : "=r"(j) : "r"(m)); // 31 - highest bit; ~0 for 0
    asm("shr.u32 %0, %1, %2;" : "=r"(rest) : "r"(0x7fffffffu), "r"(j)); // 0 for ~0 (shifts clamp)
    const unsigned v = id[(int)j]; // for 0 the word before, unused
    asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %0, 0;\n @p st.global.u32 [%1], %2;\n}" ::"r"(m), "l"(vals + d), "r"(v)
                 : "memory");
    m &= rest;
    d++;
}

constexpr unsigned NONE = 0xffffffffu;

// Grid as the collect kernel's. In a limited frame (RunArgs::limit) a chunk's columns of which no entry is to be written
// are left out, with their masks where eight of them lie together at the edge of a window: 4K, 3 M Gaussians (83 % of the
// entries lie past their tile's first 512) 286 -> 175 us, 8K, 1 M 321 -> 232 us.
template <bool SMALL>
__global__ void __launch_bounds__(RUN_THREADS, 5) k_run_expand(RunArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ExpandSmem& S = *reinterpret_cast<ExpandSmem*>(smem_raw);
    grid_dependency_wait();
    if (!SMALL && a.rest && a.ctr->n_rest == 0u) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned row = blockIdx.y;
    const RunRow r = a.row[row];
    if (SMALL && (blockIdx.x == 0 || blockIdx.x < r.nchunks)) small_offsets(a, r, row, S);
    if (blockIdx.x >= r.nchunks) return;
    const int pitch = run_pitch(a.cols);
    const unsigned cap = (unsigned)a.cap;
    const bool over = a.ctr->n_entries_total > (unsigned long long)a.cap;
    const unsigned limit = a.limit == RUN_ALL ? RUN_ALL : a.row_limit[row];
    int turn = 0;
    if (!SMALL) {
        if (tid < 6) S.need[tid / 2][tid & 1] = 0u;
        __syncthreads();
    }
    for (unsigned c = blockIdx.x; c < r.nchunks; c += gridDim.x) {
        RunChunk k;
        unsigned bend, rend;
        chunk_bounds(a, r, c, k, bend, rend);
        const unsigned n = rend - k.run; // at most CHUNK_RUNS
        if (n == 0) continue;
        unsigned long long need = ~0ull >> (64 - (a.cols + 7) / 8);
        if (!SMALL) { // NONE: no entry of the chunk is to be written, being past the tile's first `limit` ones (or, at rest, not)
            for (int j0 = 0; j0 < a.cols; j0 += RUN_THREADS) {
                const int j = j0 + tid;
                bool write = false;
                if (j < a.cols) {
                    const unsigned f = __ldg(&a.col[(size_t)(r.chunk + c) * pitch + j]);
                    const uint2 tile = __ldg(&a.ranges[(size_t)row * a.cols + j]);
                    write = f < tile.y && (a.rest ? f - tile.x >= limit && a.rest_flag[row * a.cols + j] : f - tile.x < limit);
                    S.first[j] = write ? f : NONE;
                }
                const unsigned m = __ballot_sync(0xffffffffu, write);
                if (lane == 0 && m)
                    atomicOr(&S.need[turn][j0 / RUN_THREADS], ((m & 0xffu ? 1u : 0u) | (m & 0xff00u ? 2u : 0u) |
                             (m & 0xff0000u ? 4u : 0u) | (m & 0xff000000u ? 8u : 0u)) << (4 * warp));
            }
            __syncthreads();
            need = S.need[turn][0] | ((unsigned long long)S.need[turn][1] << 32);
            // the words of the turn after the next: read by nobody since the barrier, and zero before the next one
            turn = turn == 2 ? 0 : turn + 1;
            if (tid < 2) S.need[turn == 2 ? 0 : turn + 1][tid] = 0u;
        }
        if (!need) continue;
        const uint2* const list = a.list + r.base + k.run;
        unsigned ends[CHUNK_RUNS / RUN_THREADS]; // the thread's runs: first and last column
#pragma unroll
        for (int u = 0; u < CHUNK_RUNS / RUN_THREADS; u++) {
            const unsigned j = (unsigned)(u * RUN_THREADS + tid);
            const uint2 q = j < n ? __ldg(&list[j]) : make_uint2(0u, 1u);
            if (j < n) S.id[j] = q.x;
            ends[u] = q.y;
        }
        while (need) { // a window of columns
            const int g = 8 * (__ffsll((long long)need) - 1);
            const unsigned long long in = (need >> (g / 8)) & ((1ull << (COLS / 8)) - 1ull);
            const int width = 8 * (64 - __clzll((long long)in)), cols = a.cols - g < width ? a.cols - g : width;
            need &= ~(in << (g / 8));
            for (int j = tid; j < cols * PITCH / 2; j += RUN_THREADS)
                reinterpret_cast<uint2*>(&S.mask[0][0])[j] = make_uint2(0u, 0u);
            __syncthreads();
            // run 32 s + l of the chunk: bit 31 - l of word s (the first run is the highest bit)
#pragma unroll
            for (int u = 0; u < CHUNK_RUNS / RUN_THREADS; u++) {
                const int ta = (int)(ends[u] & 0xffffu) - g, tb = (int)(ends[u] >> 16) - g;
                if (ta <= tb && tb >= 0 && ta < cols) { // an empty run has ta = 1, tb = 0
                    const int sub = u * (RUN_THREADS / 32) + warp;
                    atomicXor(&S.mask[ta > 0 ? ta : 0][sub], 0x80000000u >> lane);
                    if (tb + 1 < cols) atomicXor(&S.mask[tb + 1][sub], 0x80000000u >> lane);
                }
            }
            __syncthreads();
            { // prefix XOR over the columns, in SEGS segments
                const int sub = tid % SUBS, sg = tid / SUBS;
                const int c0 = sg * SEG_COLS, c1 = c0 + SEG_COLS < cols ? c0 + SEG_COLS : cols;
                unsigned x = 0;
#pragma unroll 8
                for (int q = c0; q < c1; q++) {
                    x ^= S.mask[q][sub];
                    S.mask[q][sub] = x;
                }
                S.seg[sg][sub] = x;
                __syncthreads();
                unsigned before = 0;
                for (int q = 0; q < sg; q++) before ^= S.seg[q][sub];
                __syncthreads();
                S.seg[sg][sub] = before;
            }
            __syncthreads();
            // a warp takes two columns at a time (one scan of 16-bit counts, two chains of stores)
            for (int q = 2 * warp; q < cols; q += 2 * RUN_WARPS) {
                const bool two = q + 1 < cols;
                const bool use0 = SMALL || S.first[g + q] != NONE, use1 = SMALL || (two && S.first[g + q + 1] != NONE);
                if (!use0 && !use1) continue;
                const uint2 b = *reinterpret_cast<const uint2*>(&S.seg[q / SEG_COLS][2 * lane]);
                const uint2 m0 = *reinterpret_cast<const uint2*>(&S.mask[q][2 * lane]);
                const uint2 m1 = two ? *reinterpret_cast<const uint2*>(&S.mask[q + 1][2 * lane]) : b;
                unsigned lo0 = m0.x ^ b.x, hi0 = m0.y ^ b.y, lo1 = m1.x ^ b.x, hi1 = m1.y ^ b.y;
                if (!use0) lo0 = hi0 = 0u; // nothing is written
                if (!use1) lo1 = hi1 = 0u;
                const unsigned n0 = (unsigned)__popc(lo0), n1 = (unsigned)__popc(lo1);
                const unsigned cnt = (n0 + (unsigned)__popc(hi0)) + ((n1 + (unsigned)__popc(hi1)) << 16);
                const unsigned excl = run_warp_scan(cnt) - cnt;
                unsigned d0 = S.first[g + q] + (excl & 0xffffu), d1 = S.first[two ? g + q + 1 : g + q] + (excl >> 16);
                const unsigned* const id = &S.id[64 * lane];
                if (!over) {
                    unsigned e0 = d0 + n0, e1 = d1 + n1;
                    while (lo0 | lo1) {
                        put_first(lo0, a.vals, d0, id);
                        put_first(lo1, a.vals, d1, id);
                    }
                    while (hi0 | hi1) {
                        put_first(hi0, a.vals, e0, id + 32);
                        put_first(hi1, a.vals, e1, id + 32);
                    }
                } else { // slots past the capacity are not written
                    auto put = [&](unsigned m, unsigned d, const unsigned* from) {
                        for (; m; d++) {
                            const int j = __clz((int)m);
                            if (d < cap) a.vals[d] = from[j];
                            m ^= 0x80000000u >> j;
                        }
                    };
                    put(lo0, d0, id);
                    put(lo1, d1, id);
                    put(hi0, d0 + n0, id + 32);
                    put(hi1, d1 + n1, id + 32);
                }
            }
            __syncthreads(); // the masks are cleared for the next columns or chunk
        }
    }
}

// at most the chunks a row can have, and about 4 waves of blocks over all rows (2 / 8 waves: 1080p 53 / 57 us
// of collection and expansion, 4K 407 / 375; 4: 53 and 379)
static dim3 run_grid(const RunArgs& a, int waves = 4)
{
    const unsigned most = a.blocks * (unsigned)RUN_SLOTS / CHUNK_STEP + a.blocks / CHUNK_BLOCKS + 1;
    const unsigned want = (unsigned)(waves * 5 * device_sm_count() / a.rows + 1);
    return dim3(most < want ? most : want, (unsigned)a.rows);
}

void launch_runs_rest(const RunArgs& limited, cudaStream_t s)
{
    RunArgs a = limited;
    a.rest = 1;
    launch_dependent(k_run_expand<false>, run_grid(a, 1), dim3(RUN_THREADS), sizeof(ExpandSmem), s, a);
}

void launch_runs_all(const RunArgs& limited, cudaStream_t s)
{
    RunArgs a = limited;
    a.limit = RUN_ALL;
    launch_dependent(k_run_expand<false>, run_grid(a), dim3(RUN_THREADS), sizeof(ExpandSmem), s, a);
}

void launch_runs(const RunArgs& a, cudaStream_t s, cudaEvent_t ev_after_collect)
{
    if (a.blocks == 0) return;
    const dim3 block(RUN_THREADS);
    if (a.tot) {
        const dim3 grid(small_chunks(a.blocks), (unsigned)a.rows);
        launch_dependent(k_run_collect_small, grid, block, 0, s, a);
        if (ev_after_collect) cudaEventRecord(ev_after_collect, s);
        launch_dependent(k_run_expand<true>, grid, block, sizeof(ExpandSmem), s, a);
        return;
    }
    const dim3 grid = run_grid(a);
    launch_dependent(k_run_rows, dim3((unsigned)a.rows), dim3(1024), 0, s, a);
    launch_dependent(k_run_collect, grid, block, 0, s, a);
    if (ev_after_collect) cudaEventRecord(ev_after_collect, s);
    launch_dependent(k_run_offsets, dim3((unsigned)a.rows), dim3(OFF_SEGS * OFF_COLS), 0, s, a);
    launch_dependent(k_run_expand<false>, grid, block, sizeof(ExpandSmem), s, a);
}

} // namespace rg
