// Algorithm 2 (Section 4.2) for node-symmetric catalogs (shapes invariant under a shift of the node index) of groups of four
// ranks: two to sixty-four groups, N = 8 .. 256.  Included by schedule.cu.
//
// One CTA decomposes one matrix at a time, in a chain of dependent activations; the time of an activation is a chain of
// shared-memory reads, integer operations and barriers, so everything here is arranged to keep that chain short.
//
//  * Credits.  Step 2 only ever looks at min(D_rem[i][j], cap_r) (Eq. 7).  N x N 16-bit cells fit shared memory (130 KB
//    at N = 256) where the residual in 32-bit granules (256 KB) does not.  A cell below F = 65,536 - M granules is
//    kept as it is; a cell of F granules or more holds F + (its index in a side list of M = 4,096 exact 32-bit
//    values).  As long as every lane capacity is below F, such a cell yields the same credit as its exact value
//    (the capacity), and the emit step keeps the side list exact until the cell drops below F and becomes ordinary.
//    Cells of rows 2p and 2p + 1 share a word, wd[p][column]: the four rows of a group at one column are two 32-bit reads
//    already packed in pairs, the four columns of a group at one row are one 128-bit read and two byte permutes.  (Row-major
//    16-bit cells took sixteen single reads, minima and multiply-adds per group in the source half of a sweep.)
//  * Scores.  Eq. (6) on a node-symmetric catalog is a sum of at most max_terms products count x C[e], where
//    C[delta][q][q'] = sum_n D-hat[(n,q)][(n+delta,q')] (the same integer as the full sum over D-hat).  The table C
//    (P S S entries, 32-bit granules) is kept in shared memory and every activation subtracts its lane volumes from
//    the entries they fall in, so D-hat itself is needed only once, for the quantum rule and the first table.
//    The terms of a shape are split by source rail into S rows, and the catalog has few distinct rows (127 per rail
//    for 4,095 shapes).  On one and two rails the first maximum is taken class by class (see (A) and big_by_class), the rows'
//    terms in registers: up to sixteen groups every task warp does it alone, without a barrier, where the block scored rows,
//    then shapes, then joined its warps behind three barriers.  16 x 64 ranks 659 -> 593 us, 1,024 x 64 ranks 1,455 -> 1,344,
//    16 x 32 ranks 306 -> 277, 512 x 256 ranks 11,760 -> 11,250.
//  * Step 2.  A (family, start) task is one or two lanes per rank group: up to four tasks share a warp, the largest are two
//    warps.  The two halves of a sweep exchange bindings as one byte per group, by shuffles wherever a task fits a warp.
//  * Emit.  An activation is first taken off the residual and off C; its plan rows and offset sums are written while the next
//    activation's tasks run, by warps without a task where the CTA has some.
//
//  * Large capacities.  When a lane capacity reaches 2^16 granules (skewed MoE matrices with many tokens), the few
//    columns that hold cells of 65,535 granules or more -- the destinations of the popular experts -- become "hot
//    columns": their cells are kept exactly, low 16 bits in the credit matrix and high 16 bits in a side array of up
//    to 32 columns, and the credits that touch them are patched after the ordinary 16-bit pass (above 32 groups, where such
//    matrices are the longest of a batch: from the words already read, and until no cell of the column is beyond 16 bits any more;
//    5.65 -> 4.2 us an activation with 256 ranks).  Every other cell of such a matrix is below 65,535 granules, so its 16-bit
//    copy is exact.  No L2 traffic is needed in this mode.
//
//  * Code size.  Instructions come from caches of about 8 KB per scheduler and 32 KB per SM; straight-line code costs 2.2
//    cycles an instruction from the first, 4 at 32 KB and 6.5 beyond, and more at every jump.  So what an ordinary
//    activation does not execute is kept out of its loop: the loop exists twice, with and without hot columns, and the 64-bit
//    scores are functions of their own.  As one loop of 65 KB with all cases inside: 16 x 64 ranks 774 -> 659 us,
//    1,024 x 64 ranks 1,591 -> 1,455, 512 x 256 ranks 12,560 -> 11,760.
//  * Instructions.  A warp that is alone on its scheduler issues one in four to five cycles, whatever it is, and a task warp executes
//    hundreds per activation.  So integer divisions and further families are out of line, rows are written at one place, a
//    warp with a single task carries no "alive" flags, the run ends as soon as a ballot says so, and the usual path is laid out
//    straight: 593 -> 532 us, 1,344 -> 1,275, 11,250 -> 10,630; 16 x 32 ranks 277 -> 247, 16 x 96 ranks 1,296 -> 1,225.
//
// A matrix that does not meet the conditions (granule below 256 bytes, a capacity of 2^22 granules or more, 2^32
// granules or more in total, more than 32 hot columns, more big cells than the side list holds) is appended to a list that
// the general kernel works through afterwards.
#pragma once

namespace {

constexpr int BIG_HOT_MAX = 32;       // columns whose cells are kept beyond 16 bits; as a column's index: none
constexpr uint32_t BIG_HOT_NONE = 0x01010101u * BIG_HOT_MAX;  // a group without a hot column
constexpr int BIG_EXCHANGE = 192;     // bytes per pair of warps: 64 source tags, 64 destination tags, words
constexpr int BIG_SMEM_LIMIT = 227 * 1024 - 2048;   // dynamic shared memory of one CTA, less room for the static variables

// Branch weights: the usual path of an activation runs straight through (every jump beyond the nearest instruction cache waits for
// the next one).
__device__ __forceinline__ bool usually(bool c) { return __builtin_expect(c, 1); }
__device__ __forceinline__ bool rarely(bool c) { return __builtin_expect(c, 0); }

template <bool V> struct BigConst { static constexpr bool value = V; };

struct BigSmem {
    int wd, hi, colmap, tbl, rs, pat, gnode, send_acc, recv_acc, red, task_f, task_den, bind, exchange, record, term, bucket, fam_task, total;
    int fill, fill_rows;      // source buffers of the asynchronous fill, offset rows per buffer (0: plain stores)
    int pat_words;            // 32-bit words of row-pattern ids per shape (two ids per word)
};

// Is the arg-max taken class by class in 32 bits (see (A) in the kernel)?  Up to sixteen groups every task warp does so by itself, a
// first and a second row per lane; above, the warps share the chunks of 32 rows, at most BIG_CHUNKS each (of four warps or more).
constexpr int BIG_CHUNKS = 3;
__host__ __device__ inline bool big_by_class(const DevCat& dc) {
    return dc.G <= 16 ? dc.lane_rows != nullptr : dc.dec != nullptr && dc.dec_stride == 4 && dc.dec_chunks <= 4 * BIG_CHUNKS;
}

__host__ __device__ inline BigSmem big_smem_layout(const DevCat& dc, const KParams& kp) {
    BigSmem L;
    const bool by_class = big_by_class(dc);
    int o = 0;
    const int wd_bytes = dc.N / 2 * big_stride(big_lanes(dc.G)) * 4, setup_bytes = dc.G * dc.G * 8 + dc.N * 24;
    L.wd = o;        o += align16(wd_bytes > setup_bytes ? wd_bytes : setup_bytes);   // set-up: D-hat, row and column sums
    L.hi = o;        o += (BIG_HOT_MAX + (dc.G > 32)) * dc.N * 2;   // high halves of the hot columns' cells (and of none of them), or the side list
    L.colmap = o;    o += align16(dc.N);                          // hot-column index of every rank
    L.tbl = o;       o += align16(dc.tbl_size * 4);
    L.rs = o;        o += align16(dc.n_patterns * 8);             // row scores of the general route, and its tables where it is the usual one
    L.pat = o;       o += by_class ? 0 : align16(dc.n_patterns * dc.max_row_terms * 4);
    L.gnode = o;     o += align16(dc.G * 2);
    L.send_acc = o;  o += dc.N * 8;
    L.recv_acc = o;  o += dc.N * 8;
    L.red = o;       o += 64 * 8;
    L.task_f = o;    o += align16(kp.max_tasks * 4);
    L.task_den = o;  o += align16(kp.max_tasks * 8);
    L.bind = o;      o += align16(kp.max_tasks * dc.N * 2);       // per task and slot: source | destination << 8
    L.exchange = o;  o += kp.big_cross ? 4 * BIG_EXCHANGE : 0;     // what the two warps of a task tell each other
    L.record = o;    o += dc.G > 32 ? dc.N * 8 + 16 : 0;           // the activation to be written out: source | destination << 8, volume
    L.pat_words = (dc.S + 1) / 2;
    L.term = o;      o += by_class ? 0 : ((dc.n_shapes + 31) & ~31) * L.pat_words * 4;
    L.bucket = o;    o += align16((dc.n_shapes + 1) * 4);
    // the families' task tables, where a CTA has its SM to itself or they are small: the tables of a new family are otherwise a
    // trip to L2 in the middle of the chain
    L.fam_task = o;  o += kp.big_stage ? dc.n_families * dc.G * 32 : 0;
    // Source buffers of the asynchronous fill: all ones, zeros (written once per CTA), the send totals and the receive
    // totals repeated fill_rows times (per matrix); the idle rows of a plan are written from them by bulk asynchronous
    // copies while the matrix is decomposed.  Only for the one-CTA-per-SM shape (more than 32 groups), in
    // whatever shared memory is left, and not below 4 KB per buffer.
    L.fill = o;
    L.fill_rows = dc.G > 32 && dc.N % 8 == 0 ? (BIG_SMEM_LIMIT - o) / 4 / (dc.N * 8) : 0;
    if (L.fill_rows > 4) L.fill_rows = 4;
    if (L.fill_rows * dc.N * 8 < 4096) L.fill_rows = 0;
    o += 4 * L.fill_rows * dc.N * 8;
    L.total = o;
    return L;
}

// Tag of row r at position q of a 4 x 4 assignment: (3 - r) in the two bits that position q owns in a byte whose
// two highest bits belong to position 0.  The four tags of a permutation add up to 255 minus the permutation written
// as a byte, so a credit sum carried as (sum << 8) + tags is largest for the largest sum and, among equal sums, for
// the first permutation in lexicographic order -- the same winner as an enumeration that keeps the first maximum.
__host__ __device__ constexpr uint32_t big_tag(int r, int q) { return (uint32_t)(3 - r) << (6 - 2 * q); }

__device__ __forceinline__ uint32_t add_max(uint32_t a, uint32_t b, uint32_t c) { return __viaddmax_u32(a, b, c); }   // max(a + b, c)

// Exact 4 x 4 assignment: v[r][q] = (credit of row r at position q) << 8 | big_tag(r, q).  Returns the largest
// sum_q v[phi(q)][q] over the permutations phi, by dynamic programming over the set of rows placed so far (positions
// 0, 1, 2, 3 in turn), 28 add / add-max operations.  The permutation byte is ~key & 255, the credit sum key >> 8.
__device__ __forceinline__ uint32_t big_best_key(const uint32_t (&v)[4][4]) {
    const uint32_t b01 = add_max(v[0][0], v[1][1], v[1][0] + v[0][1]), b02 = add_max(v[0][0], v[2][1], v[2][0] + v[0][1]);
    const uint32_t b03 = add_max(v[0][0], v[3][1], v[3][0] + v[0][1]), b12 = add_max(v[1][0], v[2][1], v[2][0] + v[1][1]);
    const uint32_t b13 = add_max(v[1][0], v[3][1], v[3][0] + v[1][1]), b23 = add_max(v[2][0], v[3][1], v[3][0] + v[2][1]);
    const uint32_t c012 = add_max(b01, v[2][2], add_max(b02, v[1][2], b12 + v[0][2]));
    const uint32_t c013 = add_max(b01, v[3][2], add_max(b03, v[1][2], b13 + v[0][2]));
    const uint32_t c023 = add_max(b02, v[3][2], add_max(b03, v[2][2], b23 + v[0][2]));
    const uint32_t c123 = add_max(b12, v[3][2], add_max(b13, v[2][2], b23 + v[1][2]));
    return add_max(c012, v[3][3], add_max(c013, v[2][3], add_max(c023, v[1][3], c123 + v[0][3])));
}

// Maximum of distinct 64-bit keys over the warp: the largest high word, then the largest low word among its holders.
__device__ __forceinline__ uint64_t big_warp_max64(uint64_t key) {
    const uint32_t hi = (uint32_t)(key >> 32), lo = (uint32_t)key;
    const uint32_t mhi = __reduce_max_sync(0xffffffffu, hi);
    const uint32_t mlo = __reduce_max_sync(0xffffffffu, hi == mhi ? lo : 0u);
    return (uint64_t)mhi << 32 | mlo;
}

// One matrix's credits as the tasks read them (shared-memory pointers).
struct BigCredits {
    const uint32_t* wd;
    const uint16_t* hi;
    const uint8_t* colmap;
    int stride, N;
    bool hot;
    // exact value of a cell as far as the matrix keeps it (a big cell yields its code, at least the capacity)
    __device__ __forceinline__ uint32_t cell(int i, int j) const {
        uint32_t c = ((const uint16_t*)wd)[((i >> 1) * stride + j) * 2 + (i & 1)];
        if (hot && colmap[j] != BIG_HOT_MAX) c |= (uint32_t)hi[(int)colmap[j] * N + i] << 16;
        return c;
    }
};

// Fills bytes [lo, hi) of dst with a repeated byte, by 16-byte stores where the address allows (all threads of the CTA).
__device__ __forceinline__ void big_fill_bytes(unsigned char* dst, size_t lo, size_t hi, unsigned char byte, int tid, int NT) {
    if (lo >= hi) return;
    const size_t head = min((size_t)((16 - ((uintptr_t)(dst + lo) & 15)) & 15), hi - lo);
    for (size_t e = lo + tid; e < lo + head; e += NT) dst[e] = byte;
    const size_t vlo = lo + head, nvec = (hi - vlo) / 16;
    const uint32_t w = 0x01010101u * byte;
    uint4* v = (uint4*)(dst + vlo);
    for (size_t e = tid; e < nvec; e += NT) v[e] = make_uint4(w, w, w, w);
    for (size_t e = vlo + nvec * 16 + tid; e < hi; e += NT) dst[e] = byte;
}

// (out of line: 64-bit division is long, and granules are powers of two in practice)
__device__ __noinline__ bool big_not_multiple(int64_t x, int64_t granule) { return x % granule != 0; }
__device__ __noinline__ int64_t big_wide_ceil_div(int64_t x, int64_t d) { return x / d + (x % d > 0); }
// Asks for a whole matrix at once (N * N * 8 is a multiple of 16): with 256 ranks the first pass is then 42,000 cycles, where each of its
// reads waited for DRAM behind the plans that others write 131,000.  (32 KB matrices gain nothing.  In line it cost the loop 2 %.)
__device__ __noinline__ void big_prefetch(const int64_t* D, int N) {
    if (threadIdx.x < 32 && ((uintptr_t)D & 15) == 0)
        for (int at = threadIdx.x * 4096; at < N * N * 8; at += 32 * 4096) bulk_prefetch((const char*)D + at, (unsigned)min(4096, N * N * 8 - at));
}
// What is wrong with the entries of rows ga * 4 .. ga * 4 + 3 (out of line: looked for only when something is).  Whole warp.
__device__ __noinline__ int big_wrong_entries(const int64_t* rows, int N, int ga, int64_t granule) {
    int flags = 0;
#pragma unroll 1
    for (int e = threadIdx.x & 31; e < 4 * N; e += 32) {
        const int64_t x = rows[e];
        const int i = e / N;
        if (x < 0) flags |= VP_ST_NEGATIVE;
        else if (x >= VP_ENTRY_LIMIT) flags |= VP_ST_OVERFLOW_RISK;
        else {
            if (e - i * N == ga * 4 + i && x != 0) flags |= VP_ST_DIAG_NONZERO;
            if (big_not_multiple(x, granule)) flags |= VP_ST_NOT_GRANULE;
        }
    }
    return flags;
}

// An offset row in rank order, whole lines for PCIe, once all of it is up to date: `threads` threads, numbered from 0, whole warps (out of
// line: for page-locked plans only, and inlined it costs the other case registers).  The barrier's number counts: an SM has 64, and a
// kernel reserves all up to its highest one (with number 9 eight small CTAs no longer fit an SM: 1.64 -> 2.43 ms).
template <int BARRIER>
__device__ __noinline__ void big_write_in_order(int64_t* row, const int64_t* acc, int N, int thread, int threads) {
    asm volatile("bar.sync %0, %1;" ::"n"(BARRIER), "r"(threads) : "memory");
    for (int r = thread; r < N; r += threads) row[r] = acc[r];
    asm volatile("bar.sync %0, %1;" ::"n"(BARRIER), "r"(threads) : "memory");
}

// Eq. (6) by the general route, in 64 bits (out of line, as the loop should stay small for the instruction caches): scores beyond
// 32 bits (up to sixteen groups), and catalogs that have no class structure (see big_by_class; the template catalogs with their shapes in
// another order, before the classes were the usual route and now: 16 and 1,024 matrices of 64 ranks 774 -> 668 and 1,567 -> 1,429 us, 148 of
// 128 ranks 2,266 -> 1,976, 16 of 256 ranks 6,308 -> 6,088).  All threads of the CTA; every
// warp gets the key of the first maximum, score << 16 | (65535 - shape): a score is at most four times what is left, so below 2^34,
// and there are fewer than 2^16 shapes.
__device__ __noinline__ uint64_t big_first_maximum(const uint32_t* tbl, uint64_t* rs, uint64_t* red, const uint32_t* pat, const uint32_t* spat,
                                                   int n_patterns, int row_terms, int n_shapes, int S) {
    const int tid = threadIdx.x, NT = blockDim.x, lane = tid & 31, ns_pad = (n_shapes + 31) & ~31;
#pragma unroll 1
    for (int p = tid; p < n_patterns; p += NT) {
        uint64_t v = 0;
#pragma unroll 1
        for (int t = 0; t < row_terms; t++) {
            const uint32_t tw = pat[p * row_terms + t];
            v += (uint64_t)tbl[tw & 0xffffu] * (tw >> 16);
        }
        rs[p] = v << 16;
    }
    __syncthreads();
    uint64_t best = 0;
#pragma unroll 1
    for (int s = tid; s < n_shapes; s += NT) {
        uint64_t key = (uint64_t)(65535 - s);
#pragma unroll 1
        for (int q = 0; q < S; q += 2) {
            const uint32_t pw = spat[q / 2 * ns_pad + s];
            key += rs[pw & 0xffffu];
            if (q + 1 < S) key += rs[pw >> 16];
        }
        best = max_v(best, key);
    }
    best = big_warp_max64(best);
    if (lane == 0) red[tid >> 5] = best;
    __syncthreads();
    return big_warp_max64(lane < NT / 32 ? red[lane] : 0ull);
}
// The same class by class in 64 bits, for the chunks of more than sixteen groups (out of line, see there): a matrix of 2^30 granules and
// more.  All threads of the CTA; the first maximal shape, -1 if all score zero.  (By the scan of all 4,095 shapes above, 16 matrices of
// 256 ranks and 1.9 x 10^9 granules took 4,630 us, here 3,660.)
__device__ __noinline__ int big_chunks_maximum(const uint32_t* tbl, uint64_t* red, const uint32_t* dec, int n_chunks, int n_classes) {
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int c = threadIdx.x >> 5; c < n_chunks; c += blockDim.x >> 5) {
        const uint4 w = __ldg((const uint4*)(dec + dec[2]) + c * 32 + lane);
        const uint64_t score = (uint64_t)tbl[w.x & 0xffffu] * (w.x >> 16) + (uint64_t)tbl[w.y & 0xffffu] * (w.y >> 16) + (uint64_t)tbl[w.z & 0xffffu] * (w.z >> 16);
        const uint64_t key = big_warp_max64(w.w == 0xffffffffu ? 0ull : (score + 1) << 16 | (0xffffu - w.w));   // (equal scores: the lowest word)
        if (lane == 0) red[c] = key;
    }
    __syncthreads();
    uint64_t sum = 0;
    if (lane < n_classes) {
        uint64_t k0 = 0, k1 = 0;
        const int c0 = (int)dec[3 + 2 * lane], c1 = (int)dec[4 + 2 * lane], c2 = (int)dec[5 + 2 * lane];
#pragma unroll 1
        for (int c = c0; c < c1; c++) k0 = max_v(k0, red[c]);
#pragma unroll 1
        for (int c = c1; c < c2; c++) k1 = max_v(k1, red[c]);
        sum = ((k0 >> 16) + (k1 >> 16)) << 16 | ((k0 & 0xffffu) + (k1 & 0xffffu) - 0xffffu);      // 65535 - (run start + place)
    }
    sum = big_warp_max64(sum);
    return (sum >> 16) > 2 ? 65535 - (int)(sum & 0xffffu) : -1;
}
// Family (of those that compete) and initial binding of a (family, start) task: h << 8 | binding, as a byte per group (see (B)).  Start t
// binds in-slot q to row (q + t) mod 4.
__device__ __noinline__ uint32_t big_family_and_start(int task, int n_start) {
    const int h = task / n_start, t = task - h * n_start;
    uint32_t dst = (uint32_t)h << 8;
#pragma unroll
    for (int q = 0; q < 4; q++) dst |= (uint32_t)(3 - ((q + t) & 3)) << (6 - 2 * q);
    return dst;
}

// Step 3 when several families compete (kept out of line: most shapes have one family, and the main loop should
// stay small for the instruction cache): best start per family (largest F, lowest start), then the family of largest
// utility F / duration by exact cross-multiplication, lowest family first among equals.  Whole warp.
// (Returns F << 32 | task: by reference the two would live in local memory, also where this is not called.)
__device__ __noinline__ uint64_t big_select_family(const uint32_t* task_f, const int64_t* task_den, int H, int n_start, int lane) {
    int64_t bf = -1, bd = 1;
    int bt = 0x7fffffff;
    for (int h = lane; h < H; h += 32) {
        int64_t ff = -1; int tt = 0;
        for (int t = 0; t < n_start; t++)
            if ((int64_t)task_f[h * n_start + t] > ff) { ff = (int64_t)task_f[h * n_start + t]; tt = h * n_start + t; }
        if (bt == 0x7fffffff || util_greater(ff, task_den[tt], bf, bd)) { bf = ff; bd = task_den[tt]; bt = tt; }
    }
#pragma unroll 1
    for (int o = 16; o; o >>= 1) {
        const int64_t of = __shfl_xor_sync(0xffffffffu, bf, o), od = __shfl_xor_sync(0xffffffffu, bd, o);
        const int ot = __shfl_xor_sync(0xffffffffu, bt, o);
        bool take = false;
        if (ot != 0x7fffffff) {
            if (bt == 0x7fffffff) take = true;
            else if (util_greater(of, od, bf, bd)) take = true;
            else if (!util_greater(bf, bd, of, od) && ot < bt) take = true;
        }
        if (take) { bf = of; bd = od; bt = ot; }
    }
    bt = __shfl_sync(0xffffffffu, bt, 0);
    bf = __shfl_sync(0xffffffffu, bf, 0);
    return (uint64_t)bf << 32 | (uint32_t)bt;
}

// Work order for a batch whose matrices differ a lot in length: CTAs that take the long matrices first leave a short tail.  An
// activation gives a group one lane over its NIC, and a family serves the same (node offset, source rail, destination rail)
// on every node, so a matrix takes at least sum over (offset, other rail) of the largest number of lanes that any node needs there,
// for its busiest rail.  That bound orders matrices like their activations (correlation 0.93 to 0.97; the number of non-zero
// cells, taken before, puts sparse matrices of 2,000 cells last that take the most activations of all), and needs the demand twice:
// lane capacity from the largest group total, then lanes per group pair.  An estimate in floats: the order does not change results.
// One CTA per matrix; a warp per source group, a lane per column.  512 matrices of 256 ranks: 13.84 -> 12.60 ms.
constexpr int BIG_KEY_THREADS = 256;
__global__ void __launch_bounds__(BIG_KEY_THREADS) big_length_kernel(DevCat dc, KParams kp, const int64_t* __restrict__ demand, const int64_t* __restrict__ tau_in,
                                                        int* __restrict__ key) {
    constexpr int CW = VP_MAX_N / 32, WARPS = BIG_KEY_THREADS / 32, GMAX = VP_MAX_N / 4;
    __shared__ float colsum[WARPS][VP_MAX_N], top[WARPS];
    __shared__ int lanes[GMAX * GMAX], rail[2 * GMAX];      // lanes per (offset, rail, rail), per rail (source, then destination)
    const int b = blockIdx.x, N = dc.N, G = dc.G, S = dc.S, P = dc.P, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t* const D = demand + (size_t)b * N * N;
    for (int e = tid; e < G * S; e += BIG_KEY_THREADS) lanes[e] = 0;
    for (int e = tid; e < 2 * S; e += BIG_KEY_THREADS) rail[e] = 0;
    float cap;
    if (tau_in && tau_in[b] > 0) {
        cap = (float)tau_in[b] * (float)dc.bw_max;
    } else {
        float col[CW], most = 0.f;
#pragma unroll
        for (int c = 0; c < CW; c++) col[c] = 0.f;
        for (int ga = warp; ga < G; ga += WARPS) {
            float sum = 0.f;
#pragma unroll
            for (int c = 0; c < CW; c++) {
                const int j = c * 32 + lane;
                if (j >= N) break;
                float s = 0.f;
#pragma unroll
                for (int r = 0; r < 4; r++) s += (float)D[(size_t)(ga * 4 + r) * N + j];
                col[c] += s; sum += s;
            }
            for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            most = fmaxf(most, sum);
        }
#pragma unroll
        for (int c = 0; c < CW; c++) colsum[warp][c * 32 + lane] = col[c];
        __syncthreads();
        float s = 0.f;
        for (int w = 0; w < WARPS; w++) s += colsum[w][tid];
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);              // a destination group's total
        most = fmaxf(most, s);
        for (int o = 16; o; o >>= 1) most = fmaxf(most, __shfl_xor_sync(0xffffffffu, most, o));
        if (lane == 0) top[warp] = most;
        __syncthreads();
        for (int w = 0; w < WARPS; w++) most = fmaxf(most, top[w]);
        cap = most / (float)kp.k_target;
    }
    const float per_lane = 1.f / fmaxf(cap, (float)kp.granule);
    __syncthreads();
    for (int ga = warp; ga < G; ga += WARPS) {
#pragma unroll
        for (int c = 0; c < CW; c++) {
            const int j = c * 32 + lane, gd = j >> 2;
            float s = 0.f;
            if (j < N)
#pragma unroll
                for (int r = 0; r < 4; r++) s += ceilf((float)D[(size_t)(ga * 4 + r) * N + j] * per_lane);
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            if (j < N && (lane & 3) == 0 && s > 0.f) {
                int delta = gd / S - ga / S;
                if (delta < 0) delta += P;
                if (P == 1 ? ga != gd : delta != 0)
                    atomicMax(&lanes[(delta * S + ga % S) * S + gd % S], (int)fminf(s, 1e6f));
            }
        }
    }
    __syncthreads();
    for (int e = tid; e < G * S; e += BIG_KEY_THREADS) {
        atomicAdd(&rail[e / S % S], lanes[e]);
        atomicAdd(&rail[S + e % S], lanes[e]);
    }
    __syncthreads();
    if (tid == 0) {
        int most = 0;
        for (int q = 0; q < 2 * S; q++) most = max_v(most, rail[q]);
        key[b] = most;
    }
}
// ... and every matrix finds its place by counting the matrices that go before it (a larger key, or the same
// and a lower index): B^2 comparisons over the whole grid, a few microseconds for a few thousand matrices.
__global__ void __launch_bounds__(256) big_rank_kernel(const int* __restrict__ key, int B, int* __restrict__ order) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= B) return;
    const int mine = key[b];
    int before = 0;
    for (int o = 0; o < B; o++) {
        const int other = __ldg(&key[o]);
        before += other > mine || (other == mine && o < b);
    }
    order[before] = b;
}

// LANES lanes per (family, start) task, SPLIT per rank group (LANES / SPLIT >= G): with two, each lane has two of the four
// columns of a tile and half the reads and byte permutes, for six shuffles more -- two thirds of the instructions on the chain,
// a quarter more in all, so it is taken while the batch leaves SMs room.  Up to 32 lanes a task is part of a warp, 64 lanes
// are two warps that meet at a barrier of their own.  Task warps are the first warps of the CTA (kp.big_task_warps),
// the threads from warp kp.big_emit_warp on emit, a slot each.
// ONE: all paths have one rate, so every slot the same capacity.  Selected per slot at run time it costs 7 to 13 %: 16 and 1,024 matrices
// of 64 ranks 519 -> 555 and 1,187 -> 1,300 us, 512 of 256 ranks 9.95 -> 11.25 ms (two rates, links of 64 and NICs of 50 B/ns: 559 us,
// 1,300 us, 11.65 ms).
template <int LANES, int SPLIT, bool ONE>
__global__ void __launch_bounds__(LANES == 64 ? 384 : (SPLIT == 2 ? LANES * 6 : LANES * 8), LANES == 64 ? 1 : 64 / LANES)
vp_schedule_big_kernel(DevCat dc, KParams kp, const int64_t* __restrict__ demand, const int64_t* __restrict__ tau_in, int B,
                       int32_t* __restrict__ n_steps, int32_t* __restrict__ chan_id, int16_t* __restrict__ lane_dst,
                       uint16_t* __restrict__ lane_inst, int64_t* __restrict__ lane_bytes, int64_t* __restrict__ send_off,
                       int64_t* __restrict__ recv_off, int64_t* __restrict__ tau_out, int32_t* __restrict__ status,
                       unsigned int* counter, int* __restrict__ todo, const int* __restrict__ order) {
    // `order` (may be null) lists the matrices in the order in which the CTAs should take them: longest first.
    constexpr bool CROSS = LANES == 64;                   // a task is two warps
    constexpr bool RECORD = CROSS && SPLIT == 1;          // task warps emit, the others write the rows
    constexpr bool EXACT = RECORD;                        // credits of hot columns from the words at hand (the other kernels lost 1 to 3 % on every matrix by it)
    constexpr bool IN_ORDER = CROSS || SPLIT == 2;        // page-locked plans: receive offsets in rank order (the kernels that pack SMs
                                                          // have no register to spare: there it cost every plan 6 %)
    constexpr int WL = CROSS ? 32 : LANES;                // a task's lanes in one warp
    constexpr int TPW = 32 / WL, QN = 4 / SPLIT;          // tasks per warp, columns per lane
    constexpr int ST = big_stride(LANES / SPLIT);         // words per row pair of the credit matrix
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = dc.N, G = dc.G, tid = threadIdx.x, NT = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, n_warps = NT >> 5;
    const BigSmem L = big_smem_layout(dc, kp);
    uint32_t* const wd = (uint32_t*)(smem_raw + L.wd);
    uint32_t* const tbl = (uint32_t*)(smem_raw + L.tbl);
    uint16_t* const Hi = (uint16_t*)(smem_raw + L.hi);
    uint8_t* const colmap = smem_raw + L.colmap;
    uint8_t* const gnode = smem_raw + L.gnode;            // per group: node index, then (at G) rail index
    int64_t* const send_acc = (int64_t*)(smem_raw + L.send_acc);
    int64_t* const recv_acc = (int64_t*)(smem_raw + L.recv_acc);
    uint64_t* const red = (uint64_t*)(smem_raw + L.red);
    uint32_t* const task_f = (uint32_t*)(smem_raw + L.task_f);
    int64_t* const task_den = (int64_t*)(smem_raw + L.task_den);
    uint16_t* const bindings = (uint16_t*)(smem_raw + L.bind);
    uint32_t* const bucket = (uint32_t*)(smem_raw + L.bucket);
    // Big cells (16-bit mode): a cell of big_floor granules or more holds big_floor + its index in the side list, where
    // its exact value is kept.  Every capacity is below big_floor, so such a cell gives the same credit as its value.
    uint32_t* const side = (uint32_t*)(smem_raw + L.hi);
    const int big_max = min(BIG_HOT_MAX * N / 2, 4096), big_floor = 65536 - big_max;
    __shared__ int s_b, s_flags, s_mode, s_nhot, s_nbig;           // s_mode: 0 leave to the general kernel, 1 plain, 2 hot columns
    __shared__ int s_hot, s_beyond[BIG_HOT_MAX];          // cells that are 2^16 granules or more still, in all and per hot column
    __shared__ int64_t s_tau, s_left;
    __shared__ int2 s_pick;                               // first family and families of the shape chosen (none: nothing is covered)
    __shared__ int64_t s_tscale[VP_MAX_CLASSES];
    __shared__ uint32_t s_cap[VP_MAX_CLASSES];
    __shared__ __align__(8) unsigned long long s_stage_bar;
    unsigned long long n_act = 0;
    unsigned n_done = 0;
    Counters cnt;                                         // phase cycle counts (only with VP_PHASE_TIMING)
    cnt.t_mark = 0;
    for (int i = 0; i < 6; i++) cnt.cyc[i] = 0;
    const int ns_pad = (dc.n_shapes + 31) & ~31;
    const int S = dc.S, P = dc.P;
    const bool by_class = big_by_class(dc);

    const double inv_bw = 1.0 / (double)dc.bw_max;
    // ---- stage the catalog once per CTA: bulk asynchronous copies (TMA) onto one mbarrier; should the bounded wait give
    // up, plain loads fetch the same arrays
    {
        const void* from[4] = {dc.bucket_ptr, dc.shape_pat, dc.pat_term, dc.fam_task};
        const int at[4] = {L.bucket, L.term, L.pat, L.fam_task};
        const int bytes[4] = {align16((dc.n_shapes + 1) * 4), by_class ? 0 : ns_pad * L.pat_words * 4,
                              by_class ? 0 : align16(dc.n_patterns * dc.max_row_terms * 4), kp.big_stage ? dc.n_families * G * 32 : 0};
        const unsigned bar = smem_u32(&s_stage_bar);
        if (tid == 0) {
            mbar_init(bar, 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            unsigned all = 0;
            for (int i = 0; i < 4; i++) all += (unsigned)bytes[i];
            mbar_expect_tx(bar, all);
            for (int i = 0; i < 4; i++)
                if (bytes[i]) bulk_load(smem_u32(smem_raw + at[i]), from[i], (unsigned)bytes[i], bar);
        }
        __syncthreads();
        if (!__syncthreads_and(mbar_wait_bounded(bar, 0, 1u << 20))) {
            for (int i = 0; i < 4; i++)
                for (int e = tid; e < bytes[i] / 4; e += NT) ((uint32_t*)(smem_raw + at[i]))[e] = ((const uint32_t*)from[i])[e];
        }
        for (int a = tid; a < G; a += NT) { gnode[a] = (uint8_t)(a / S); gnode[G + a] = (uint8_t)(a % S); }
        for (int e = tid; e < L.fill_rows * N * 8 / 16; e += NT) {       // fill buffers: all ones, then zeros
            ((uint4*)(smem_raw + L.fill))[e] = make_uint4(0xffffffffu, 0xffffffffu, 0xffffffffu, 0xffffffffu);
            ((uint4*)(smem_raw + L.fill + L.fill_rows * N * 8))[e] = make_uint4(0u, 0u, 0u, 0u);
        }
        __syncthreads();
    }
    // ---- what a thread keeps of the catalog for Step 1 (see (A) below)
    uint64_t* const rs = (uint64_t*)(smem_raw + L.rs);
    const uint32_t* const pat = by_class ? dc.pat_term : (const uint32_t*)(smem_raw + L.pat);
    const uint32_t* const spat = by_class ? dc.shape_pat : (const uint32_t*)(smem_raw + L.term);
    constexpr bool BY_LANE = LANES / SPLIT <= 16;         // a first and a second row per lane, else up to BIG_CHUNKS chunks per warp
    constexpr int ROWS = BY_LANE ? 2 : BIG_CHUNKS;
    uint4 row[ROWS];
    int unit0 = 0, unit0_end = 0, unit1 = 0, unit1_end = 0, unit_span = 1;   // lane = class: chunks of its two units; most chunks of a unit
    if (by_class) {
        if constexpr (BY_LANE) {
            row[0] = __ldg((const uint4*)dc.lane_rows + lane);
            row[1] = __ldg((const uint4*)dc.lane_rows + 32 + lane);
        } else {
#pragma unroll
            for (int i = 0; i < ROWS; i++) {
                const int c = warp + i * n_warps;
                row[i] = __ldg((const uint4*)(dc.dec + dc.dec[2]) + min(c, dc.dec_chunks - 1) * 32 + lane);
            }
            if (lane < dc.dec_classes) {
                unit0 = (int)dc.dec[3 + 2 * lane]; unit0_end = unit1 = (int)dc.dec[4 + 2 * lane]; unit1_end = (int)dc.dec[5 + 2 * lane];
            }
            unit_span = (int)__reduce_max_sync(0xffffffffu, (unsigned)max(1, max(unit0_end - unit0, unit1_end - unit1)));
        }
    }
    auto row_score = [&](const uint4& w) {
        return tbl[w.x & 0xffffu] * (w.x >> 16) + tbl[w.y & 0xffffu] * (w.y >> 16) + tbl[w.z & 0xffffu] * (w.z >> 16);
    };
    constexpr bool one_class = ONE;
    const int n_task_warps = kp.big_task_warps, emit_warp = kp.big_emit_warp;
    const int r_emit = tid - emit_warp * 32;              // this thread's slot when it emits
    const int emit_threads = (N + 31) & ~31;              // whole warps
    const bool emits = r_emit >= 0 && r_emit < N, emit_warps = r_emit >= 0 && r_emit < emit_threads;
    // this thread's place in Step 2: task group (warp, or pair of warps), lane of the task, rank group and columns
    const int wg = CROSS ? warp >> 1 : warp, sub = CROSS ? warp & 1 : 0, n_tg = CROSS ? n_task_warps >> 1 : n_task_warps;
    const int tl = CROSS ? sub * 32 + lane : lane & (WL - 1), tsub = CROSS ? 0 : lane / WL, a = tl / SPLIT, part = tl - a * SPLIT;
    const unsigned tmask = WL == 32 ? 0xffffffffu : ((1u << (WL & 31)) - 1u) << (tsub * WL);   // the task's lanes
    unsigned my_sweeps = 0;
    // this lane's first task: its family (of those that compete) and initial binding
    const uint32_t first_task = big_family_and_start(wg * TPW + tsub, kp.n_start), dst_1 = first_task & 0xffu;
    const int h_1 = (int)(first_task >> 8);
    const int ag = a < G ? a : 0;                         // (spare lanes repeat group 0 and are ignored)
    uint8_t* const ex_src = smem_raw + L.exchange + wg * BIG_EXCHANGE;
    uint8_t* const ex_dst = ex_src + 64;
    volatile uint32_t* const ex_word = (volatile uint32_t*)(ex_src + 128);
    volatile int64_t* const ex_time = (volatile int64_t*)(ex_src + 160);
    auto task_sync = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(1 + wg) : "memory"); };
    uint32_t tags[3][QN];                                 // big_tag of this lane's columns (two lanes per group)
#pragma unroll
    for (int r = 0; r < 3; r++)
#pragma unroll
        for (int i = 0; i < QN; i++) tags[r][i] = (uint32_t)(3 - r) << (6 - 2 * (part * QN + i));
    const int fill_warp = n_warps - 1;                    // issues the fill (only in CTAs with warps that hold no task)

    for (;;) {
        if (tid == 0) {
            const unsigned at = atomicAdd(counter, 1u);
            s_b = at < (unsigned)B ? (order ? order[at] : (int)at) : B;
            s_flags = 0;
        }
        __syncthreads();
        const int b = s_b;
        if (b >= B) break;
#ifdef VP_PHASE_TIMING
        cnt.t_mark = clock64();
#endif
        const int64_t* D = demand + (size_t)b * N * N;
        if (RECORD) big_prefetch(D, N);
        const size_t lane_base = (size_t)b * kp.k_max * N, off_base = (size_t)b * (kp.k_max + 1) * N;
        int32_t* chan_id_b = chan_id + (size_t)b * kp.k_max;
        int16_t* lane_dst_b = lane_dst + lane_base;
        uint16_t* lane_inst_b = lane_inst + lane_base;
        int64_t* lane_bytes_b = lane_bytes + lane_base;
        int64_t* send_off_b = send_off + off_base;
        int64_t* recv_off_b = recv_off ? recv_off + off_base : nullptr;

        // ---- pass 1 over D: validate; row sums, column sums and group sums (Eq. 5) into the set-up area
        int64_t* Dhat = (int64_t*)(smem_raw + L.wd);
        int64_t* rowsum = Dhat + G * G;
        int64_t* colsum = rowsum + N;
        int64_t* colmax = colsum + N;
        uint32_t* const colpart = (uint32_t*)colsum;          // [j] low 24 bits of the column's parts, [N + j] the rest (added up below)
        uint32_t* const coltop = (uint32_t*)colmax;           // largest entry of the column >> 8
        for (int i = tid; i < N; i += NT) { colpart[i] = 0; colpart[N + i] = 0; coltop[i] = 0; send_acc[i] = 0; recv_acc[i] = 0; colmap[i] = BIG_HOT_MAX; if (EXACT) Hi[BIG_HOT_MAX * N + i] = 0; }
        if (EXACT) for (int i = tid; i < BIG_HOT_MAX; i += NT) s_beyond[i] = 0;
        if (tid == 0) { s_nhot = 0; s_nbig = 0; if (EXACT) s_hot = 0; }
        __syncthreads();
        int flags = 0;
        // One warp per source group, 32 columns per load, four rows in flight at once (one of eight pieces) and their sums side by side.
        // An entry's checks are bits that must not be there: of its value from 2^40 on, of the diagonal, of the difference to the next
        // multiple of the granule (entries are below 2^40, so a product with the reciprocal rounds to the quotient of a multiple).
        // Column sums as two 32-bit atomics, as 64-bit ones are loops.  Row by row, with 64-bit remainders, this and the second
        // pass took 45,000 of 912,000 cycles of a matrix of 64 ranks, 134,000 of 1,600,000 with eight CTAs on the SM.
        constexpr int CW = LANES / SPLIT * 4 / 32;           // 32-column pieces of a row
        constexpr int RB = CW <= 4 ? 4 : 1;                  // (256 ranks: with two rows the loop behind lost 1 % to registers)
        const double inv_granule = kp.inv_granule;
        const auto col_sum = [&](int j) { return ((int64_t)colpart[N + j] << 24) + colpart[j]; };
        for (int ga = warp; ga < G; ga += n_warps) {
            int64_t colv[CW];
            uint32_t colm[CW];
            uint64_t wrong = 0;
#pragma unroll
            for (int m = 0; m < CW; m++) { colv[m] = 0; colm[m] = 0; }
#pragma unroll 1
            for (int i4 = 0; i4 < 4; i4 += RB) {
                const int64_t* row = D + (size_t)(ga * 4 + i4) * N;
                int64_t v[RB][CW], rsum[RB];
#pragma unroll
                for (int r = 0; r < RB; r++)
#pragma unroll
                    for (int m = 0; m < CW; m++) v[r][m] = m * 32 + lane < N ? row[r * N + m * 32 + lane] : 0;
#pragma unroll
                for (int r = 0; r < RB; r++) {
                    rsum[r] = 0;
#pragma unroll
                    for (int m = 0; m < CW; m++) {
                        const int64_t x = v[r][m];
                        wrong |= (uint64_t)x >> 40 | (uint64_t)(__double2ll_rn((double)x * inv_granule) * kp.granule ^ x);
                        if (m * 32 + lane == ga * 4 + i4 + r) wrong |= (uint64_t)x;
                        rsum[r] += x;
                        colv[m] += x;
                        colm[m] = max_v(colm[m], (uint32_t)(x >> 8));
                    }
                }
#pragma unroll
                for (int o = 16; o; o >>= 1)
#pragma unroll
                    for (int r = 0; r < RB; r++) rsum[r] += __shfl_xor_sync(0xffffffffu, rsum[r], o);
                if (lane == 0)
#pragma unroll
                    for (int r = 0; r < RB; r++) rowsum[ga * 4 + i4 + r] = rsum[r];   // (rows of this group belong to this warp alone)
            }
#pragma unroll
            for (int m = 0; m < CW; m++) {
                const int j = m * 32 + lane;
                int64_t pair = colv[m];                          // sum over a destination group's four columns
                pair += __shfl_xor_sync(0xffffffffu, pair, 1);
                pair += __shfl_xor_sync(0xffffffffu, pair, 2);
                if (j < N) {
                    atomicAdd(&colpart[j], (uint32_t)colv[m] & 0xffffffu);
                    atomicAdd(&colpart[N + j], (uint32_t)(colv[m] >> 24));
                    atomicMax(&coltop[j], colm[m]);
                    if ((lane & 3) == 0) Dhat[ga * G + (j >> 2)] = pair;
                }
            }
            if (__any_sync(0xffffffffu, wrong != 0)) flags |= big_wrong_entries(D + (size_t)ga * 4 * N, N, ga, kp.granule);
        }
        const int64_t tau_given = tau_in ? tau_in[b] : 0;
        if (tid == 0 && (tau_given < 0 || tau_given > VP_ENTRY_LIMIT)) flags |= VP_ST_BAD_TAU;
        if (flags) atomicOr(&s_flags, flags);
        for (int i = tid; i < N; i += NT) {
            send_off_b[i] = 0;
            if (recv_off_b) recv_off_b[i] = 0;
        }
        __syncthreads();
        int st = s_flags;
        int k = 0;
        int64_t tau = 0;
        bool deferred = false;
        if (st == 0) {
            // ---- quantum (Section 5) and capacities
            const RowDiv by_bw{dc.bw_max, inv_bw};
            const auto ceil_div = [](int64_t x, const RowDiv& by) {
                if (rarely(x >= (int64_t)1 << 52)) return big_wide_ceil_div(x, by.d);
                int64_t rem;
                const int64_t q = by.div(x, rem);
                return q + (rem > 0);
            };
            int64_t tot = 0, most = 0;
            for (int i = tid; i < N; i += NT) {
                tot += rowsum[i];
                most = max_v(most, max_v(rowsum[i], col_sum(i)));
            }
            int64_t est = ceil_div(most, by_bw);
            for (int l = tid; l < dc.n_res; l += NT) {
                const uint32_t bwl = dc.forced_bw[l];
                if (!bwl) continue;
                int64_t f = 0;
                const uint32_t e1 = dc.forced_ptr[l + 1];
#pragma unroll 4
                for (uint32_t e = dc.forced_ptr[l]; e < e1; e++) f += Dhat[dc.forced_cell[e]];
                est = max_v(est, ceil_div(f, bwl == (uint32_t)dc.bw_max ? by_bw : RowDiv{(int64_t)bwl, 1.0 / (double)bwl}));
            }
            est = warp_max_i64(est);
            tot = warp_sum_i64(tot);
            if (lane == 0) { red[warp] = (uint64_t)est; red[32 + warp] = (uint64_t)tot; }
            __syncthreads();
            if (tid == 0) {
                int64_t e = 0, t = 0;
                for (int w = 0; w < n_warps; w++) { e = max_v(e, (int64_t)red[w]); t += (int64_t)red[32 + w]; }
                const RowDiv by_granule{kp.granule, inv_granule};
                int64_t rem;
                const int64_t tq = tau_given > 0 ? tau_given : max_v((int64_t)1, ceil_div(e, RowDiv{(int64_t)kp.k_target, 1.0 / (double)kp.k_target}));
                int64_t cap_max = 0;
                for (int cl = 0; cl < dc.n_classes; cl++) {
                    // in granules, at least one (rate x quantum may exceed what the reciprocal divides exactly)
                    const int64_t x = tq * dc.class_bw[cl];
                    const int64_t cp = max_v((int64_t)1, x < ((int64_t)1 << 52) ? by_granule.div(x, rem) : x / kp.granule);
                    cap_max = max_v(cap_max, cp);
                    s_cap[cl] = (uint32_t)min_v(cp, (int64_t)0xffffffffll);
                    s_tscale[cl] = dc.class_wdiv[cl] * kp.granule;
                }
                // 16-bit credits need capacities below 2^16 granules, hot columns capacities below 2^22 (four credits and
                // a tag share 32 bits); the 32-bit table needs fewer than 2^32 granules in all
                s_left = t < ((int64_t)1 << 52) ? by_granule.div(t, rem) : t / kp.granule;
                const bool fits = kp.granule >= 256 && s_left < ((int64_t)1 << 32);
                s_mode = !fits ? 0 : (cap_max < big_floor ? 1 : (cap_max < ((int64_t)1 << 22) ? 2 : 0));
                s_tau = tq;
            }
            __syncthreads();
            tau = s_tau;
            if (s_mode == 2) {                               // hot columns: those with a cell of 65,535 granules or more
                for (int j = tid; j < N; j += NT)
                    if (coltop[j] >= (uint32_t)min_v(65535 * kp.granule >> 8, (int64_t)0xffffffffll)) {   // (multiples of a granule of 256 or more)
                        const int at = atomicAdd(&s_nhot, 1);
                        if (at < BIG_HOT_MAX) colmap[j] = (uint8_t)at;
                    }
                __syncthreads();
                if (tid == 0 && s_nhot > BIG_HOT_MAX) s_mode = 0;
                __syncthreads();
            }
            deferred = s_mode == 0;
        }
        if (deferred) {
            // the general kernel takes this matrix (it validates and derives the quantum again)
            if (tid == 0) todo[atomicAdd(counter + 1, 1u)] = b;
            __syncthreads();
            continue;
        }
        // Idle rows are filled from the end of the plan towards the activations while the matrix is decomposed (fill_warp,
        // a block of 4 fill_rows rows per iteration): fill_lo is the first row already filled.
        const bool fills = RECORD && L.fill_rows > 0 && st == 0 && !kp.host_rows &&
            (((uintptr_t)lane_dst_b | (uintptr_t)lane_inst_b | (uintptr_t)lane_bytes_b | (uintptr_t)send_off_b |
              (uintptr_t)(recv_off_b ? recv_off_b : send_off_b)) & 15) == 0;
        const unsigned chunk = (unsigned)(L.fill_rows * N * 8);
        int fill_lo = kp.k_max;
        // rows [lo, hi) of one block, one copy per lane; hi - lo <= 4 fill_rows
        auto fill_block = [&](int lo, int hi) {
            const int R = L.fill_rows;
            int arr = lane, r0 = lo, r1 = hi, width = 2;
            if (lane >= 2) { arr = 2 + (lane - 2) / 4; r0 = lo + ((lane - 2) & 3) * R; r1 = min(r0 + R, hi); width = 8; }
            if (lane < 14 && r1 > r0) {
                unsigned char* const dst = arr == 0 ? (unsigned char*)lane_dst_b : arr == 1 ? (unsigned char*)lane_inst_b
                                         : arr == 2 ? (unsigned char*)lane_bytes_b : arr == 3 ? (unsigned char*)(send_off_b + N)
                                                    : (recv_off_b ? (unsigned char*)(recv_off_b + N) : nullptr);
                if (dst) bulk_store(dst + (size_t)r0 * N * width, smem_u32(smem_raw + L.fill) + (arr < 2 ? 0u : (unsigned)(arr - 1) * chunk),
                                    (unsigned)((r1 - r0) * N * width));
            }
            bulk_commit();
        };
        if (fills) {
            if (warp == fill_warp) bulk_wait_read<0>();      // the last matrix's copies have read the totals
            __syncthreads();
            unsigned char* const buf = smem_raw + L.fill;
            for (unsigned e = tid; e < chunk / 16; e += NT) {
                const int i2 = (int)(e % (unsigned)(N / 2));
                ((longlong2*)(buf + 2 * chunk))[e] = ((const longlong2*)rowsum)[i2];
                ((longlong2*)(buf + 3 * chunk))[e] = make_longlong2(col_sum(2 * i2), col_sum(2 * i2 + 1));
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        if (st == 0) {
            // ---- first score table from D-hat, in granules
            for (int e = tid; e < dc.tbl_size; e += NT) {
                const int q2 = e % S, q = (e / S) % S, delta = e / (S * S);
                int64_t s = 0;
                for (int n = 0; n < P; n++) {
                    int n2 = n + delta; if (n2 >= P) n2 -= P;
                    s += Dhat[(size_t)(n * S + q) * G + n2 * S + q2];
                }
                tbl[e] = (uint32_t)__double2ll_rn((double)s * inv_granule);      // (a multiple)
            }
            __syncthreads();
            // ---- pass 2 over D: the residual in granules as 16-bit cells (big cells through the side list)
            const bool hot_mode = s_mode == 2;
            uint16_t* const cells = (uint16_t*)wd;
            // a warp per pair of rows (a word of the matrix per column), 8 or 16 loads in flight
            constexpr int PU = CW >= 4 ? 1 : 4 / CW;
#pragma unroll 1
            for (int p0 = warp; p0 < N / 2; p0 += PU * n_warps) {
                int64_t raw[PU][2][CW];
#pragma unroll
                for (int u = 0; u < PU; u++)
#pragma unroll
                    for (int m = 0; m < CW; m++) {
                        const int p = p0 + u * n_warps, j = m * 32 + lane;
                        const bool in = p < N / 2 && j < N;
                        raw[u][0][m] = in ? D[2 * p * N + j] : 0;
                        raw[u][1][m] = in ? D[(2 * p + 1) * N + j] : 0;
                    }
#pragma unroll
                for (int u = 0; u < PU; u++)
#pragma unroll
                    for (int m = 0; m < CW; m++) {
                        const int p = p0 + u * n_warps, j = m * 32 + lane;
                        if (p >= N / 2 || j >= N) continue;
                        uint32_t v[2];
#pragma unroll
                        for (int r = 0; r < 2; r++) v[r] = (uint32_t)__double2ll_rn((double)raw[u][r][m] * inv_granule);
                        if (!hot_mode) {
                            if (rarely(max_v(v[0], v[1]) >= (uint32_t)big_floor)) {
#pragma unroll 1
                                for (int r = 0; r < 2; r++) {
                                    const uint32_t x = r ? v[1] : v[0];
                                    if (x < (uint32_t)big_floor) continue;   // a big cell: exact value in the side list, its index in the matrix
                                    const int at = atomicAdd(&s_nbig, 1);
                                    const uint32_t code = (uint32_t)big_floor + (uint32_t)min_v(at, big_max - 1);
                                    if (at < big_max) side[at] = x;
                                    if (r) v[1] = code; else v[0] = code;
                                }
                            }
                        } else if (colmap[j] != BIG_HOT_MAX) {   // exact: 32 bits in a hot column, below 65,535 elsewhere
#pragma unroll 1
                            for (int r = 0; r < 2; r++) {
                                const uint32_t high = (r ? v[1] : v[0]) >> 16;
                                Hi[(int)colmap[j] * N + 2 * p + r] = (uint16_t)high;
                                if (EXACT && high) { atomicAdd(&s_beyond[colmap[j]], 1); atomicAdd(&s_hot, 1); }
                            }
                        }
                        wd[p * ST + j] = __byte_perm(v[0], v[1], 0x5410);
                    }
            }
            __syncthreads();
            if (s_nbig > big_max) {                          // more big cells than the side list holds: the general kernel's
                if (tid == 0) todo[atomicAdd(counter + 1, 1u)] = b;
                __syncthreads();
                continue;
            }
            // The loop, with and without hot columns: two copies, each with a short path (see "Code size" above).
            auto decompose = [&](auto hot_columns) {
                constexpr bool HOT = decltype(hot_columns)::value;
                uint32_t left = (uint32_t)s_left;                  // (below 2^32 granules, see s_mode)
                const uint32_t by_class_below = by_class ? 1u << 30 : 0u;
                const BigCredits cr{wd, Hi, colmap, ST, N, HOT};
                const uint32_t cap0 = s_cap[0], cap2 = min_v(cap0, 65535u) * 0x00010001u;
                // An activation is first taken off the residual; its rows are written while the next one's tasks run: by the thread
                // that emitted the slot (p_*), or (RECORD) by the warps without a task, from the record of the slot.
                bool pend = false;
                int p_fam = 0;
                uint32_t p_bind = 0, p_x = 0;
                uint2* const record = (uint2*)(smem_raw + L.record);
                auto write_slot = [&](int kk, int r, int fam, uint32_t bind, uint32_t x, uint32_t inst) {
                    const int i = (int)(bind & 0xffu), j = (int)(bind >> 8);
                    const size_t row = (size_t)kk * N, orow = (size_t)(kk + 1) * N;
                    const int64_t bytes = (int64_t)x * kp.granule;
                    const int64_t sa = send_acc[i] + bytes, ra = recv_acc[j] + bytes;
                    send_acc[i] = sa;                             // (src and dst are permutations: every rank is written once)
                    recv_acc[j] = ra;
                    lane_dst_b[row + i] = x ? (int16_t)j : (int16_t)-1;
                    lane_bytes_b[row + i] = bytes;
                    send_off_b[orow + i] = sa;
                    if (recv_off_b && !(IN_ORDER && kp.host_rows)) recv_off_b[orow + j] = ra;
                    lane_inst_b[row + i] = x ? (uint16_t)inst : (uint16_t)0xFFFF;
                    if (r == 0) chan_id_b[kk] = fam;
            };
                auto write_row = [&](int kk, uint32_t inst) {
                    if (RECORD) {
                        const int fam = (int)record[N].x;
                        for (int r = tid - n_task_warps * 32; r < N; r += NT - n_task_warps * 32)
                            write_slot(kk, r, fam, record[r].x, record[r].y, __ldg(dc.fam_slot + (size_t)fam * N + r));
                    } else {
                        if (emit_warp > 0 && emits) inst = __ldg(dc.fam_slot + (size_t)p_fam * N + r_emit);
                        if (emits) write_slot(kk, r_emit, p_fam, p_bind, p_x, inst);
                    }
                    // (every lane of the writing warps comes here once per activation: pend is the same in a warp)
                    if (IN_ORDER && kp.host_rows && recv_off_b) {
                        const int first = RECORD ? n_task_warps * 32 : emit_warp * 32;
                        big_write_in_order<CROSS ? 5 : 1>(recv_off_b + (size_t)(kk + 1) * N, recv_acc, N, tid - first, RECORD ? NT - first : emit_threads);
                    }
                    pend = false;
                };
                VP_TICK(0);

                int f0 = 0, H = 0;                                 // first family and families of the shape chosen
                for (;;) {
                    if (rarely(left == 0 || k == kp.k_max)) {
                        if (left != 0) st |= VP_ST_STEP_LIMIT;
                        break;
                    }
                    // path instance of the slot to be written out, where task warps write it: a trip to L2 that ends long before then
                    const uint32_t inst = !RECORD && emit_warp == 0 && pend && emits ? __ldg(dc.fam_slot + (size_t)p_fam * N + r_emit) : 0u;
                    // (A) Eq. (6), class by class (two rails).  A shape is a first row p0 and a second row p1 from the list of p0's class, and
                    // its index grows with p0's place in shape order first, p1's place in the list second.  So within a class the
                    // first maximum is (first maximal p0, first maximal p1 of the list): two independent maxima.  32 bits hold every
                    // score while what is left is below 2^30 (a score is at most four times that); 1 is added so that any row beats none.
                    int best_s = -1;
                    if (usually(left < by_class_below)) {
                        if constexpr (BY_LANE) {
                            // Every task warp by itself, a first and a second row per lane: no barrier.  A first row adds the largest second row
                            // of its class; among equal sums the lowest run start is the lowest shape, as the runs do not overlap.
                            if (warp < n_task_warps) {
                                const uint32_t v0 = row_score(row[0]) + 1u, v1 = row_score(row[1]) + 1u;
                                uint32_t m1[5], sum = 0;
#pragma unroll
                                for (int cl = 0; cl < 5; cl++) {
                                    m1[cl] = __reduce_max_sync(0xffffffffu, row[1].w >> cl & 1u ? v1 : 0u);
                                    if ((row[0].w & 7u) == (uint32_t)cl) sum = v0 + m1[cl];
                                }
                                const uint32_t best = __reduce_max_sync(0xffffffffu, sum);
                                const uint32_t first = __reduce_min_sync(0xffffffffu, sum == best ? row[0].w : 0xffffffffu);
                                const uint32_t cl = first & 7u;
                                uint32_t most = m1[0];
#pragma unroll
                                for (int o = 1; o < 5; o++) if (cl == (uint32_t)o) most = m1[o];
                                const uint32_t place = __reduce_min_sync(0xffffffffu, (row[1].w >> cl & 1u) && v1 == most ? row[1].w >> (5u + 5u * cl) & 31u : 31u);
                                if (best > 2u) best_s = (int)((first >> 3) + place);
                            }
                        } else {
                            // A warp per chunk of 32 rows, in shape order: the first lane with the chunk's largest score leaves it with its
                            // tie-break word (run start or place in the list); every task warp combines them, a class per lane.
                            uint2* const chunk_best = (uint2*)red;
#pragma unroll
                            for (int i = 0; i < ROWS; i++) {
                                const int c = warp + i * n_warps;
                                if (c < dc.dec_chunks) {
                                    const uint32_t v = row[i].w == 0xffffffffu ? 0u : row_score(row[i]) + 1u, m = __reduce_max_sync(0xffffffffu, v);
                                    const unsigned who = __ballot_sync(0xffffffffu, v == m);
                                    if (lane == __ffs((int)who) - 1) chunk_best[c] = make_uint2(m, row[i].w);
                                }
                            }
                            __syncthreads();
                            if (warp < n_task_warps) {
                                uint2 k0 = chunk_best[unit0], k1 = chunk_best[unit1];
                                for (int i = 1; i < unit_span; i++) {          // (units of more than 32 rows)
                                    const uint2 x0 = chunk_best[min(unit0 + i, dc.dec_chunks - 1)], x1 = chunk_best[min(unit1 + i, dc.dec_chunks - 1)];
                                    if (unit0 + i < unit0_end && x0.x > k0.x) k0 = x0;
                                    if (unit1 + i < unit1_end && x1.x > k1.x) k1 = x1;
                                }
                                const uint32_t sum = lane < dc.dec_classes ? k0.x + k1.x : 0u, best = __reduce_max_sync(0xffffffffu, sum);
                                const uint32_t s = __reduce_min_sync(0xffffffffu, sum == best ? k0.y + k1.y : 0xffffu);
                                if (best > 2u) best_s = (int)s;
                            }
                        }
                    } else if (!BY_LANE && by_class) {
                        best_s = big_chunks_maximum(tbl, red, dc.dec, dc.dec_chunks, dc.dec_classes);
                    } else {
                        const uint64_t key = big_first_maximum(tbl, rs, red, pat, spat, dc.n_patterns, dc.max_row_terms, dc.n_shapes, S);
                        if (warp < n_task_warps && (key >> 16) != 0) best_s = 65535 - (int)(key & 0xffffu);
                    }
                    f0 = (int)bucket[max(best_s, 0)];              // (warps without a task learn them after Step 2)
                    H = best_s >= 0 ? (int)bucket[best_s + 1] - f0 : 0;
                    if (tid == 0) s_pick = make_int2(f0, H);
                    const int n_tasks = H * kp.n_start;
                    VP_TICK(1);

                    const bool hot = EXACT && HOT && s_hot > 0;            // (none beyond 16 bits left: the 16-bit credits are exact)
                    // (B) MultiStartAA: LANES lanes per (family, start), SPLIT of them per rank group.
                    //
                    // A binding travels as the low byte of a group's best key: the tag 3 - row of position 0 in its two highest bits,
                    // of position 3 in the lowest.  An in-slot finds the tag of its slot in the byte of the slot's source group, an
                    // out-slot the tag of its destination likewise: by a shuffle inside a warp, through shared memory between two.
                    // Slot words (see DevCat::fam_task): place of the cells for tag 0, owning group, class, shift of the tag.
                    uint32_t uo[QN], ui[QN];
                    auto fetch_slots = [&](int f) {
                        const unsigned at = ((unsigned)f * (unsigned)G + (unsigned)ag) * 32u + (SPLIT == 2 ? 8u * (unsigned)part : 0u);
                        auto take = [&](const unsigned char* row) {
                            if constexpr (SPLIT == 1) {
                                const uint4 o = *(const uint4*)row, i = *(const uint4*)(row + 16);
                                uo[0] = o.x; uo[1] = o.y; uo[QN - 2] = o.z; uo[QN - 1] = o.w;
                                ui[0] = i.x; ui[1] = i.y; ui[QN - 2] = i.z; ui[QN - 1] = i.w;
                            } else {
                                const uint2 o = *(const uint2*)row, i = *(const uint2*)(row + 16);
                                uo[0] = o.x; uo[1] = o.y;
                                ui[0] = i.x; ui[1] = i.y;
                            }
                        };
                        if (SPLIT == 2 ? usually(kp.big_stage) : rarely(kp.big_stage)) take(smem_raw + L.fam_task + at);
                        else take((const unsigned char*)dc.fam_task + at);
                    };
                    int task0 = warp < n_task_warps ? wg * TPW : n_tasks;
                    uint32_t dst = dst_1;
                    if (usually(task0 < n_tasks)) fetch_slots(f0 + min(h_1, H - 1));     // (a lane without a task repeats another's reads)
                    // ---- rows of the last activation, while the tables travel, and a block of the fill
                    if (SPLIT == 2 || RECORD ? rarely(pend) : usually(pend)) write_row(k - 1, inst);
                    if (RECORD && fills && warp == fill_warp) {
                        if (fill_lo <= k + 1) {                    // the activations have reached filled rows: those copies must be over
                            bulk_wait_all();
                            asm volatile("fence.proxy.async;" ::: "memory");
                        } else if (fill_lo - 2 * L.fill_rows >= k + 64) {       // (8 rows: with 16 the SMs write 5.9 TB/s in bursts, 512 x 256 ranks 10.57 -> 10.71 ms; with 4 10.8)
                            fill_block(fill_lo - 2 * L.fill_rows, fill_lo);
                            fill_lo -= 2 * L.fill_rows;
                        }
                    }

                    if (usually(task0 < n_tasks)) {
                        for (;;) {
                            const int task = min(task0 + tsub, n_tasks - 1);
                            const bool mine = TPW == 1 || task0 + tsub < n_tasks, act = mine && a < G;
                            uint32_t src = 0x100u;                 // (no binding yet)
                            int dt[QN];                            // tag (3 - row) each out-slot's destination has
                            auto fetch_dst = [&]() {
#pragma unroll
                                for (int i = 0; i < QN; i++) {
                                    if (CROSS) dt[i] = (int)(((unsigned)ex_dst[(uo[i] >> 16) & 0xffu] >> (uo[i] >> 28)) & 3u);
                                    else dt[i] = (int)((__shfl_sync(0xffffffffu, dst, (int)(uo[i] >> (17 - SPLIT)), WL) >> (uo[i] >> 28)) & 3u);
                                }
                            };
                            // best key of the group's 4 x 4 tile: v holds this lane's columns
                            auto best_key = [&](const uint32_t (&v)[4][QN]) {
                                if constexpr (SPLIT == 1) {
                                    return big_best_key(v);
                                } else {                           // both columns of a pair of rows; the other lane has the other two columns
                                    const uint32_t p01 = add_max(v[0][0], v[1][1], v[1][0] + v[0][1]), p02 = add_max(v[0][0], v[2][1], v[2][0] + v[0][1]);
                                    const uint32_t p03 = add_max(v[0][0], v[3][1], v[3][0] + v[0][1]), p12 = add_max(v[1][0], v[2][1], v[2][0] + v[1][1]);
                                    const uint32_t p13 = add_max(v[1][0], v[3][1], v[3][0] + v[1][1]), p23 = add_max(v[2][0], v[3][1], v[3][0] + v[2][1]);
                                    const uint32_t o01 = __shfl_xor_sync(0xffffffffu, p01, 1), o02 = __shfl_xor_sync(0xffffffffu, p02, 1);
                                    const uint32_t o03 = __shfl_xor_sync(0xffffffffu, p03, 1), o12 = __shfl_xor_sync(0xffffffffu, p12, 1);
                                    const uint32_t o13 = __shfl_xor_sync(0xffffffffu, p13, 1), o23 = __shfl_xor_sync(0xffffffffu, p23, 1);
                                    const uint32_t m0 = add_max(p01, o23, add_max(p02, o13, p03 + o12)), m1 = add_max(p12, o03, add_max(p13, o02, p23 + o01));
                                    return max_v(m0, m1);
                                }
                            };
                            auto tile_column = [&](uint32_t (&v)[4][QN], int i, uint32_t lo, uint32_t hi) {
                                v[0][i] = __byte_perm(lo, SPLIT == 1 ? big_tag(0, i) : tags[0][i], 0x5104);      // (low half) << 8 | tag
                                v[1][i] = __byte_perm(lo, SPLIT == 1 ? big_tag(1, i) : tags[1][i], 0x5324);      // (high half) << 8 | tag
                                v[2][i] = __byte_perm(hi, SPLIT == 1 ? big_tag(2, i) : tags[2][i], 0x5104);
                                v[3][i] = __byte_perm(hi, 0u, 0x5324);                                           // (row 3 has tag 0)
                            };
                            auto cap_of = [&](uint32_t w) { return one_class ? cap0 : s_cap[(w >> 24) & 0xfu]; };
                            auto cap2_of = [&](uint32_t w) { return one_class ? cap2 : min_v(s_cap[(w >> 24) & 0xfu], 65535u) * 0x00010001u; };
                            // exact credit in place of the 16-bit one (the tag byte stays)
                            auto hot_credit = [&](uint32_t& key, uint32_t cell, uint32_t cap) { key = __byte_perm(key, min_v(cell, cap), 0x6540); };
                            // source half: one exact assignment per source group
                            auto source_half = [&]() {
                                uint32_t v[4][QN];
#pragma unroll
                                for (int i = 0; i < QN; i++) {
                                    const uint32_t* const at = wd + ((int)(uo[i] & 0xffffu) - dt[i]);
                                    const uint32_t c2 = cap2_of(uo[i]);
                                    tile_column(v, i, __vminu2(at[0], c2), __vminu2(at[ST], c2));
                                }
                                if (!EXACT && HOT) {          // out-slots bound to a hot column: exact 32-bit cells
#pragma unroll
                                    for (int i = 0; i < QN; i++) {
                                        const int j = (int)((uo[i] >> 16) & 0xffu) * 4 + 3 - dt[i];
                                        if (colmap[j] != BIG_HOT_MAX) {
#pragma unroll
                                            for (int r = 0; r < 4; r++)
                                                v[r][i] = min_v(cr.cell(ag * 4 + r, j), cap_of(uo[i])) * 256u + (v[r][i] & 0xffu);
                                        }
                                    }
                                }
                                if (hot) {                         // the same from the words at hand
#pragma unroll
                                    for (int i = 0; i < QN; i++) {
                                        const int col = colmap[((uo[i] >> 16) & 0xffu) * 4 + 3 - dt[i]];
                                        if (col != BIG_HOT_MAX) {
                                            const uint2 h = *(const uint2*)(Hi + col * N + ag * 4);
                                            const uint32_t* const at = wd + ((int)(uo[i] & 0xffffu) - dt[i]);
                                            const uint32_t lo = at[0], hi = at[ST], cap = cap_of(uo[i]);
                                            hot_credit(v[0][i], __byte_perm(lo, h.x, 0x5410), cap);
                                            hot_credit(v[1][i], __byte_perm(lo, h.x, 0x7632), cap);
                                            hot_credit(v[2][i], __byte_perm(hi, h.y, 0x5410), cap);
                                            hot_credit(v[3][i], __byte_perm(hi, h.y, 0x7632), cap);
                                        }
                                    }
                                }
                                return best_key(v) & 0xffu;
                            };
#pragma unroll
                            for (int i = 0; i < QN; i++) dt[i] = (int)((dst >> (uo[i] >> 28)) & 3u);   // (every group starts from the same binding)
                            uint32_t src_new = source_half();
                            int F_old = -1;                        // this lane's task; the same in all its lanes, as alive is
                            bool alive = mine;                     // (the only task of a warp lives until its loop ends)
                            for (int sweep = 0; ; sweep++) {
                                // If no source binding of a task moved, the destination half would see what it saw last sweep and
                                // return the same binding and the same F: the run ends here exactly as it would after computing that.
                                // (Spare lanes follow group 0, so they need no mask.)
                                unsigned who = __ballot_sync(0xffffffffu, alive && src_new != src);
                                if (alive) src = src_new;
                                if (CROSS) {
                                    if (SPLIT == 1 || part == 0) ex_src[a] = (uint8_t)src;
                                    if (lane == 0) ex_word[sub] = who;
                                    task_sync();
                                    who = ex_word[0] | ex_word[1];
                                }
                                if constexpr (TPW == 1) {
                                    if (who == 0) { my_sweeps++; break; }
                                } else {
                                    if (alive && !(who & tmask)) { my_sweeps++; alive = false; }
                                    if (!__any_sync(0xffffffffu, alive)) break;
                                }
                                // destination half: the tags of the in-slots' sources, the cells of their rows
                                uint32_t v[4][QN];
                                unsigned tag[QN];
#pragma unroll
                                for (int i = 0; i < QN; i++) {
                                    if (CROSS) tag[i] = (unsigned)ex_src[(ui[i] >> 16) & 0xffu] >> (ui[i] >> 28);
                                    else tag[i] = __shfl_sync(0xffffffffu, src, (int)(ui[i] >> (17 - SPLIT)), WL) >> (ui[i] >> 28);
                                    const uint4 w = *(const uint4*)(wd + ((int)(ui[i] & 0xffffu) - (int)((tag[i] >> 1) & 1u) * ST));
                                    const unsigned sel = 0x7632u - (tag[i] & 1u) * 0x2222u;        // high or low halves
                                    const uint32_t c2 = cap2_of(ui[i]);
                                    tile_column(v, i, __vminu2(__byte_perm(w.x, w.y, sel), c2), __vminu2(__byte_perm(w.z, w.w, sel), c2));
                                }
                                if (!EXACT && HOT && *((const uint32_t*)colmap + ag) != BIG_HOT_NONE) {
#pragma unroll
                                    for (int r = 0; r < 4; r++)
                                        if (colmap[ag * 4 + r] != BIG_HOT_MAX) {
#pragma unroll
                                            for (int i = 0; i < QN; i++)
                                                v[r][i] = min_v(cr.cell((int)((ui[i] >> 16) & 0xffu) * 4 + 3 - (int)(tag[i] & 3u), ag * 4 + r), cap_of(ui[i])) * 256u +
                                                          (v[r][i] & 0xffu);
                                        }
                                }
                                uint32_t cols;                     // hot columns among the ranks of this group
                                if (hot && (cols = *((const uint32_t*)colmap + ag)) != BIG_HOT_NONE) {
#pragma unroll
                                    for (int i = 0; i < QN; i++) {
                                        const uint16_t* const h = Hi + ((ui[i] >> 16) & 0xffu) * 4 + 3 - (tag[i] & 3u);
                                        const uint4 w = *(const uint4*)(wd + ((int)(ui[i] & 0xffffu) - (int)((tag[i] >> 1) & 1u) * ST));
                                        const unsigned sel = 0x5410u + (~tag[i] & 1u) * 0x0022u;   // its half, then the high half from the side array
                                        const uint32_t cap = cap_of(ui[i]);
                                        hot_credit(v[0][i], __byte_perm(w.x, h[(cols & 0xffu) * N], sel), cap);
                                        hot_credit(v[1][i], __byte_perm(w.y, h[(cols >> 8 & 0xffu) * N], sel), cap);
                                        hot_credit(v[2][i], __byte_perm(w.z, h[(cols >> 16 & 0xffu) * N], sel), cap);
                                        hot_credit(v[3][i], __byte_perm(w.w, h[(cols >> 24) * N], sel), cap);
                                    }
                                }
                                const uint32_t key = best_key(v);
                                unsigned who2 = __ballot_sync(0xffffffffu, alive && ((key ^ dst) & 0xffu) != 0);
                                if (alive) dst = key & 0xffu;
                                // Eq. (8): at most 2^8 lanes of less than 2^22 granules.  The next sweep's source half needs no F: it runs while
                                // the sum is under way and is dropped if the run ends.
                                const bool more = sweep + 1 < kp.i_aa;
                                uint32_t F = (TPW == 1 ? a < G && (SPLIT == 1 || part == 0) : act) ? key >> 8 : 0u;
                                if constexpr (TPW == 1) F = __reduce_add_sync(0xffffffffu, F);
                                if (CROSS) {
                                    if (SPLIT == 1 || part == 0) ex_dst[a] = (uint8_t)dst;
                                    if (lane == 0) { ex_word[2 + sub] = who2; ex_word[4 + sub] = F; }
                                    task_sync();
                                    who2 = ex_word[2] | ex_word[3];
                                    F = ex_word[4] + ex_word[5];
                                }
                                fetch_dst();
                                if (more && (TPW > 1 || who2 != 0)) src_new = source_half();
                                if constexpr (TPW > 1) {           // (both lanes of a group hold its credit)
#pragma unroll
                                    for (int o = SPLIT; o < WL; o <<= 1) F += __shfl_xor_sync(0xffffffffu, F, o);
                                }
                                // If no destination binding moved, the next sweep would be a repetition of this one (same sources, same
                                // destinations, same F) and would end the run, so it is counted and skipped.
                                if constexpr (TPW == 1) {
                                    my_sweeps++;
                                    const bool up = (int)F > F_old && more;
                                    F_old = (int)F;
                                    if (!up) break;
                                    if (who2 == 0) { my_sweeps++; break; }
                                } else {
                                    if (alive) {
                                        my_sweeps++;
                                        alive = (int)F > F_old && more;
                                        F_old = (int)F;
                                        if (alive && !(who2 & tmask)) { my_sweeps++; alive = false; }
                                    }
                                    if (!__any_sync(0xffffffffu, alive)) break;
                                }
                            }
                            // Eq. (9) volumes of the binding as it stands and the slowest lane of Eq. (10): only needed when several
                            // families compete on utility
                            int64_t tmax = 0;
                            uint32_t bind[QN];                     // source and destination rank of every out-slot
#pragma unroll
                            for (int i = 0; i < QN; i++)
                                bind[i] = (uint32_t)(ag * 4 + 3 - (int)((src >> (6 - 2 * (part * QN + i))) & 3u)) |
                                          (uint32_t)((int)((uo[i] >> 16) & 0xffu) * 4 + 3 - dt[i]) << 8;
                            if (rarely(H > 1)) {
                                if (act) {
#pragma unroll
                                    for (int i = 0; i < QN; i++) {
                                        const uint32_t cl = (uo[i] >> 24) & 0xfu;
                                        tmax = max_v(tmax, (int64_t)min_v(cr.cell((int)(bind[i] & 0xffu), (int)(bind[i] >> 8)), s_cap[cl]) * s_tscale[cl]);
                                    }
                                }
#pragma unroll
                                for (int o = WL / 2; o; o >>= 1) tmax = max_v(tmax, __shfl_xor_sync(0xffffffffu, tmax, o));
                                if (CROSS) {
                                    if (lane == 0) ex_time[sub] = tmax;
                                    task_sync();
                                    tmax = max_v(ex_time[0], ex_time[1]);
                                }
                            }
                            if (act) {
                                uint32_t* const at = (uint32_t*)(bindings + (size_t)task * N + a * 4 + part * QN);
                                at[0] = bind[0] | bind[1] << 16;
                                if (QN == 4) at[1] = bind[QN - 2] | bind[QN - 1] << 16;
                            }
                            if (tl == 0 && mine) {
                                n_done++;
                                task_f[task] = (uint32_t)F_old;
                                if (H > 1) task_den[task] = F_old > 0 ? kp.lambda_ns * dc.W + tmax : 1;
                            }
                            task0 += n_tg * TPW;
                            if (usually(task0 >= n_tasks)) break;
                            // (further families)
                            const uint32_t next = big_family_and_start(min(task0 + tsub, n_tasks - 1), kp.n_start);
                            dst = next & 0xffu;
                            fetch_slots(f0 + (int)(next >> 8));
                            if (CROSS) task_sync();                // (the last task's bytes have been read)
                        }
                    }
                    __syncthreads();
                    VP_TICK(2);

                    // (C) best start per family (largest F, lowest t), then largest utility, lowest family
                    if (warp >= n_task_warps) { f0 = s_pick.x; H = s_pick.y; }
                    int wtask, wfam = f0;
                    uint32_t wF;
                    if (rarely(H == 0)) { st |= VP_ST_UNCOVERED; break; }
                    if (usually(H == 1 && kp.n_start == 4)) {                 // one family, four starts: best start, no utilities to compare
                        const uint4 f4 = *(const uint4*)task_f;
                        const uint32_t m01 = max_v(f4.x, f4.y), m23 = max_v(f4.z, f4.w);
                        wF = max_v(m01, m23);
                        wtask = m01 >= m23 ? (f4.x >= f4.y ? 0 : 1) : (f4.z >= f4.w ? 2 : 3);
                    } else if (H == 1) {
                        wtask = 0; wF = task_f[0];
#pragma unroll 1
                        for (int t = 1; t < kp.n_start; t++)
                            if (task_f[t] > wF) { wF = task_f[t]; wtask = t; }
                    } else {
                        const uint64_t chosen = big_select_family(task_f, task_den, H, kp.n_start, lane);
                        wtask = (int)(uint32_t)chosen; wF = (uint32_t)(chosen >> 32);
                        wfam += (int)(big_family_and_start(wtask, kp.n_start) >> 8);
                    }
                    if (rarely(wF == 0)) { st |= VP_ST_NO_PROGRESS; break; }
                    VP_TICK(3);

                    // (D) activation k: its volumes off the residual and off the score table
                    if (emits) {
                        const uint32_t bw = bindings[(size_t)wtask * N + r_emit];
                        const int i = (int)(bw & 0xffu), j = (int)(bw >> 8);
                        uint16_t* const cell = cells + ((i >> 1) * ST + j) * 2 + (i & 1);
                        uint32_t c = *cell, now_cell;
                        // the table entry of the slot's group pair
                        int entry;
                        if (S == 2) {
                            int delta = (j >> 3) - (r_emit >> 3);
                            if (delta < 0) delta += P;
                            entry = delta * 4 + ((r_emit >> 2) & 1) * 2 + ((j >> 2) & 1);
                        } else {
                            const int ga = r_emit >> 2, gd = j >> 2;
                            int delta = (int)gnode[gd] - (int)gnode[ga];
                            if (delta < 0) delta += P;
                            entry = (delta * S + gnode[G + ga]) * S + gnode[G + gd];
                        }
                        p_fam = wfam;
                        uint32_t cap = cap0;
                        if (!one_class) cap = s_cap[__ldg(dc.fam_cls + (size_t)p_fam * N + r_emit)];
                        if (!HOT) {
                            const uint32_t x = min_v(cap, c);
                            p_x = x;
                            if (rarely(c >= (uint32_t)big_floor)) {           // a big cell: exact value in the side list
                                const uint32_t now = side[c - big_floor] - x;
                                if (now >= (uint32_t)big_floor) { side[c - big_floor] = now; now_cell = c; }
                                else now_cell = now;                  // (an ordinary cell from here on)
                            } else {
                                now_cell = c - x;
                            }
                            *cell = (uint16_t)now_cell;
                        } else {
                            const int col = colmap[j];
                            uint16_t* const hcell = col != BIG_HOT_MAX ? Hi + col * N + i : nullptr;
                            if (hcell) c |= (uint32_t)*hcell << 16;   // a hot column: the exact 32-bit cell
                            p_x = min_v(cap, c);
                            *cell = (uint16_t)(c - p_x);
                            if (hcell) *hcell = (uint16_t)((c - p_x) >> 16);
                            if (EXACT && HOT && c >= 65536u && c - p_x < 65536u) {   // one less; a column without any is like the others from here on
                                atomicSub(&s_hot, 1);                 // (this column is this thread's for this activation)
                                if (--s_beyond[col] == 0) colmap[j] = BIG_HOT_MAX;
                            }
                        }
                        atomicSub(&tbl[entry], p_x);                  // (an idle lane takes zero)
                        p_bind = bw;
                        if (RECORD) {
                            record[r_emit] = make_uint2(bw, p_x);
                            if (r_emit == 0) record[N] = make_uint2((uint32_t)p_fam, 0u);
                        }
                    }
                    pend = RECORD ? warp >= n_task_warps : emit_warps;   // plan rows and offset sums follow (write_row)
                    left -= wF;
                    k++;
                    __syncthreads();
                    VP_TICK(4);
                }
                if (pend) write_row(k - 1, RECORD || !emits ? 0u : __ldg(dc.fam_slot + (size_t)p_fam * N + r_emit));   // the last activation of the matrix
            };
            if (hot_mode) decompose(BigConst<true>()); else decompose(BigConst<false>());
        }
        __syncthreads();
        // ---- idle rows beyond n_steps; offset rows repeat the totals
        if (fills && st == 0) {
            if (warp == fill_warp)                               // (the copies go on while the next matrix is decomposed)
                for (int hi = fill_lo; hi > k; hi -= 4 * L.fill_rows) fill_block(max(hi - 4 * L.fill_rows, k), hi);
        } else if (!kp.host_rows) {
            if (fills && warp == fill_warp) {                    // incomplete plan: the totals are not the demand's, fill again
                bulk_wait_all();
                asm volatile("fence.proxy.async;" ::: "memory");
            }
            __syncthreads();
            const bool off_aligned = (((uintptr_t)send_off_b | (uintptr_t)(recv_off_b ? recv_off_b : send_off_b)) & 15) == 0;
            const size_t lo = (size_t)k * N, hi = (size_t)kp.k_max * N;
            big_fill_bytes((unsigned char*)lane_dst_b, lo * 2, hi * 2, 0xff, tid, NT);
            big_fill_bytes((unsigned char*)lane_inst_b, lo * 2, hi * 2, 0xff, tid, NT);
            big_fill_bytes((unsigned char*)lane_bytes_b, lo * 8, hi * 8, 0x00, tid, NT);
            if (off_aligned) {                                   // N is a multiple of four: rows are whole 16-byte pairs
                const int half = N / 2, step = NT % half;
                int i2 = (int)((unsigned)(lo / 2 + tid) % (unsigned)half) - step;
                for (size_t e = lo / 2 + tid; e < hi / 2; e += NT) {
                    i2 += step;
                    if (i2 >= half) i2 -= half;
                    ((longlong2*)(send_off_b + N))[e] = ((const longlong2*)send_acc)[i2];
                    if (recv_off_b) ((longlong2*)(recv_off_b + N))[e] = ((const longlong2*)recv_acc)[i2];
                }
            } else {
                for (size_t e = lo + tid; e < hi; e += NT) {
                    const int i = (int)(e % N);
                    send_off_b[N + e] = send_acc[i];
                    if (recv_off_b) recv_off_b[N + e] = recv_acc[i];
                }
            }
        }
        for (int kk = k + tid; kk < kp.k_max && !kp.host_rows; kk += NT) chan_id_b[kk] = -1;
        if (tid == 0) {
            n_act += (unsigned long long)k;
            n_steps[b] = k;
            status[b] = st;
            if (tau_out) tau_out[b] = tau;
        }
        __syncthreads();
        VP_TICK(5);
    }
    bulk_wait_all();
    unsigned long long* stats = (unsigned long long*)(counter + 4);
    if (tid == 0 && n_act) atomicAdd(&stats[0], n_act);
    const unsigned long long n_tasks_done = (unsigned long long)warp_sum_i64((int64_t)n_done);   // (counted by the first lane of every task)
    const unsigned long long n_sweeps = (unsigned long long)warp_sum_i64(tl == 0 && warp < n_task_warps ? (int64_t)my_sweeps : 0);
    if (lane == 0 && n_tasks_done) { atomicAdd(&stats[1], n_tasks_done); atomicAdd(&stats[2], n_sweeps); }
#ifdef VP_PHASE_TIMING
    if (tid == 0) for (int i = 0; i < 6; i++) atomicAdd(&stats[3 + i], (unsigned long long)cnt.cyc[i]);
#endif
}

}  // namespace
