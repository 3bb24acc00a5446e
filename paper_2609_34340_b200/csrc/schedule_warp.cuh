// Algorithm 2 with ONE WARP per demand matrix, for catalogs of at most four groups of four ranks (N <= 16).
//
// A matrix this small has too little work per phase for a whole CTA: with several warps per matrix most of an
// iteration is spent in block barriers and in hand-overs through shared memory.  Here a warp owns a matrix from
// the first to the last activation and nothing but __syncwarp orders its phases.  Two forms of the main loop:
//
//  * decompose_units: capacities below 2^22 granules (granules of at least 256 bytes, so as a rule).  Bound by the chain of
//    dependent instructions of one activation, so each phase is cut to few of them, and what an ordinary activation does not
//    execute (families that compete, 64-bit scores) is out of line, because instructions come from small caches:
//    (A) a lane scores one row pattern of the catalog (source group x lane counts per destination group: at most 32), then
//        every shape is the sum of four row scores; two warp reductions leave the first maximum (Eq. 6);
//    (B) four starts at a time, two lanes per rank group: a lane reads two of the four columns of its group's 4 x 4 tile (one
//        16-byte read each, from credits kept ready) and the pair joins its halves of the exact assignment (Eq. 7) by six
//        shuffles.  A binding travels as one byte per group, by shuffle.  The next source half runs while Eq. (8) is summed;
//    (C) one warp maximum of F and start leaves the best start;
//    (D) sixteen lanes take the activation off the residual, the credits (row-major and transposed) and D-hat; its plan rows
//        are written in the shadow of the next activation's tasks.
//    One matrix of 8 ranks 38.1 -> 29.4 us, 256 of 16 ranks 104.6 -> 81.1, 4,096 of 8 ranks 147.9 -> 111.5 by the code out of
//    line, the credits kept ready and the last sweep's source half left out.
//  * decompose_bytes: any other matrix, the same algorithm on 64-bit bytes with a lane per rank group.
//
// A CTA is one to four such warps that share only the staged catalog.  Included by schedule.cu.
#pragma once

namespace {


struct WarpSmem {                           // byte offsets; the per-warp block comes first, once per warp
    int drem, dremT, cred, dhat, send_acc, recv_acc, rs, cap64, tscale, cap32, bind, bind_dst, per_warp;
    int rows, shape_rows, fam_task, term, fam_in, fam_cls, fam_slot, bucket, total;
};

// units: the tables of decompose_units are staged, otherwise those of decompose_bytes.
__host__ __device__ inline WarpSmem warp_smem_layout(const DevCat& dc, const KParams& kp, int n_warps, bool units) {
    WarpSmem L;
    const int ns_pad = (dc.n_shapes + 31) & ~31;
    int o = 0;
    // bytes: rows padded by one element, no bank conflicts down a column; 32-bit granules: residual, credits and their transpose
    L.drem = o;      o += align16(dc.N * (dc.N + 1) * 8 > 3 * dc.N * dc.N * 4 ? dc.N * (dc.N + 1) * 8 : 3 * dc.N * dc.N * 4);
    L.dremT = L.drem + dc.N * dc.N * 4;
    L.cred = L.dremT + dc.N * dc.N * 4;
    L.dhat = o;      o += align16(dc.G * dc.G * 8);
    L.send_acc = o;  o += dc.N * 8;
    L.recv_acc = o;  o += dc.N * 8;
    L.rs = o;        o += 272;                                 // row scores: 33 of 64 bits
    L.cap64 = o;     o += VP_MAX_CLASSES * 8;
    L.tscale = o;    o += VP_MAX_CLASSES * 8;
    L.cap32 = o;     o += VP_MAX_CLASSES * 4;
    L.bind = o;      o += align16(kp.max_tasks * dc.N);        // bytes: source of every slot; granules: with bind_dst, source | destination << 8
    L.bind_dst = o;  o += align16(kp.max_tasks * dc.N);
    L.per_warp = align16(o);
    o = L.per_warp * n_warps;
    L.rows = o;        o += dc.row_term ? 32 * 16 : 0;
    L.shape_rows = o;  o += dc.row_term ? ns_pad * 4 : 0;
    L.fam_task = o;    o += units ? dc.n_families * dc.G * 32 : 0;
    L.term = o;        o += units ? 0 : ns_pad * dc.max_terms * 4;
    L.fam_slot = o;    o += units ? 0 : align16(dc.n_families * dc.N * 4);
    L.fam_in = o;      o += units ? 0 : align16(dc.n_families * dc.N * 2);
    L.fam_cls = o;     o += units ? 0 : align16(dc.n_families * dc.N);
    L.bucket = o;      o += align16((dc.n_shapes + 1) * 4);
    L.total = o;
    return L;
}


extern __shared__ __align__(16) unsigned char vp_wsmem[];   // the CTA's dynamic shared memory

// Shared-memory byte offsets (into vp_wsmem), table and output pointers of one warp's matrix.  Offsets rather than
// pointers: every access is then provably a shared-memory access with a 32-bit address.
struct WCtx {
    int N, G, lane;
    unsigned o_drem, o_dremT, o_cred, o_dhat, o_send_acc, o_recv_acc, o_rs, o_cap64, o_cap32, o_tscale, o_bind, o_bind_dst;
    unsigned o_rows, o_shape_rows, o_fam_task, o_bucket;
    const uint32_t *term, *fam_slot;                            // (decompose_bytes: shared or global memory)
    const uint16_t* fam_in;
    const uint8_t* fam_cls;
    int32_t* chan_id_b;
    int16_t* lane_dst_b;
    uint16_t* lane_inst_b;
    int64_t *lane_bytes_b, *send_off_b, *recv_off_b;
};

template <typename T> __device__ __forceinline__ T* ws(unsigned off) { return (T*)(vp_wsmem + off); }

// Sum and maximum over the four lanes of a team (lane & ~3 .. lane | 3); every lane gets it.
__device__ __forceinline__ int64_t team_sum(int64_t v) {
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    return v + __shfl_xor_sync(0xffffffffu, v, 2);
}
__device__ __forceinline__ int64_t team_max(int64_t v) {
    v = max_v(v, __shfl_xor_sync(0xffffffffu, v, 1));
    return max_v(v, __shfl_xor_sync(0xffffffffu, v, 2));
}

// Eq. (6) by row patterns: this lane's pattern, and the patterns of its up to four shapes (a byte per source group; pattern 32 scores
// zero).
struct RowScores {
    bool on;
    unsigned rs;
    int n_shapes;
    uint4 row;
    uint32_t shape[4];
    __device__ __forceinline__ void load(const DevCat& dc, const WCtx& c) {
        on = dc.row_term != nullptr && dc.n_shapes <= 128;
        rs = c.o_rs;
        n_shapes = dc.n_shapes;
        if (c.lane == 0) ws<int64_t>(rs)[32] = 0;
        row = make_uint4(0u, 0u, 0u, 0u);
        if (on) row = *(ws<uint4>(c.o_rows) + c.lane);
#pragma unroll
        for (int u = 0; u < 4; u++) shape[u] = on && c.lane + 32 * u < n_shapes ? ws<uint32_t>(c.o_shape_rows)[c.lane + 32 * u] : 0x20202020u;
    }
    // largest score and, in best_s, the lane's first shape that has it (low words of D-hat); the scores travel by shuffles
    __device__ __forceinline__ uint32_t narrow(const uint32_t* dhat32, int lane, int& best_s) const {
        const uint32_t mine = dhat32[2 * (row.x & 0xffffu)] * (row.x >> 16) + dhat32[2 * (row.y & 0xffffu)] * (row.y >> 16) +
                              dhat32[2 * (row.z & 0xffffu)] * (row.z >> 16) + dhat32[2 * (row.w & 0xffffu)] * (row.w >> 16);
        uint32_t best = 0;
#pragma unroll
        for (int u = 0; u < 4; u++)
            if (u == 0 || n_shapes > (u < 3 ? 32 : 96)) {        // (a few shapes: one per lane)
                const uint32_t w = shape[u];                    // (a shuffle takes the source lane from the low five bits)
                uint32_t v = __shfl_sync(0xffffffffu, mine, (int)w) + __shfl_sync(0xffffffffu, mine, (int)(w >> 8)) +
                             __shfl_sync(0xffffffffu, mine, (int)(w >> 16)) + __shfl_sync(0xffffffffu, mine, (int)(w >> 24));
                if ((w & 0x20u) == 0 && v > best) { best = v; best_s = lane + 32 * u; }
            }
        return best;
    }
    __device__ __forceinline__ void wide(const int64_t* Dhat, int lane, int64_t& best, int& best_s) const {
        ws<int64_t>(rs)[lane] = Dhat[row.x & 0xffffu] * (int64_t)(row.x >> 16) + Dhat[row.y & 0xffffu] * (int64_t)(row.y >> 16) +
                                Dhat[row.z & 0xffffu] * (int64_t)(row.z >> 16) + Dhat[row.w & 0xffffu] * (int64_t)(row.w >> 16);
        __syncwarp();
#pragma unroll
        for (int u = 0; u < 4; u++)
            if (lane + 32 * u < n_shapes) {
                int64_t v = 0;
#pragma unroll
                for (int r = 0; r < 4; r++) v += ws<int64_t>(rs)[(shape[u] >> (8 * r)) & 0xffu];
                if (v > best) { best = v; best_s = lane + 32 * u; }
            }
    }
};

// Eq. (6) from the terms themselves, for catalogs with more patterns or shapes than that: first maximum of this lane's shapes.
__device__ __forceinline__ void score_terms(int n_shapes, int max_terms, const uint32_t* term, const int64_t* Dhat, int lane, int64_t& best, int& best_s) {
    const int ns_pad = (n_shapes + 31) & ~31;               // row stride of the transposed term table
    for (int s0 = lane; s0 < n_shapes; s0 += 128) {         // four shapes per lane in flight
        int64_t score[4] = {0, 0, 0, 0};
        const uint32_t* tp = term + s0;                        // term e of shape s is at [e][s]: lanes read neighbours
        const int last = n_shapes - 1 - s0;                 // shapes beyond the catalog re-read the last one
        int du[4];
#pragma unroll
        for (int u = 0; u < 4; u++) du[u] = min(32 * u, last);
#pragma unroll 4
        for (int e = 0; e < max_terms; e++) {
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const uint32_t w = tp[e * ns_pad + du[u]];
                score[u] += *(const int64_t*)((const char*)Dhat + (w & 0xffffu)) * (int64_t)(w >> 16);
            }
        }
#pragma unroll
        for (int u = 0; u < 4; u++)
            if (s0 + 32 * u < n_shapes && score[u] > best) { best = score[u]; best_s = s0 + 32 * u; }
    }
}

// Eq. (6) in 64 bits, from the terms (out of line): first maximal shape, -1 if nothing is covered.
__device__ __noinline__ int warp_first_shape(int n_shapes, int max_terms, const uint32_t* term, const int64_t* Dhat, int lane) {
    int64_t best = -1;
    int best_s = 0x7fffffff;
    score_terms(n_shapes, max_terms, term, Dhat, lane, best, best_s);
    warp_argmax_first(best, best_s);
    return best > 0 ? best_s : -1;
}

// What a warp's tasks read: the residual in granules (row i at D + i * N); the credits min(residual, largest capacity) << 8, row-major
// (C) and transposed (CT), so that a tile needs no minimum and no shift on one path rate; the capacities.
struct WarpUnits {
    const uint32_t *D, *C, *CT, *cap;
    int N;
};

// MultiStartAA of four tasks at a time, two lanes per rank group (eight lanes per task).  uo, ui: slot words of the lane's two
// out-slots and in-slots (see DevCat::fam_task); dst: the task's initial binding; mine: the lane belongs to a task; act: and to a group.
//
// A binding travels as the low byte of a group's best key: the tag 3 - row of position 0 in its two highest bits, of position 3 in the
// lowest.  Spare lanes repeat group 0.  Returns the task's F; src, dt0, dt1: its final binding (dt: tags of the out-slots' destinations).
template <bool ONE>
__device__ __forceinline__ uint32_t warp_tasks(const WarpUnits& m, const uint2 uo, const uint2 ui, uint32_t dst, bool mine, bool act, int part,
                                               unsigned gmask, int i_aa, unsigned& n_sweeps, uint32_t& src, int& dt0, int& dt1) {
    auto cap_of = [&](uint32_t w) { return ONE ? 0xffffffffu : m.cap[(w >> 24) & 0xfu] << 8; };
    const uint32_t oc0 = cap_of(uo.x), oc1 = cap_of(uo.y), ic0 = cap_of(ui.x), ic1 = cap_of(ui.y);
    // tags of the lane's two columns: (3 - row) << (6 - 2 column), row 3 has none
    const uint32_t t10 = part ? 1u << 2 : 1u << 6, t11 = t10 >> 2;
    // best key of the tile whose columns 2 part, 2 part + 1 are x and y: both columns on every pair of rows; the other lane
    // of the group has the other two columns
    auto best_key = [&](const uint4& x, uint32_t cx, const uint4& y, uint32_t cy) {
        const uint32_t x0 = min_v(x.x, cx) + 3u * t10, x1 = min_v(x.y, cx) + 2u * t10, x2 = min_v(x.z, cx) + t10, x3 = min_v(x.w, cx);
        const uint32_t y0 = min_v(y.x, cy) + 3u * t11, y1 = min_v(y.y, cy) + 2u * t11, y2 = min_v(y.z, cy) + t11, y3 = min_v(y.w, cy);
        const uint32_t p01 = add_max(x0, y1, x1 + y0), p02 = add_max(x0, y2, x2 + y0), p03 = add_max(x0, y3, x3 + y0);
        const uint32_t p12 = add_max(x1, y2, x2 + y1), p13 = add_max(x1, y3, x3 + y1), p23 = add_max(x2, y3, x3 + y2);
        const uint32_t o01 = __shfl_xor_sync(0xffffffffu, p01, 1), o02 = __shfl_xor_sync(0xffffffffu, p02, 1);
        const uint32_t o03 = __shfl_xor_sync(0xffffffffu, p03, 1), o12 = __shfl_xor_sync(0xffffffffu, p12, 1);
        const uint32_t o13 = __shfl_xor_sync(0xffffffffu, p13, 1), o23 = __shfl_xor_sync(0xffffffffu, p23, 1);
        const uint32_t m0 = add_max(p01, o23, add_max(p02, o13, p03 + o12)), m1 = add_max(p12, o03, add_max(p13, o02, p23 + o01));
        return max_v(m0, m1);
    };
    auto tag_of = [&](uint32_t bytes, uint32_t w) { return (int)((__shfl_sync(0xffffffffu, bytes, (int)(w >> 15), 8) >> (w >> 28)) & 3u); };
    auto source_half = [&]() {                               // credits of group a towards its out-slots' destinations
        return best_key(*(const uint4*)(m.CT + ((int)(uo.x & 0xffffu) - dt0 * m.N)), oc0, *(const uint4*)(m.CT + ((int)(uo.y & 0xffffu) - dt1 * m.N)), oc1) & 0xffu;
    };
    dt0 = (int)((dst >> (uo.x >> 28)) & 3u);                 // (every group starts from the same binding)
    dt1 = (int)((dst >> (uo.y >> 28)) & 3u);
    uint32_t src_new = source_half(), F_old = 0;             // (0: a first F of zero ends the run as -1 would: the sweep after it repeats it)
    src = 0x100u;                                            // (no binding yet)
    bool alive = mine;                                       // the same in a task's eight lanes, as F is
#pragma unroll 1
    for (int sweep = 1; ; sweep++) {
        // If no source binding of a task moved, the destination half would see what it saw last sweep and return the same
        // binding and the same F: the run ends here exactly as it would after computing that.
        const unsigned who = __ballot_sync(0xffffffffu, alive && src_new != src);
        if (alive) src = src_new;
        if (alive && !(who & gmask)) { n_sweeps++; alive = false; }
        if (who == 0) break;
        // destination half: credits into group a from its in-slots' sources
        const int s0 = tag_of(src, ui.x), s1 = tag_of(src, ui.y);
        const uint32_t key = best_key(*(const uint4*)(m.C + ((int)(ui.x & 0xffffu) - s0 * m.N)), ic0, *(const uint4*)(m.C + ((int)(ui.y & 0xffffu) - s1 * m.N)), ic1);
        const unsigned who2 = __ballot_sync(0xffffffffu, alive && ((key ^ dst) & 0xffu) != 0);
        if (alive) dst = key & 0xffu;
        uint32_t F = act ? key >> 8 : 0u;                    // Eq. (8); both lanes of a group hold its credit
        F += __shfl_xor_sync(0xffffffffu, F, 2);
        dt0 = tag_of(dst, uo.x);
        dt1 = tag_of(dst, uo.y);
        // the next sweep's source half needs no F: it runs while that is summed and is dropped if the run ends
        const bool more = sweep < i_aa && who2 != 0;
        if (more) src_new = source_half();
        F += __shfl_xor_sync(0xffffffffu, F, 4);
        // If no destination binding moved, the next sweep would be a repetition of this one and would end the run, so it is
        // counted and skipped.
        if (alive) {
            n_sweeps++;
            alive = (sweep == 1 || F > F_old) && sweep < i_aa;
            F_old = F;
            if (alive && !(who2 & gmask)) { n_sweeps++; alive = false; }
        }
        if (!more || !__any_sync(0xffffffffu, alive)) break;
    }
    return F_old;
}

// Steps 2 and 3 by the general route (out of line): any number of families and starts, four tasks at a time.  Returns F << 32 | task
// of the best start of the best family (F = 0: none), whose binding is at bindings + task * N then (source | destination << 8 per slot).
template <bool ONE>
__device__ __noinline__ uint64_t warp_families(const WarpUnits m, const uint32_t* fam_task, const int64_t* tscale, uint16_t* bindings, int f0, int H, int G,
                                               int n_start, int i_aa, int64_t lambda_w, int lane, unsigned& sweeps_out) {
    const int tsub = lane >> 3, a = (lane & 7) >> 1, part = lane & 1, ag = a < G ? a : 0, n_tasks = H * n_start;
    int64_t bf = -1, bd = 1, ff = -1, fd = 1;                // best family so far; best start of the current family
    int bt = -1, ft = -1, cur_h = -1;
    unsigned n_sweeps = 0;
#pragma unroll 1
    for (int task0 = 0; task0 < n_tasks; task0 += 4) {
        const int task = min(task0 + tsub, n_tasks - 1), h = H == 1 ? 0 : task / n_start, t = task - h * n_start;
        const bool mine = task0 + tsub < n_tasks, act = mine && a < G;
        const uint32_t* const fam = fam_task + ((f0 + h) * G + ag) * 8 + part * 2;
        const uint2 uo = *(const uint2*)fam, ui = *(const uint2*)(fam + 4);
        uint32_t src;
        int dt0, dt1;
        const uint32_t F = warp_tasks<ONE>(m, uo, ui, big_family_and_start(t, n_start) & 0xffu, mine, act, part, 0xffu << (8 * tsub), i_aa, n_sweeps, src, dt0, dt1);
        const uint32_t bind = (uint32_t)(ag * 4 + 3 - (int)((src >> (6 - 4 * part)) & 3u)) | (uint32_t)((int)((uo.x >> 16) & 0xffu) * 4 + 3 - dt0) << 8 |
                              (uint32_t)(ag * 4 + 3 - (int)((src >> (4 - 4 * part)) & 3u)) << 16 | (uint32_t)((int)((uo.y >> 16) & 0xffu) * 4 + 3 - dt1) << 24;
        if (act) *(uint32_t*)(bindings + task * m.N + a * 4 + part * 2) = bind;
        if (H == 1) {                                        // largest F, lowest start (F is 0 without a task)
            const uint32_t best = __reduce_max_sync(0xffffffffu, F << 2 | (uint32_t)(3 - tsub));
            if ((int64_t)(best >> 2) > bf) { bf = best >> 2; bt = task0 + 3 - (int)(best & 3u); }
            continue;
        }
        // Evaluate (Eq. 9, 10): slowest lane under the final bindings
        int64_t tmax = 0;
        if (act) {
#pragma unroll
            for (int i = 0; i < 2; i++) {
                const uint32_t bw = bind >> (16 * i), cl = ((i ? uo.y : uo.x) >> 24) & 0xfu;
                const uint32_t x = min_v(m.D[(int)(bw & 0xffu) * m.N + (int)((bw >> 8) & 0xffu)], m.cap[cl]);
                tmax = max_v(tmax, (int64_t)x * tscale[cl]);
            }
        }
        tmax = team_max(tmax);
        tmax = max_v(tmax, __shfl_xor_sync(0xffffffffu, tmax, 4));
        const int64_t den = F > 0 ? lambda_w + tmax : 1;
        // the round's results in task order (every lane follows along)
#pragma unroll 1
        for (int s = 0; s < 4; s++) {
            const int64_t Fs = __shfl_sync(0xffffffffu, F, 8 * s), ds = __shfl_sync(0xffffffffu, den, 8 * s);
            const int tk = task0 + s, ht = tk / n_start;
            if (tk < n_tasks) {
                if (ht != cur_h) {                           // a new family starts: settle the previous one
                    if (cur_h >= 0 && (bt < 0 || util_greater(ff, fd, bf, bd))) { bf = ff; bd = fd; bt = ft; }
                    cur_h = ht; ff = -1; fd = 1; ft = -1;
                }
                if (Fs > ff) { ff = Fs; fd = ds; ft = tk; }  // largest F, lowest start
            }
        }
    }
    if (cur_h >= 0 && (bt < 0 || util_greater(ff, fd, bf, bd))) { bf = ff; bd = fd; bt = ft; }   // lowest family on ties
    sweeps_out = n_sweeps;
    __syncwarp();
    return (uint64_t)bf << 32 | (uint32_t)bt;
}

template <bool NARROW> struct WarpLeft { typedef uint32_t type; };
template <> struct WarpLeft<false> { typedef int64_t type; };

// Main loop for a matrix held in 32-bit granules (`total` of them) with capacities below 2^22 granules.  Two copies: while scores need
// 64 bits, and from then on; what an ordinary activation does not execute is out of line (instructions come from small caches, see
// schedule_big.cuh).  ONE: all paths have one rate.
template <bool ONE>
__device__ __forceinline__ void decompose_units(const DevCat& dc, const KParams& kp, const WCtx& c, int64_t total, int& k_out, int& st, Counters& cnt) {
    const int N = c.N, G = c.G, lane = c.lane;
    uint32_t* const D = ws<uint32_t>(c.o_drem);
    uint32_t* const C = ws<uint32_t>(c.o_cred);
    uint32_t* const CT = ws<uint32_t>(c.o_dremT);              // CT[j * N + i] = C[i * N + j]
    int64_t* const Dhat = ws<int64_t>(c.o_dhat);
    const uint32_t* const dhat32 = ws<uint32_t>(c.o_dhat);     // (low words)
    const uint32_t* const s_cap = ws<uint32_t>(c.o_cap32);
    uint16_t* const bindings = ws<uint16_t>(c.o_bind);
    const uint32_t* const fam_task = ws<uint32_t>(c.o_fam_task);
    const uint32_t cap0 = s_cap[0];
    const WarpUnits units{D, C, CT, s_cap, N};
    uint32_t cap_most = cap0;
    if (!ONE)
        for (int cl = 1; cl < dc.n_classes; cl++) cap_most = max_v(cap_most, s_cap[cl]);
    for (int e = lane; e < N * N; e += 32) {                   // (D and its transpose are given)
        C[e] = min_v(D[e], cap_most) << 8;
        CT[e] = min_v(CT[e], cap_most) << 8;
    }
    __syncwarp();
    // this lane's place in Step 2: task of four, rank group, columns 2 part and 2 part + 1 of the group's tile
    const int tsub = lane >> 3, a = (lane & 7) >> 1, part = lane & 1, ag = a < G ? a : 0;
    const unsigned gmask = 0xffu << (8 * tsub);
    const uint32_t dst_1 = big_family_and_start(tsub, 4) & 0xffu;
    const uint32_t my_fam = (uint32_t)(ag * 8 + part * 2);
    const bool mine_1 = tsub < kp.n_start, act = mine_1 && a < G;
    const int my_slot = lane < N ? lane : 0;
    unsigned n_sweeps = 0, n_done = 0;
    RowScores by_rows;
    by_rows.load(dc, c);
    int k = 0;
    // the activation taken off the residual whose rows are still to be written (slot `lane`)
    bool pend = false;
    int p_fam = 0;
    uint32_t p_bind = 0, p_x = 0;
    auto write_row = [&](int kk, uint32_t inst) {
        if (lane < N) {
            const int i = (int)(p_bind & 0xffu), j = (int)(p_bind >> 8);
            const size_t row = (size_t)kk * N, orow = (size_t)(kk + 1) * N;
            const int64_t bytes = (int64_t)p_x * kp.granule;
            const int64_t sa = ws<int64_t>(c.o_send_acc)[i] + bytes, ra = ws<int64_t>(c.o_recv_acc)[j] + bytes;
            ws<int64_t>(c.o_send_acc)[i] = sa;
            ws<int64_t>(c.o_recv_acc)[j] = ra;
            c.lane_dst_b[row + i] = p_x ? (int16_t)j : (int16_t)-1;
            c.lane_bytes_b[row + i] = bytes;
            c.send_off_b[orow + i] = sa;
            if (c.recv_off_b) c.recv_off_b[orow + j] = ra;
            c.lane_inst_b[row + i] = p_x ? (uint16_t)inst : (uint16_t)0xFFFF;
            if (lane == 0) c.chan_id_b[kk] = p_fam;
        }
    };

    auto slot_inst = [&]() { return __ldg(dc.fam_slot + (unsigned)(p_fam * N + my_slot)); };

    auto run = [&](auto scores) {
        constexpr bool NARROW = decltype(scores)::value;         // every score (at most g x what is left) fits 32 bits
        typedef typename WarpLeft<NARROW>::type left_t;
        left_t left = (left_t)total;
        for (;;) {
            if (rarely(left == 0 || k == kp.k_max || (!NARROW && left < ((left_t)1 << 30)))) break;
            // path instance of the slot to be written out: a trip to L2 that ends long before write_row needs it
            const uint32_t inst = slot_inst();
            // (A) Eq. (6): shape scores, first maximum
            int best_s = 0x7fffffff;
            if (NARROW && usually(by_rows.on)) {
                const uint32_t best = by_rows.narrow(dhat32, lane, best_s), m = __reduce_max_sync(0xffffffffu, best);
                best_s = (int)__reduce_min_sync(0xffffffffu, best == m ? (uint32_t)best_s : 0x7fffffffu);
                if (m == 0) best_s = -1;
            } else {
                best_s = warp_first_shape(dc.n_shapes, dc.max_terms, dc.term_t, Dhat, lane);
            }
            VP_TICK(0);
            if (rarely(best_s < 0)) { st |= VP_ST_UNCOVERED; break; }
            const int f0 = (int)ws<uint32_t>(c.o_bucket)[best_s], H = (int)ws<uint32_t>(c.o_bucket)[best_s + 1] - f0;
            VP_TICK(1);

            // (B) MultiStartAA, (C) best start per family, best family
            uint32_t wF, bind;                                   // F of the best start, source | destination << 8 of slot `lane`
            int wfam = f0;
            // One family, one round: largest F, lowest start; bindings stay in registers.  (Fewer starts than four leave lanes without a
            // task, whose F is 0.  By the route out of line 256 matrices of 16 ranks took 128 and 139 us with one start and three, here 74 and 84.)
            if (usually(H == 1 && kp.n_start <= 4)) {
                const uint32_t* const fam = fam_task + (uint32_t)(f0 * G) * 8u + my_fam;
                const uint2 uo = *(const uint2*)fam, ui = *(const uint2*)(fam + 4);
                if (usually(pend)) write_row(k - 1, inst);
                uint32_t src;
                int dt0, dt1;
                const uint32_t F = warp_tasks<ONE>(units, uo, ui, dst_1, mine_1, act, part, gmask, kp.i_aa, n_sweeps, src, dt0, dt1);
                VP_TICK(2);
                const uint32_t mine = (uint32_t)(ag * 4 + 3 - (int)((src >> (6 - 4 * part)) & 3u)) | (uint32_t)((int)((uo.x >> 16) & 0xffu) * 4 + 3 - dt0) << 8 |
                                      (uint32_t)(ag * 4 + 3 - (int)((src >> (4 - 4 * part)) & 3u)) << 16 | (uint32_t)((int)((uo.y >> 16) & 0xffu) * 4 + 3 - dt1) << 24;
                n_done += (unsigned)kp.n_start;
                const uint32_t best = __reduce_max_sync(0xffffffffu, F << 2 | (uint32_t)(3 - tsub));     // (F is at most sixteen lanes of 2^22 granules)
                wF = best >> 2;
                bind = (__shfl_sync(0xffffffffu, mine, (int)(3u - (best & 3u)) << 3 | ((lane >> 1) & 7)) >> (16 * (lane & 1))) & 0xffffu;
            } else {
                if (pend) write_row(k - 1, inst);
                unsigned more_sweeps;
                const uint64_t chosen = warp_families<ONE>(units, fam_task, ws<int64_t>(c.o_tscale), bindings, f0, H, G, kp.n_start, kp.i_aa, kp.lambda_ns * dc.W, lane, more_sweeps);
                n_sweeps += more_sweeps;
                n_done += (unsigned)(H * kp.n_start);
                wF = (uint32_t)(chosen >> 32);
                wfam += (int)(big_family_and_start((int)(uint32_t)chosen, kp.n_start) >> 8);
                bind = lane < N ? bindings[(int)(uint32_t)chosen * N + lane] : 0u;
            }
            pend = false;
            if (rarely(wF == 0)) { st |= VP_ST_NO_PROGRESS; break; }
            VP_TICK(3);

            // (D) activation k off the residual and off D-hat (Eq. 5)
            __syncwarp();
            if (lane < N) {
                const int i = (int)(bind & 0xffu), j = (int)(bind >> 8);
                uint32_t cap = cap0;
                if (!ONE) cap = s_cap[__ldg(dc.fam_cls + (size_t)wfam * N + lane)];
                const uint32_t cell = D[i * N + j], x = min_v(cap, cell);
                const uint32_t credit = min_v(cell - x, cap_most) << 8;
                D[i * N + j] = cell - x;
                C[i * N + j] = credit;
                CT[j * N + i] = credit;
                int64_t* const sum = &Dhat[(lane >> 2) * G + (j >> 2)];
                if (NARROW) atomicSub((unsigned int*)sum, x);    // (high word is zero, low word >= x)
                else atomicAdd((unsigned long long*)sum, (unsigned long long)(-(int64_t)x));
                p_x = x;
            }
            p_bind = bind;
            p_fam = wfam;
            pend = true;
            left -= wF;
            k++;
            __syncwarp();
            VP_TICK(4);
        }
        total = (int64_t)left;
    };
    if (total >= ((int64_t)1 << 30)) run(BigConst<false>());
    if (st == 0 && k < kp.k_max && total < ((int64_t)1 << 30)) run(BigConst<true>());
    if (st == 0 && total != 0) st |= VP_ST_STEP_LIMIT;
    if (pend) write_row(k - 1, slot_inst());
    k_out = k;
    if (lane == 0) cnt.tasks += n_done;
    if ((lane & 7) == 0) cnt.sweeps += n_sweeps;
}

// Main loop for any other matrix, in 64-bit bytes (`left` of them): eight (family, start) tasks at a time, a team of four lanes
// per task, one lane per rank group, which enumerates its group's 24 permutations.
__device__ __forceinline__ void decompose_bytes(const DevCat& dc, const KParams& kp, const WCtx& c, int64_t left, int& k, int& st, Counters& cnt) {
    const int N = c.N, G = c.G, lane = c.lane;
    const int ld = N + 1;                                // row stride of D_rem
    const int team = lane >> 2, a = lane & 3;
    const bool active = a < G;
    const int ns_shift = (kp.n_start & (kp.n_start - 1)) == 0 ? 31 - __clz(kp.n_start) : -1;
    int64_t* const Drem = ws<int64_t>(c.o_drem);
    const int64_t* const cap = ws<int64_t>(c.o_cap64);
    int64_t* const Dhat = ws<int64_t>(c.o_dhat);
    RowScores by_rows;
    by_rows.load(dc, c);

    for (;;) {
        if (left == 0) break;
        if (k == kp.k_max) { st |= VP_ST_STEP_LIMIT; break; }
        // (A) Eq. (6): shape scores, first maximum
        int64_t best = -1;
        int best_s = 0x7fffffff;
        if (by_rows.on) by_rows.wide(Dhat, lane, best, best_s);
        else score_terms(dc.n_shapes, dc.max_terms, c.term, Dhat, lane, best, best_s);
        VP_TICK(0);
        warp_argmax_first(best, best_s);
        if (best <= 0) { st |= VP_ST_UNCOVERED; break; }
        const int f0 = (int)ws<uint32_t>(c.o_bucket)[best_s], H = (int)ws<uint32_t>(c.o_bucket)[best_s + 1] - f0;
        const int n_tasks = H * kp.n_start;
        VP_TICK(1);

        // (B) MultiStartAA, eight (family, start) tasks at a time; (C) best start per family, best family
        int64_t bf = -1, bd = 1, ff = -1, fd = 1;        // best family so far; best start of the current family
        int bt = -1, ft = -1, cur_h = -1;
        for (int task0 = 0; task0 < n_tasks; task0 += 8) {
            const int task = min(task0 + team, n_tasks - 1);
            const bool has = task0 + team < n_tasks && active;
            const int h = ns_shift >= 0 ? task >> ns_shift : task / kp.n_start, tt = task - h * kp.n_start, f = f0 + h;
            uint8_t* const srcb = ws<uint8_t>(c.o_bind) + task * N;
            uint8_t* const dstb = ws<uint8_t>(c.o_bind_dst) + task * N;
            int64_t cap_out[4], cap_in[4];
            int rq[4], cls_in[4];
            const int ag = active ? a : 0;                   // (spare lanes read group 0's tables and write nothing)
            const uint2 fin4 = *(const uint2*)(c.fam_in + f * N + ag * 4);        // four in-slots, 16 bits each
            const uint32_t fcls4 = *(const uint32_t*)(c.fam_cls + f * N + ag * 4);  // four out-slot classes
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const unsigned w = ((q < 2 ? fin4.x : fin4.y) >> (16 * (q & 1))) & 0xffffu;
                cap_out[q] = cap[(fcls4 >> (8 * q)) & 0xffu];
                rq[q] = (int)(w & 0xffu);
                cls_in[q] = (int)(w >> 8);
                cap_in[q] = cap[cls_in[q]];
                if (has) dstb[rq[q]] = (uint8_t)(a * 4 + ((q + tt) & 3));     // start t rotates the in-slots of every group
            }
            __syncwarp();
            VP_TICK(2);
            int64_t F_old = -1, F_new = -1;
            bool alive = has;
            for (int sweep = 0; sweep < kp.i_aa && __any_sync(0xffffffffu, alive); sweep++) {
                if (alive) {                                  // source half: credits of group a towards its out-slots' destinations
                    const uint32_t d4 = *(const uint32_t*)(dstb + a * 4);
                    int64_t cm[4][4];
#pragma unroll
                    for (int q = 0; q < 4; q++) {
                        const int dq = (int)((d4 >> (8 * q)) & 0xffu);
                        const int64_t* col = Drem + (a * 4) * ld + dq;
#pragma unroll
                        for (int i = 0; i < 4; i++) cm[i][q] = min_v(col[i * ld], cap_out[q]);
                    }
                    unsigned bpk;
                    best_assignment<4, int64_t>(cm, bpk);
                    const uint32_t rows4 = (bpk & 3u) | ((bpk >> 2) & 3u) << 8 | ((bpk >> 4) & 3u) << 16 | ((bpk >> 6) & 3u) << 24;   // the row bound to position q, in byte q
                    *(uint32_t*)(srcb + a * 4) = (uint32_t)(a * 4) * 0x01010101u + rows4;
                }
                __syncwarp();
                int64_t part = 0;
                if (alive) {                                  // destination half: credits into group a from its in-slots' sources
                    int64_t cm[4][4];
#pragma unroll
                    for (int q = 0; q < 4; q++) {
                        const int64_t* row = Drem + (int)srcb[rq[q]] * ld + a * 4;
#pragma unroll
                        for (int i = 0; i < 4; i++) cm[i][q] = min_v(row[i], cap_in[q]);
                    }
                    unsigned bpk;
                    part = best_assignment<4, int64_t>(cm, bpk);
#pragma unroll
                    for (int q = 0; q < 4; q++) dstb[rq[q]] = (uint8_t)(a * 4 + ((bpk >> (2 * q)) & 3u));
                }
                const int64_t Fn = team_sum(part);   // Eq. (8)
                if (alive) {
                    F_new = Fn;
                    if (a == 0) cnt.sweeps++;
                    if (Fn <= F_old) alive = false;           // the run ends; its bindings stay as this sweep left them
                    else F_old = Fn;
                }
                __syncwarp();
            }
            VP_TICK(3);
            // Evaluate (Eq. 9, 10), needed only when several families compete: the volume of every in-slot of this
            // lane's group under the final bindings, the slowest lane over the team
            int64_t den = 1;
            if (H > 1) {
                int64_t tmax = 0;
                if (has) {
#pragma unroll
                    for (int q = 0; q < 4; q++) {
                        const int64_t x = min_v(Drem[(int)srcb[rq[q]] * ld + (int)dstb[rq[q]]], cap_in[q]);
                        tmax = max_v(tmax, x * ws<int64_t>(c.o_tscale)[cls_in[q]]);
                    }
                }
                tmax = team_max(tmax);
                den = F_new > 0 ? kp.lambda_ns * dc.W + tmax : 1;
            }
            if (has && a == 0) cnt.tasks++;
            if (H == 1 && n_tasks <= 8) {
                // one family, one round: the best start is the largest F, the lowest start among equals -- one maximum of
                // F << 3 | (7 - start) over the warp (F is below 2^42)
                const uint64_t key = has && a == 0 ? (uint64_t)F_new << 3 | (uint64_t)(7 - team) : 0ull;
                const uint32_t hi = (uint32_t)(key >> 32), lo = (uint32_t)key;
                const uint32_t mhi = __reduce_max_sync(0xffffffffu, hi);
                const uint32_t mlo = __reduce_max_sync(0xffffffffu, hi == mhi ? lo : 0u);
                const uint64_t mkey = (uint64_t)mhi << 32 | mlo;
                bf = (int64_t)(mkey >> 3); bd = 1; bt = 7 - (int)(mkey & 7u);
                cur_h = -1;                                       // (settled)
                break;
            }
            // the teams' results in task order (every lane follows along)
            const int in_round = min(8, n_tasks - task0);
            for (int t = 0; t < in_round; t++) {
                const int64_t Ft = __shfl_sync(0xffffffffu, F_new, t * 4), dt = __shfl_sync(0xffffffffu, den, t * 4);
                const int tk = task0 + t, ht = ns_shift >= 0 ? tk >> ns_shift : tk / kp.n_start;
                if (ht != cur_h) {                             // a new family starts: settle the previous one
                    if (cur_h >= 0 && (bt < 0 || util_greater(ff, fd, bf, bd))) { bf = ff; bd = fd; bt = ft; }
                    cur_h = ht; ff = -1; fd = 1; ft = -1;
                }
                if (Ft > ff) { ff = Ft; fd = dt; ft = tk; }    // largest F, lowest start
            }
        }
        if (cur_h >= 0 && (bt < 0 || util_greater(ff, fd, bf, bd))) { bf = ff; bd = fd; bt = ft; }   // lowest family on ties
        if (bf <= 0) { st |= VP_ST_NO_PROGRESS; break; }
        VP_TICK(4);

        // (D) emit activation k, D_rem -= X(E), write offset row k+1, re-sum D-hat
        {
            const int h = ns_shift >= 0 ? bt >> ns_shift : bt / kp.n_start;
            const size_t row = (size_t)k * N, orow = (size_t)(k + 1) * N;
            if (lane < N) {
                const int r = lane;
                const uint32_t w = c.fam_slot[(f0 + h) * N + r];
                const int i = ws<uint8_t>(c.o_bind)[bt * N + r], j = ws<uint8_t>(c.o_bind_dst)[bt * N + r];
                const int64_t bytes = min_v(cap[(w >> 24) & 0xf], Drem[i * ld + j]);
                // straight-line: an idle lane (x = 0) writes the idle values and adds zero
                const bool busy = bytes > 0;
                const int64_t sa = ws<int64_t>(c.o_send_acc)[i] + bytes, ra = ws<int64_t>(c.o_recv_acc)[j] + bytes;
                c.lane_dst_b[row + i] = busy ? (int16_t)j : (int16_t)-1;
                c.lane_inst_b[row + i] = busy ? (uint16_t)(w & 0xffffu) : (uint16_t)0xFFFF;
                c.lane_bytes_b[row + i] = bytes;
                Drem[i * ld + j] -= bytes;
                if (busy) atomicAdd((unsigned long long*)&Dhat[(i >> 2) * G + (j >> 2)], (unsigned long long)(-bytes));   // Eq. (5)
                ws<int64_t>(c.o_send_acc)[i] = sa;
                ws<int64_t>(c.o_recv_acc)[j] = ra;
                c.send_off_b[orow + i] = sa;
                if (c.recv_off_b) c.recv_off_b[orow + j] = ra;
            }
            if (lane == 0) c.chan_id_b[k] = f0 + h;
            left -= bf;
            __syncwarp();
        }
        k++;
        __syncwarp();
        VP_TICK(5);
    }
}

// UNITS: the granule is at least 256 bytes, so the matrices run in decompose_units as a rule, whose tables are staged; the odd
// matrix of larger capacities reads those of decompose_bytes from global memory.  Otherwise decompose_bytes and its tables.
// `slots`: per warp three counters for vp_schedule_read_stats, given when there is a warp for every matrix: the launch then needs
// no counter and nothing zeroed.
template <bool UNITS, bool ONE>
__global__ void __launch_bounds__(128, 3)
vp_schedule_warp_kernel(DevCat dc, KParams kp, const int64_t* __restrict__ demand, const int64_t* __restrict__ tau_in, int B,
                        int32_t* __restrict__ n_steps, int32_t* __restrict__ chan_id, int16_t* __restrict__ lane_dst,
                        uint16_t* __restrict__ lane_inst, int64_t* __restrict__ lane_bytes, int64_t* __restrict__ send_off,
                        int64_t* __restrict__ recv_off, int64_t* __restrict__ tau_out, int32_t* __restrict__ status,
                        unsigned int* counter, unsigned long long* slots) {
    unsigned char* const smem_raw = vp_wsmem;
    const int N = dc.N, G = dc.G, tid = threadIdx.x, NT = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, n_warps = NT >> 5;
    const int ld = N + 1;
    const WarpSmem L = warp_smem_layout(dc, kp, n_warps, UNITS);
    // ---- stage the catalog (shared by the warps of the CTA): bulk asynchronous copies (TMA) of whole arrays onto one
    // mbarrier; plain loads if the bounded wait gives up.  The catalog was uploaded when it was loaded: no need to wait for the
    // kernel ahead.
    {
        const int ns_pad = (dc.n_shapes + 31) & ~31;
        const void* from[7] = {dc.bucket_ptr, dc.row_term, dc.shape_rows, dc.fam_task, dc.term_t, dc.fam_slot, dc.fam_in};
        const int at[7] = {L.bucket, L.rows, L.shape_rows, L.fam_task, L.term, L.fam_slot, L.fam_in};
        const int bytes[7] = {align16((dc.n_shapes + 1) * 4), dc.row_term ? 32 * 16 : 0, dc.row_term ? ns_pad * 4 : 0, UNITS ? dc.n_families * G * 32 : 0,
                              UNITS ? 0 : ns_pad * dc.max_terms * 4, UNITS ? 0 : align16(dc.n_families * N * 4), UNITS ? 0 : align16(dc.n_families * N * 2)};
        const int b_cls = UNITS ? 0 : align16(dc.n_families * N);
        __shared__ __align__(8) unsigned long long s_stage_bar;
        const unsigned bar = smem_u32(&s_stage_bar);
        if (tid == 0) {
            mbar_init(bar, 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            unsigned total = (unsigned)b_cls;
#pragma unroll
            for (int i = 0; i < 7; i++) total += (unsigned)bytes[i];
            mbar_expect_tx(bar, total);
#pragma unroll
            for (int i = 0; i < 7; i++)
                if (bytes[i]) bulk_load(smem_u32(smem_raw + at[i]), from[i], (unsigned)bytes[i], bar);
            if (b_cls) bulk_load(smem_u32(smem_raw + L.fam_cls), dc.fam_cls, (unsigned)b_cls, bar);
        }
        __syncthreads();
        if (!__syncthreads_and(mbar_wait_bounded(bar, 0, 1u << 20))) {
#pragma unroll
            for (int i = 0; i < 7; i++)
                for (int e = tid; e < bytes[i] / 4; e += NT) ((uint32_t*)(smem_raw + at[i]))[e] = ((const uint32_t*)from[i])[e];
            for (int e = tid; e < b_cls / 4; e += NT) ((uint32_t*)(smem_raw + L.fam_cls))[e] = ((const uint32_t*)dc.fam_cls)[e];
        }
    }
    // quantum rule: the cells that cross this lane's resource (at most sixteen cells and resources), as a mask
    uint32_t forced = 0, forced_bw = 0;
    if (lane < dc.n_res) {
        forced_bw = dc.forced_bw[lane];
        if (forced_bw)
            for (uint32_t e = dc.forced_ptr[lane]; e < dc.forced_ptr[lane + 1]; e++) forced |= 1u << dc.forced_cell[e];
    }
    const bool masks = dc.n_res <= 32;                     // (else the lists are read for every matrix)
    // reciprocals, while the kernel ahead still runs (worked out behind the wait they and the addresses took 1,400 cycles of a call)
    const RowDiv granule{kp.granule, kp.inv_granule}, bw_max{dc.bw_max, 1.0 / (double)dc.bw_max}, by_target{(int64_t)kp.k_target, 1.0 / (double)kp.k_target};
    const RowDiv by_forced{(int64_t)max(forced_bw, 1u), 1.0 / (double)max(forced_bw, 1u)};
    __syncthreads();
    grid_wait();
    WCtx c;
    c.N = N; c.G = G; c.lane = lane;
    const unsigned base = (unsigned)warp * (unsigned)L.per_warp;
    c.o_drem = base + L.drem; c.o_dremT = base + L.dremT; c.o_cred = base + L.cred; c.o_dhat = base + L.dhat; c.o_send_acc = base + L.send_acc; c.o_recv_acc = base + L.recv_acc;
    c.o_rs = base + L.rs; c.o_cap64 = base + L.cap64; c.o_cap32 = base + L.cap32; c.o_tscale = base + L.tscale;
    c.o_bind = base + L.bind; c.o_bind_dst = base + L.bind_dst;
    c.o_rows = L.rows; c.o_shape_rows = L.shape_rows; c.o_fam_task = L.fam_task; c.o_bucket = L.bucket;
    c.term = UNITS ? dc.term_t : ws<const uint32_t>(L.term);
    c.fam_slot = UNITS ? dc.fam_slot : ws<const uint32_t>(L.fam_slot);
    c.fam_in = UNITS ? dc.fam_in : ws<const uint16_t>(L.fam_in);
    c.fam_cls = UNITS ? dc.fam_cls : ws<const uint8_t>(L.fam_cls);
    int64_t* const Drem = ws<int64_t>(c.o_drem);
    uint32_t* const D32 = ws<uint32_t>(c.o_drem);
    uint32_t* const DT32 = ws<uint32_t>(c.o_dremT);
    int64_t* const Dhat = ws<int64_t>(c.o_dhat);
    int64_t* const send_acc = ws<int64_t>(c.o_send_acc);
    int64_t* const recv_acc = ws<int64_t>(c.o_recv_acc);
    int64_t* const cap64 = ws<int64_t>(c.o_cap64);
    int64_t* const tscale = ws<int64_t>(c.o_tscale);
    uint32_t* const cap32 = ws<uint32_t>(c.o_cap32);
    auto ceil_div = [](int64_t x, const RowDiv& by) {      // x below 2^52
        int64_t rem;
        const int64_t q = by.div(x, rem);
        return q + (rem > 0);
    };
    const unsigned inv_n = 65536u / (unsigned)N + 1u;      // e / N for e < 256
    unsigned long long n_act = 0;
    Counters cnt;
    cnt.tasks = 0; cnt.sweeps = 0; cnt.t_mark = 0;
    for (int i = 0; i < 6; i++) cnt.cyc[i] = 0;

    for (int round = 0; ; round++) {
        int b = (int)blockIdx.x * n_warps + warp;
        if (slots) {
            if (round) break;
        } else {
            if (lane == 0) b = (int)atomicAdd(counter, 1u);
            b = __shfl_sync(0xffffffffu, b, 0);
        }
        if (b >= B) break;
        const int64_t* D = demand + (size_t)b * N * N;
        const size_t lane_base = (size_t)b * kp.k_max * N, off_base = (size_t)b * (kp.k_max + 1) * N;
        c.chan_id_b = chan_id + (size_t)b * kp.k_max;
        c.lane_dst_b = lane_dst + lane_base;
        c.lane_inst_b = lane_inst + lane_base;
        c.lane_bytes_b = lane_bytes + lane_base;
        c.send_off_b = send_off + off_base;
        c.recv_off_b = recv_off ? recv_off + off_base : nullptr;

        // ---- validate; D in granules and its transpose
        int flags = 0;
        int64_t v[8];
#pragma unroll
        for (int u = 0; u < 8; u++) v[u] = lane + 32 * u < N * N ? D[lane + 32 * u] : 0;
        const int64_t tau_given = tau_in ? tau_in[b] : 0;
#pragma unroll
        for (int u = 0; u < 8; u++) {
            const int e = lane + 32 * u;
            if (e >= N * N) continue;
            const int i = (int)(((unsigned)e * inv_n) >> 16), j = e - i * N;
            int64_t q = 0, rem = 0;
            if (v[u] < 0) flags |= VP_ST_NEGATIVE;
            else if (v[u] >= VP_ENTRY_LIMIT) flags |= VP_ST_OVERFLOW_RISK;
            else {
                q = granule.div(v[u], rem);
                if (i == j && v[u] != 0) flags |= VP_ST_DIAG_NONZERO;
                if (rem) flags |= VP_ST_NOT_GRANULE;
            }
            if (UNITS) {
                D32[e] = (uint32_t)q;
                DT32[j * N + i] = (uint32_t)q;
            } else {
                Drem[i * ld + j] = v[u];
            }
        }
        if (tau_given < 0 || tau_given > VP_ENTRY_LIMIT) flags |= VP_ST_BAD_TAU;
        flags = (int)__reduce_or_sync(0xffffffffu, (unsigned)flags);
        for (int i = lane; i < N; i += 32) {
            send_acc[i] = 0; recv_acc[i] = 0;
            c.send_off_b[i] = 0;
            if (c.recv_off_b) c.recv_off_b[i] = 0;
        }
        __syncwarp();
        int st = flags, k = 0;
        int64_t tau = 0;
#ifdef VP_PHASE_TIMING
        cnt.t_mark = clock64();
#endif
        if (st == 0) {
            // ---- row sums (lanes 0..), column sums (lanes 16..), group sums (Eq. 5), quantum (Section 5), all in bytes
            int64_t est = 0, tot = 0;
            if ((lane & 15) < N) {
                const int i = lane & 15;
                int64_t s = 0;
                if (UNITS) {
                    const uint4* const x = (const uint4*)((lane < 16 ? D32 : DT32) + i * N);
                    for (int m = 0; m < N / 4; m++) {
                        const uint4 w = x[m];
                        s += (int64_t)w.x + w.y + ((int64_t)w.z + w.w);
                    }
                    s *= kp.granule;
                } else {
                    for (int m = 0; m < N; m++) s += lane < 16 ? Drem[i * ld + m] : Drem[m * ld + i];
                }
                est = ceil_div(s, bw_max);
                if (lane < 16) tot = s;
            }
            if (lane < G * G) {
                const int ga = lane / G, gd = lane - ga * G;
                int64_t s = 0;
                if (UNITS) {
#pragma unroll
                    for (int i = 0; i < 4; i++) {
                        const uint4 w = *(const uint4*)(D32 + (ga * 4 + i) * N + gd * 4);
                        s += (int64_t)w.x + w.y + ((int64_t)w.z + w.w);
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 4; i++)
#pragma unroll
                        for (int j = 0; j < 4; j++) s += Drem[(ga * 4 + i) * ld + gd * 4 + j];
                }
                Dhat[lane] = s;                              // (granules or bytes, as the matrix is held)
            }
            __syncwarp();
            const int64_t unit = UNITS ? kp.granule : 1;
            if (masks) {
                if (forced) {
                    int64_t f = 0;
                    for (uint32_t m = forced; m; m &= m - 1) f += Dhat[__ffs((int)m) - 1];
                    est = max_v(est, ceil_div(f * unit, by_forced));
                }
            } else {
                for (int l = lane; l < dc.n_res; l += 32) {
                    const uint32_t bwl = dc.forced_bw[l];
                    if (!bwl) continue;
                    int64_t f = 0;
                    for (uint32_t e = dc.forced_ptr[l]; e < dc.forced_ptr[l + 1]; e++) f += Dhat[dc.forced_cell[e]];
                    est = max_v(est, ceil_div(f * unit, RowDiv{(int64_t)bwl, 1.0 / (double)bwl}));
                }
            }
            est = (int64_t)big_warp_max64((uint64_t)est);
            tot = warp_sum_i64(tot);
            const int64_t tq = tau_given > 0 ? tau_given : max_v((int64_t)1, ceil_div(est, by_target));
            // capacities in granules, at least one (rate x quantum may exceed what the reciprocal divides exactly)
            int64_t cap_gr = 0;
            if (lane < dc.n_classes) {
                const int64_t x = tq * dc.class_bw[lane];
                int64_t rem;
                cap_gr = x < ((int64_t)1 << 52) ? granule.div(x, rem) : x / kp.granule;
                cap_gr = max_v(cap_gr, (int64_t)1);
            }
            // 32-bit granules: capacities below 2^22 granules (four credits and a permutation byte share 32 bits)
            const bool units = UNITS && !__any_sync(0xffffffffu, cap_gr >= ((int64_t)1 << 22));
            if (lane < dc.n_classes) {
                cap64[lane] = cap_gr * kp.granule;
                cap32[lane] = (uint32_t)cap_gr;
                tscale[lane] = dc.class_wdiv[lane] * (units ? kp.granule : 1);
            }
            tau = tq;
            __syncwarp();
            if (units) {
                int64_t rem;
                decompose_units<ONE>(dc, kp, c, granule.div(tot, rem), k, st, cnt);
            } else {
                if (UNITS) {                                 // (back to bytes)
                    for (int e = lane; e < N * N; e += 32) {
                        const int i = (int)(((unsigned)e * inv_n) >> 16);
                        Drem[i * ld + e - i * N] = D[e];
                    }
                    for (int cell = lane; cell < G * G; cell += 32) Dhat[cell] *= kp.granule;
                    __syncwarp();
                }
                decompose_bytes(dc, kp, c, tot, k, st, cnt);
            }
        }
        __syncwarp();
        // ---- idle rows beyond n_steps; offset rows repeat the totals
        const size_t rows = kp.host_rows ? 0 : (size_t)(kp.k_max - k) * N;      // elements per array
        if ((((uintptr_t)c.lane_dst_b | (uintptr_t)c.lane_inst_b | (uintptr_t)c.lane_bytes_b | (uintptr_t)c.send_off_b |
              (uintptr_t)(c.recv_off_b ? c.recv_off_b : c.send_off_b)) & 15) == 0 && (32 % N) == 0 && N >= 8) {
            // whole rows of 2 N bytes and 8 N bytes in 16-byte vectors (N = 8 or 16: a warp's stride keeps a lane's ranks)
            const uint4 ones = make_uint4(0xffffffffu, 0xffffffffu, 0xffffffffu, 0xffffffffu);
            uint4* const ld4 = (uint4*)(c.lane_dst_b + (size_t)k * N);
            uint4* const li4 = (uint4*)(c.lane_inst_b + (size_t)k * N);
            for (size_t e = lane; e < rows / 8; e += 32) { ld4[e] = ones; li4[e] = ones; }
            const int i2 = (2 * lane) & (N - 1);
            const longlong2 sa = *(const longlong2*)(send_acc + i2), ra = *(const longlong2*)(recv_acc + i2);
            longlong2* const lb2 = (longlong2*)(c.lane_bytes_b + (size_t)k * N);
            longlong2* const so2 = (longlong2*)(c.send_off_b + (size_t)(k + 1) * N);
            longlong2* const ro2 = c.recv_off_b ? (longlong2*)(c.recv_off_b + (size_t)(k + 1) * N) : nullptr;
#pragma unroll 4
            for (size_t e = lane; e < rows / 2; e += 32) {
                lb2[e] = make_longlong2(0, 0);
                so2[e] = sa;
                if (ro2) ro2[e] = ra;
            }
        } else {
            for (size_t e = (size_t)k * N + lane; e < (size_t)k * N + rows; e += 32) {
                c.lane_dst_b[e] = -1;
                c.lane_inst_b[e] = 0xFFFF;
                c.lane_bytes_b[e] = 0;
                const int i = (int)(e % N);
                c.send_off_b[N + e] = send_acc[i];
                if (c.recv_off_b) c.recv_off_b[N + e] = recv_acc[i];
            }
        }
        for (int kk = k + lane; kk < kp.k_max && !kp.host_rows; kk += 32) c.chan_id_b[kk] = -1;
        if (lane == 0) {
            n_act += (unsigned long long)k;
            n_steps[b] = k;
            status[b] = st;
            if (tau_out) tau_out[b] = tau;
        }
        __syncwarp();
    }
    cnt.tasks = (unsigned long long)warp_sum_i64((int64_t)cnt.tasks);      // (counted by one lane, or the first lane of every team)
    cnt.sweeps = (unsigned long long)warp_sum_i64((int64_t)cnt.sweeps);
    if (lane == 0) {
        if (slots) {
            unsigned long long* const mine = slots + 3 * ((size_t)blockIdx.x * n_warps + warp);
            mine[0] = n_act; mine[1] = cnt.tasks; mine[2] = cnt.sweeps;
            if (blockIdx.x == 0 && warp == 0) {
                const uint32_t warps = gridDim.x * (uint32_t)n_warps;
                counter[3] = warps;
                ((uint64_t*)counter)[kStatsTagWord] = vp_stats_tag((uint64_t)(uintptr_t)counter, warps);
            }
        } else {
            unsigned long long* const stats = (unsigned long long*)(counter + 4);
            if (n_act) atomicAdd(&stats[0], n_act);
            if (cnt.tasks) { atomicAdd(&stats[1], cnt.tasks); atomicAdd(&stats[2], cnt.sweeps); }
        }
#ifdef VP_PHASE_TIMING
        for (int i = 0; i < 6; i++) atomicAdd((unsigned long long*)(counter + 4) + 3 + i, (unsigned long long)cnt.cyc[i]);
#endif
    }
}

}  // namespace
