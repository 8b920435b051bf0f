// Small batches: one row per thread-block cluster.  Included by albireo_sample.cu.
//
// With a CTA per row a small batch leaves most of the chip idle, and a row of 300 KB takes the 7 us
// that one SM needs to stream it.  Here a row is shared by up to 16 CTAs.  Each copies its slice into
// shared memory once (one bulk copy per piece, no ring: the slice stays there, so the further passes of
// a wide row cost no memory traffic at all), overwrites the penalised tokens in it with -inf and keeps
// them in a list of their own with their scores.  What the CTAs exchange are a few words (distributed
// shared memory, two or three cluster barriers) and their short candidate lists; CTA 0 finishes the row.
//
// The threshold of the candidates is the better of two bounds on the row's k-th largest score: the
// largest of the slices' own k-th largest values, and the smallest of their ceil(k / size)-th largest.

constexpr int SLICE_MIN = 18 * 1024;      // the final stage's scratch lies in CTA 0's slice when that is done with
constexpr int X_LEAST = 1024;             // penalised tokens and unaligned ends of a slice that are listed on chip, at least
constexpr int X_ENDS = 16;                // most unaligned ends of a row (14), rounded up
constexpr int GENERAL_BYTES = HIST_BINS * 16 + GL_CAP * 8 + 4096;      // what the general path lays over the front

// 32-bit words of the tables behind a slice of n elements: bitmap, coarse prefix; then the list_words of the launch for
// counts (then scores) and ids, as many as there can be of them or as there is room for
__host__ __device__ constexpr int slice_coarse_off(int n) { return (((n + 31) / 32) + 4) & ~3; }
__host__ __device__ constexpr int slice_counts_off(int n) { return slice_coarse_off(n) + ((n + 31) / 32 + 7) / 8 + 1; }

// The largest 1 / T at which rows are counted by value.  Top-p rows with a Zipf prior over ids, us without and with counting: 32 of 128256, slices of
// 64 KB, T = 0.2 16.5 and 18.4, 0.25 17.3 and 18.4, 0.3 17.8 and 18.5, 0.35 18.1 and 18.3, 0.7 19.6 and 19.5, 1 27.5 and 24.1; 64 of 152064, 152 KB,
// 21.9 and 22.5, 24.4 and 22.6, at 0.3 26.0 and 22.4, 1 42.4 and 32.2.  (A row whose maximum is 29 and more above all else is as quick without at
// any temperature, 14.3 and 17.7, but that is known too late.)
__host__ __device__ constexpr float counted_inv_t(int slice_bytes) { return slice_bytes >= 96 * 1024 ? 4.0f : 3.0f; }

// Bytes of what lies between a slice and the scores of its penalised tokens: those tables, or, when they are done with, what counted rows need.
__host__ __device__ constexpr int slice_tables(bool counted, bool with_history, int n) {
    const int tables = with_history ? 4 * slice_counts_off(n) : 0;
    return counted && tables < (int)sizeof(CountedSegs) ? (int)sizeof(CountedSegs) : tables;
}

// The k-th and the kp-th largest of the block's per-thread maxima `mk` (0: none), from below: the
// smallest maximum of the value-linear bin in which the count from the top gets there (see
// warm_select).  0 where there are fewer maxima.
__device__ void slice_select(const CandSmem &cs, uint32_t mk, int k, int kp, uint32_t kmin, uint32_t kmax,
                             uint32_t &tau, uint32_t &tau_part) {
    BlockScratch &s = block_scratch();
    uint32_t *binmin = (uint32_t *)(cs.cand + SEL_BINS);
    const float zmin = unkey(kmin), d = unkey(kmax) - zmin;
    const float scale = (d > 0.0f && d <= 3.0e38f) ? __fdividef((float)(SEL_BINS - 1), d) : 0.0f;
    if (mk) {
        int q = (int)((unkey(mk) - zmin) * scale);
        q = q < 0 ? 0 : (q > SEL_BINS - 1 ? SEL_BINS - 1 : q);
        atomicAdd(&cs.hist[q], 1u);
        atomicMin(&binmin[q], mk);
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        constexpr int PER = SEL_BINS / 32;
        uint32_t cn[PER], sum = 0;
#pragma unroll
        for (int q = 0; q < PER; q += 4) {
            const uint4 v = *(const uint4 *)(cs.hist + PER * lane + q);
            cn[q] = v.x; cn[q + 1] = v.y; cn[q + 2] = v.z; cn[q + 3] = v.w;
            sum += v.x + v.y + v.z + v.w;
        }
        uint32_t suf = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const uint32_t t = __shfl_down_sync(0xFFFFFFFFu, suf, o); if (lane + o < 32) suf += t; }
        auto pick = [&](uint32_t want) -> uint32_t {       // in exactly one lane, if there are that many
            uint32_t above = suf - sum;
            if (!(above < want && suf >= want)) return 0u;
            int q = PER - 1;
#pragma unroll
            for (int j = PER - 1; j > 0; --j) { if (above + cn[j] < want && q == j) { above += cn[j]; q = j - 1; } }
            return binmin[PER * lane + q];
        };
        const uint32_t a = __reduce_max_sync(0xFFFFFFFFu, pick((uint32_t)k)), b2 = __reduce_max_sync(0xFFFFFFFFu, pick((uint32_t)kp));
        if (lane == 0) { s.found_digit = a; s.found_cnt = b2; }
    }
    __syncthreads();
    tau = s.found_digit; tau_part = s.found_cnt;
}

// The slice's penalised tokens: how often each occurs (bitmap over the slice, ranks, counts), then
// their scores from the raw logits in shared memory, which they leave with -inf in their place.
// Returns how many there are, or -1 if there is no room for them.  Where the list on chip holds the scores but not
// the ids as well, the ids go to the workspace (`xid` points there then): the row has a word per history id in it, and
// a slice's part begins after as many words as the history has ids ahead of the slice.  (Such rows went to the general
// path: 64 rows of 152064 with 8192-id histories and top-k 40 took 260 us.)  Ends with a barrier.  The row's unaligned ends
// (ids below id_lo or from id_hi on, CTA 0 only) are counted in s.red: occurrences in the output, and in
// the high word whether there are any in the prompt.
// `landed()` waits for the slice; everything before it overlaps the copy.
template <int DT, class W>
__device__ __noinline__ int slice_history(RowCtx c, const int32_t *ids, int len, int out_start, int slice_off, int id0, int nids,
                                          int id_lo, int id_hi, int tab_off, int xz_off, int list_words, uint32_t *ws, int64_t ws_cap, int64_t ws_off,
                                          W landed, bool &ok, int *&xid) {
    typedef Elem<DT> E;
    BlockScratch &s = block_scratch();
    extern __shared__ __align__(128) unsigned char smem[];
    const int nwords = (nids + 31) >> 5, ncoarse = (nwords + 7) >> 3;
    uint32_t *bitmap = (uint32_t *)(smem + tab_off), *coarse = bitmap + slice_coarse_off(nids), *counts = (uint32_t *)(smem + xz_off);
    uint32_t ahead = 0, own = 0;           // history ids ahead of the slice and in it
    for (int w = threadIdx.x; w <= nwords; w += NT) bitmap[w] = 0;
    __syncthreads();
    for (int j = threadIdx.x; j < len; j += NT) {
        const int id = __ldg(ids + j);
        const uint32_t t = (uint32_t)(id - id0);
        ahead += id >= 0 && id < id0;
        own += t < (uint32_t)nids;
        if (id < id_lo ? id >= 0 : id >= id_hi && id < c.V) {
            // (32-bit adds: the first ids of a vocabulary are most of many a history, and a 64-bit add in shared
            // memory is a compare-and-swap loop, 18 us for 2700 ids)
            uint32_t *e = (uint32_t *)&s.red[id < id_lo ? id : id_lo + (id - id_hi)];
            if (j >= out_start) atomicAdd(e, 1u); else e[1] = 1u;
        }
        if (t < (uint32_t)nids) {
            const uint32_t bit = 1u << (t & 31);
            if (!(*(volatile uint32_t *)&bitmap[t >> 5] & bit)) atomicOr(&bitmap[t >> 5], bit);
        }
    }
    __syncthreads();
    uint32_t U = 0;
    for (int base = 0; base < ncoarse; base += NT) {
        const int cb = base + threadIdx.x;
        uint32_t pc = 0;
        if (cb < ncoarse) for (int w = cb << 3; w < min(nwords, (cb << 3) + 8); ++w) pc += __popc(bitmap[w]);
        uint32_t tot;
        const uint32_t ex = block_exscan_u32(pc, tot);
        if (cb < ncoarse) coarse[cb] = U + ex;
        U += tot;
    }
    c.bitmap = bitmap; c.coarse = coarse; c.counts = counts; c.n_distinct = U; c.ncoarse = ncoarse;
    bool fits = 2u * (U + X_ENDS) <= (uint32_t)list_words;
    if (!fits && U + X_ENDS <= (uint32_t)list_words) {
        uint32_t at, n_own;
        block_exscan_u32(ahead, at);
        block_exscan_u32(own, n_own);
        fits = ws && ws_off >= 0 && U + X_ENDS <= n_own && ws_off + (int64_t)at + (int64_t)n_own <= ws_cap;
        if (fits) xid = (int *)ws + ws_off + at;
    }
    if (fits) for (uint32_t u = threadIdx.x; u < U; u += NT) counts[u] = 0;
    __syncthreads();
    if (fits) {
        for (int j = max(out_start, 0) + (int)threadIdx.x; j < len; j += NT) {
            const uint32_t t = (uint32_t)(__ldg(ids + j) - id0);
            if (t < (uint32_t)nids) atomicAdd(&counts[hist_rank(c, (int)t)], 1u);
        }
    }
    ok = landed();
    __syncthreads();
    if (!fits) return -1;
    if (ok) {
        for (uint32_t r = threadIdx.x; r < U; r += NT) {
            const int t = hist_id_of_rank(c, r);
            const float x = E::load_plain(smem + slice_off, t);
            const float z = __fmul_rn(penalise_counted(c, x, counts[r]), c.invT);
            ((float *)counts)[r] = z;
            xid[r] = id0 + t;
            if (E::SIZE == 4) ((uint32_t *)(smem + slice_off))[t] = 0xFF800000u;
            else ((unsigned short *)(smem + slice_off))[t] = (unsigned short)(VecTest<DT>::fill().x & 0xFFFFu);
        }
    }
    __syncthreads();
    return (int)U;
}

template <int DT, class SRC, class TEAM>
__device__ __noinline__ RowOut team_wide_row(SRC src, TEAM tm, RowParams rp, float invT, uint32_t kmax, uint32_t n_fin, int b, uint32_t status) {
    return wide_row<DT>(block_scratch(), src, tm, rp, invT, kmax, n_fin, b, status);
}

// COUNTED: with the code for rows counted by value (see counted_row) and the table for it in front of the slice; launches whose slices are too small,
// or whose rows are not counted, do without (see COUNTED_SLICE, may_count_rows): beside that code their top-p rows took 1.4 us longer, 18.7
// against 17.2 for 8 rows of 32000.
template <int DT, bool COUNTED>
__global__ void __launch_bounds__(NT, 1) albireo_cluster_kernel(const __grid_constant__ SampleArgs a) {
    typedef Elem<DT> E;
    typedef VecTest<DT> T;
    extern __shared__ __align__(128) unsigned char smem[];
    BlockScratch &s = block_scratch();
    constexpr int SLICE_OFF = slice_off(COUNTED);
    ClusterTeam<COUNTED> tm;
    tm.rank = (int)cg::this_cluster().block_rank(); tm.size = (int)cg::this_cluster().num_blocks();
    const int b = blockIdx.x / tm.size, V = a.V, lane = threadIdx.x & 31;
    uint64_t *bar = (uint64_t *)(smem + SLICE_OFF + a.slice_bytes);
    const int tab_off = SLICE_OFF + a.slice_bytes + 16;

    CandSmem cs;
    cs.cand = (u64 *)smem;
    cs.hist = (uint32_t *)(smem + CAND_CAP * 8);
    cs.sorted = (u64 *)(smem + SLICE_OFF);
    cs.efx = cs.sorted + SORT_MAX;
    cs.gsc = cs.efx + SORT_MAX;

    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if constexpr (COUNTED) s.seg_off = tab_off;
        s.cand_cnt = 0; s.runmax = 0; s.race.bound = NO_BOUND; s.mm_max = 0; s.mm_min = 0xFFFFFFFFu; s.list_cnt = 0;
        tm.x->far_cand = 0; tm.x->far_list = 0;
    }
    if (threadIdx.x < NWARPS) s.red[threadIdx.x] = 0;
    cs.hist[threadIdx.x] = 0;
    ((uint32_t *)(cs.cand + SEL_BINS))[threadIdx.x] = 0xFFFFFFFFu;
    // (waited for before the first access to another CTA's shared memory: by then every CTA runs)
    asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory");
    // the next kernel in the stream may be scheduled from here on (it waits for this one to finish), and
    // nothing is read or written before the kernel ahead has finished
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");

    RowParams rp;
    RowCtx c;
    const uint32_t bad_param = load_row<DT>(a, b, s.seg_base, rp, c);
    if (a.nseg > 1 && threadIdx.x == 0) {
        const size_t row_off = (size_t)(a.seg_row_offset + b) * (size_t)a.row_stride * E::SIZE;
        for (int j = 0; j < a.nseg; ++j)
            s.seg_base[j] = a.seg_ptr_count > 0 ? (const char *)a.seg_ptr[j] + row_off
                                                : (const char *)c.row + (size_t)j * (size_t)a.seg_stride * E::SIZE;
    }
    const uintptr_t addr = (uintptr_t)c.row;
    int head = (int)(((16u - (uint32_t)(addr & 15u)) & 15u) / E::SIZE);
    if (head > V) head = V;
    const int nvec = (V - head) / E::PER_VEC;
    const int per = (nvec + tm.size - 1) / tm.size;
    const int v0 = min(nvec, tm.rank * per), nv = min(nvec, v0 + per) - v0;
    const int id0 = head + v0 * E::PER_VEC, tail0 = head + nvec * E::PER_VEC;
    if (threadIdx.x == 0) {
        if (nv > 0) {
            Ring rg;
            rg.vps = a.vps; rg.seg_base = s.seg_base;
            mbar_expect_tx(bar, (uint32_t)nv * 16u);
            ring_copy(rg, smem + SLICE_OFF, (const uint4 *)((const char *)c.row + (size_t)head * E::SIZE), v0, nv, bar);
        } else asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
    }
    int o0 = 0, o1 = 0, ostart = 0;
    const bool tables = a.hist_ids && a.hist_off;
    if (tables) { o0 = a.hist_off[b]; o1 = a.hist_off[b + 1]; if (a.out_start) ostart = a.out_start[b]; }

    RowOut out;
    out.token = 0; out.logprob = 0.0f; out.n_keep = 0; out.n_topk = 0; out.status = bad_param;
    if (tm.rank == 0) {
        if (a.dbg_topk_ids) for (int j = threadIdx.x; j < a.dbg_cap; j += NT) a.dbg_topk_ids[(int64_t)b * a.dbg_cap + j] = -1;
        if (a.num_top > 0) for (int j = threadIdx.x; j < a.num_top; j += NT) {
            a.out_top_ids[(int64_t)b * a.num_top + j] = -1;
            a.out_top_logprobs[(int64_t)b * a.num_top + j] = __uint_as_float(0xFF800000u);
        }
    }
    if (threadIdx.x == 0) fill_general_args(s.ga, a);
    __syncthreads();

    const uint32_t fin_thr = T::finite_threshold(c.invT);       // (while the slice travels)
    // the slice: penalised tokens and (CTA 0) the row's unaligned ends move to the list of extras
    bool landed = true, fits = true;
    int nx = 0;
    const int n_slice_ids = nv * E::PER_VEC;
    SmemSlice<DT> src;
    src.vec_off = SLICE_OFF; src.nvec = nv; src.id0 = id0;
    // (a launch without histories has no tables: only the row's unaligned ends are listed)
    src.xz_off = tab_off + slice_tables(COUNTED, tables, n_slice_ids);
    int *xid = (int *)(smem + src.xz_off) + (a.list_words >> 1);
    // (Rows are counted by value where a cut or a list has to be found, and in slices that are worth clearing and adding up a
    // table of 8192 counts: 32 top-p rows of 128256 by 4 CTAs 26.6 -> 23.7 us, but 13 of 50257 by 8 21.2 -> 23.1.  With no cut
    // the pass of masses and race is faster than counting and race, 22.4 us against 24.5 for 64 rows of 152064.  At low temperatures
    // hardly a vector has any mass, and the pass of masses passes over the others: see counted_inv_t.)
    const bool cand_row = candidate_eligible(rp, a), counted = COUNTED && !cand_row && !nothing_cut(rp, a) && counted_eligible<DT>(rp, c, a) && c.invT <= counted_inv_t(a.slice_bytes);
    if (o1 > o0) {
        nx = slice_history<DT>(c, a.hist_ids + o0, o1 - o0, ostart, SLICE_OFF, id0, n_slice_ids, tm.rank == 0 ? head : 0,
                               tm.rank == 0 ? tail0 : V, tab_off, src.xz_off, a.list_words, a.ws_counts, a.ws_counts_cap, (int64_t)o0,
                               [&] { return mbar_wait(bar, 0); }, landed, xid);
        if (nx < 0) { nx = 0; fits = false; }
    } else landed = mbar_wait(bar, 0);
    const uint32_t distinct = (uint32_t)nx;
    if (tm.rank == 0 && head + (V - tail0) > 0) {
        const int nscal = head + (V - tail0), q = threadIdx.x;      // at most 14
        if (q < nscal) {
            const int i = q < head ? q : tail0 + (q - head);
            const u64 seen = s.red[q];
            const float x = E::load(elem_ptr<DT>(c, i), 0);
            xid[nx + q] = i;
            ((float *)(smem + src.xz_off))[nx + q] = __fmul_rn(seen ? penalise_counted(c, x, (uint32_t)seen) : x, c.invT);
            if (seen) atomicAdd(&tm.x->far_list, 1u);              // (distinct ids among them; far_list starts over below)
        }
        nx += nscal;
        __syncthreads();
    }
    src.nx = nx; src.xid = xid;

    // the slice's maximum, its number of finite scores and every thread's own maximum
    const bool full_lp = (a.flags & ALBIREO_FLAG_LOGPROB_FULL_VOCAB) != 0, full_list = full_lp && a.num_top > 0;
    const bool has_topk = rp.greedy || (rp.top_k >= 1 && rp.top_k < V);
    const int k = rp.greedy ? 1 : rp.top_k, k_eff = full_list ? max(k, a.num_top) : k;
    uint32_t mk = 0, nfin = 0;
    if (counted) {
        if constexpr (COUNTED) {
            counted_clear(src);
            __syncthreads();
            if (__all_sync(0xFFFFFFFFu, landed)) counting_pass<0, false>(src, c.invT, 0.0f);
        }
    } else if (landed) {
        // (the number of finite scores is wanted for rows that may turn out to be wide, and by calls that ask for the top-k stage's size)
        const bool count = !cand_row || !has_topk || a.out_num_topk;
        typename T::Run run = T::run_start();
        if (count) src.vectors([&](const uint4 &q, int) {
            T::run_take(run, q, c.invT);
            nfin += (uint32_t)E::PER_VEC - T::count_not_finite(q, fin_thr, c.invT);
        });
        else {
            const uint4 *vec = (const uint4 *)(smem + SLICE_OFF);
#pragma unroll 4
            for (int v = threadIdx.x; v < nv; v += NT) T::run_take(run, vec[v], c.invT);
        }
        mk = T::run_key(run, c.invT);
        src.extras([&](int, float z) {
            const uint32_t kk = key_of(z);
            mk = kk > mk ? kk : mk;
            nfin += (kk >= KEY_MIN_FINITE && kk < KEY_POS_INF);
        });
    }
    if (mk < KEY_MIN_FINITE || mk >= KEY_POS_INF) mk = 0;
    {
        const uint32_t wmx = __reduce_max_sync(0xFFFFFFFFu, mk), wmn = __reduce_min_sync(0xFFFFFFFFu, mk ? mk : 0xFFFFFFFFu);
        const uint32_t wn = __reduce_add_sync(0xFFFFFFFFu, nfin);
        if (lane == 0) { if (wmx) { atomicMax(&s.mm_max, wmx); atomicMin(&s.mm_min, wmn); } if (wn) atomicAdd(&s.list_cnt, wn); }
    }
    const bool any_late = __syncthreads_or(!landed) != 0;
    uint32_t kmax = s.mm_max, tau_s = 0, tau_p = 0, counted_flags = 0, n_vec = 0;
    if constexpr (COUNTED) { if (counted) n_vec = counted_finite(src, s, c.invT, distinct, counted_flags); }
    if (cand_row && has_topk && kmax) slice_select(cs, mk, k_eff, (k_eff + tm.size - 1) / tm.size, s.mm_min, kmax, tau_s, tau_p);
    asm volatile("barrier.cluster.wait;" ::: "memory");            // (the arrival at the start)
    if ((int)threadIdx.x < tm.size) {
        const int r = threadIdx.x;
        *tm.at(&tm.x->kmax[tm.rank], r) = kmax;
        *tm.at(&tm.x->tau[tm.rank], r) = tau_s;
        *tm.at(&tm.x->tau_part[tm.rank], r) = tau_p;
        *tm.at(&tm.x->nfin[tm.rank], r) = s.list_cnt + n_vec;
        *tm.at(&tm.x->flags[tm.rank], r) = (any_late ? 0x80000000u : 0u) | (fits ? 0u : 0x40000000u) | counted_flags | (distinct + tm.x->far_list);
    }
    tm.sync();
    // (a slot per lane: a loop over the slots would be a chain of shared-memory latencies)
    const bool has_slot = lane < tm.size;
    kmax = __reduce_max_sync(0xFFFFFFFFu, has_slot ? tm.x->kmax[lane] : 0u);
    uint32_t tau = __reduce_max_sync(0xFFFFFFFFu, has_slot ? tm.x->tau[lane] : 0u);
    const uint32_t tau_part = __reduce_min_sync(0xFFFFFFFFu, has_slot ? tm.x->tau_part[lane] : 0xFFFFFFFFu);
    const uint32_t n_fin = __reduce_add_sync(0xFFFFFFFFu, has_slot ? tm.x->nfin[lane] : 0u);
    const uint32_t flags_r = has_slot ? tm.x->flags[lane] : 0u;
    const uint32_t bad = __reduce_or_sync(0xFFFFFFFFu, flags_r) & 0xF0000000u, distinct_row = __reduce_add_sync(0xFFFFFFFFu, flags_r & 0x0FFFFFFFu);
    // what only the one-CTA path decides: too many distinct ids for the tables or for the caller's workspace
    const bool to_general = (bad & 0x40000000u) || kmax == 0 || !(cand_row || wide_eligible(rp, a)) ||
                            (distinct_row > (uint32_t)CNT_CAP && (int64_t)o0 + distinct_row > a.ws_counts_cap);
    bool done = false;
    if (bad & 0x80000000u) {
        mbar_wait(bar, 0);                      // (a copy still in flight gets as long again before its memory is given up)
        out.status |= ALBIREO_ROW_TIMEOUT; out.token = -1; out.logprob = __uint_as_float(0x7FC00000u);
        done = true;
    } else if (!to_general) {
        bool wide = !cand_row;
        if (cand_row) {
            const bool stream_minp = floor_while_streaming<true>(rp, a, has_topk, full_list);
            tau = max(tau, tau_part);
            if (!has_topk || tau < KEY_MIN_FINITE) tau = KEY_MIN_FINITE;
            if (stream_minp) tau = max(tau, min(kmax, minp_key(unkey(kmax), rp.ln_min_p)));
            const uint32_t thr = T::raw_threshold(tau, c.invT);
            // a thread's survivors of a vector (most have none, the rest one or two) take their places in the list together
            src.vectors([&](const uint4 &q, int i0) {
                uint32_t bits = T::may_pass(q, thr, c.invT) ? T::elem_bits(q, thr, c.invT) : 0u;
                if (!bits) return;
                auto key_at = [&](int x) { return key_of(__fmul_rn(pick_element<DT>(q, x), c.invT)); };
                uint32_t in = 0;
                for (uint32_t r = bits; r; r &= r - 1u) { const uint32_t key = key_at(__ffs(r) - 1); in |= key >= tau && key < KEY_POS_INF ? r & -r : 0u; }
                uint32_t slot = in ? atomicAdd(&s.cand_cnt, (uint32_t)__popc(in)) : 0u;
                for (; in; in &= in - 1u, ++slot) {
                    const int x = __ffs(in) - 1;
                    if (slot < (uint32_t)CAND_CAP) cs.cand[slot] = comp_of(key_at(x), i0 + x);
                }
            });
            src.extras([&](int i, float z) {
                const uint32_t key = key_of(z);
                if (key >= tau && key < KEY_POS_INF) {
                    const uint32_t slot = atomicAdd(&s.cand_cnt, 1u);
                    if (slot < (uint32_t)CAND_CAP) cs.cand[slot] = comp_of(key, i);
                }
            });
            if (full_lp) {
                u64 S_all, same;
                mass_pass<DT, SUM_ONLY, false>(src, c.invT, unkey(kmax), 0.0f, 0u, 0, S_all, same);
                S_all = block_sum_u64(S_all);
                if (threadIdx.x == 0) *tm.at(&tm.x->S_all[tm.rank], 0) = S_all;
            }
            __syncthreads();
            const int n_mine = (int)s.cand_cnt;
            if ((int)threadIdx.x < tm.size) *tm.at(&tm.x->ncand[tm.rank], (int)threadIdx.x) = (uint32_t)n_mine;
            if (tm.rank != 0 && n_mine <= CAND_CAP) {
                if (threadIdx.x == 0) s.found_digit = n_mine ? atomicAdd(tm.at(&tm.x->far_cand, 0), (uint32_t)n_mine) : 0u;
                __syncthreads();
                const int at = CAND_CAP - 1 - (int)s.found_digit;
                u64 *cand0 = tm.at(cs.cand, 0);
                for (int j = threadIdx.x; j < n_mine; j += NT) if (at - j >= 0) cand0[at - j] = cs.cand[j];
            }
            tm.sync();
            int n = (int)__reduce_add_sync(0xFFFFFFFFu, has_slot ? tm.x->ncand[lane] : 0u);
            // a min-p that keeps more than the final stage takes is a wide row; the team stays together for it
            wide = !has_topk && n > SORT_MAX;
            if (!wide && tm.rank == 0 && n <= CAND_CAP) {
                n = close_gap(cs.cand, CAND_CAP, n_mine, n - n_mine);
                u64 full_fx = 0;
                if (full_lp) for (int r = 0; r < tm.size; ++r) full_fx += tm.x->S_all[r];
                done = candidate_finish<true>(s, cs, n, tau, kmax, rp, a, b, out, full_fx, n_fin);
            }
        }
        if (wide) {
            const uint32_t status = out.status;
            if constexpr (COUNTED) out.status |= ROW_NOT_COUNTED;
            if constexpr (COUNTED) {
                // (out of line beside the code for counted rows, which else leaves the others spilling: 30 rows of 152064 with a top-k 10.5 us instead
                // of 10.2.  Top-p rows that are not counted lose by it, 17.5 to 18.0 us for 8 rows of 32000: so not in the other kernel.)
                if (counted) out = counted_row(src, tm, rp, c.invT, kmax, n_fin, bad, b, status);
                if (out.status & ROW_NOT_COUNTED) out = team_wide_row<DT>(src, tm, rp, c.invT, kmax, n_fin, b, status);
            } else out = wide_row<DT>(s, src, tm, rp, c.invT, kmax, n_fin, b, status);
            done = !(out.status & ROW_NOT_DONE);
            if (!done) out.status = status;
        }
    }
    if (tm.rank != 0) return;
    if (!done) {
        // the one-CTA path, from global memory, with tables over the whole row
        __syncthreads();
        if (threadIdx.x == 0) asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
        __syncthreads();
        HistSmem hs;
        const int nw = (V + 31) >> 5, nc = (nw + 7) >> 3;
        hs.bitmap = (uint32_t *)(smem + GENERAL_BYTES);
        hs.coarse = hs.bitmap + (nw + 1);
        hs.counts = hs.coarse + (nc + 1);
        if (o1 > o0) {
            hist_prefetch(a.hist_ids + o0, o1 - o0, (int32_t *)smem);
            c.has_hist = build_history(hs, c, a.hist_ids + o0, o1 - o0, ostart, (const int32_t *)smem, a.ws_counts, a.ws_counts_cap, (int64_t)o0);
            if (!c.has_hist) out.status |= ALBIREO_ROW_HISTORY_OVERFLOW;
        }
        __syncthreads();
        out = general_path_call<DT>(&s, smem, c, rp, b, out.status);
    }
    store_row(a, b, out);
}
