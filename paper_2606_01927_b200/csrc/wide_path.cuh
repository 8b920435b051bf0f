// Wide rows: rows whose kept set has no small bound (top-p alone, no cut at all, a min-p that keeps
// thousands).  Included by albireo_sample.cu.
//
// What such a row costs is instructions: every element needs its mass, and with no cut a share of a Philox block.  So the row
// is passed over as few times as the definition allows and each pass does one short fixed sequence per element.  Rows of
// bfloat16 are counted by value (counted_row, below); in general:
//   mass    e = exp(z - zmax) summed in fixed point, and, where a cut or a list has to be found, one
//           32-bit shared-memory add per element into a histogram of masses over bins that are linear
//           in log2 e (32 per octave);
//   locate  the window of bins in which the wanted mass (or rank) is reached, from prefix sums; a window
//           that may hold more than the list takes is split again (one more pass that adds only the
//           window's elements);
//   final   the elements above the window are kept for sure: their exact mass, their number, the race.
//           Those in the window go to an on-chip list, in which the cut is found exactly; the exact
//           masses check that the histogram had located it (otherwise the row goes to the general path).
// With no cut the first and the last pass are the same pass.  A row may be shared by the CTAs of a
// cluster (a Team), each holding a slice; what they exchange is the histogram and a few words.

// ------------------------------------------------------------------ teams

constexpr int MAX_TEAM = 16;

// Words that the CTAs of a row exchange: slot r is written by CTA r, in every CTA or only in CTA 0's copy.
struct TeamWords {
    uint32_t kmax[MAX_TEAM], tau[MAX_TEAM], tau_part[MAX_TEAM], nfin[MAX_TEAM], flags[MAX_TEAM];   // in every CTA
    uint32_t ncand[MAX_TEAM];         // (rows counted by value: whether the table cannot tell)
    u64 ahead[MAX_TEAM];                                                                                           // in every CTA
    u64 S[MAX_TEAM], S_all[MAX_TEAM], M[MAX_TEAM], G[MAX_TEAM];                                                    // in CTA 0's
    uint32_t n[MAX_TEAM];
    float z[MAX_TEAM];
    uint32_t far_cand, far_list;      // CTA 0: entries that the others have put at the far end of its lists
};

// (COUNTED here and below: in a kernel with the table of rows counted by value, which lies in front of them)
template <bool COUNTED> __device__ __forceinline__ TeamWords &team_words();
template <bool COUNTED>
struct TeamWordsHere {                // this CTA's (named anew at every use, see block_scratch)
    __device__ __forceinline__ TeamWords *operator->() const { return &team_words<COUNTED>(); }
    __device__ __forceinline__ TeamWords &operator*() const { return team_words<COUNTED>(); }
};
template <bool COUNTED>
struct SoloTeam {                     // a CTA that has the row to itself
    TeamWordsHere<COUNTED> x;
    static constexpr bool ALONE = true;
    static constexpr int rank = 0, size = 1;
    __device__ __forceinline__ void sync() const { __syncthreads(); }
    template <class P> __device__ __forceinline__ P *at(P *p, int) const { return p; }
};
template <bool COUNTED>
struct ClusterTeam {                  // the CTAs of a thread-block cluster
    TeamWordsHere<COUNTED> x;
    static constexpr bool ALONE = false;
    int rank, size;
    __device__ __forceinline__ void sync() const {
        asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    }
    template <class P> __device__ __forceinline__ P *at(P *p, int r) const { return cg::this_cluster().map_shared_rank(p, r); }
};

// ------------------------------------------------------------------ reductions with few instructions

// sum of the warp's values, each below 2^58, in every lane: three 32-bit reductions instead of ten shuffles
__device__ __forceinline__ u64 warp_total(u64 v) {
    const uint32_t a = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)v & 0x7FFFFFu), b = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)(v >> 23) & 0x7FFFFFu);
    const uint32_t c = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)(v >> 46));
    return (u64)a + ((u64)b << 23) + ((u64)c << 46);
}
// the largest G of the warp and its z, in every lane
__device__ __forceinline__ void warp_best(u64 &G, float &z) {
    const uint32_t hi = __reduce_max_sync(0xFFFFFFFFu, (uint32_t)(G >> 32));
    const uint32_t lo = __reduce_max_sync(0xFFFFFFFFu, (uint32_t)(G >> 32) == hi ? (uint32_t)G : 0u);
    const uint32_t who = __ballot_sync(0xFFFFFFFFu, (uint32_t)(G >> 32) == hi && (uint32_t)G == lo);
    z = __shfl_sync(0xFFFFFFFFu, z, __ffs(who) - 1);
    G = ((u64)hi << 32) | lo;
}
// what a pass leaves in each thread, added up: masses, number and race of the kept elements
struct Partial {
    u64 M, G;
    uint32_t n;
    float z;
    __device__ __forceinline__ void over_warp() { M = warp_total(M); n = __reduce_add_sync(0xFFFFFFFFu, n); warp_best(G, z); }
};
// The block's totals, in every lane of warp 0 (the other warps have handed in theirs).  One barrier.
__device__ __forceinline__ void block_partial(BlockScratch &s, Partial &p) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    p.over_warp();
    if (lane == 0) { s.red[wid] = p.M; s.red2[wid] = p.G; s.r32a[wid] = p.n; s.r32b[wid] = __float_as_uint(p.z); }
    __syncthreads();
    if (wid == 0) {
        const bool in = lane < NWARPS;
        p.M = in ? s.red[lane] : 0ull; p.G = in ? s.red2[lane] : 0ull; p.n = in ? s.r32a[lane] : 0u; p.z = in ? __uint_as_float(s.r32b[lane]) : 0.0f;
        p.over_warp();
    }
}

// ------------------------------------------------------------------ what a CTA reads of its row

template <int DT>
__device__ __forceinline__ uint4 kill_elements(uint4 q, uint32_t m) {      // elements of the mask become -inf
    if constexpr (Elem<DT>::PER_VEC == 4) {
        if (m & 1u) q.x = 0xFF800000u;
        if (m & 2u) q.y = 0xFF800000u;
        if (m & 4u) q.z = 0xFF800000u;
        if (m & 8u) q.w = 0xFF800000u;
    } else {
        const uint32_t ninf = VecTest<DT>::fill().x;
        auto word = [&](uint32_t w, uint32_t mm) {
            if (mm & 1u) w = (w & 0xFFFF0000u) | (ninf & 0xFFFFu);
            if (mm & 2u) w = (w & 0x0000FFFFu) | (ninf & 0xFFFF0000u);
            return w;
        };
        q.x = word(q.x, m); q.y = word(q.y, m >> 2); q.z = word(q.z, m >> 4); q.w = word(q.w, m >> 6);
    }
    return q;
}
// element x of a vector, x not known at compile time
template <int DT>
__device__ __forceinline__ float pick_element(const uint4 &q, int x) {
    constexpr int PV = Elem<DT>::PER_VEC;
    const uint32_t w = x < PV / 2 ? (x < PV / 4 ? q.x : q.y) : (x < 3 * PV / 4 ? q.z : q.w);
    return Elem<DT>::get(make_uint4(w, w, w, w), PV == 4 ? 0 : (x & 1));
}

// A callee that takes two vectors gets two of a thread's at a time from global memory, and elsewhere one and nothing (-inf, id -1).
template <class F> constexpr bool by_pairs = std::is_invocable<F, uint4, uint4, int, int>::value;
// A callee may come with a test of two vectors at once: where no lane's answer is true the callee is not called for them (it must
// have nothing to do there).
struct NoTest {};

// The whole row from global memory (from the L2 after the first pass), in plain 16-byte loads that wait in registers: AHEAD of a thread's
// vectors are on their way while it works on another.  Penalised tokens are masked out of the vectors
// and come from the history tables.  Both loops have the same trip count in every lane of a warp (lanes
// past the end see -inf), so that the callee may use warp collectives, but no block barriers.
// How many wait is what the registers of the passes leave room for: 4 where the callee keeps a sum or a maximum, else 2 (with 4, the functions around the passes spilled 124 bytes instead of
// 32 to 60), 1 where whole vectors are raced; 2 and 2 where pairs are tested.  148 rows of 128256, top-p, us with 4 everywhere and so: fp32 98.5 and 93.3, f16 77.8 and 72.8; 256 rows of fp32, which
// the L2 does not hold, 143.9 and 134.7 (136.9 from a ring); with 2 for the largest element, too, rows without a cut 55.1 -> 59.
// (What the loop does not touch per vector stays in shared memory: a pass needs its registers for the elements.)
// What bounds a pass is shared memory and issue slots, not the loads: with the vectors brought into shared memory by bulk copies, as before,
// both the copies and the reads back were in the way of the callee's own accesses, and each tile of 32 KB cost a hand-shake of all
// warps.  A row of 152064 bfloat16 logits by one CTA, in the L2, us including the launch, from a ring and from registers: largest element
// 8.3 and 6.2, counted by value 19.5 and 12.4, exponentials summed 13.2 and 12.4; two rows per SM 10.3 and 8.2, 32.8 and 22.4, 23.7 and 20.5.
struct RowShared {
    RowCtx c;
    RowParams rp;
    const uint4 *vp;
    int head, nvec;
    int vps;                      // vectors per piece
};
template <int DT> __device__ __forceinline__ RowShared &row_shared();
template <int DT> __device__ __forceinline__ constexpr int row_segments();
// which of the n elements from i0 on are in the history, from the bitmap's address in shared memory
template <int N>
__device__ __forceinline__ uint32_t history_mask(uint32_t bitmap, int i0) {
    uint32_t w0, w1;
    asm volatile("ld.shared.u32 %0, [%2];\n\tld.shared.u32 %1, [%2 + 4];" : "=r"(w0), "=r"(w1) : "r"(bitmap + 4u * ((uint32_t)i0 >> 5)));
    return __funnelshift_r(w0, w1, i0 & 31) & ((1u << N) - 1u);
}
template <int DT>
struct RowSlice {
    typedef Elem<DT> E;
    static constexpr bool SPARE_REGISTERS = false;      // 64 per thread
    __device__ __forceinline__ int first_id() const { return row_shared<DT>().head; }
    __device__ __forceinline__ int end_id() const { return row_shared<DT>().head + row_shared<DT>().nvec * E::PER_VEC; }
    __device__ __forceinline__ int elements() const { return row_shared<DT>().nvec * E::PER_VEC; }
    __device__ __forceinline__ int segments() const { return row_segments<DT>(); }      // (counted rows: see CountedSegs)
    // vector v by itself (v < 0: none)
    __device__ __forceinline__ uint4 vector(int v) const {
        if (v < 0) return VecTest<DT>::fill();
        const RowShared &r = row_shared<DT>();
        uint4 q = __ldg(vec_ptr<DT>(r.c, r.vp, v));
        if (r.c.has_hist) {
            const uint32_t m = history_mask<E::PER_VEC>(smem_u32(r.c.bitmap), r.head + v * E::PER_VEC);
            if (m) q = kill_elements<DT>(q, m);
        }
        return q;
    }
    // The row's vectors, piece after piece (lanes past the end of one see -inf and the id behind the last).
    template <int AHEAD = 2, class F, class T = NoTest> __device__ __forceinline__ void vectors(F &&f, T &&test = T()) const {
        constexpr bool PAIRS = by_pairs<F>, TESTED = !std::is_same<std::decay_t<T>, NoTest>::value;
        const RowShared &r = row_shared<DT>();
        const int head = r.head, end_id = head + r.nvec * E::PER_VEC;
        const uint32_t bitmap = r.c.has_hist ? smem_u32(r.c.bitmap) : 0u;
        auto masked = [&](uint4 q, int i0) -> uint4 {
            if (bitmap && i0 < end_id) {
                const uint32_t m = history_mask<E::PER_VEC>(bitmap, i0);
                if (m) q = kill_elements<DT>(q, m);
            }
            return q;
        };
#pragma unroll 1
        for (int j = 0; j < r.c.nseg; ++j) {
            const bool whole = r.c.nseg == 1;
            const int lo = whole ? 0 : j * r.vps, hi = whole ? r.nvec : min(r.nvec, lo + r.vps);
            const uint4 *const vp = (whole ? r.vp : (const uint4 *)r.c.seg_base[j]) - lo;
            auto load = [&](int v) -> uint4 { return v < hi ? __ldg(vp + v) : VecTest<DT>::fill(); };
            auto id_of = [&](int v) { return v < hi ? head + v * E::PER_VEC : end_id; };
            if constexpr (TESTED) {
                // two at a time, the next two on their way
                uint4 q0 = load(lo + (int)threadIdx.x), q1 = load(lo + (int)threadIdx.x + NT);
#pragma unroll 1
                for (int v0 = lo + (int)threadIdx.x; v0 - (int)threadIdx.x < hi; v0 += 2 * NT) {
                    const uint4 x = q0, y = q1;
                    q0 = load(v0 + 2 * NT); q1 = load(v0 + 3 * NT);
                    if (!__any_sync(0xFFFFFFFFu, test(x, y))) continue;
#pragma unroll 1
                    for (int u = 0; u < 2; ++u) {
                        const int i0 = id_of(v0 + u * NT);
                        f(masked(u ? y : x, i0), i0);
                    }
                }
            } else {
                uint4 q[AHEAD];
#pragma unroll
                for (int u = 0; u < AHEAD; ++u) q[u] = load(lo + (int)threadIdx.x + u * NT);
#pragma unroll 1
                for (int v0 = lo + (int)threadIdx.x; v0 - (int)threadIdx.x < hi; v0 += AHEAD * NT) {
#pragma unroll
                    for (int u = 0; u < AHEAD; u += PAIRS ? 2 : 1) {
                        const int v = v0 + u * NT, i0 = id_of(v);
                        const uint4 x = masked(q[u], i0);
                        q[u] = load(v + AHEAD * NT);
                        if constexpr (PAIRS) {
                            const int i1 = id_of(v + NT);
                            const uint4 y = masked(q[u + 1], i1);
                            q[u + 1] = load(v + (AHEAD + 1) * NT);
                            f(x, y, i0, i1);
                        } else f(x, i0);
                    }
                }
            }
        }
        __syncthreads();
    }
    template <class F> __device__ __forceinline__ void extras(F &&f) const {
        const RowShared &r = row_shared<DT>();
        const RowCtx &c = r.c;
        const int head = r.head, tail0 = head + r.nvec * E::PER_VEC, nscal = head + (c.V - tail0);
        const int total = nscal + (c.has_hist ? (int)c.n_distinct : 0);
#pragma unroll 1
        for (int base = 0; base < total; base += NT) {
            const int q = base + (int)threadIdx.x;
            int i = 0; float z = -INFINITY;
            if (q < nscal) {
                i = q < head ? q : tail0 + (q - head);
                if (!(c.has_hist && ((c.bitmap[i >> 5] >> (i & 31)) & 1u))) z = __fmul_rn(E::load(elem_ptr<DT>(c, i), 0), c.invT);
            } else if (q < total) {
                const uint32_t rank = (uint32_t)(q - nscal);
                i = hist_id_of_rank(c, rank);
                z = c.scored ? __uint_as_float(c.counts[rank]) : __fmul_rn(penalise_counted(c, E::load(elem_ptr<DT>(c, i), 0), c.counts[rank]), c.invT);
            }
            f(i, z);
        }
    }
};

// A slice of the row that lies in shared memory, its penalised tokens already overwritten with -inf;
// they and the row's unaligned ends are in a list of (id, score).  Both loops have the same trip count
// in every lane of a warp (lanes past the end see -inf), so that the callee may use warp collectives,
// but no block barriers.
template <int DT>
struct SmemSlice {
    typedef Elem<DT> E;
    static constexpr bool SPARE_REGISTERS = true;       // 128 per thread
    int vec_off, nvec, id0;       // where the slice and the list lie in the dynamic shared memory
    const int *xid;               // (in the workspace where there are too many for both lists on chip)
    int xz_off, nx;
    __device__ __forceinline__ int first_id() const { return id0; }
    __device__ __forceinline__ int end_id() const { return id0 + nvec * E::PER_VEC; }
    __device__ __forceinline__ int elements() const { return nvec * E::PER_VEC; }
    __device__ __forceinline__ int segments() const { return block_scratch().seg_off; }      // (in a register it was spilled)
    __device__ __forceinline__ uint4 vector(int v) const {
        extern __shared__ __align__(128) unsigned char smem[];
        return v < 0 ? VecTest<DT>::fill() : ((const uint4 *)(smem + vec_off))[v];
    }
    template <int AHEAD = 2, class F, class T = NoTest> __device__ __forceinline__ void vectors(F &&f, T && = T()) const {
        extern __shared__ __align__(128) unsigned char smem[];
        const uint4 *vec = (const uint4 *)(smem + vec_off);
        constexpr bool PAIRS = by_pairs<F>;
#pragma unroll 1
        for (int base = 0; base < nvec; base += NT) {
            const int v = base + (int)threadIdx.x, i0 = id0 + v * E::PER_VEC;
            const uint4 q = v < nvec ? vec[v] : VecTest<DT>::fill();
            if constexpr (PAIRS) f(q, VecTest<DT>::fill(), i0, -1);
            else f(q, i0);
        }
    }
    template <class F> __device__ __forceinline__ void extras(F &&f) const {
        extern __shared__ __align__(128) unsigned char smem[];
        const float *xz = (const float *)(smem + xz_off);
#pragma unroll 1
        for (int r0 = 0; r0 < nx; r0 += NT) {
            const int r = r0 + (int)threadIdx.x;
            f(r < nx ? xid[r] : 0, r < nx ? xz[r] : -INFINITY);
        }
    }
};

// ------------------------------------------------------------------ masses and their order codes

// Code of an element: F = -log2(e) in 1/65536 octaves, rounded; a larger z never has a larger F (every
// step is one monotone rounding).  Kept with the exponent of the magic number added: code(z = zmax) is
// F_ZERO.  Beyond 128 octaves the sum leaves the integer range of the mantissa and only keeps the order.
constexpr uint32_t F_ZERO = 0x4B000000u;               // bits of 2^23
constexpr int W_SHIFT = 11;                            // 65536 / 2^11 = 32 bins per octave
constexpr int W_BINS = 1344;                           // 42 octaves
constexpr int W_PER = 4;                               // bins per thread in the scans (one 16-byte load; the last threads have none)
constexpr int W_LIST = CAND_CAP;                       // entries of the top-N list and, beside it, of the window's list
constexpr int W_LIST_ALONE = 2 * W_LIST;               // entries of the window's list where there is no top-N list

__device__ __forceinline__ float ex2_ftz(float t) { float e; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(t)); return e; }
__device__ __forceinline__ float log2_mass(float z, float zmax) { return __fmul_rn(__fsub_rn(z, zmax), 1.4426950408889634f); }
// (of two elements: one rounding per step as well, so the same bits)
__device__ __forceinline__ float2 log2_mass2(float2 z, float zmax) {
    return mul_pair(add_pair(z, pair_of(-zmax)), pair_of(1.4426950408889634f));
}
__device__ __forceinline__ uint2 code_of2(float2 t2) {
    const float2 c = fma_pair(t2, pair_of(-65536.0f), pair_of(8388608.0f));
    return make_uint2(__float_as_uint(c.x), __float_as_uint(c.y));
}
__device__ __forceinline__ uint32_t code_of(float t2) { return __float_as_uint(__fmaf_rn(t2, -65536.0f, 8388608.0f)); }
// A bin's masses are added up as 12-bit fractions of the bin's octave (at most 2^19 elements: no
// overflow).  `octave_code` = code >> 16 carries the magic exponent, which turns into the sign bit.
__device__ __forceinline__ uint32_t mass12(float e, uint32_t octave_code) {
    const float neg = __uint_as_float(__float_as_uint(e) + (octave_code << 23));
    return __float_as_uint(2048.0f - neg) - 0x45000000u;
}
__device__ __forceinline__ u64 mass_of_bin(uint32_t q, uint32_t octave) { return octave < 60u ? ((u64)q << 28) >> octave : 0ull; }   // 2^-40 units
// hist[bin] += v if bin < W_BINS, without a branch
__device__ __forceinline__ void hist_add_if(uint32_t hist_addr, uint32_t bin, uint32_t v) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.lt.u32 p, %1, %2;\n\t@p red.shared.add.u32 [%0], %3;\n\t}"
                 ::"r"(hist_addr + bin * 4u), "r"(bin), "n"(W_BINS), "r"(v) : "memory");
}

struct WideSmem {
    u64 *top;             // W_LIST composites: the top-N list
    u64 *list;            // W_LIST composites: the window
    uint32_t *hist;       // W_BINS words
    u64 *queue;           // 64 entries per warp, later masses of the window's list
};
// The front of the dynamic shared memory, whatever the kernel keeps behind it
// (the candidate list and its select bins lie where the top-N list does).
constexpr int WIDE_LIST_OFF = COMMON_BYTES, WIDE_HIST_OFF = WIDE_LIST_OFF + W_LIST * 8;
constexpr int WIDE_QUEUE_OFF = WIDE_HIST_OFF + W_BINS * 4, WIDE_BYTES = WIDE_QUEUE_OFF + NWARPS * 64 * 8;
static_assert(W_LIST_ALONE * 8 <= WIDE_HIST_OFF, "the window's list alone lies over both lists and the select bins");
// Rows of bfloat16 whose values are counted (see counted_row): the table of counts lies over all of the above, the queues of the last
// pass, when it is done with, behind the lists.  What else they need (CountedSegs) lies where the kernel has room: in a cluster
// over the tables of the history, of which only the scores are still wanted.
constexpr int CT_BINS = 8192, CT_ODD = 254, CT_BYTES = CT_BINS * 4;
constexpr int CT_QUEUE_OFF = WIDE_LIST_OFF + W_LIST * 8;
constexpr int FINAL_QUEUE = (CT_BYTES - CT_QUEUE_OFF) / 2 / NT * NT;      // vectors that wait in the last pass, by their numbers (at most 2^16)
static_assert(WIDE_BYTES <= CT_BYTES && ALBIREO_MAX_VOCAB / 8 <= 65536, "lists and queue in front of the team's words");
// Where the cut and the list end, the same in every CTA.
struct CountedCut {
    uint32_t thr_any, thr_win, thr_sure, thr_top;     // raw, packed twice: values from there on matter, are in the window or kept, are kept, are listed
    uint32_t key_lo, key_hi;                          // the window's order keys, both inclusive: above it kept
    uint32_t key_seg;                                 // extras above it are in M and n
    uint32_t key_top;
    u64 M; uint32_t n;                                // kept for sure, all but the extras above the window and not above key_seg
    uint32_t n_any;                                   // no more elements of vectors than this are at or above thr_any (all ones: not known)
    uint32_t fail;                                    // (0 ahead of the counting pass: any thread may set it from there on)
};
struct alignas(16) CountedSegs {
    u64 mass[NT];                     // by segments of 16 values; with no cut the list of the race (RACE_LIST) lies here
    uint32_t cnt[NT];
    uint32_t zeros[2];                // +0 and -0
    uint32_t n_odd, odd[CT_ODD];      // other values that have no place in the table
    uint32_t lost;                    // there are more of them than that
    uint32_t high;                    // some of them are above the table's
    CountedCut cut;
};
// The slices of a cluster begin behind the team's words, by one CTA the row's own block does.  (At 128 bytes: 30 rows
// of 152064 with a top-k took 10.7 us with slices at 16, 10.3 so.)
__host__ __device__ constexpr int team_off(bool counted) { return counted ? CT_BYTES : WIDE_BYTES; }
__host__ __device__ constexpr int slice_off(bool counted) { return (team_off(counted) + (int)sizeof(TeamWords) + 127) & ~127; }
template <bool COUNTED> __device__ __forceinline__ TeamWords &team_words() { extern __shared__ __align__(128) unsigned char smem[]; return *(TeamWords *)(smem + team_off(COUNTED)); }
__host__ __device__ constexpr bool counts_rows(int dt) { return dt == ALBIREO_BF16; }      // the kernel of one CTA per row
__host__ __device__ constexpr int row_off(int dt) { return slice_off(counts_rows(dt)) + (counts_rows(dt) ? (int)sizeof(CountedSegs) : 0); }
// (the tables of the history, which the passes ask, lie behind the ring of at least two stages)
constexpr int row_end(int dt) { return row_off(dt) + (int)sizeof(RowShared); }
static_assert(row_end(ALBIREO_F32) <= COMMON_BYTES + 2 * STAGE_BYTES && row_end(ALBIREO_BF16) <= COMMON_BYTES + 2 * STAGE_BYTES && row_end(ALBIREO_F16) <= COMMON_BYTES + 2 * STAGE_BYTES, "a wide row in front of its tables");
template <int DT> __device__ __forceinline__ constexpr int row_segments() { return slice_off(counts_rows(DT)); }
template <int DT> __device__ __forceinline__ RowShared &row_shared() { extern __shared__ __align__(128) unsigned char smem[]; return *(RowShared *)(smem + row_off(DT)); }
static_assert(sizeof(CountedSegs) % 16 == 0 && sizeof(RowShared) % 8 == 0, "what follows is aligned");
__device__ __forceinline__ WideSmem wide_smem() {
    extern __shared__ __align__(128) unsigned char smem[];
    WideSmem w;
    w.top = (u64 *)smem; w.list = (u64 *)(smem + WIDE_LIST_OFF);
    w.hist = (uint32_t *)(smem + WIDE_HIST_OFF); w.queue = (u64 *)(smem + WIDE_QUEUE_OFF);
    return w;
}

// One pass of masses.  FIRST_LEVEL: every element into its bin (1/32 octave; what lies more than 42
// octaves below the maximum is in none: 2^19 such elements weigh 1e-7 of it).  INSIDE_WINDOW: only
// elements with code in [lo, lo + (W_BINS << shift)), into bins of 2^shift.  S: the masses of the
// elements with z >= zfloor (inside a window: of those ahead of it), S_all: of all.
// About 19 instructions per element and, on the first level, a shared-memory add (3 to 5 bank cycles per warp).
enum MassMode { SUM_ONLY, FIRST_LEVEL, INSIDE_WINDOW };
template <int DT, int MODE, bool FLOOR, class SRC>
__device__ __forceinline__ void mass_pass(const SRC &src, float invT, float zmax, float zfloor, uint32_t lo, int shift, u64 &S_out, u64 &S_all_out) {
    typedef Elem<DT> E;
    const uint32_t hist = smem_u32(wide_smem().hist);
    const float minus0 = minus_zero(invT);
    MassSum S, S_all;
    // an element's place in the histogram, and whether its mass counts towards S
    auto place = [&](float z, float e, uint32_t f) -> bool {
        bool in = true;
        if (FLOOR) { in = z >= zfloor; f = in ? f : 0xFFFFFFFFu; }
        if (MODE == INSIDE_WINDOW) in = f < lo;
        if (MODE == FIRST_LEVEL) hist_add_if(hist, (f >> W_SHIFT) - (F_ZERO >> W_SHIFT), mass12(e, f >> 16));
        if (MODE == INSIDE_WINDOW) hist_add_if(hist, f >= lo ? (f - lo) >> shift : 0xFFFFFFFFu, mass12(e, f >> 16));
        return in;
    };
    auto add2 = [&](float2 z) {
        const float2 t2 = log2_mass2(z, zmax);
        const float2 e = make_float2(ex2_ftz(t2.x), ex2_ftz(t2.y));
        const uint2 f = code_of2(t2);
        const bool in0 = place(z.x, e.x, f.x), in1 = place(z.y, e.y, f.y);
        S.add2(make_float2(in0 ? e.x : 0.0f, in1 ? e.y : 0.0f));
        if (FLOOR && MODE != INSIDE_WINDOW) S_all.add2(e);
    };
    const uint32_t thr = VecTest<DT>::raw_threshold(key_of(zmax - 29.5f), invT);
    src.template vectors<MODE == SUM_ONLY ? 4 : 2>([&](const uint4 &q, int) {
        if (!VecTest<DT>::may_pass(q, thr, invT)) return;          // nothing within 42 octaves of the maximum
#pragma unroll
        for (int j = 0; j < E::PER_VEC; j += 2) add2(scores_of(E::get(q, j), E::get(q, j + 1), invT, minus0));
    });
    src.extras([&](int, float z) { add2(make_float2(z, -INFINITY)); });
    S_out = S.total(); S_all_out = FLOOR ? S_all.total() : S_out;
}

// The passes out of line, for the kernel that has 64 registers per thread: each gets them all to itself.
struct PassOut { u64 a, b; };
template <int DT, int MODE, bool FLOOR>
__device__ __noinline__ PassOut solo_mass_pass(float invT, float zmax, float zfloor, uint32_t lo, int shift) {
    PassOut o;
    mass_pass<DT, MODE, FLOOR>(RowSlice<DT>(), invT, zmax, zfloor, lo, shift, o.a, o.b);
    return o;
}

// One level of the search: where the running total of the team's histogram (masses, or lower bounds of
// the element counts) reaches its target, give or take the rounding of the histogram: 2^-slack_shift of
// its total on both sides, or so many elements (targets beyond the total are cut down to it).  On the first level of a search
// by mass the target is the share `frac` of the histogram's own total.  (A bin's mass is cut off at 2^-40: W_BINS units at most.)
struct Window {
    uint32_t lo, hi;      // codes, both inclusive
    uint32_t id_lo, id_hi;      // of the elements with code lo only ids from id_lo on, of those with code hi only up to id_hi
    u64 before;           // running total ahead of lo
    uint32_t most;        // no more elements than this lie in [lo, hi]
    uint32_t ahead_most;  // nor than this ahead of it (first level)
    bool found;
};
template <class TEAM>
__device__ __noinline__ Window find_window(TEAM tm, bool by_count, uint32_t base, int shift, double frac, u64 target, int slack_shift) {
    BlockScratch &s = block_scratch();
    uint32_t *hist = wide_smem().hist;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t q[W_PER] = {0, 0, 0, 0};
    if ((int)threadIdx.x < W_BINS / W_PER) {
#pragma unroll 4
        for (int r = 0; r < tm.size; ++r) {
            const uint4 h = *((const uint4 *)tm.at(hist, r) + threadIdx.x);
            q[0] += h.x; q[1] += h.y; q[2] += h.z; q[3] += h.w;
        }
    }
    u64 v[W_PER], local = 0;
    uint32_t cnt = 0;
#pragma unroll
    for (int j = 0; j < W_PER; ++j) {
        const uint32_t code = base + ((uint32_t)(threadIdx.x * W_PER + j) << shift);
        v[j] = by_count ? (u64)((q[j] + 4095u) >> 12) : mass_of_bin(q[j], (code - F_ZERO) >> 16);
        local += v[j];
        q[j] = (q[j] + 2039u) / 2040u;                   // upper bound of the bin's count (a member adds 2047 or more)
        cnt += q[j];
    }
    u64 inc = local;
    uint32_t cinc = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const u64 t = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        const uint32_t tc = __shfl_up_sync(0xFFFFFFFFu, cinc, o);
        if (lane >= o) { inc += t; cinc += tc; }
    }
    if (lane == 31) { s.red[wid] = inc; s.r32a[wid] = cinc; }
    if (threadIdx.x == 0) { s.found_digit = 0xFFFFFFFFu; s.found_cnt = 0xFFFFFFFFu; }
    __syncthreads();
    const u64 wt = lane < NWARPS ? s.red[lane] : 0ull;
    const uint32_t wc = lane < NWARPS ? s.r32a[lane] : 0u;
    const u64 tot = warp_total(wt);
    u64 run = warp_total(lane < wid ? wt : 0ull) + inc - local;
    uint32_t crun = __reduce_add_sync(0xFFFFFFFFu, lane < wid ? wc : 0u) + cinc - cnt;
    if (frac > 0.0) target = (u64)(frac * (double)tot);
    const u64 slack = by_count ? (u64)slack_shift : (tot >> slack_shift) + W_BINS;
    u64 t_lo = target > slack ? target - slack : 1, t_hi = target + slack;
    if (t_hi > tot) t_hi = tot;
    if (t_lo < 1) t_lo = 1;
    if (t_lo > t_hi) t_lo = t_hi;
#pragma unroll
    for (int j = 0; j < W_PER; ++j) {
        const u64 nx = run + v[j];
        if (run < t_lo && t_lo <= nx) { s.found_digit = threadIdx.x * W_PER + j; s.found_above = run; s.list_cnt = crun; }
        if (run < t_hi && t_hi <= nx) { s.found_cnt = threadIdx.x * W_PER + j; s.cand_cnt = crun + q[j]; }
        run = nx; crun += q[j];
    }
    __syncthreads();
    const uint32_t a = s.found_digit, b2 = s.found_cnt;
    Window w;
    w.found = tot > 0 && a != 0xFFFFFFFFu && b2 != 0xFFFFFFFFu;
    w.lo = base + (a << shift); w.hi = base + (b2 << shift) + ((1u << shift) - 1u); w.id_lo = 0; w.id_hi = 0xFFFFFFFFu;
    w.before = s.found_above; w.most = s.cand_cnt - s.list_cnt; w.ahead_most = s.list_cnt;
    __syncthreads();
    return w;
}
template <int DT, bool FLOOR>
__device__ __forceinline__ void window_mass_pass(const SmemSlice<DT> &src, float invT, float zmax, float zfloor, uint32_t lo, int shift, u64 &ahead) {
    u64 all;
    mass_pass<DT, INSIDE_WINDOW, FLOOR>(src, invT, zmax, zfloor, lo, shift, ahead, all);
}
template <int DT, bool FLOOR>
__device__ __forceinline__ void window_mass_pass(const RowSlice<DT> &, float invT, float zmax, float zfloor, uint32_t lo, int shift, u64 &ahead) {
    ahead = solo_mass_pass<DT, INSIDE_WINDOW, FLOOR>(invT, zmax, zfloor, lo, shift).a;
}
constexpr int TIE_SHIFT = 9;      // ids per bin when equal scores are told apart by them: 512 (2^19 ids at most: 1024 bins)
// The elements of a few codes, counted in bins of their ids (4096 each, the unit of find_window's counts),
// their smallest and largest order key, and the exact mass of all that are ahead of them.
template <int DT, class SRC>
__device__ __noinline__ void tie_pass(SRC src, float invT, float zmax, float zfloor, uint32_t lo, uint32_t hi, u64 &ahead, uint32_t &kmin, uint32_t &kmax) {
    typedef Elem<DT> E;
    const uint32_t hist = smem_u32(wide_smem().hist);
    MassSum S;
    uint32_t mn = 0xFFFFFFFFu, mx = 0;
    auto see = [&](int i, float z) {
        const float t2 = log2_mass(z, zmax);
        const uint32_t f = code_of(t2);
        if (!(z >= zfloor)) return;
        S.add(f < lo ? ex2_ftz(t2) : 0.0f);
        if (f >= lo && f <= hi) {
            const uint32_t k = key_of(z);
            mn = k < mn ? k : mn; mx = k > mx ? k : mx;
            hist_add_if(hist, (uint32_t)i >> TIE_SHIFT, 4096u);
        }
    };
    src.vectors([&](const uint4 &q, int i0) {
#pragma unroll
        for (int j = 0; j < E::PER_VEC; ++j) see(i0 + j, __fmul_rn(E::get(q, j), invT));
    });
    src.extras([&](int i, float z) { see(i, z); });
    ahead = S.total(); kmin = mn; kmax = mx;
}
// Narrows a window until no more than `cap` elements can be in it (or the codes run out).  The pass over
// the elements also gives the exact mass ahead of the window, so that the histogram's rounding counts
// only inside it: without that a cut far down a long tail (top-p 0.999) could not be told apart from
// thousands of tail elements.  `target`: an exact mass in 2^-40 units, or a count.
template <int DT, bool FLOOR, class SRC, class TEAM>
__device__ __noinline__ bool narrow_window(SRC src, TEAM tm, float invT, float zmax, float zfloor, bool by_count, u64 target,
                                           uint32_t cap, Window *wp) {
    BlockScratch &s = block_scratch();
    Window w = *wp;
    const uint32_t ahead_most = w.ahead_most;
    uint32_t *hist = wide_smem().hist;
    const int lane = threadIdx.x & 31;
    bool try_ties = !by_count;
#pragma unroll 1
    for (int it = 0; it < 6 && w.most > cap; ++it) {
        const uint32_t width = w.hi - w.lo + 1;
        int shift = 0;
        while (((width - 1) >> shift) >= (uint32_t)W_BINS) ++shift;
        const bool ties = try_ties && width <= 16u;
        if (!ties && width == 1u) return false;
        tm.sync();                                       // everybody has read the histograms
        for (int i = threadIdx.x; i < W_BINS; i += NT) hist[i] = 0;
        __syncthreads();
        if (ties) {
            // Thousands of equal scores at the cut (16-bit logits far from zero: the bulk of a vocabulary falls
            // on a few hundred values).  They all weigh the same, so the cut among them is a count, and they
            // are in order of their ids: the window becomes a range of ids.
            try_ties = width > 1u;                       // (once more if they turn out not to be equal)
            u64 ahead;
            uint32_t kmin, kmax;
            tie_pass<DT>(src, invT, zmax, zfloor, w.lo, w.hi, ahead, kmin, kmax);
            ahead = block_sum_u64(ahead);
            kmax = (uint32_t)block_max_u64(kmax);
            kmin = ~(uint32_t)block_max_u64(~kmin);
            if ((int)threadIdx.x < tm.size) {
                const int r = (int)threadIdx.x;
                *tm.at(&tm.x->ahead[tm.rank], r) = ahead; *tm.at(&tm.x->kmax[tm.rank], r) = kmax; *tm.at(&tm.x->tau[tm.rank], r) = ~kmin;
            }
            tm.sync();
            const bool in = lane < tm.size;
            ahead = warp_total(in ? tm.x->ahead[lane] : 0ull);
            kmax = __reduce_max_sync(0xFFFFFFFFu, in ? tm.x->kmax[lane] : 0u);
            kmin = ~__reduce_max_sync(0xFFFFFFFFu, in ? tm.x->tau[lane] : 0u);
            const u64 each = __float2ull_rn(ex2_ftz(log2_mass(unkey(kmax), zmax)) * FX_SCALE);
            if (each == 0) return false;
            if (kmin == kmax) {
                const u64 rest = target > ahead ? target - ahead : 1ull;
                const Window t = find_window(tm, true, 0u, TIE_SHIFT, 0.0, (rest + each - 1) / each, 1);
                if (!t.found) return false;
                w.lo = w.hi = code_of(log2_mass(unkey(kmax), zmax));
                w.id_lo = t.lo; w.id_hi = t.hi; w.most = t.most;
                break;
            }
            if (width == 1u) return false;
            tm.sync();
            for (int i = threadIdx.x; i < W_BINS; i += NT) hist[i] = 0;
            __syncthreads();
        }
        u64 ahead;
        window_mass_pass<DT, FLOOR>(src, invT, zmax, zfloor, w.lo, shift, ahead);
        ahead = block_sum_u64(ahead);
        if ((int)threadIdx.x < tm.size) *tm.at(&tm.x->ahead[tm.rank], (int)threadIdx.x) = ahead;
        tm.sync();
        ahead = warp_total(lane < tm.size ? tm.x->ahead[lane] : 0ull);
        const u64 before = w.before;
        const u64 rest = by_count ? target - before : (target > ahead ? target - ahead : 1ull);
        w = find_window(tm, by_count, w.lo, shift, 0.0, rest, by_count ? 0 : 11);
        if (!w.found) return false;
        w.before += before;                              // (a count; by mass the next level measures it anew)
    }
    w.ahead_most = ahead_most;
    *wp = w;
    return w.most <= cap;
}

// ------------------------------------------------------------------ the race

// What the generator's first two rounds leave that does not depend on the token (two of their four products), and
// the keys of the third.
__device__ __forceinline__ PhiloxRow philox_row(uint64_t seed, uint32_t R, uint64_t step) {
    PhiloxRow r;
    const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    const uint64_t p1 = (uint64_t)(uint32_t)step * 0xCD9E8D57u;
    const uint64_t p0 = (uint64_t)((uint32_t)(p1 >> 32) ^ R ^ k0) * 0xD2511F53u;
    r.x0 = (uint32_t)p1 ^ (k0 + 0x9E3779B9u); r.x1 = (uint32_t)(step >> 32) ^ k1;
    r.x2 = (uint32_t)(p0 >> 32) ^ (k1 + 0xBB67AE85u); r.x3 = (uint32_t)p0;
    r.k0 = k0 + 2u * 0x9E3779B9u; r.k1 = k1 + 2u * 0xBB67AE85u;
    return r;
}
// N blocks of the generator at once share its key schedule; each product is one wide multiplication, and those are
// what the race is bound by (a quarter of the rate of other instructions: 18 a block, 5 cycles each measured).
template <int N>
__device__ __forceinline__ void philox_blocks(const PhiloxRow &r, uint32_t block, uint32_t (&w)[4 * N]) {
    uint32_t k0 = r.k0, k1 = r.k1;
    uint32_t c0[N], c1[N], c2[N], c3[N];
#pragma unroll
    for (int n = 0; n < N; ++n) {
        const uint64_t p0 = (uint64_t)(block + n) * 0xD2511F53u, p1 = (uint64_t)((uint32_t)(p0 >> 32) ^ r.x1) * 0xCD9E8D57u;
        c0[n] = (uint32_t)(p1 >> 32) ^ r.x0; c1[n] = (uint32_t)p1; c2[n] = (uint32_t)p0 ^ r.x2; c3[n] = r.x3;
    }
#pragma unroll
    for (int i = 2; i < 10; ++i) {
#pragma unroll
        for (int n = 0; n < N; ++n) {
            const uint64_t p0 = (uint64_t)c0[n] * 0xD2511F53u, p1 = (uint64_t)c2[n] * 0xCD9E8D57u;
            c0[n] = (uint32_t)(p1 >> 32) ^ c1[n] ^ k0; c1[n] = (uint32_t)p1;
            c2[n] = (uint32_t)(p0 >> 32) ^ c3[n] ^ k1; c3[n] = (uint32_t)p0;
        }
        k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
    }
#pragma unroll
    for (int n = 0; n < N; ++n) { w[4 * n] = c0[n]; w[4 * n + 1] = c1[n]; w[4 * n + 2] = c2[n]; w[4 * n + 3] = c3[n]; }
}

// The best race score of this CTA so far is shared by its threads (order code in s.runmax).  An
// element can only beat it if E < exp(d - best), and E = -log1p(-v) >= v: so a compare of the uniform
// v with e * exp(-best) decides almost every element without a logarithm.
struct Racer {
    float K;              // exp(-best) with a margin for the rounding of e
    uint32_t seen;        // order code K was computed from
    u64 G;                // this thread's best: order code of the score, ~id
    float z;              // and its z
    __device__ __forceinline__ void start(float K0 = 3.0e34f) { K = K0; seen = 0; G = 0; z = 0.0f; }
    __device__ __forceinline__ void refresh(const uint32_t *best) {
        const uint32_t now = *(const volatile uint32_t *)best;
        if (now != seen) { seen = now; K = fminf(1.0001f * ex2_ftz(-unkey(now) * 1.4426950408889634f), K); }
    }
    __device__ __forceinline__ void take(uint32_t *best, int i, float z_, float g) {
        const u64 g64 = ((u64)orderable_f32(g) << 32) | (uint32_t)(~(uint32_t)i);
        if (g64 > G) {
            G = g64; z = z_;
            if ((uint32_t)(g64 >> 32) > *(volatile uint32_t *)best) atomicMax(best, (uint32_t)(g64 >> 32));
        }
    }
    // no larger word lets an element of mass e win
    __device__ __forceinline__ uint32_t word_bound(float e) const { return __float2uint_ru(e * K * 4294967296.0f); }
};
__device__ __forceinline__ float unit_above(uint32_t w) { return __uint_as_float((w >> 9) | 0x3F800000u); }      // 1 + (v rounded down)
constexpr float RACE_LUCK = 24.5f;    // exp(3.2): the winner of a row of mass S has a score above ln S - 3.2 (ln S - ln E) but for 2e-11 of all rows
__device__ __noinline__ float nle_once(uint32_t w) { return neg_log_exp1_fast(w); }      // (where it is rare: one copy of the code)

__device__ __forceinline__ float race_bound(uint32_t best) {      // Racer::K of a best score's order code
    return best ? fminf(1.0001f * ex2_ftz(-unkey(best) * 1.4426950408889634f), 3.0e34f) : 3.0e34f;
}
__device__ __forceinline__ void list_append(u64 *list, int cap, uint32_t *cnt, float z, int i) {
    const uint32_t slot = atomicAdd(cnt, 1u);
    if (slot < (uint32_t)cap) list[slot] = comp_of(key_of(z), i);
}

// Mass and race element by element in one pass: of the whole row (no cut), or (CUT, arguments in s.fa) of
// the elements kept for sure where those are a good part of the row, the window's going to the list.
// OFF: id of a vector's first element modulo 4 (the generator's blocks are 4 ids).
// What decides is the smallest of a vector's words against the bound of its largest mass: 9 wide multiplications per
// 2 elements, 8 instructions an element for its mass, and little else.
template <int DT, int OFF, bool CUT, class SRC>
__device__ __forceinline__ void race_all(const SRC &src, BlockScratch &s, Partial &p) {
    typedef Elem<DT> E;
    constexpr int PV = E::PER_VEC, NB = PV / 4 + (OFF ? 1 : 0);
    uint32_t *best = &s.runmax;
    const float invT = s.fa.invT, zmax = s.fa.zmax, minus0 = minus_zero(invT);
    const uint32_t sure = CUT ? s.fa.sure : 0u, win_hi = CUT ? s.fa.win_hi : 0u;
    MassSum S;
    uint32_t n = 0;
    Racer rc;
    rc.start(RACE_LUCK);
    const PhiloxRow pr = s.race.philox;
    // an element by itself
    auto race_one = [&](int i, float z, float e) {
        uint32_t w[4];
        philox_blocks<1>(pr, (uint32_t)i >> 2, w);
        const uint32_t x = (i & 3) == 0 ? w[0] : (i & 3) == 1 ? w[1] : (i & 3) == 2 ? w[2] : w[3];
        if (e > 0.0f && x <= rc.word_bound(e)) rc.take(best, i, z, __fsub_rn(z, zmax) + nle_once(x));
    };
    // an element at the edge: in the window, or an equal of its first code with a lower id
    auto edge = [&](int i, float z, float t2, uint32_t f) {
        const FinalArgs &fa = s.fa;
        if (!(z >= fa.zfloor)) return;
        if (f == sure && (uint32_t)i < fa.id_lo) { const float e = ex2_ftz(t2); S.add(e); ++n; race_one(i, z, e); }
        else if (f < win_hi || (f == win_hi && (uint32_t)i <= fa.id_hi)) list_append(fa.list, fa.list_cap, &s.list_cnt, z, i);
    };
    src.template vectors<1>([&](const uint4 &q, int i0) {
        float e[PV], top = 0.0f;
        uint32_t at_edge = 0;
#pragma unroll
        for (int j = 0; j < PV; j += 2) {
            const float2 t2 = log2_mass2(scores_of(E::get(q, j), E::get(q, j + 1), invT, minus0), zmax);
            e[j] = ex2_ftz(t2.x); e[j + 1] = ex2_ftz(t2.y);
            if constexpr (CUT) {
                const uint2 f = code_of2(t2);
                at_edge |= (uint32_t)(f.x >= sure && f.x <= win_hi) << j | (uint32_t)(f.y >= sure && f.y <= win_hi) << (j + 1);
                e[j] = f.x < sure ? e[j] : 0.0f; e[j + 1] = f.y < sure ? e[j + 1] : 0.0f;
                n += (f.x < sure) + (f.y < sure);
            }
            S.add2(make_float2(e[j], e[j + 1]));
            top = fmaxf(top, fmaxf(e[j], e[j + 1]));
        }
        if constexpr (CUT) {
            while (at_edge) {
                const int x = __ffs(at_edge) - 1;
                at_edge &= at_edge - 1;
                const float z = __fmul_rn(pick_element<DT>(q, x), invT), t2 = log2_mass(z, zmax);
                edge(i0 + x, z, t2, code_of(t2));
            }
            __syncwarp();
        }
        rc.refresh(best);
        if (!__any_sync(0xFFFFFFFFu, top * rc.K >= 1.16e-10f)) return;      // v is at least 2^-33
        uint32_t w[4 * NB], least = 0xFFFFFFFFu;
        philox_blocks<NB>(pr, (uint32_t)(i0 >> 2), w);
#pragma unroll
        for (int j = 0; j < PV; ++j) least = min(least, w[OFF + j]);
        if (!__any_sync(0xFFFFFFFFu, least <= rc.word_bound(top))) return;
        uint32_t hits = 0;
#pragma unroll
        for (int j = 0; j < PV; ++j) hits |= (uint32_t)(e[j] > 0.0f && w[OFF + j] <= rc.word_bound(e[j])) << j;
        // rare after the first vectors: the exact score, one element per lane at a time, the bound renewed in between
        while (__any_sync(0xFFFFFFFFu, hits != 0)) {
            if (hits) {
                const int x = __ffs(hits) - 1;
                hits &= hits - 1;
                uint32_t wx = w[OFF];
#pragma unroll
                for (int j = 1; j < PV; ++j) wx = x == j ? w[OFF + j] : wx;
                const float z = __fmul_rn(pick_element<DT>(q, x), invT), d = __fsub_rn(z, zmax);
                if (wx <= rc.word_bound(ex2_ftz(d * 1.4426950408889634f))) rc.take(best, i0 + x, z, d + nle_once(wx));
            }
            __syncwarp();
            rc.refresh(best);
        }
    });
    src.extras([&](int i, float z) {
        const float d = __fsub_rn(z, zmax);
        if (!(d > -3.0e38f)) return;
        const float t2 = log2_mass(z, zmax);
        const uint32_t f = code_of(t2);
        bool in = true;
        if constexpr (CUT) in = f < sure;
        rc.refresh(best);
        if (in) { const float e = ex2_ftz(t2); S.add(e); ++n; race_one(i, z, e); }
        else if (f <= win_hi) edge(i, z, t2, f);        // (CUT only)
    });
    p.M = S.total(); p.n = CUT ? n : 0; p.G = rc.G; p.z = rc.z;
}

// An element of mass e can only beat a score g if E < e exp(-g), and E = -log1p(-v) >= v: so comparing v / e with
// K = exp(-g) decides almost every element without a logarithm.  Nor does K take one: an element's own E / e is an upper
// bound of it, and E <= v (1 + v) up to v = 1/2.  The smallest K of a CTA so far is shared by its threads (s.race.bound,
// the float's bits).  It starts from a score that the winner of a row of mass S reaches but for 2e-11 of all rows, ln S - 3.2 (the winner's
// score is ln S - ln E); a row in which none did goes to the general path.
// (With K from the exact scores alone batches of vectors stopped for several of them, a few hundred cycles each, while the first
// batches of all warps were under way: 32 top-p rows of 128256 spent 6.0 us in the last pass, 5.4 so.)
constexpr uint32_t NO_BOUND = 0x7F7FFFFFu;
__device__ __forceinline__ float unit_below(uint32_t w) { return __uint_as_float((w >> 9) | 0x3F800000u) - 1.0f; }      // v rounded down to 2^-23
// an upper bound of E / e from v (rounded down) and 1 / e
__device__ __forceinline__ float race_cap(float v, float inv_e) {
    const float up = v + 1.1920929e-7f;
    return v < 0.5f ? 1.0002f * (__fmaf_rn(up, up, up) * inv_e) : 3.0e38f;
}
// What the race needs across the vectors of a pass: the generator's row and each thread's best element (order code of the score, ~id, and its z) in
// registers where there are some to spare (IN_REGS: 128 per thread), else in shared memory, the best by warps where block_partial takes it from -
// held across the passes' loops they were spilled, and what is spilled comes back from the L2.  (By the other kernel's way
// 64 rows of 152064 without a cut took 24.5 us instead of 21.9.)
// LISTED: the reference is not the row's maximum.  A score is z - maximum + (-ln E), rounded, and an equal one by another reference may be
// rounded otherwise, so the elements that pass the bound are listed (their score and id) and raced when the maximum is known.  The bound
// has a margin of 2e-4 in the score: rounding does not reach it where the winner is no more than 88 above the reference, and
// above that all elements pass, their mass being infinite (and the list, mostly, runs over).
__device__ __forceinline__ u64 *race_list() { extern __shared__ __align__(128) unsigned char smem[]; return ((CountedSegs *)(smem + row_segments<ALBIREO_BF16>()))->mass; }
enum RaceBest { IN_REGS, IN_SHARED, LISTED };
constexpr int RACE_LIST = NT;         // entries, where the segments' masses would lie
template <RaceBest BEST>
struct CountedRacer {
    static constexpr bool REGS = BEST == IN_REGS;
    BlockScratch &s;
    PhiloxRow kept;
    u64 G;
    float z;
    __device__ __forceinline__ explicit CountedRacer(BlockScratch &s_) : s(s_), G(0), z(0.0f) {
        if constexpr (BEST == LISTED) return;
        if constexpr (REGS) { kept = s.race.philox; return; }
        if ((threadIdx.x & 31) == 0) { s.red2[threadIdx.x >> 5] = 0; s.r32b[threadIdx.x >> 5] = 0; }
        __syncwarp();
    }
    __device__ __forceinline__ PhiloxRow row() const {
        if constexpr (REGS) return kept;
        const volatile PhiloxRow &v = s.race.philox;
        PhiloxRow r;
        r.x0 = v.x0; r.x1 = v.x1; r.x2 = v.x2; r.x3 = v.x3; r.k0 = v.k0; r.k1 = v.k1;
        return r;
    }
    __device__ __forceinline__ float K() const { return __uint_as_float(*(const volatile uint32_t *)&s.race.bound); }
    // no larger word lets an element of mass e win
    __device__ __forceinline__ static uint32_t word_bound(float e, float K) { return __float2uint_ru(e * K * 4294967296.0f); }
    // by whole warps: the lanes' bounds; gives the smallest of all.  (Never 0: masses relative to a reference far below the maximum can be infinite.)
    __device__ __forceinline__ float tighten(float cap) const {
        const uint32_t least = __reduce_min_sync(0xFFFFFFFFu, __float_as_uint(fminf(fmaxf(cap, 1e-37f), 3.0e38f)));
        const float now = K();
        if (__uint_as_float(least) < now && (threadIdx.x & 31) == 0) atomicMin(&s.race.bound, least);
        return fminf(__uint_as_float(least), now);
    }
    // by whole warps: the lanes' best elements (0: none)
    __device__ __forceinline__ void take(u64 g, float zg) {
        if constexpr (REGS) { if (g > G) { G = g; z = zg; } return; }
        if (!__any_sync(0xFFFFFFFFu, g != 0)) return;
        warp_best(g, zg);
        const int wid = threadIdx.x >> 5;
        if ((threadIdx.x & 31) == 0 && g > s.red2[wid]) { s.red2[wid] = g; s.r32b[wid] = __float_as_uint(zg); }
        __syncwarp();
    }
    __device__ __forceinline__ void list(int i, float z_) {
        const uint32_t at = atomicAdd(&s.cand_cnt, 1u);
        if (at < (uint32_t)RACE_LIST) race_list()[at] = comp_of(key_of(z_), i);
    }
    __device__ __forceinline__ static u64 code_of_score(float g, int i) { return ((u64)orderable_f32(g) << 32) | (uint32_t)(~(uint32_t)i); }
    // One element per lane by itself, by whole warps: of log2 mass t2 and d = z - reference (`in`: if it is there at all).
    __device__ __forceinline__ void race(bool in, int i, float zi, float d, float t2) {
        uint32_t w[4];
        philox_blocks<1>(row(), (uint32_t)i >> 2, w);
        const uint32_t x = (i & 3) == 0 ? w[0] : (i & 3) == 1 ? w[1] : (i & 3) == 2 ? w[2] : w[3];
        const float v = unit_below(x), inv_e = in ? ex2_ftz(-t2) : INFINITY;
        if (!__any_sync(0xFFFFFFFFu, v * inv_e <= K())) return;                         // (0 x infinity is no hit)
        const float least = tighten(in ? race_cap(v, inv_e) : 3.0e38f);
        if constexpr (BEST == LISTED) {
            if (v * inv_e <= least) list(i, zi);
            __syncwarp();
        } else take(v * inv_e <= least ? code_of_score(d + nle_once(x), i) : 0ull, zi);
    }
    // The elements of a vector, their words w[OFF ..], by whole warps: `inv_mass` of element j gives 1 / e, infinity for one that does not take part.
    template <int DT, int OFF, int N, class F>
    __device__ __forceinline__ void race_hits(const uint32_t (&w)[N], const uint4 &q, int i0, float invT, float zref, F &&inv_mass) {
        constexpr int PV = Elem<DT>::PER_VEC;
        float cap = 3.0e38f;
#pragma unroll
        for (int j = 0; j < PV; ++j) cap = fminf(cap, race_cap(unit_below(w[OFF + j]), inv_mass(j)));
        const float K = tighten(cap);
        uint32_t hits = 0;
#pragma unroll
        for (int j = 0; j < PV; ++j) hits |= (uint32_t)(unit_below(w[OFF + j]) * inv_mass(j) <= K) << j;
        u64 best = 0;
        float zbest = 0.0f;
        while (hits) {
            const int x = __ffs(hits) - 1;
            hits &= hits - 1;
            const float zx = __fmul_rn(pick_element<DT>(q, x), invT);
            if constexpr (BEST == LISTED) { list(i0 + x, zx); continue; }
            uint32_t wx = w[OFF];
#pragma unroll
            for (int j = 1; j < PV; ++j) wx = x == j ? w[OFF + j] : wx;
            const u64 g = code_of_score(__fsub_rn(zx, zref) + nle_once(wx), i0 + x);
            if (g > best) { best = g; zbest = zx; }
        }
        __syncwarp();
        if constexpr (BEST != LISTED) take(best, zbest);
    }
    __device__ __forceinline__ void finish(Partial &p) const {
        if constexpr (REGS) { p.G = G; p.z = z; return; }
        __syncwarp();
        const bool first = (threadIdx.x & 31) == 0;
        p.G = first ? s.red2[threadIdx.x >> 5] : 0ull; p.z = first ? __uint_as_float(s.r32b[threadIdx.x >> 5]) : 0.0f;
        __syncwarp();
    }
};

// The same for the kernel with 64 registers per thread, what the race needs in shared memory. (With the row's words and the bound
// held across the loop 68 to 104 bytes were spilled, and what is spilled comes back from the L2.)
template <int DT, int OFF, bool CUT, class SRC>
__device__ __forceinline__ void race_all_shared(const SRC &src, BlockScratch &s, Partial &p) {
    typedef Elem<DT> E;
    constexpr int PV = E::PER_VEC, NB = PV / 4 + (OFF ? 1 : 0);
    const float invT = s.fa.invT, zmax = s.fa.zmax, minus0 = minus_zero(invT);
    const uint32_t sure = CUT ? s.fa.sure : 0u, win_hi = CUT ? s.fa.win_hi : 0u;
    MassSum S;
    uint32_t n = 0;
    CountedRacer<IN_SHARED> rc(s);
    // an element at the edge: in the window, or (true) an equal of its first code with a lower id
    auto edge = [&](int i, float z, uint32_t f) -> bool {
        const FinalArgs &fa = s.fa;
        if (!(z >= fa.zfloor)) return false;
        if (f == sure && (uint32_t)i < fa.id_lo) return true;
        if (f < win_hi || (f == win_hi && (uint32_t)i <= fa.id_hi)) list_append(fa.list, fa.list_cap, &s.list_cnt, z, i);
        return false;
    };
    src.template vectors<1>([&](const uint4 &q, int i0) {
        float e[PV], top = 0.0f;
        uint32_t at_edge = 0;
#pragma unroll
        for (int j = 0; j < PV; j += 2) {
            const float2 t2 = log2_mass2(scores_of(E::get(q, j), E::get(q, j + 1), invT, minus0), zmax);
            e[j] = ex2_ftz(t2.x); e[j + 1] = ex2_ftz(t2.y);
            if constexpr (CUT) {
                const uint2 f = code_of2(t2);
                at_edge |= (uint32_t)(f.x >= sure && f.x <= win_hi) << j | (uint32_t)(f.y >= sure && f.y <= win_hi) << (j + 1);
                e[j] = f.x < sure ? e[j] : 0.0f; e[j + 1] = f.y < sure ? e[j + 1] : 0.0f;
                n += (f.x < sure) + (f.y < sure);
            }
            S.add2(make_float2(e[j], e[j + 1]));
            top = fmaxf(top, fmaxf(e[j], e[j + 1]));
        }
        if constexpr (CUT) {
            // (equals kept for sure are put back among the kept ones)
            while (at_edge) {
                const int x = __ffs(at_edge) - 1;
                at_edge &= at_edge - 1;
                const float z = __fmul_rn(pick_element<DT>(q, x), invT), t2 = log2_mass(z, zmax);
                if (edge(i0 + x, z, code_of(t2))) {
                    const float ex = ex2_ftz(t2);
                    S.add(ex); ++n;
                    top = fmaxf(top, ex);
#pragma unroll
                    for (int j = 0; j < PV; ++j) e[j] = x == j ? ex : e[j];
                }
            }
            __syncwarp();
        }
        const float K = rc.K();
        if (!__any_sync(0xFFFFFFFFu, top * K >= 1.16e-10f)) return;      // v is at least 2^-33
        uint32_t w[4 * NB], least = 0xFFFFFFFFu;
        philox_blocks<NB>(rc.row(), (uint32_t)(i0 >> 2), w);
#pragma unroll
        for (int j = 0; j < PV; ++j) least = min(least, w[OFF + j]);
        if (!__any_sync(0xFFFFFFFFu, least <= rc.word_bound(top, K))) return;
        rc.template race_hits<DT, OFF>(w, q, i0, invT, zmax, [&](int j) { return e[j] > 0.0f ? __fdividef(1.0f, e[j]) : INFINITY; });
    });
    src.extras([&](int i, float z) {
        const float d = __fsub_rn(z, zmax), t2 = log2_mass(z, zmax);
        bool in = d > -3.0e38f;
        if constexpr (CUT) {
            const uint32_t f = code_of(t2);
            if (in && f >= sure) in = f <= win_hi && edge(i, z, f);
        }
        if (in) { S.add(ex2_ftz(t2)); ++n; }
        rc.race(in, i, z, d, t2);
    });
    p.M = S.total(); p.n = CUT ? n : 0;
    rc.finish(p);
}

// Mass, number and race of the elements kept for sure, and the lists (arguments in s.fa).  Kept elements
// are scattered over the lanes, and the race term is long: each warp collects them in a queue and works
// off 32 at a time.  Without registers to spare, what has been summed up stays in shared memory, a slot per
// warp: kept in registers across the scan it was spilled, and local memory of 1024 threads does not fit what the shared memory
// leaves of the L1 (60 us for a row of 238016 with 64 kept elements, now a third of that).
template <int DT, class SRC>
__device__ __forceinline__ void final_pass(const SRC &src, BlockScratch &s, Partial &p) {
    typedef Elem<DT> E;
    const WideSmem ws = wide_smem();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    u64 *queue = ws.queue + wid * 64;
    int qn = 0;                                          // the same in every lane
    constexpr bool REGS = SRC::SPARE_REGISTERS;
    u64 S = 0;
    uint32_t n_kept = 0;
    Racer rc;
    rc.start();
    if (!REGS && lane == 0) { s.red[wid] = 0; s.red2[wid] = 0; s.r32a[wid] = 0; s.r32b[wid] = 0; }
    __syncwarp();
    auto work = [&](int keep) {                          // works the queue off until no more than `keep` are left
        const FinalArgs &fa = s.fa;
#pragma unroll 1
        while (qn > keep) {
            const int cnt = qn < 32 ? qn : 32;
            qn -= cnt;
            __syncwarp();
            float K;
            if constexpr (REGS) { rc.refresh(&s.runmax); K = rc.K; }
            else K = race_bound(*(volatile uint32_t *)&s.runmax);
            int i = 0; float z = -INFINITY;
            if (lane < cnt) { const u64 en = queue[qn + lane]; i = (int)(uint32_t)en; z = __uint_as_float((uint32_t)(en >> 32)); }
            const float t2 = log2_mass(z, fa.zmax), e = ex2_ftz(t2);
            const uint32_t f = code_of(t2);
            const bool alive = z >= fa.zfloor, sure = alive && (f < fa.sure || (f == fa.sure && (uint32_t)i < fa.id_lo));
            if (alive && !sure && (f < fa.win_hi || (f == fa.win_hi && (uint32_t)i <= fa.id_hi))) list_append(fa.list, fa.list_cap, &s.list_cnt, z, i);
            if (alive && f <= fa.top_hi) list_append(ws.top, W_LIST, &s.cand_cnt, z, i);
            uint32_t w = 0;
            bool may = sure;
            if (sure && !fa.exp1_row) {
                w = race_word(fa.seed, fa.R, fa.step, i);
                may = unit_above(w) <= __fmaf_rn(e, K, 1.0f);
            }
            if constexpr (REGS) {
                if (sure) { S += __float2ull_rn(e * FX_SCALE); ++n_kept; }
                if (may) rc.take(&s.runmax, i, z, __fsub_rn(z, fa.zmax) + (fa.exp1_row ? -logf(__ldg(fa.exp1_row + i)) : nle_once(w)));
                __syncwarp();
                continue;
            }
            const u64 mass = warp_total(sure ? __float2ull_rn(e * FX_SCALE) : 0ull);
            const uint32_t n = (uint32_t)__popc(__ballot_sync(0xFFFFFFFFu, sure));
            u64 G = 0;
            if (__any_sync(0xFFFFFFFFu, may)) {
                if (may) {
                    const float g = __fsub_rn(z, fa.zmax) + (fa.exp1_row ? -logf(__ldg(fa.exp1_row + i)) : nle_once(w));
                    G = ((u64)orderable_f32(g) << 32) | (uint32_t)(~(uint32_t)i);
                }
                __syncwarp();
                warp_best(G, z);
            }
            if (lane == 0) {
                s.red[wid] += mass; s.r32a[wid] += n;
                if (G > s.red2[wid]) {
                    s.red2[wid] = G; s.r32b[wid] = __float_as_uint(z);
                    if ((uint32_t)(G >> 32) > *(volatile uint32_t *)&s.runmax) atomicMax(&s.runmax, (uint32_t)(G >> 32));
                }
            }
            __syncwarp();
        }
    };
    // Called by whole warps.  Everything about an element but its place in the queue is worked out 32
    // elements at a time.
    auto push = [&](int i, float z, bool in) {
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, in);
        if (in) queue[qn + __popc(m & ((1u << lane) - 1u))] = ((u64)__float_as_uint(z) << 32) | (uint32_t)i;
        qn += __popc(m);
        if (qn >= 32) work(31);
    };
    {
        const uint32_t thr = s.fa.vec_thr;
        const float invT = s.fa.invT;
        src.vectors([&](const uint4 &q, int i0) {
            uint32_t bits = VecTest<DT>::may_pass(q, thr, invT) ? VecTest<DT>::elem_bits(q, thr, invT) : 0u;
            while (__any_sync(0xFFFFFFFFu, bits != 0)) {     // one element per lane at a time
                const int x = __ffs(bits | 0x80000000u) - 1;
                push(i0 + x, __fmul_rn(pick_element<DT>(q, x), invT), bits != 0);
                bits &= bits - 1u;
            }
        }, [&](const uint4 &x, const uint4 &y) { return VecTest<DT>::may_pass(x, thr, invT) || VecTest<DT>::may_pass(y, thr, invT); });
    }
    src.extras([&](int i, float z) { push(i, z, z >= s.fa.zfloor); });
    work(0);
    p.M = S; p.n = n_kept; p.G = rc.G; p.z = rc.z;
    if (!REGS && lane == 0) { p.M = s.red[wid]; p.n = s.r32a[wid]; p.G = s.red2[wid]; p.z = __uint_as_float(s.r32b[wid]); }
    __syncwarp();
}

template <int DT, int OFF, bool CUT>
__device__ __noinline__ Partial solo_race_all() {
    Partial p;
    race_all_shared<DT, OFF, CUT>(RowSlice<DT>(), block_scratch(), p);
    return p;
}
template <int DT>
__device__ __noinline__ Partial solo_final_pass() {
    Partial p;
    final_pass<DT>(RowSlice<DT>(), block_scratch(), p);
    return p;
}
template <int DT, bool FLOOR>
__device__ __forceinline__ void first_mass_pass(const SmemSlice<DT> &src, float invT, float zmax, float zfloor, u64 &S, u64 &S_all) {
    mass_pass<DT, FIRST_LEVEL, FLOOR>(src, invT, zmax, zfloor, F_ZERO, W_SHIFT, S, S_all);
}
template <int DT, bool FLOOR>
__device__ __forceinline__ void first_mass_pass(const RowSlice<DT> &, float invT, float zmax, float zfloor, u64 &S, u64 &S_all) {
    const PassOut o = solo_mass_pass<DT, FIRST_LEVEL, FLOOR>(invT, zmax, zfloor, F_ZERO, W_SHIFT);
    S = o.a; S_all = o.b;
}
// (out of line in clusters too: code that is fetched only when it runs leaves the other passes' code together. With the races without a
// cut inlined 64 such rows of 152064 took 21.9 us instead of 21.5, 13 mixed rows of 50257 21.4 instead of 21.2.)
template <int DT, int OFF, bool CUT>
__device__ __noinline__ Partial team_race_all(SmemSlice<DT> src) {
    Partial p;
    race_all<DT, OFF, CUT>(src, block_scratch(), p);
    return p;
}
template <int DT, int OFF, bool CUT>
__device__ __forceinline__ void run_race_all(const SmemSlice<DT> &src, BlockScratch &s, Partial &p) { p = team_race_all<DT, OFF, CUT>(src); }
template <int DT, int OFF, bool CUT>
__device__ __forceinline__ void run_race_all(const RowSlice<DT> &, BlockScratch &s, Partial &p) { p = solo_race_all<DT, OFF, CUT>(); }
template <int DT, bool CUT, class SRC>
__device__ __forceinline__ void run_race(const SRC &src, BlockScratch &s, Partial &p) {
    switch (src.first_id() & 3) {
        case 0: run_race_all<DT, 0, CUT>(src, s, p); break;
        case 1: run_race_all<DT, 1, CUT>(src, s, p); break;
        case 2: run_race_all<DT, 2, CUT>(src, s, p); break;
        default: run_race_all<DT, 3, CUT>(src, s, p); break;
    }
}
template <int DT> __device__ __forceinline__ void run_final_pass(const SmemSlice<DT> &src, BlockScratch &s, Partial &p) { final_pass<DT>(src, s, p); }
template <int DT> __device__ __forceinline__ void run_final_pass(const RowSlice<DT> &, BlockScratch &s, Partial &p) { p = solo_final_pass<DT>(); }

// ------------------------------------------------------------------ one wide row

constexpr uint32_t ROW_NOT_DONE = 0x80000000u;      // internal status bit: the general path has to take the row

// the mass that the kept prefix has to reach
__device__ __forceinline__ u64 topp_target(float top_p, u64 S) {
    const double t = ceil((double)top_p * (double)S);
    const u64 target = t <= 1.0 ? 1ull : (u64)t;
    return target > S ? (S < 1 ? 1ull : S) : target;
}

// CTA 0: moves the entries that the others put at the far end of `buf` behind its own n0; returns the number of all
// (more than `cap`, which only +inf or NaN among the logits can bring about: nothing is moved).
__device__ __forceinline__ int close_gap(u64 *buf, int cap, int n0, int nfar) {
    if (nfar == 0 || n0 + nfar > cap) return n0 + nfar;
    u64 keep[W_LIST_ALONE / NT];
#pragma unroll
    for (int q = 0; q < W_LIST_ALONE / NT; ++q) { const int j = threadIdx.x + q * NT; keep[q] = j < nfar ? buf[cap - 1 - j] : 0ull; }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < W_LIST_ALONE / NT; ++q) { const int j = threadIdx.x + q * NT; if (j < nfar && n0 + j < cap) buf[n0 + j] = keep[q]; }
    __syncthreads();
    return n0 + nfar;
}

// Sorts list[0..n) in descending order (a bitonic network over the next power of two, which it returns and
// up to which the list is filled with zeros): 1 to 4 us where counting every entry's rank took 45 at 540.
__device__ __noinline__ int list_sort(u64 *list, int n) {
    int P = 2;
    while (P < n) P <<= 1;
    for (int i = n + (int)threadIdx.x; i < P; i += NT) list[i] = 0ull;
    __syncthreads();
    for (int k = 2; k <= P; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int t = threadIdx.x; t < (P >> 1); t += NT) {
                const int i = ((t & ~(j - 1)) << 1) | (t & (j - 1)), l = i | j;
                const u64 a = list[i], b2 = list[l];
                if ((i & k) == 0 ? a < b2 : a > b2) { list[i] = b2; list[l] = a; }
            }
            __syncthreads();
        }
    }
    return P;
}

__device__ __forceinline__ bool all_keys_are(const u64 *list, int n, uint32_t key) {
    bool same = true;
    for (int i = threadIdx.x; i < n; i += NT) same &= (uint32_t)(list[i] >> 32) == key;
    return same;
}
// The `want`-th lowest id of list[0..n), 1 <= want <= n <= W_LIST_ALONE, the same in every thread: ids counted in bins of 1024, and the entries of one bin by
// their bits.  (16-bit logits far from zero have hundreds of elements at the score of the cut; sorted, 1250 of them took 20 us.)
__device__ __noinline__ uint32_t lowest_ids(const u64 *list, int n, uint32_t want) {
    BlockScratch &s = block_scratch();
    uint32_t *bins = (uint32_t *)wide_smem().queue;      // NT bins, then 32 words of one bin's ids
    static_assert(NT * 1024 >= ALBIREO_MAX_VOCAB && NWARPS * 64 * 8 >= (NT + 32) * 4, "a bin per thread, over the queues");
    bins[threadIdx.x] = 0u;
    if (threadIdx.x < 32) bins[NT + threadIdx.x] = 0u;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += NT) atomicAdd(&bins[(uint32_t)comp_idx(list[i]) >> 10], 1u);
    __syncthreads();
    const uint32_t mine = bins[threadIdx.x];
    uint32_t tot;
    const uint32_t ahead = block_exscan_u32(mine, tot);
    if (ahead < want && want <= ahead + mine) { s.found_digit = threadIdx.x; s.found_cnt = want - ahead; }
    __syncthreads();
    const uint32_t bin = s.found_digit;
    for (int i = threadIdx.x; i < n; i += NT) {
        const uint32_t id = (uint32_t)comp_idx(list[i]);
        if (id >> 10 == bin) atomicOr(&bins[NT + ((id >> 5) & 31u)], 1u << (id & 31u));
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        const uint32_t w = bins[NT + threadIdx.x], c = __popc(w), k = s.found_cnt;
        uint32_t inc = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const uint32_t x = __shfl_up_sync(0xFFFFFFFFu, inc, o); if ((int)threadIdx.x >= o) inc += x; }
        if (inc - c < k && k <= inc) s.list_cnt = (bin << 10) + (threadIdx.x << 5) + __fns(w, 0, (int)(k - (inc - c)));
    }
    __syncthreads();
    return s.list_cnt;
}

// What the passes of a wide row leave behind, apart from each thread's sums and the lists.
struct WideEnd {
    u64 M0; uint32_t n0;                 // mass and number of elements kept for sure that the sums do not contain
    u64 S, S_all;                        // the mass that top-p is a share of, the whole row's
    float zmax;
    uint32_t n_fin;
    bool summed, in_team, all_kept, topp, full;   // the sums contain the whole row's mass; S and S_all are in the team's words; every finite score is kept
    float race_from;                     // a winner's score below this: one that was passed over may be ahead of it (-infinity: none was)
};
constexpr float RACE_FROM = -3.1977f;    // for a race whose bound started from RACE_LUCK: 0.001 - 3.1987 (ln 24.5)
// From there to the result, which is CTA 0's, in its warp 0.
template <class TEAM>
__device__ __forceinline__ RowOut wide_finish_in(TEAM tm, float top_p, uint64_t seed, uint32_t R, Partial p, const WideEnd &w, u64 *list, int list_cap,
                                                 const float *exp1_row, int b, RowOut out) {
    BlockScratch &s = block_scratch();
    const WideSmem ws = wide_smem();
    const int lane = threadIdx.x & 31;
    const bool want_list = s.ga.num_top > 0, topp = w.topp, full = w.full;
    const float zmax = w.zmax;
    block_partial(s, p);                                 // (its barrier also ends the appends)
    const int n_list = (int)s.list_cnt, n_top = (int)s.cand_cnt;
    if (threadIdx.x == 0) {
        const int r = tm.rank;
        *tm.at(&tm.x->M[r], 0) = p.M; *tm.at(&tm.x->n[r], 0) = p.n; *tm.at(&tm.x->G[r], 0) = p.G; *tm.at(&tm.x->z[r], 0) = p.z;
    }
    if (tm.size > 1 && tm.rank != 0 && (topp || want_list)) {
        // the lists' entries go to the far ends of CTA 0's lists (each list's sum is within its capacity)
        if (threadIdx.x == 32) {
            s.found_digit = n_list ? atomicAdd(tm.at(&tm.x->far_list, 0), (uint32_t)n_list) : 0u;
            s.found_cnt = n_top ? atomicAdd(tm.at(&tm.x->far_cand, 0), (uint32_t)n_top) : 0u;
        }
        __syncthreads();
        const int at_list = list_cap - 1 - (int)s.found_digit, at_top = W_LIST - 1 - (int)s.found_cnt;
        u64 *list0 = tm.at(list, 0), *top0 = tm.at(ws.top, 0);
        for (int j = threadIdx.x; j < n_list; j += NT) if (at_list - j >= 0) list0[at_list - j] = list[j];
        for (int j = threadIdx.x; j < n_top; j += NT) if (at_top - j >= 0) top0[at_top - j] = ws.top[j];
    }
    tm.sync();
    if (tm.rank != 0) return out;

    // CTA 0 has everything
    const TeamWords &x = *tm.x;
    const bool in = lane < tm.size;
    p.M = in ? x.M[lane] : 0ull; p.n = in ? x.n[lane] : 0u; p.G = in ? x.G[lane] : 0ull; p.z = in ? x.z[lane] : 0.0f;
    p.over_warp();
    p.M += w.M0; p.n = w.all_kept ? w.n_fin : p.n + w.n0;
    u64 S = w.S, S_all = w.summed ? p.M : w.S_all;
    if (w.in_team) { S = warp_total(in ? x.S[lane] : 0ull); S_all = warp_total(in ? x.S_all[lane] : 0ull); }
    if (topp) {
        const u64 target = topp_target(top_p, S);
        const int L = close_gap(list, list_cap, n_list, (int)x.far_list);
        if (p.M >= target || L < 1 || L > list_cap) { out.status |= ROW_NOT_DONE; return out; }
        auto mass_of = [&](u64 C) { return __float2ull_rn(ex2_ftz(log2_mass(unkey((uint32_t)(C >> 32)), zmax)) * FX_SCALE); };
        Partial k;
        k.M = 0; k.n = 0; k.G = 0; k.z = 0.0f;
        auto keep = [&](u64 C, u64 own) {
            k.M += own; ++k.n;
            const float zq = unkey((uint32_t)(C >> 32));
            const float g = __fsub_rn(zq, zmax) + race_nle(seed, R, s.ga.step, exp1_row, comp_idx(C));
            const u64 gq = ((u64)orderable_f32(g) << 32) | (uint32_t)C;
            if (gq > k.G) { k.G = gq; k.z = zq; }
        };
        // An entry is kept while the mass ahead of it in the order, with the mass kept for sure, is short of
        // the target.  A short list: every entry adds that mass up (masses over the queues, done with by now),
        // one barrier in all; from 192 entries on a sort and a prefix sum are faster (2 us against 3 at 300).
        bool reached;
        if (L <= 192) {
            // (two or four threads share an entry's comparisons where there are more than 64)
            u64 *mass = ws.queue;
            if ((int)threadIdx.x < L) mass[threadIdx.x] = mass_of(list[threadIdx.x]);
            __syncthreads();
            const int sh = L <= 64 ? 0 : L <= 128 ? 2 : 1, j = (int)threadIdx.x >> sh, part = (int)threadIdx.x & ((1 << sh) - 1);
            const u64 C = j < L ? list[j] : 0ull;
            u64 ahead = 0, reach = 0;
            if (j < L) {
#pragma unroll 4
                for (int q = part; q < L; q += 1 << sh) ahead += list[q] > C ? mass[q] : 0ull;
            }
            for (int o = 1; o < 1 << sh; o <<= 1) ahead += __shfl_xor_sync(0xFFFFFFFFu, ahead, o);
            ahead += p.M;
            if (j < L) {
                const u64 own = mass[j];
                reach = ahead + own;
                if (part == 0 && ahead < target) keep(C, own);
            }
            reached = __syncthreads_or(reach >= target) != 0;
        } else if (__syncthreads_and(all_keys_are(list, L, (uint32_t)(list[0] >> 32)))) {
            // elements of one score: so many of the lowest ids are kept as are short of the target
            const u64 each = mass_of(list[0]), want = each ? (target - p.M + each - 1) / each : 0ull;
            reached = want > 0 && want <= (u64)L;
            if (reached) {
                const uint32_t last = lowest_ids(list, L, (uint32_t)want);
                for (int q = threadIdx.x; q < L; q += NT) if ((uint32_t)comp_idx(list[q]) <= last) keep(list[q], each);
            }
            __syncthreads();
        } else {
            const int P = list_sort(list, L), per = (P + NT - 1) / NT, q0 = (int)threadIdx.x * per, q1 = min(L, q0 + per);
            u64 local = 0, tot;
            for (int q = q0; q < q1; ++q) local += mass_of(list[q]);
            u64 run = p.M + block_exscan_u64(local, tot);
            reached = p.M + tot >= target;
#pragma unroll 1
            for (int q = q0; q < q1 && run < target; ++q) {
                const u64 C = list[q], own = mass_of(C);
                run += own;
                keep(C, own);
            }
            __syncthreads();
        }
        if (!reached) { out.status |= ROW_NOT_DONE; return out; }
        block_partial(s, k);
        p.M += k.M; p.n += k.n;
        if (k.G > p.G) { p.G = k.G; p.z = k.z; }
    }
    if (w.race_from > -INFINITY && __syncthreads_or(threadIdx.x == 0 && !(unkey((uint32_t)(p.G >> 32)) >= w.race_from))) { out.status |= ROW_NOT_DONE; return out; }
    double lnS = 0.0;
    if (threadIdx.x < 32) {
        const u64 S_ref = full ? S_all : p.M;
        lnS = log((double)S_ref) - LN2_40;
        const int tok = comp_idx(p.G);
        out.token = tok < 0 ? 0 : tok;                  // (NaN logits: any id in range)
        out.n_keep = (int32_t)p.n;
        out.logprob = (p.n == 1 && !full) ? 0.0f : (float)(((double)p.z - (double)zmax) - lnS);
    }
    if (want_list) {
        if (threadIdx.x == 0) { s.bcast[0] = (u64)__double_as_longlong(lnS); s.found_cnt = p.n; }
        const int n_all = close_gap(ws.top, W_LIST, n_top, (int)x.far_cand);
        __syncthreads();
        const double lnS_all = __longlong_as_double((long long)s.bcast[0]);
        const uint32_t members = full ? w.n_fin : s.found_cnt;
        if ((uint32_t)n_all < min((uint32_t)s.ga.num_top, members) || n_all > W_LIST) { out.status |= ROW_NOT_DONE; return out; }      // (the same in every thread)
#pragma unroll 1
        for (int j = threadIdx.x; j < n_all; j += NT) {
            const u64 C = ws.top[j];
            uint32_t rank = 0;
#pragma unroll 4
            for (int q = 0; q < n_all; ++q) rank += ws.top[q] > C;
            if (rank < (uint32_t)s.ga.num_top && rank < members) {
                const int64_t o = (int64_t)b * s.ga.num_top + rank;
                s.ga.out_top_ids[o] = comp_idx(C);
                s.ga.out_top_logprobs[o] = (members == 1 && !full) ? 0.0f : (float)(((double)unkey((uint32_t)(C >> 32)) - (double)zmax) - lnS_all);
            }
        }
    }
    return out;
}

template <bool COUNTED>
__device__ __noinline__ RowOut wide_finish_call(float top_p, uint64_t seed, uint32_t R, Partial p, WideEnd w, u64 *list, int list_cap, const float *exp1_row,
                                                int b, RowOut out) {
    return wide_finish_in(SoloTeam<COUNTED>(), top_p, seed, R, p, w, list, list_cap, exp1_row, b, out);
}
// (with 64 registers per thread out of line; of rows that have been counted)
template <class TEAM>
__device__ __forceinline__ RowOut wide_finish(const TEAM &tm, float top_p, uint64_t seed, uint32_t R, const Partial &p, const WideEnd &w, u64 *list, int list_cap,
                                              const float *exp1_row, int b, const RowOut &out) {
    if constexpr (TEAM::ALONE) return wide_finish_call<true>(top_p, seed, R, p, w, list, list_cap, exp1_row, b, out);
    else return wide_finish_in(tm, top_p, seed, R, p, w, list, list_cap, exp1_row, b, out);
}

// The row's kept set, token and log-probability; the result is CTA 0's, in its warp 0.  `kmax`, `n_fin`:
// the row's largest order key and its number of finite scores (the same in every CTA).
template <int DT, class SRC, class TEAM>
__device__ __forceinline__ RowOut wide_row(BlockScratch &s, const SRC &src, const TEAM &tm, const RowParams &rp, float invT,
                                           uint32_t kmax, uint32_t n_fin, int b, uint32_t status) {
    const WideSmem ws = wide_smem();
    const int lane = threadIdx.x & 31;
    RowOut out;
    out.token = 0; out.logprob = 0.0f; out.n_keep = 0; out.n_topk = (int32_t)n_fin; out.status = status | ALBIREO_ROW_GENERAL_PATH;
    const float zmax = unkey(kmax);
    const bool full = (s.ga.flags & ALBIREO_FLAG_LOGPROB_FULL_VOCAB) != 0, want_list = s.ga.num_top > 0;
    const bool topp = rp.top_p < 1.0f, minp = rp.min_p > 0.0f;
    const float *exp1_row = s.ga.exp1 ? s.ga.exp1 + (int64_t)b * s.ga.exp1_stride : nullptr;
    const uint32_t kfloor = minp ? minp_key(zmax, rp.ln_min_p) : KEY_MIN_FINITE;
    if (kfloor > kmax || (minp && full && want_list)) { out.status |= ROW_NOT_DONE; return out; }
    const float zfloor = unkey(kfloor);
    u64 *const list = want_list ? ws.list : ws.top;
    const int list_cap = want_list ? W_LIST : W_LIST_ALONE;

    if (threadIdx.x == 0) { s.runmax = 0; tm.x->far_cand = 0; tm.x->far_list = 0; }
    const bool need_hist = topp || want_list || (full && minp);
    Window win, top;
    win.lo = win.hi = top.lo = top.hi = 0;
    if (need_hist) {
        for (int i = threadIdx.x; i < W_BINS; i += NT) ws.hist[i] = 0;
        __syncthreads();
        u64 S, S_all;
        if (minp) first_mass_pass<DT, true>(src, invT, zmax, zfloor, S, S_all);
        else first_mass_pass<DT, false>(src, invT, zmax, zfloor, S, S_all);
        S = warp_total(S);
        S_all = minp ? warp_total(S_all) : S;
        if (lane == 0) { s.red[threadIdx.x >> 5] = S; s.red2[threadIdx.x >> 5] = S_all; }
        __syncthreads();
        if (threadIdx.x < 32) {
            S = warp_total(lane < NWARPS ? s.red[lane] : 0ull);
            S_all = warp_total(lane < NWARPS ? s.red2[lane] : 0ull);
            if (lane == 0) { *tm.at(&tm.x->S[tm.rank], 0) = S; *tm.at(&tm.x->S_all[tm.rank], 0) = S_all; }
        }
        tm.sync();
        bool ok = true;
        const u64 want = (u64)(s.ga.num_top < (int32_t)n_fin ? s.ga.num_top : (int32_t)n_fin);
        const bool all_listed = want_list && n_fin <= (uint32_t)(W_LIST / 2);
        if (want_list) {
            if (all_listed) top.hi = 0xFFFFFFFEu;
            else {
                // (the histogram ends 42 octaves down: a row with fewer entries than wanted ahead of that is the
                // general path's; what the bounds of the counts leave open shows when the list is there)
                top = find_window(tm, true, F_ZERO, W_SHIFT, 0.0, want, 0);
                ok = top.found && (u64)top.ahead_most + top.most >= want;
            }
        }
        if (topp && ok) {
            // (a member's rounding is up to 2^-12 of it, 2^-14 of the total with those of the others)
            win = find_window(tm, false, F_ZERO, W_SHIFT, fmax((double)rp.top_p, 1e-12), 0ull, 14);
            ok = win.found;
        }
        if (topp && ok && win.most > (uint32_t)list_cap) {
            const u64 target = topp_target(rp.top_p, warp_total(lane < tm.size ? *tm.at(&tm.x->S[lane], 0) : 0ull));
            ok = minp ? narrow_window<DT, true>(src, tm, invT, zmax, zfloor, false, target, list_cap, &win)
                      : narrow_window<DT, false>(src, tm, invT, zmax, zfloor, false, target, list_cap, &win);
        }
        // (ahead of the list's last bin there are fewer than 2 num_top + 1 elements)
        const uint32_t top_cap = (uint32_t)(W_LIST - 2 * ALBIREO_MAX_NUM_TOP - 32);
        if (want_list && ok && !all_listed && top.most > top_cap)
            ok = minp ? narrow_window<DT, true>(src, tm, invT, zmax, zfloor, true, want, top_cap, &top)
                      : narrow_window<DT, false>(src, tm, invT, zmax, zfloor, true, want, top_cap, &top);
        if (!ok) { tm.sync(); out.status |= ROW_NOT_DONE; return out; }          // (the same in every CTA)
    }
    if (threadIdx.x == 0) { s.list_cnt = 0; s.cand_cnt = 0; }
    __syncthreads();

    const bool no_cut = !topp && !minp && !want_list && !exp1_row;
    // kept elements that are a good part of the row are raced in place: 25 instructions per element of the
    // row against about 40 per kept element through the queues (`ahead_most` is up to twice their number)
    const bool dense = topp && !minp && !want_list && !exp1_row && win.ahead_most > n_fin / 4;
    if ((no_cut || dense) && threadIdx.x == 32) { s.race.philox = philox_row(rp.seed, rp.R, s.ga.step); s.race.bound = __float_as_uint(RACE_LUCK); }
    if (threadIdx.x == 0) {
        FinalArgs &fa = s.fa;
        fa.invT = invT; fa.zmax = zmax; fa.zfloor = zfloor;
        fa.sure = topp ? win.lo : 0xFFFFFFFFu;
        fa.win_hi = topp ? win.hi : 0u;
        fa.id_lo = topp ? win.id_lo : 0u; fa.id_hi = topp ? win.id_hi : 0u;
        fa.top_hi = want_list ? top.hi : 0u;
        fa.list = list; fa.list_cap = list_cap;
        fa.seed = rp.seed; fa.step = s.ga.step; fa.R = rp.R; fa.exp1_row = exp1_row;
        // the vector test lets through everything with a code up to the largest that matters
        uint32_t key = kfloor;
        const uint32_t deepest = fa.win_hi > fa.top_hi ? fa.win_hi : fa.top_hi;
        if (fa.sure != 0xFFFFFFFFu && deepest < F_ZERO + (128u << 16)) {
            const float zlow = zmax - ((float)(deepest - F_ZERO + 2) * (0.6931472f / 65536.0f) * 1.00001f + 1e-6f * fabsf(zmax));
            const uint32_t k2 = key_of(zlow);
            key = k2 > key ? k2 : key;
        }
        fa.vec_thr = VecTest<DT>::raw_threshold(key, invT);
    }
    __syncthreads();
    Partial p;
    if (no_cut) run_race<DT, false>(src, s, p);
    else if (dense) run_race<DT, true>(src, s, p);
    else run_final_pass<DT>(src, s, p);
    WideEnd w;
    w.M0 = 0; w.n0 = 0; w.S = 0; w.S_all = 0; w.zmax = zmax; w.n_fin = n_fin; w.summed = !need_hist; w.in_team = need_hist; w.all_kept = !need_hist && !minp;
    w.topp = topp; w.full = full; w.race_from = no_cut || dense ? RACE_FROM : -INFINITY;
    return wide_finish_in(tm, rp.top_p, rp.seed, rp.R, p, w, list, list_cap, exp1_row, b, out);
}

// ------------------------------------------------------------------ rows of bfloat16: counted by value
//
// A bfloat16 logit has few values: from 2^-26 up to 64 either sign has 4096, and elements of one value have one mass.
// So the row's masses are a count per value - one shared-memory increment per element, 4 instructions, where the
// exponential, its exact sum and a histogram of masses take 19 - times an exponential per value, worked out
// afterwards, when the maximum is known.  One pass gives the maximum, the number of finite scores, the exact
// mass and, from prefix sums, the very value at which a cut or a list ends; with no cut the race is in the same
// pass.  (Increments of one warp meet in 3.5 bank cycles on average, which bounds the pass: 3620 cycles per 32768 elements
// in one SM against 6940 for the pass of masses and 690 for the maximum.)
// What has no place in the table: zeros, which have counts of their own; values of 64 and more, or nearer to zero than 2^-26, which are
// listed, up to CT_ODD of them (a row with more is done as rows of other types are); all from -63.75 down are counted together, and
// weigh nothing unless the maximum is as low.  The scores of the extras (penalised tokens, unaligned ends) lie between those of the values:
// they are added to the segment of 16 values that they belong to, and stay open in the segment of the cut.

constexpr int CT_PER = CT_BINS / NT;                   // values per thread: a segment
constexpr uint32_t CT_LOW = 0xC27Fu;                   // -63.75: this value and everything below
constexpr uint32_t ROW_NOT_COUNTED = 0x40000000u;      // internal status bit: the table does not hold the row (the same in every CTA)
static_assert(CT_PER == 16 && CT_ODD + 2 <= NT, "a segment is 16 values; a thread to each value without a place");

__device__ __forceinline__ uint32_t *counted_table() { extern __shared__ __align__(128) unsigned char smem[]; return (uint32_t *)smem; }
template <class SRC> __device__ __forceinline__ CountedSegs &counted_segs(const SRC &src) {
    extern __shared__ __align__(128) unsigned char smem[];
    return *(CountedSegs *)(smem + src.segments());
}
__device__ __forceinline__ uint32_t ct_index(uint32_t c) { return (c & 0xFFFu) | ((c >> 3) & 0x1000u); }
// the j-th value in descending order, and one step up from a value
__device__ __forceinline__ uint32_t ct_code(int j) { return j < 4096 ? 0x427Fu - (uint32_t)j : 0xB280u + (uint32_t)(j - 4096); }
__device__ __forceinline__ uint32_t ct_above(uint32_t c) { return c & 0x8000u ? c - 1u : c + 1u; }
// which place an element takes whose score lies above that of the next lower value than c and not above that of c
__device__ __forceinline__ int ct_place(uint32_t c) {
    const uint32_t mag = c & 0x7FFFu;
    if (mag < 0x3280u) return 4095;
    if (mag >= 0x4280u) return c & 0x8000u ? CT_BINS - 1 : 0;
    return c & 0x8000u ? 4096 + (int)(mag - 0x3280u) : (int)(0x427Fu - mag);
}
__device__ __forceinline__ float ct_score(uint32_t c, float invT) { return __fmul_rn(__uint_as_float(c << 16), invT); }
__device__ __forceinline__ u64 mass_fx(float z, float zmax) { return __float2ull_rn(ex2_ftz(log2_mass(z, zmax)) * FX_SCALE); }

// (by whole blocks; a barrier must follow)
template <class SRC>
__device__ __forceinline__ void counted_clear(const SRC &src) {
    CountedSegs &c = counted_segs(src);
#pragma unroll
    for (int i = 0; i < CT_PER / 4; ++i) ((uint4 *)counted_table())[i * NT + threadIdx.x] = make_uint4(0, 0, 0, 0);
    c.mass[threadIdx.x] = 0ull; c.cnt[threadIdx.x] = 0u;
    if (threadIdx.x == 0) { c.zeros[0] = c.zeros[1] = 0u; c.n_odd = 0u; c.lost = 0u; c.high = 0u; c.cut.fail = 0u; }
}
template <class SRC>
__device__ __noinline__ void count_odd_vector(SRC src, uint4 q) {
    CountedSegs &c = counted_segs(src);
    if (*(volatile uint32_t *)&c.lost) {               // (then only the values at CT_LOW are still wanted)
        const uint32_t low = VecTest<ALBIREO_BF16>::count_not_finite(q, (CT_LOW - 1u) * 0x10001u, 1.0f);
        if (low) atomicAdd(&counted_table()[ct_index(CT_LOW)], low);
        return;
    }
#pragma unroll 1
    for (int j = 0; j < 8; ++j) {
        const uint32_t v = __float_as_uint(pick_element<ALBIREO_BF16>(q, j)) >> 16, mag = v & 0x7FFFu;
        if (mag == 0u) atomicAdd(&c.zeros[v >> 15], 1u);
        else if (mag >= 0x3280u && mag < 0x4280u) atomicAdd(&counted_table()[ct_index(v)], 1u);
        else {
            const uint32_t at = atomicAdd(&c.n_odd, 1u);
            if (at < (uint32_t)CT_ODD) c.odd[at] = v; else c.lost = 1u;
            if (mag >= 0x4280u) { c.high = 1u; if (mag >= 0x7F80u) c.lost = 1u; }
        }
    }
}
// counts the vector's values; `top` is its largest of each half
template <class SRC>
__device__ __forceinline__ void count_vector(const SRC &src, uint4 q, __nv_bfloat162 top) {
    typedef __nv_bfloat162 H2;
    uint32_t *count = counted_table();
    const uint32_t low2 = CT_LOW | (CT_LOW << 16), high2 = 0x42804280u, tiny2 = 0x32803280u;
    auto h = [](const uint32_t &w) { return *reinterpret_cast<const H2 *>(&w); };
    const H2 least = __hmin2(__hmin2(__habs2(h(q.x)), __habs2(h(q.y))), __hmin2(__habs2(h(q.z)), __habs2(h(q.w))));
    const bool plain = (__hlt2_mask(top, h(high2)) & __hge2_mask(least, h(tiny2))) == 0xFFFFFFFFu;
    auto clamp = [&](uint32_t &w) { const H2 x = __hmax2(h(w), h(low2)); w = *reinterpret_cast<const uint32_t *>(&x); };
    clamp(q.x); clamp(q.y); clamp(q.z); clamp(q.w);
    if (!plain) { count_odd_vector(src, q); return; }
    auto add = [&](uint32_t w) {
        const uint32_t i = ((w & 0x0FFF0FFFu) | ((w >> 3) & 0xF000F000u)) & 0x1FFF1FFFu;
        atomicAdd(&count[i & 0xFFFFu], 1u);
        atomicAdd(&count[i >> 16], 1u);
    };
    add(q.x); add(q.y); add(q.z); add(q.w);
}
// The race of a vector's elements from `from` on (see race_all), by whole warps.
template <int OFF, class RACER>
__device__ __forceinline__ void race_vector(RACER &rc, const uint4 &q, int i0, __nv_bfloat162 top2, float from, float invT, float zref) {
    constexpr int NB = 2 + (OFF ? 1 : 0);
    const float xtop = fmaxf(__low2float(top2), __high2float(top2)), top = xtop >= from ? ex2_ftz(log2_mass(__fmul_rn(xtop, invT), zref)) : 0.0f;
    const float K = rc.K();
    if (!__any_sync(0xFFFFFFFFu, top * K >= 1.16e-10f)) return;
    uint32_t w[4 * NB], least = 0xFFFFFFFFu;
    philox_blocks<NB>(rc.row(), (uint32_t)(i0 >> 2), w);
#pragma unroll
    for (int j = 0; j < 8; ++j) least = min(least, w[OFF + j]);
    if (!__any_sync(0xFFFFFFFFu, least <= rc.word_bound(top, K))) return;
    rc.template race_hits<ALBIREO_BF16, OFF>(w, q, i0, invT, zref, [&](int j) {
        const float x = Elem<ALBIREO_BF16>::get(q, j);
        return x >= from ? ex2_ftz(-log2_mass(__fmul_rn(x, invT), zref)) : INFINITY;
    });
}

// The first pass: values counted, s.mm_max the largest order key, s.list_cnt the finite scores among the extras.
// RACE (no cut; see race_reference): the race as well, against zref in the place of the maximum: its candidates are listed (see CountedRacer).
template <int OFF, bool RACE, class SRC>
__device__ __noinline__ void counting_pass(SRC src, float invT, float zref) {
    BlockScratch &s = block_scratch();
    const int end = src.end_id();
    __nv_bfloat162 most = __halves2bfloat162(__ushort_as_bfloat16(0xFF80), __ushort_as_bfloat16(0xFF80));
    [[maybe_unused]] CountedRacer<LISTED> rc(s);
    if constexpr (!RACE) src.template vectors<4>([&](const uint4 &q0, const uint4 &q1, int i0, int i1) {
        const __nv_bfloat162 top0 = VecTest<ALBIREO_BF16>::vmax(q0), top1 = VecTest<ALBIREO_BF16>::vmax(q1);
        most = __hmax2(most, __hmax2(top0, top1));
        if (i0 < end) count_vector(src, q0, top0);
        if (i1 >= 0 && i1 < end) count_vector(src, q1, top1);
    });
    else src.template vectors<1>([&](const uint4 &q, int i0) {
        const __nv_bfloat162 top = VecTest<ALBIREO_BF16>::vmax(q);
        most = __hmax2(most, top);
        if (i0 < end) count_vector(src, q, top);
        __syncwarp();
        race_vector<OFF>(rc, q, i0, top, -INFINITY, invT, zref);
    });
    uint32_t kbest = key_of(__fmul_rn(fmaxf(__low2float(most), __high2float(most)), invT)), nfin = 0;
    src.extras([&](int i, float z) {
        const uint32_t k = key_of(z);
        kbest = k > kbest ? k : kbest;
        nfin += (k >= KEY_MIN_FINITE && k < KEY_POS_INF);
        if constexpr (RACE) {
            const float d = __fsub_rn(z, zref);
            rc.race(d > -3.0e38f, i, z, d, d * 1.4426950408889634f);
        }
    });
    if (kbest < KEY_MIN_FINITE || kbest >= KEY_POS_INF) kbest = 0;
    kbest = __reduce_max_sync(0xFFFFFFFFu, kbest);
    nfin = __reduce_add_sync(0xFFFFFFFFu, nfin);
    if ((threadIdx.x & 31) == 0) { atomicMax(&s.mm_max, kbest); if (nfin) atomicAdd(&s.list_cnt, nfin); }
}
template <class SRC>
__device__ __forceinline__ void run_counting(const SRC &src, BlockScratch &s, bool race, float invT, float zref) {
    if (!race) { counting_pass<0, false>(src, invT, 0.0f); return; }
    switch (src.first_id() & 3) {
        case 0: counting_pass<0, true>(src, invT, zref); break;
        case 1: counting_pass<1, true>(src, invT, zref); break;
        case 2: counting_pass<2, true>(src, invT, zref); break;
        default: counting_pass<3, true>(src, invT, zref); break;
    }
}
// What the race of a row without a cut is run against in the place of the maximum, which is not known yet: the largest score of the block's
// vectors `q`, one per thread (0 where they have none, and then no bound to start from).  The generator and the race's bound
// are set up as well.  Contains a barrier, and one has to follow.
__device__ __forceinline__ float race_reference(BlockScratch &s, const uint4 &q, float invT, const RowParams &rp) {
    const uint32_t k = __reduce_max_sync(0xFFFFFFFFu, VecTest<ALBIREO_BF16>::vmax_key(q, invT));
    if ((threadIdx.x & 31) == 0) s.r32a[threadIdx.x >> 5] = k;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const float top = unkey(__reduce_max_sync(0xFFFFFFFFu, lane < NWARPS ? s.r32a[lane] : 0u));
    const bool some = fabsf(top) < 3.0e38f;
    if (threadIdx.x == 0) { s.race.philox = philox_row(rp.seed, rp.R, s.ga.step); s.race.bound = some ? __float_as_uint(RACE_LUCK) : NO_BOUND; s.cand_cnt = 0; }
    return some ? top : 0.0f;
}
// which wide rows are counted (the temperature's bound keeps the scores of different values apart)
template <int DT>
__device__ __forceinline__ bool counted_eligible(const RowParams &rp, const RowCtx &c, const SampleArgs &a) {
    return DT == ALBIREO_BF16 && wide_eligible(rp, a) && !a.exp1 && !(rp.min_p > 0.0f && (a.flags & ALBIREO_FLAG_LOGPROB_FULL_VOCAB)) &&
           c.invT > 1e-18f && c.invT < 1e18f;
}
__device__ __forceinline__ bool nothing_cut(const RowParams &rp, const SampleArgs &a) { return !(rp.top_p < 1.0f) && !(rp.min_p > 0.0f) && a.num_top <= 0; }
// How many of the vectors' elements have a finite score, where not all of those counted at CT_LOW are the `killed`
// penalised tokens.  Ends with a barrier.
template <class SRC>
__device__ __noinline__ uint32_t count_finite(SRC src, float invT) {
    BlockScratch &s = block_scratch();
    const uint32_t thr = VecTest<ALBIREO_BF16>::finite_threshold(invT);
    uint32_t n = 0;
    src.template vectors<4>([&](const uint4 &q, int) { n += 8u - VecTest<ALBIREO_BF16>::count_not_finite(q, thr, invT); });
    return (uint32_t)block_sum_u64(n);
}
// Row (or slice) after the counting pass and a barrier: the number of finite scores among the vectors' elements, and what
// the table cannot tell (bit 29), or only if the maximum is far above -63.75 (bit 28).  The same in every thread.
// `exact`: else only those above -63.75 are wanted where there may be others.
template <class SRC>
__device__ __forceinline__ uint32_t counted_finite(const SRC &src, BlockScratch &s, float invT, uint32_t killed, uint32_t &flags, bool exact = true) {
    const CountedSegs &c = counted_segs(src);
    const uint32_t low = counted_table()[ct_index(CT_LOW)];
    flags = c.lost ? 0x20000000u : 0u;
    const uint32_t rest = (uint32_t)src.elements() - low;
    if (low == killed) return rest;
    if (!exact) { flags |= 0x10000000u; return rest; }
    const uint32_t n = count_finite(src, invT);
    if (n != rest) flags |= 0x10000000u;
    return n;
}

// which halves of a word are in the window
__device__ __forceinline__ uint32_t edge_mask(uint32_t w, uint32_t thr_win, uint32_t thr_sure) {
    typedef __nv_bfloat162 H2;
    const H2 h = *reinterpret_cast<const H2 *>(&w);
    return __hge2_mask(h, *reinterpret_cast<const H2 *>(&thr_win)) & ~__hge2_mask(h, *reinterpret_cast<const H2 *>(&thr_sure));
}
// and the elements that they stand for
__device__ __forceinline__ uint32_t edge_bits(uint32_t x, uint32_t y, uint32_t z, uint32_t w) {
    auto two = [](uint32_t m) { return (m & 1u) | ((m >> 15) & 2u); };
    return two(x) | two(y) << 2 | two(z) << 4 | two(w) << 6;
}
// Mass, number and lists of the extras, the race of all that is kept for sure, the window's elements to their list.
// Where few vectors have something that matters they are listed by their number, and the list is worked off by all warps alike: where they lie close together
// (the head of a vocabulary) they would else be a few warps' work.  Where they may be more than the list holds every vector is worked on as it comes. (100 rows of 152064,
// us of this pass, listed in parts and as they come: 49000 kept 53 and 37, 23000 43 and 35.)
// (out of line: few vectors have any)
__device__ __noinline__ void append_elements(uint4 q, int i0, uint32_t bits, float invT) {
    BlockScratch &s = block_scratch();
    while (bits) {
        const int x = __ffs(bits) - 1;
        bits &= bits - 1u;
        list_append(wide_smem().top, W_LIST, &s.cand_cnt, __fmul_rn(pick_element<ALBIREO_BF16>(q, x), invT), i0 + x);
    }
    __syncwarp();
}
template <int OFF, class SRC>
__device__ __noinline__ Partial counted_final_pass(SRC src) {
    typedef VecTest<ALBIREO_BF16> T;
    extern __shared__ __align__(128) unsigned char smem[];
    BlockScratch &s = block_scratch();
    const CountedCut &cut = counted_segs(src).cut;
    const WideSmem ws = wide_smem();
    // (worked out anew where they are used: held across the loop they were spilled)
    auto lane_now = [] { int l; asm volatile("mov.u32 %0, %%laneid;" : "=r"(l)); return l; };
    uint16_t *queue = (uint16_t *)(smem + CT_QUEUE_OFF);
    CountedRacer<SRC::SPARE_REGISTERS ? IN_REGS : IN_SHARED> rc(s);
    auto work = [&](const uint4 &q, int i0) {
        const volatile CountedCut &c = cut;
        const float invT = *(const volatile float *)&s.fa.invT;
        const uint32_t thr_sure = c.thr_sure, thr_win = c.thr_win;
        if (s.ga.num_top > 0) {
            const uint32_t bits = T::elem_bits(q, c.thr_top, invT);
            if (__any_sync(0xFFFFFFFFu, bits != 0u)) append_elements(q, i0, bits, invT);
        }
        uint32_t in = edge_bits(edge_mask(q.x, thr_win, thr_sure), edge_mask(q.y, thr_win, thr_sure), edge_mask(q.z, thr_win, thr_sure), edge_mask(q.w, thr_win, thr_sure));
        while (in) {
            const int x = __ffs(in) - 1;
            in &= in - 1u;
            list_append(s.fa.list, s.fa.list_cap, &s.list_cnt, __fmul_rn(pick_element<ALBIREO_BF16>(q, x), invT), i0 + x);
        }
        __syncwarp();
        race_vector<OFF>(rc, q, i0, T::vmax(q), __uint_as_float(thr_sure << 16), invT, *(const volatile float *)&s.fa.zmax);
    };
    if (cut.n_any <= (uint32_t)FINAL_QUEUE) {
        {
            const uint32_t thr_any = cut.thr_any;
            const int first_id = src.first_id(), end = src.end_id();
            src.template vectors<4>([&](const uint4 &q, int i0) {
                const bool in = T::may_pass(q, thr_any, 1.0f) && i0 < end;
                const uint32_t m = __ballot_sync(0xFFFFFFFFu, in);
                if (m == 0) return;
                const int lane = lane_now();
                uint32_t at = 0;
                if (lane == 0) at = atomicAdd(&s.runmax, (uint32_t)__popc(m));
                at = __shfl_sync(0xFFFFFFFFu, at, 0) + __popc(m & ((1u << lane) - 1u));
                if (in && at < (uint32_t)FINAL_QUEUE) queue[at] = (uint16_t)((uint32_t)(i0 - first_id) / 8u);
            });
        }
        __syncthreads();
        // (never more than there is room for, see n_any; else the row is given up)
        const int n = (int)min(s.runmax, (uint32_t)FINAL_QUEUE);
        if (s.runmax > (uint32_t)FINAL_QUEUE) s.list_cnt = 0x10000000u;
        uint4 ahead = src.vector((int)threadIdx.x < n ? (int)queue[threadIdx.x] : -1);
#pragma unroll 1
        for (int at = (int)threadIdx.x, v = at < n ? (int)queue[at] : -1; at - lane_now() < n; at += NT) {
            // (the next one is fetched while this one is worked on)
            const uint4 q = ahead;
            const int i0 = v < 0 ? 0 : src.first_id() + v * 8;
            v = at + NT < n ? (int)queue[at + NT] : -1;
            ahead = src.vector(v);
            work(q, i0);
        }
    } else src.template vectors<1>(work);
    Partial p;
    p.M = 0; p.n = 0;
    const float zmax = s.fa.zmax;
    const bool listed = s.ga.num_top > 0;
    src.extras([&](int i, float z) {
        const uint32_t k = key_of(z);
        const bool finite = k < KEY_POS_INF && k >= KEY_MIN_FINITE, sure = finite && k > cut.key_hi;
        if (listed && finite && k >= cut.key_top) list_append(ws.top, W_LIST, &s.cand_cnt, z, i);
        if (sure && k <= cut.key_seg) { p.M += mass_fx(z, zmax); ++p.n; }
        if (finite && !sure && k >= cut.key_lo) list_append(s.fa.list, s.fa.list_cap, &s.list_cnt, z, i);
        __syncwarp();
        const float d = __fsub_rn(z, zmax);
        if (__any_sync(0xFFFFFFFFu, sure)) rc.race(sure, i, z, d, d * 1.4426950408889634f);
    });
    rc.finish(p);
    return p;
}

// A segment's 16 values by one warp: where the running total from the top of the order (masses, or counts) reaches `need` of what the
// segment adds.  Which values are ahead of that for sure, which may be the one: lo <= hi, 16 for what follows the segment's last value.
struct SegmentEnd { int lo, hi; u64 mass_ahead; uint32_t cnt_ahead, cnt_most; };
template <class TEAM>
__device__ __forceinline__ SegmentEnd end_in_segment(const TEAM &tm, int seg, bool by_mass, u64 need, u64 seg_mass, uint32_t seg_cnt, float invT, float zmax, float zfloor) {
    const int lane = threadIdx.x & 31;
    const uint32_t code = ct_code(seg * CT_PER + (lane & 15));
    const float z = ct_score(code, invT);
    uint32_t cnt = 0;
    if (lane < CT_PER && z >= zfloor)
        for (int r = 0; r < tm.size; ++r) cnt += *tm.at(&counted_table()[ct_index(code)], r);
    u64 mass = (u64)cnt * mass_fx(z, zmax);
#pragma unroll
    for (int o = 1; o < CT_PER; o <<= 1) {
        const u64 t = __shfl_up_sync(0xFFFFFFFFu, mass, o);
        const uint32_t tc = __shfl_up_sync(0xFFFFFFFFu, cnt, o);
        if (lane >= o) { mass += t; cnt += tc; }
    }
    const u64 open_mass = seg_mass - __shfl_sync(0xFFFFFFFFu, mass, CT_PER - 1);
    const uint32_t open_cnt = seg_cnt - __shfl_sync(0xFFFFFFFFu, cnt, CT_PER - 1);
    const u64 have = by_mass ? mass : (u64)cnt, open = by_mass ? open_mass : (u64)open_cnt;
    const uint32_t lo = __ballot_sync(0xFFFFFFFFu, lane < CT_PER && have + open >= need), hi = __ballot_sync(0xFFFFFFFFu, lane < CT_PER && have >= need);
    SegmentEnd e;
    e.lo = lo ? __ffs(lo) - 1 : CT_PER - 1; e.hi = hi ? __ffs(hi) - 1 : CT_PER;
    e.mass_ahead = __shfl_sync(0xFFFFFFFFu, mass, max(e.lo - 1, 0)); e.cnt_ahead = __shfl_sync(0xFFFFFFFFu, cnt, max(e.lo - 1, 0));
    if (e.lo == 0) { e.mass_ahead = 0; e.cnt_ahead = 0; }
    e.cnt_most = __shfl_sync(0xFFFFFFFFu, cnt, min(e.hi, CT_PER - 1)) + open_cnt;
    return e;
}
// the order key from which on elements belong to the first hi + 1 values of a segment (hi = 16: to the whole of it)
__device__ __forceinline__ uint32_t ct_key_down_to(int seg, int hi, float invT) {
    const int j = seg * CT_PER + hi;
    if (j >= CT_BINS) return KEY_MIN_FINITE;
    return key_of(ct_score(ct_code(j), invT)) + (hi == CT_PER ? 1u : 0u);
}

// The masses of a counted row: its extras' and its values', by segments (in shared memory; cut.fail set where an extra has no place), or, with no
// cut, each thread's share of the sum.
template <class SRC>
__device__ __noinline__ u64 counted_masses(SRC src, float invT, float zmax, uint32_t kfloor, bool no_cut) {
    BlockScratch &s = block_scratch();
    CountedSegs &ct = counted_segs(src);
    const int t = threadIdx.x, n_odd = (int)ct.n_odd;
    const float zfloor = unkey(kfloor);
    u64 sum = 0;
    // (64 bits as two words, the carry by whoever makes the low one wrap: any number of masses may meet in a segment. A
    // 64-bit add in shared memory is a compare-and-swap loop.)
    auto in_segment = [&](int seg, u64 m, uint32_t n = 1u) {
        uint32_t *w = (uint32_t *)&ct.mass[seg];
        const uint32_t lo = (uint32_t)m, was = atomicAdd(&w[0], lo), hi = (uint32_t)(m >> 32) + (was + lo < lo);
        if (hi) atomicAdd(&w[1], hi);
        atomicAdd(&ct.cnt[seg], n);
    };
    src.extras([&](int, float z) {
        const uint32_t k = key_of(z);
        if (k >= KEY_POS_INF || k < kfloor) return;
        const u64 m = mass_fx(z, zmax);
        if (no_cut) { sum += m; return; }
        const uint32_t raw = VecTest<ALBIREO_BF16>::raw_threshold(k, invT) & 0xFFFFu;
        if (raw == 0xFF80u) ct.cut.fail = 1u; else in_segment(ct_place(raw) / CT_PER, m);
    });
    if (t < n_odd || t >= NT - 2) {
        const uint32_t code = t < n_odd ? ct.odd[t] : (uint32_t)(t - (NT - 2)) << 15, n = t < n_odd ? 1u : ct.zeros[t - (NT - 2)];
        const float z = ct_score(code, invT);
        if (n != 0u && z >= zfloor) {
            const u64 m = (u64)n * mass_fx(z, zmax);
            if (no_cut) sum += m; else in_segment(ct_place(code) / CT_PER, m, n);
        }
    }
    __syncthreads();
    const uint32_t first = t < 256 ? 0x4270u - 16u * (uint32_t)t : 0xB280u + 16u * (uint32_t)(t - 256);      // the smallest magnitude
    const uint4 *words = (const uint4 *)&counted_table()[ct_index(first)];
    u64 mass = 0;
    uint32_t cnt = 0;
#pragma unroll
    for (int i = 0; i < CT_PER / 4; ++i) {
        const uint4 w = words[i];
        if ((w.x | w.y | w.z | w.w) == 0u) continue;
        const uint32_t v[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float z = ct_score(first + 4 * i + j, invT);
            if (z >= zfloor) { cnt += v[j]; mass += (u64)v[j] * mass_fx(z, zmax); }
        }
    }
    if (no_cut) return sum + mass;
    ct.mass[t] += mass;
    ct.cnt[t] += cnt;
    return 0;
}
// From the segments of all CTAs to the cut (see CountedCut), the same in every CTA; s.bcast[2] and [3]: the mass above the floor and the one to
// be reached.  False: the table does not tell.
template <class SRC, class TEAM>
__device__ __noinline__ bool counted_locate(SRC src, TEAM tm, float invT, float zmax, uint32_t kfloor, bool minp, float top_p, uint32_t n_fin, int list_cap, bool high) {
    typedef VecTest<ALBIREO_BF16> T;
    BlockScratch &s = block_scratch();
    CountedSegs &ct = counted_segs(src);
    CountedCut &cut = ct.cut;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, t = threadIdx.x;
    const bool topp = top_p < 1.0f, listed = s.ga.num_top > 0;
    const float zfloor = unkey(kfloor);
    u64 mass = 0;
    uint32_t cnt = 0;
#pragma unroll 4
    for (int r = 0; r < tm.size; ++r) { mass += *tm.at(&ct.mass[t], r); cnt += *tm.at(&ct.cnt[t], r); }
    u64 run = mass;
    uint32_t crun = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const u64 tt = __shfl_up_sync(0xFFFFFFFFu, run, o);
        const uint32_t tc = __shfl_up_sync(0xFFFFFFFFu, crun, o);
        if (lane >= o) { run += tt; crun += tc; }
    }
    if (lane == 31) { s.red[wid] = run; s.r32a[wid] = crun; }
    __syncthreads();
    const u64 wt = lane < NWARPS ? s.red[lane] : 0ull;
    const uint32_t wc = lane < NWARPS ? s.r32a[lane] : 0u;
    const u64 S = warp_total(wt);
    run += warp_total(lane < wid ? wt : 0ull) - mass;
    crun += __reduce_add_sync(0xFFFFFFFFu, lane < wid ? wc : 0u) - cnt;
    const u64 target = topp ? topp_target(top_p, S) : S;
    const u64 want = (u64)min((uint32_t)s.ga.num_top, n_fin);
    if (topp && run < target && target <= run + mass) { s.found_digit = (uint32_t)t; s.found_above = run; s.bcast[0] = mass; s.r32b[0] = crun; s.r32b[1] = cnt; }
    if (listed && (u64)crun < want && want <= (u64)crun + cnt) { s.found_cnt = (uint32_t)t; s.bcast[1] = mass; s.r32b[2] = crun; s.r32b[3] = cnt; }
    __syncthreads();
    if (wid == 0) {
        // the cut: the window's values, and those above it
        const uint32_t n_all = __reduce_add_sync(0xFFFFFFFFu, wc);
        CountedCut c;
        c.n_any = 0xFFFFFFFFu;
        c.M = S; c.n = n_all; c.key_lo = 0xFFFFFFFFu; c.key_hi = kfloor - 1u; c.key_seg = c.key_hi; c.fail = 0;
        c.thr_sure = c.thr_win = T::fill().x;             // (everything: -inf has no mass and does not win)
        if (minp && !topp) { c.thr_sure = c.thr_win = T::raw_threshold(kfloor, invT); c.n_any = n_all; }      // (all that is above the floor has been counted)
        if (topp) {
            const int seg = (int)s.found_digit;
            if (seg < 0) c.fail = 1u;
            else {
                SegmentEnd e = end_in_segment(tm, seg, true, target - s.found_above, s.bcast[0], s.r32b[1], invT, zmax, zfloor);
                // (values above the table's are in its first segment: where the cut is there too, the window begins with them)
                const bool from_top = seg == 0 && high;
                if (from_top) { e.lo = 0; e.mass_ahead = 0; e.cnt_ahead = 0; }
                const uint32_t above = ct_code(seg * CT_PER + e.lo);
                c.M = s.found_above + e.mass_ahead; c.n = s.r32b[0] + e.cnt_ahead;
                c.key_hi = from_top ? 0xFFFFFFFFu : key_of(ct_score(above, invT));
                c.key_lo = max(ct_key_down_to(seg, e.hi, invT), kfloor);
                c.key_seg = seg == 0 ? 0xFFFFFFFFu : key_of(ct_score(ct_code(seg * CT_PER), invT));
                c.thr_sure = (from_top ? 0x7F80u : ct_above(above)) * 0x10001u;
                c.thr_win = e.hi < CT_PER ? ct_code(seg * CT_PER + e.hi) * 0x10001u : T::raw_threshold(c.key_lo, invT);
                c.n_any = s.r32b[0] + e.cnt_most;
                if (e.cnt_most - e.cnt_ahead > (uint32_t)list_cap) c.fail = 1u;
            }
        }
        if (lane == 0) {
            cut.M = c.M; cut.n = c.n; cut.key_lo = c.key_lo; cut.key_hi = c.key_hi; cut.key_seg = c.key_seg;
            cut.thr_sure = c.thr_sure; cut.thr_win = c.thr_win; cut.n_any = c.n_any; cut.fail = c.fail;
        }
    } else if (wid == 1) {
        // the list: everything down to the value at which the wanted number is reached
        uint32_t key_top = kfloor, fail = 0, n_top = 0xFFFFFFFFu;
        if (listed && n_fin > (uint32_t)(W_LIST / 2)) {
            const int seg = (int)s.found_cnt;
            if (seg < 0) fail = !(minp || topp);         // (fewer than wanted: all that are kept)
            else {
                const SegmentEnd e = end_in_segment(tm, seg, false, want - s.r32b[2], s.bcast[1], s.r32b[3], invT, zmax, zfloor);
                key_top = max(ct_key_down_to(seg, e.hi, invT), kfloor);
                n_top = s.r32b[2] + e.cnt_most;
                if (n_top > (uint32_t)W_LIST) fail = 1u;
            }
        }
        if (lane == 0) { cut.key_top = key_top; cut.thr_top = listed ? T::raw_threshold(key_top, invT) : 0u; s.r32b[8] = fail; s.r32b[9] = n_top; }
    } else if (t == 64) {
        s.fa.invT = invT; s.fa.zmax = zmax; s.fa.list_cap = list_cap; s.fa.exp1_row = nullptr;
        s.fa.list = listed ? wide_smem().list : wide_smem().top;
        s.race.bound = __float_as_uint(RACE_LUCK / ((float)target * (1.0f / FX_SCALE)));
        s.bcast[2] = S; s.bcast[3] = target;
    }
    tm.sync();                                           // (everybody has read the tables; lists and queues lie over them)
    if (cut.fail | s.r32b[8]) return false;
    if (t == 0) {
        const float win = __uint_as_float(cut.thr_win << 16), top = __uint_as_float(cut.thr_top << 16);
        cut.thr_any = listed && top < win ? cut.thr_top : cut.thr_win;
        if (listed && top < win) cut.n_any = s.r32b[9];
    }
    __syncthreads();
    return true;
}

// A row (or a team's slices of it) whose values have been counted; by one CTA with no cut, it has been raced as well.
// `flags`: see counted_finite, of all CTAs.  As wide_row otherwise.
template <class SRC, class TEAM>
__device__ __noinline__ RowOut counted_row(SRC src, TEAM tm, const RowParams rp, float invT, uint32_t kmax, uint32_t n_fin,
                                           uint32_t flags, int b, uint32_t status) {
    BlockScratch &s = block_scratch();
    const int lane = threadIdx.x & 31, t = threadIdx.x;
    RowOut out;
    out.token = 0; out.logprob = 0.0f; out.n_keep = 0; out.n_topk = (int32_t)n_fin; out.status = status | ALBIREO_ROW_GENERAL_PATH;
    const float zmax = unkey(kmax);
    const bool topp = rp.top_p < 1.0f, minp = rp.min_p > 0.0f, listed = s.ga.num_top > 0, no_cut = !topp && !minp && !listed;
    const uint32_t kfloor = minp ? minp_key(zmax, rp.ln_min_p) : KEY_MIN_FINITE;
    const float zlow = ct_score(CT_LOW, invT);
    const bool raced = TEAM::ALONE && no_cut;
    // (values that are counted together must weigh nothing and be below the floor; a race that is listed as a whole)
    if ((raced && s.cand_cnt > (uint32_t)RACE_LIST) || (flags & 0x20000000u) || kfloor > kmax || ((flags & 0x10000000u) && (!(zmax - zlow > 29.0f) || (minp && unkey(kfloor) <= zlow)))) {
        out.status |= ROW_NOT_COUNTED;
        return out;
    }
    const CountedCut &cut = counted_segs(src).cut;
    if (t == 0) {
        counted_table()[ct_index(CT_LOW)] = 0;
        tm.x->far_cand = 0; tm.x->far_list = 0;
    }
    Partial p;
    p.M = counted_masses(src, invT, zmax, kfloor, raced);
    p.n = 0; p.G = 0; p.z = 0.0f;
    WideEnd w;
    w.M0 = 0; w.n0 = 0; w.S = 0; w.S_all = 0; w.zmax = zmax; w.n_fin = n_fin; w.summed = raced; w.in_team = false; w.all_kept = !topp && !minp; w.topp = topp;
    w.full = (s.ga.flags & ALBIREO_FLAG_LOGPROB_FULL_VOCAB) != 0;
    w.race_from = RACE_FROM;
    const int list_cap = listed ? W_LIST : W_LIST_ALONE;
    if (raced) {
        if (t < (int)s.cand_cnt) {
            const u64 C = race_list()[t];
            const int i = comp_idx(C);
            p.z = unkey((uint32_t)(C >> 32));
            p.G = CountedRacer<LISTED>::code_of_score(__fsub_rn(p.z, zmax) + race_nle(rp.seed, rp.R, s.ga.step, nullptr, i), i);
        }
    } else {
        if (t < tm.size) *tm.at(&tm.x->ncand[tm.rank], t) = cut.fail | (counted_segs(src).high ? 2u : 0u);       // (a barrier has ended the extras)
        if (t == 0) { s.found_digit = 0xFFFFFFFFu; s.found_cnt = 0xFFFFFFFFu; s.list_cnt = 0; s.cand_cnt = 0; s.runmax = 0; s.race.philox = philox_row(rp.seed, rp.R, s.ga.step); }
        tm.sync();
        const uint32_t told = __reduce_or_sync(0xFFFFFFFFu, lane < tm.size ? tm.x->ncand[lane] : 0u);
        if ((told & 1u) || !counted_locate(src, tm, invT, zmax, kfloor, minp, rp.top_p, n_fin, list_cap, (told & 2u) != 0u)) { out.status |= ROW_NOT_COUNTED; return out; }
        w.S = w.S_all = s.bcast[2];
        w.race_from = 0.001f - logf(RACE_LUCK / ((float)s.bcast[3] * (1.0f / FX_SCALE)));
        switch (src.first_id() & 3) {
            case 0: p = counted_final_pass<0>(src); break;
            case 1: p = counted_final_pass<1>(src); break;
            case 2: p = counted_final_pass<2>(src); break;
            default: p = counted_final_pass<3>(src); break;
        }
        w.M0 = cut.M; w.n0 = cut.n;
    }
    return wide_finish(tm, rp.top_p, rp.seed, rp.R, p, w, listed ? wide_smem().list : wide_smem().top, list_cap, nullptr, b, out);
}
