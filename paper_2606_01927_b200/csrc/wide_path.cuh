// Wide rows: rows whose kept set has no small bound (top-p alone, no cut at all, a min-p that keeps
// thousands).  Included by albireo_sample.cu.
//
// What such a row costs is instructions: every element needs an exponential (its mass), and with
// no cut a share of a Philox block; 41 (no cut) to 65 per logit in all, at 28 to 41 % of the issue slots (the largest
// stalls are instruction fetch, fixed latencies and barriers).  So the row is passed over as few times as the definition allows
// and each pass does one short fixed sequence per element:
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
    uint32_t kmax[MAX_TEAM], tau[MAX_TEAM], tau_part[MAX_TEAM], nfin[MAX_TEAM], flags[MAX_TEAM], ncand[MAX_TEAM];   // in every CTA
    u64 ahead[MAX_TEAM];                                                                                           // in every CTA
    u64 S[MAX_TEAM], S_all[MAX_TEAM], M[MAX_TEAM], G[MAX_TEAM];                                                    // in CTA 0's
    uint32_t n[MAX_TEAM];
    float z[MAX_TEAM];
    uint32_t far_cand, far_list;      // CTA 0: entries that the others have put at the far end of its lists
};

struct SoloTeam {                     // a CTA that has the row to itself
    TeamWords *x;
    static constexpr int rank = 0, size = 1;
    __device__ __forceinline__ void sync() const { __syncthreads(); }
    template <class P> __device__ __forceinline__ P *at(P *p, int) const { return p; }
};
struct ClusterTeam {                  // the CTAs of a thread-block cluster
    TeamWords *x;
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

// The whole row, streamed from global memory (from the L2 after the first pass) through a ring of bulk
// copies: next to CTAs that stream their own rows a plain load comes back after 1.5 to 3 us, and only the
// copies of whole tiles keep enough of them in flight.  Penalised tokens are masked out of the vectors
// and come from the history tables.  Both loops have the same trip count in every lane of a warp (lanes
// past the end see -inf), so that the callee may use warp collectives, but no block barriers.
// (A pass needs its registers for the elements: what the loop does not touch per vector stays in shared memory.)
// (a tile is 4 vectors per thread, 32 KiB, where two of them fit, else 2: what a tile costs is the hand-shake)
constexpr int WIDE_VEC_BYTES = NT * 16;
constexpr int WIDE_MAX_STAGES = 6;
struct RowShared {
    RowCtx c;
    RowParams rp;
    const uint4 *vp;
    int head, nvec, vps, nst, tv; // stages of the ring, vectors per thread and tile
    uint32_t tiles;               // tiles of the passes so far
    uint32_t issued;              // tiles of this pass whose copy has been issued
    uint32_t timeout;             // a wait on a copy expired
    uint32_t done[WIDE_MAX_STAGES];
    uint64_t bar[WIDE_MAX_STAGES];
};
__device__ __forceinline__ RowShared &row_shared();
__device__ __forceinline__ unsigned char *wide_stage(int st);
template <int DT>
struct RingSlice {
    typedef Elem<DT> E;
    static constexpr bool SPARE_REGISTERS = false;      // 64 per thread
    __device__ __forceinline__ int first_id() const { return row_shared().head; }
    __device__ __forceinline__ static void issue(RowShared &r, int t, int st) {
        Ring rg;
        rg.vps = r.vps; rg.seg_base = r.c.seg_base;
        const int v0 = t * (NT * r.tv), nv = min(r.nvec - v0, NT * r.tv);
        mbar_expect_tx(&r.bar[st], (uint32_t)nv * 16u);
        ring_copy(rg, wide_stage(st * r.tv), r.vp, v0, nv, &r.bar[st]);
    }
    // The tiles of all passes are numbered through, which gives stage and phase; the last warp done with a
    // stage refills it.  A wait that expires marks the row, and nothing more is copied.
    template <class F> __device__ __forceinline__ void vectors(F &&f) const {
        RowShared &r = row_shared();
        const uint32_t first = r.tiles;
        const int nvec = r.nvec, head = r.head, nst = r.nst, tv = r.tv, ntiles = (nvec + NT * tv - 1) / (NT * tv);
        const uint32_t *bitmap = r.c.has_hist ? r.c.bitmap : nullptr;
        int st = (int)(first % (uint32_t)nst);
        uint32_t parity = (first / (uint32_t)nst) & 1u;
        if (threadIdx.x == 0) {
            const int npre = r.timeout ? 0 : min(ntiles, nst);
            r.issued = (uint32_t)npre;
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
#pragma unroll 1
            for (int t = 0, q = st; t < npre; ++t) { issue(r, t, q); q = q + 1 == nst ? 0 : q + 1; }
        }
        __syncwarp();       // (the other lanes of the issuing warp, spinning on the first copy, could keep the issuing lane from running)
#pragma unroll 1
        for (int t = 0; t < ntiles; ++t) {
            if (*(volatile uint32_t *)&r.timeout == 0u && !mbar_wait(&r.bar[st], parity)) r.timeout = 1u;
            __syncwarp();
            const uint4 *stage = (const uint4 *)wide_stage(st * tv);
#pragma unroll 1
            for (int u = 0; u < tv; ++u) {
                const int v = (t * tv + u) * NT + (int)threadIdx.x, i0 = head + v * E::PER_VEC;
                uint4 q = VecTest<DT>::fill();
                if (v < nvec) {
                    q = stage[u * NT + threadIdx.x];
                    if (bitmap) {
                        const uint32_t m = __funnelshift_r(bitmap[i0 >> 5], bitmap[(i0 >> 5) + 1], i0 & 31) & ((1u << E::PER_VEC) - 1u);
                        if (m) q = kill_elements<DT>(q, m);
                    }
                }
                f(q, i0);
            }
            __syncwarp();
            if ((threadIdx.x & 31) == 0) {
                __threadfence_block();
                if (atomicAdd(&r.done[st], 1u) == (uint32_t)(NWARPS - 1)) {
                    r.done[st] = 0;
                    __threadfence_block();
                    if (t + nst < ntiles && *(volatile uint32_t *)&r.timeout == 0u) {
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        issue(r, t + nst, st);
                        atomicMax(&r.issued, (uint32_t)(t + nst + 1));
                    }
                }
            }
            __syncwarp();
            if (++st == nst) { st = 0; parity ^= 1u; }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            // (after an expired wait: the copies in flight land, or get as long again, before the CTA moves on)
            if (r.timeout)
                for (uint32_t t = r.issued > (uint32_t)nst ? r.issued - (uint32_t)nst : 0u; t < r.issued; ++t)
                    mbar_wait(&r.bar[(first + t) % (uint32_t)nst], ((first + t) / (uint32_t)nst) & 1u);
            r.tiles = first + (uint32_t)ntiles;
        }
        __syncthreads();
    }
    template <class F> __device__ __forceinline__ void extras(F &&f) const {
        const RowShared &r = row_shared();
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
                z = __fmul_rn(penalise_counted(c, E::load(elem_ptr<DT>(c, i), 0), c.counts[rank]), c.invT);
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
    template <class F> __device__ __forceinline__ void vectors(F &&f) const {
        extern __shared__ __align__(128) unsigned char smem[];
        const uint4 *vec = (const uint4 *)(smem + vec_off);
#pragma unroll 1
        for (int base = 0; base < nvec; base += NT) {
            const int v = base + (int)threadIdx.x;
            f(v < nvec ? vec[v] : VecTest<DT>::fill(), id0 + v * E::PER_VEC);
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
    u64 *queue;           // 64 entries per warp
};
// The front of the dynamic shared memory, whatever the kernel keeps behind it
// (the candidate list and its select bins lie where the top-N list does).
constexpr int WIDE_LIST_OFF = COMMON_BYTES, WIDE_HIST_OFF = WIDE_LIST_OFF + W_LIST * 8;
constexpr int WIDE_QUEUE_OFF = WIDE_HIST_OFF + W_BINS * 4, WIDE_BYTES = WIDE_QUEUE_OFF + NWARPS * 64 * 8;
static_assert(W_LIST_ALONE * 8 <= WIDE_HIST_OFF, "the window's list alone lies over both lists and the select bins");
constexpr int TEAM_OFF = WIDE_BYTES, SLICE_OFF = (TEAM_OFF + (int)sizeof(TeamWords) + 127) & ~127;
// (a CTA that has the row to itself: the row's own block and the ring of its passes follow)
constexpr int ROW_OFF = SLICE_OFF, WIDE_RING_OFF = (ROW_OFF + (int)sizeof(RowShared) + 127) & ~127;
__device__ __forceinline__ RowShared &row_shared() { extern __shared__ __align__(128) unsigned char smem[]; return *(RowShared *)(smem + ROW_OFF); }
__device__ __forceinline__ unsigned char *wide_stage(int st) { extern __shared__ __align__(128) unsigned char smem[]; return smem + WIDE_RING_OFF + st * WIDE_VEC_BYTES; }
// (taken from the kernel's own shared array, so that the compiler knows the address space)
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
    src.vectors([&](const uint4 &q, int) {
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
    mass_pass<DT, MODE, FLOOR>(RingSlice<DT>(), invT, zmax, zfloor, lo, shift, o.a, o.b);
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
__device__ __noinline__ Window find_window(BlockScratch *sp, TEAM tm, bool by_count, uint32_t base, int shift, double frac, u64 target, int slack_shift) {
    BlockScratch &s = *sp;
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
__device__ __forceinline__ void window_mass_pass(const RingSlice<DT> &, float invT, float zmax, float zfloor, uint32_t lo, int shift, u64 &ahead) {
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
__device__ __noinline__ bool narrow_window(BlockScratch *sp, SRC src, TEAM tm, float invT, float zmax, float zfloor, bool by_count, u64 target,
                                           uint32_t cap, Window *wp) {
    BlockScratch &s = *sp;
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
            ahead = block_sum_u64(s, ahead);
            kmax = (uint32_t)block_max_u64(s, kmax);
            kmin = ~(uint32_t)block_max_u64(s, ~kmin);
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
                const Window t = find_window(sp, tm, true, 0u, TIE_SHIFT, 0.0, (rest + each - 1) / each, 1);
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
        ahead = block_sum_u64(s, ahead);
        if ((int)threadIdx.x < tm.size) *tm.at(&tm.x->ahead[tm.rank], (int)threadIdx.x) = ahead;
        tm.sync();
        ahead = warp_total(lane < tm.size ? tm.x->ahead[lane] : 0ull);
        const u64 before = w.before;
        const u64 rest = by_count ? target - before : (target > ahead ? target - ahead : 1ull);
        w = find_window(sp, tm, by_count, w.lo, shift, 0.0, rest, by_count ? 0 : 11);
        if (!w.found) return false;
        w.before += before;                              // (a count; by mass the next level measures it anew)
    }
    w.ahead_most = ahead_most;
    *wp = w;
    return w.most <= cap;
}

// ------------------------------------------------------------------ the race

// N blocks of the generator at once share its key schedule; each product is one wide multiplication.
template <int N>
__device__ __forceinline__ void philox_blocks(uint64_t seed, uint32_t R, uint64_t step, uint32_t block, uint32_t (&w)[4 * N]) {
    uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    uint32_t c0[N], c1[N], c2[N], c3[N];
#pragma unroll
    for (int n = 0; n < N; ++n) { c0[n] = block + n; c1[n] = R; c2[n] = (uint32_t)step; c3[n] = (uint32_t)(step >> 32); }
#pragma unroll
    for (int i = 0; i < 10; ++i) {
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
    __device__ __forceinline__ void start() { K = 3.0e34f; seen = 0; G = 0; z = 0.0f; }
    __device__ __forceinline__ void refresh(const uint32_t *best) {
        const uint32_t now = *(const volatile uint32_t *)best;
        if (now != seen) { seen = now; K = fminf(1.0001f * ex2_ftz(-unkey(now) * 1.4426950408889634f), 3.0e34f); }
    }
    __device__ __forceinline__ void take(uint32_t *best, int i, float z_, float g) {
        const u64 g64 = ((u64)orderable_f32(g) << 32) | (uint32_t)(~(uint32_t)i);
        if (g64 > G) {
            G = g64; z = z_;
            if ((uint32_t)(g64 >> 32) > *(volatile uint32_t *)best) atomicMax(best, (uint32_t)(g64 >> 32));
        }
    }
};
__device__ __forceinline__ float unit_above(uint32_t w) { return __uint_as_float((w >> 9) | 0x3F800000u); }      // 1 + (v rounded down)
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
// OFF: id of a vector's first element modulo 4 (the generator's blocks are 4 ids).  About 20
// instructions per element, half of them Philox; vectors that could not win with the luckiest word skip it.
template <int DT, int OFF, bool CUT, class SRC>
__device__ __forceinline__ void race_all(const SRC &src, BlockScratch &s, Partial &p) {
    typedef Elem<DT> E;
    constexpr int PV = E::PER_VEC, NB = PV / 4 + (OFF ? 1 : 0);
    uint32_t *best = &s.runmax;
    const float invT = s.fa.invT, zmax = s.fa.zmax, minus0 = minus_zero(invT);
    const uint64_t seed = s.fa.seed, step = s.fa.step;
    const uint32_t R = s.fa.R;
    const uint32_t sure = CUT ? s.fa.sure : 0u, win_hi = CUT ? s.fa.win_hi : 0u;
    MassSum S;
    uint32_t n = 0;
    Racer rc;
    rc.start();
    // an element at the edge: in the window, or an equal of its first code with a lower id
    auto edge = [&](int i, float z, float t2, uint32_t f) {
        const FinalArgs &fa = s.fa;
        if (!(z >= fa.zfloor)) return;
        if (f == sure && (uint32_t)i < fa.id_lo) {
            S.add(ex2_ftz(t2)); ++n;
            const uint32_t w = race_word(seed, R, step, i);
            if (unit_above(w) <= __fmaf_rn(ex2_ftz(t2), rc.K, 1.0f)) rc.take(best, i, z, __fsub_rn(z, zmax) + nle_once(w));
        } else if (f < win_hi || (f == win_hi && (uint32_t)i <= fa.id_hi)) list_append(fa.list, fa.list_cap, &s.list_cnt, z, i);
    };
    src.vectors([&](const uint4 &q, int i0) {
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
        uint32_t w[4 * NB];
        philox_blocks<NB>(seed, R, step, (uint32_t)(i0 >> 2), w);
        uint32_t hits = 0;
#pragma unroll
        for (int j = 0; j < PV; ++j) hits |= (uint32_t)((!CUT || e[j] > 0.0f) && unit_above(w[OFF + j]) <= __fmaf_rn(e[j], rc.K, 1.0f)) << j;
        // rare after the first vectors: the exact score, one element per lane at a time, the bound renewed in between
        while (__any_sync(0xFFFFFFFFu, hits != 0)) {
            if (hits) {
                const int x = __ffs(hits) - 1;
                hits &= hits - 1;
                uint32_t wx = w[OFF];
#pragma unroll
                for (int j = 1; j < PV; ++j) wx = x == j ? w[OFF + j] : wx;
                const float z = __fmul_rn(pick_element<DT>(q, x), invT), d = __fsub_rn(z, zmax);
                if (d > -3.0e38f && unit_above(wx) <= __fmaf_rn(ex2_ftz(d * 1.4426950408889634f), rc.K, 1.0f)) rc.take(best, i0 + x, z, d + nle_once(wx));
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
        if (in) {
            S.add(ex2_ftz(t2)); ++n;
            rc.take(best, i, z, d + race_nle(seed, R, step, nullptr, i));
        } else if (f <= win_hi) edge(i, z, t2, f);        // (CUT only)
    });
    p.M = S.total(); p.n = CUT ? n : 0; p.G = rc.G; p.z = rc.z;
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
        });
    }
    src.extras([&](int i, float z) { push(i, z, z >= s.fa.zfloor); });
    work(0);
    p.M = S; p.n = n_kept; p.G = rc.G; p.z = rc.z;
    if (!REGS && lane == 0) { p.M = s.red[wid]; p.n = s.r32a[wid]; p.G = s.red2[wid]; p.z = __uint_as_float(s.r32b[wid]); }
    __syncwarp();
}

template <int DT, int OFF, bool CUT>
__device__ __noinline__ Partial solo_race_all(BlockScratch *sp) {
    Partial p;
    race_all<DT, OFF, CUT>(RingSlice<DT>(), *sp, p);
    return p;
}
template <int DT>
__device__ __noinline__ Partial solo_final_pass(BlockScratch *sp) {
    Partial p;
    final_pass<DT>(RingSlice<DT>(), *sp, p);
    return p;
}
template <int DT, bool FLOOR>
__device__ __forceinline__ void first_mass_pass(const SmemSlice<DT> &src, float invT, float zmax, float zfloor, u64 &S, u64 &S_all) {
    mass_pass<DT, FIRST_LEVEL, FLOOR>(src, invT, zmax, zfloor, F_ZERO, W_SHIFT, S, S_all);
}
template <int DT, bool FLOOR>
__device__ __forceinline__ void first_mass_pass(const RingSlice<DT> &, float invT, float zmax, float zfloor, u64 &S, u64 &S_all) {
    const PassOut o = solo_mass_pass<DT, FIRST_LEVEL, FLOOR>(invT, zmax, zfloor, F_ZERO, W_SHIFT);
    S = o.a; S_all = o.b;
}
// (out of line in clusters too: code that is fetched only when it runs leaves the other passes' code together)
template <int DT, int OFF>
__device__ __noinline__ Partial team_race_cut(SmemSlice<DT> src, BlockScratch *sp) {
    Partial p;
    race_all<DT, OFF, true>(src, *sp, p);
    return p;
}
template <int DT, int OFF, bool CUT>
__device__ __forceinline__ void run_race_all(const SmemSlice<DT> &src, BlockScratch &s, Partial &p) {
    if constexpr (CUT) p = team_race_cut<DT, OFF>(src, &s); else race_all<DT, OFF, CUT>(src, s, p);
}
template <int DT, int OFF, bool CUT>
__device__ __forceinline__ void run_race_all(const RingSlice<DT> &, BlockScratch &s, Partial &p) { p = solo_race_all<DT, OFF, CUT>(&s); }
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
template <int DT> __device__ __forceinline__ void run_final_pass(const RingSlice<DT> &, BlockScratch &s, Partial &p) { p = solo_final_pass<DT>(&s); }

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
                top = find_window(&s, tm, true, F_ZERO, W_SHIFT, 0.0, want, 0);
                ok = top.found && (u64)top.ahead_most + top.most >= want;
            }
        }
        if (topp && ok) {
            // (a member's rounding is up to 2^-12 of it, 2^-14 of the total with those of the others)
            win = find_window(&s, tm, false, F_ZERO, W_SHIFT, fmax((double)rp.top_p, 1e-12), 0ull, 14);
            ok = win.found;
        }
        if (topp && ok && win.most > (uint32_t)list_cap) {
            const u64 target = topp_target(rp.top_p, warp_total(lane < tm.size ? *tm.at(&tm.x->S[lane], 0) : 0ull));
            ok = minp ? narrow_window<DT, true>(&s, src, tm, invT, zmax, zfloor, false, target, list_cap, &win)
                      : narrow_window<DT, false>(&s, src, tm, invT, zmax, zfloor, false, target, list_cap, &win);
        }
        // (ahead of the list's last bin there are fewer than 2 num_top + 1 elements)
        const uint32_t top_cap = (uint32_t)(W_LIST - 2 * ALBIREO_MAX_NUM_TOP - 32);
        if (want_list && ok && !all_listed && top.most > top_cap)
            ok = minp ? narrow_window<DT, true>(&s, src, tm, invT, zmax, zfloor, true, want, top_cap, &top)
                      : narrow_window<DT, false>(&s, src, tm, invT, zmax, zfloor, true, want, top_cap, &top);
        if (!ok) { tm.sync(); out.status |= ROW_NOT_DONE; return out; }          // (the same in every CTA)
    }
    if (threadIdx.x == 0) { s.list_cnt = 0; s.cand_cnt = 0; }
    __syncthreads();

    Partial p;
    const bool no_cut = !topp && !minp && !want_list && !exp1_row;
    // kept elements that are a good part of the row are raced in place: 25 instructions per element of the
    // row against about 40 per kept element through the queues (`ahead_most` is up to twice their number)
    const bool dense = topp && !minp && !want_list && !exp1_row && win.ahead_most > n_fin / 4;
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
    if (no_cut) run_race<DT, false>(src, s, p);
    else if (dense) run_race<DT, true>(src, s, p);
    else run_final_pass<DT>(src, s, p);
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
    u64 S = 0, S_all = p.M;
    if (need_hist) { S = warp_total(in ? x.S[lane] : 0ull); S_all = warp_total(in ? x.S_all[lane] : 0ull); }
    else if (!minp) p.n = n_fin;
    if (topp) {
        const u64 target = topp_target(rp.top_p, S);
        const int L = close_gap(list, list_cap, n_list, (int)x.far_list);
        if (p.M >= target || L < 1 || L > list_cap) { out.status |= ROW_NOT_DONE; return out; }
        auto mass_of = [&](u64 C) { return __float2ull_rn(ex2_ftz(log2_mass(unkey((uint32_t)(C >> 32)), zmax)) * FX_SCALE); };
        Partial k;
        k.M = 0; k.n = 0; k.G = 0; k.z = 0.0f;
        auto keep = [&](u64 C, u64 own) {
            k.M += own; ++k.n;
            const float zq = unkey((uint32_t)(C >> 32));
            const float g = __fsub_rn(zq, zmax) + race_nle(rp.seed, rp.R, s.ga.step, exp1_row, comp_idx(C));
            const u64 gq = ((u64)orderable_f32(g) << 32) | (uint32_t)C;
            if (gq > k.G) { k.G = gq; k.z = zq; }
        };
        // An entry is kept while the mass ahead of it in the order, with the mass kept for sure, is short of
        // the target.  A short list: every entry adds that mass up (masses over the queues, done with by now),
        // one barrier in all; from 192 entries on a sort and a prefix sum are faster (2 us against 3 at 300).
        bool reached;
        if (L <= 192) {
            u64 *mass = ws.queue;
            if ((int)threadIdx.x < L) mass[threadIdx.x] = mass_of(list[threadIdx.x]);
            __syncthreads();
            u64 reach = 0;
            if ((int)threadIdx.x < L) {
                const u64 C = list[threadIdx.x], own = mass[threadIdx.x];
                u64 ahead = p.M;
#pragma unroll 4
                for (int q = 0; q < L; ++q) ahead += list[q] > C ? mass[q] : 0ull;
                reach = ahead + own;
                if (ahead < target) keep(C, own);
            }
            reached = __syncthreads_or(reach >= target) != 0;
        } else {
            const int P = list_sort(list, L), per = (P + NT - 1) / NT, q0 = (int)threadIdx.x * per, q1 = min(L, q0 + per);
            u64 local = 0, tot;
            for (int q = q0; q < q1; ++q) local += mass_of(list[q]);
            u64 run = p.M + block_exscan_u64(s, local, tot);
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
        const uint32_t members = full ? n_fin : s.found_cnt;
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
