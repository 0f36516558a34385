// Kept-score tabu search (chap_tabu_run): included by kernels.cu inside
// namespace chap.
//
// A move changes only the residuals of the moved column's rows, so inside one
// run the flip scores need no second evaluation from scratch: they are
// integer sums over the halves of a column, and the walk over the entries of
// the changed rows adds (term after) - (term before) to every column it
// meets (exact: the sums stay equal to a fresh evaluation).  The kept values
// live for one run: every chap_tabu_run call evaluates all of them first
// (k_keep_*).  k_search then runs the iterations in one launch of a single
// CTA or of one thread-block cluster: select, apply and walk, separated by
// __syncthreads or the cluster's hardware barrier (no spinning on memory).
//
//  * Selection: positions are summarised in blocks of kSrBlk; a block's best
//    score regardless of tabu sits in the shared memory of the CTA that owns
//    it, and only blocks the walk changed are summarised again.  The best
//    block's variable is the move when tabu and aspiration admit it;
//    otherwise the blocks that can hold the best admissible flip are scanned.
//  * Apply: one thread per row of the moved column computes the row state
//    after the move into a shared-memory record (every CTA all of them, so
//    that no list crosses CTAs; the row states are written back after the
//    walk).  A weight update records the violated rows of each CTA's blocks
//    of rows, found through a count per kSrBlk rows.
//  * Walk: the records' rows are cut into chunks of kSrChunk entries, one
//    warp per chunk.
//  * A column of more than kSrRows rows, or a weight update of many rows,
//    lists its records in global memory; when that walk is longer than
//    kSrBigWalk chunks per warp it leaves the launch and is done by the whole
//    GPU (k_search_walk).

constexpr int kSrThreads = 512;
constexpr int kSrWarps = kSrThreads / 32;
constexpr int kSrBlk = 256;      // positions of one summary block, rows of one violation count
constexpr int kSrChunk = 256;    // row entries of one walk chunk (8 per lane)
constexpr int kSrBigWalk = 16;   // chunks per warp above which the whole GPU walks
constexpr int kSrMaxCluster = 16;
constexpr int kSrRows = kSrThreads;     // rows of a move, or of a batch of a weight update, recorded in shared memory
constexpr int kSrFlipWords = 16384;     // words of the flip bits in shared memory (524,288 positions; more: in global memory)
constexpr int kSrMaxTops = 4096;        // summary blocks one CTA owns at most

// Result of a CTA or of the cluster: larger s wins, then lower var.
struct __align__(16) SrBest {
    long long s;
    int var, q;
};

struct SrShared {
    SrBest wslot[2][kSrWarps];
    SrBest slot[2][kSrMaxCluster];
    long long sum[2][kSrMaxCluster];
    int wsum[2][kSrWarps];
    int wtot[kSrWarps];                 // chunks of each warp's records
    int incl[kSrRows];                  // chunks up to and with each record, inside its warp
    int nrec;
    int nlist[2];                       // stale blocks of the iteration
    SrRec rec[kSrRows];
};

__device__ __forceinline__ bool sr_better(const SrBest &a, const SrBest &b) { return cand_better(a.s, a.var, b.s, b.var); }

// Best of the warp's lanes (s >= 0) in every lane: three warp reductions, no
// butterfly of 64-bit shuffles.
__device__ __forceinline__ SrBest sr_warp_best(SrBest b)
{
    const unsigned hi = (unsigned)((unsigned long long)b.s >> 32);
    const unsigned mhi = __reduce_max_sync(FULLMASK, hi);
    const unsigned lo = hi == mhi ? (unsigned)b.s : 0u;
    const unsigned mlo = __reduce_max_sync(FULLMASK, lo);
    const bool top = hi == mhi && lo == mlo;
    const int mv = __reduce_min_sync(FULLMASK, top ? b.var : INT_MAX);
    const unsigned who = __ballot_sync(FULLMASK, top && b.var == mv);
    const int q = __shfl_sync(FULLMASK, b.q, __ffs(who) - 1);
    return SrBest{(long long)(((unsigned long long)mhi << 32) | mlo), mv, q};
}

// The CTAs of the search: one (nct = 1) or a cluster.
struct SrTeam {
    int nct, rank, par, lg;   // nct = 2^lg
    SrShared *sh;
    __device__ __forceinline__ void sync() const
    {
        if (nct == 1) __syncthreads();
        else cooperative_groups::this_cluster().sync();
    }
    // Best of all threads of the team, in every thread; a team barrier.
    __device__ __forceinline__ SrBest best(SrBest b)
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        b = sr_warp_best(b);
        if (lane == 0) sh->wslot[par][warp] = b;
        __syncthreads();
        if (nct > 1) {
            if (warp == 0) {
                b = sr_warp_best(sh->wslot[par][lane & (kSrWarps - 1)]);
                if (lane < nct) *cooperative_groups::this_cluster().map_shared_rank(&sh->slot[par][rank], lane) = b;
            }
            sync();
            b = sh->slot[par][lane & (nct - 1)];
        } else {
            b = sh->wslot[par][lane & (kSrWarps - 1)];
        }
        par ^= 1;
        return sr_warp_best(b);
    }
    // Sum over the CTA's threads, in every thread; a CTA barrier.
    __device__ __forceinline__ int add_cta(int v)
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        v = __reduce_add_sync(FULLMASK, v);
        if (lane == 0) sh->wsum[par][warp] = v;
        __syncthreads();
        v = lane < kSrWarps ? sh->wsum[par][lane] : 0;
        par ^= 1;
        return __reduce_add_sync(FULLMASK, v);
    }
    // Sum over all threads of the team, in every thread; a team barrier.
    __device__ __forceinline__ long long add(int v)
    {
        const int lane = threadIdx.x & 31;
        const int p = par;
        long long t = add_cta(v);
        if (nct == 1) return t;
        if (threadIdx.x < nct) *cooperative_groups::this_cluster().map_shared_rank(&sh->sum[p][rank], threadIdx.x) = t;
        sync();
        t = lane < nct ? sh->sum[p][lane] : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(FULLMASK, t, o);
        return t;
    }
};

// The CTA's part of the selection state and the flip bits, in dynamic shared
// memory: per owned summary block (block b belongs to CTA b % nct, place
// b / nct) its best and a stale mark, and one bit per binary position (1: the
// flip raises x), every CTA's the same.
struct SrLocal {
    SrBest *tops;
    unsigned char *stale;
    int *list;           // stale blocks of the iteration
    unsigned *up;        // null: d.bup is read instead
    int nl;              // owned blocks
};

// Layout of the dynamic shared memory: SrShared, tops, flip bits, list, marks.
__host__ __device__ constexpr int sr_stale_offset(int nl, int flip_words)
{
    return (int)sizeof(SrShared) + nl * ((int)sizeof(SrBest) + 4) + 4 * flip_words;
}
__host__ __device__ constexpr int sr_smem_bytes(int nl, int flip_words)
{
    return sr_stale_offset(nl, flip_words) + nl;
}

__device__ __forceinline__ bool sr_up(const Dev &d, const SrLocal &L, int q)
{
    if (L.up) return (L.up[q >> 5] >> (q & 31)) & 1u;
    return __ldcg(d.bup + q) != 0;
}

// Marks the summary block of position q stale in the CTA that owns it; outside
// k_search (no CTA owns blocks) in the global marks.
__device__ __forceinline__ void sr_mark(const Search &S, const SrTeam *T, const SrLocal &L, int q)
{
    const int b = q / kSrBlk;
    if (!T) S.bdirty[b] = 1;
    else if (T->nct == 1) L.stale[b] = 1;
    else *cooperative_groups::this_cluster().map_shared_rank(&L.stale[b >> T->lg], b & (T->nct - 1)) = 1;
}

// ------------------------------------------------------------- kept values

// Row entries with the position of their column and the coefficient as int64
// (integral rows) or double bits (others); one warp per row, once per handle.
__global__ void k_keep_entries(Dev d, int *epos, long long *eval)
{
    const int lane = threadIdx.x & 31;
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < d.m; i += (gridDim.x * blockDim.x) >> 5) {
        const bool integ = d.row_int[i] != 0;
        for (long long e = d.row_ptr[i] + lane; e < d.row_ptr[i + 1]; e += 32) {
            epos[e] = d.vpos[d.col_idx[e]];
            const double a = d.row_val[e];
            eval[e] = integ ? dbl_int(a) : __double_as_longlong(a);
        }
    }
}

// The first kSrHead integral entries (row, coefficient) of every binary
// position at an address known from the position alone, so that a move's rows
// are loaded without waiting for the column pointers; once per handle.
__global__ void k_keep_heads(Dev d, Search S)
{
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < (long long)S.bc * kSrHead; t += (long long)gridDim.x * blockDim.x) {
        const int q = (int)(t / kSrHead), e = d.ci_ptr[q] + (int)(t % kSrHead);
        S.head[t] = e < d.ci_ptr[q + 1] ? make_int2(d.ci_row[e], d.ci_val[e]) : make_int2(0, 0);
    }
}

// Flip score and violation change of every binary position.
template <int G>
__global__ void __launch_bounds__(kEvalThreads) k_keep_bin(Dev d, Search S)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int CPW = 32 / G;
    const int g = lane / G, sub = lane & (G - 1);
    const int nquad = (S.bc + CPW - 1) / CPW;
    for (int qd = blockIdx.x * kEvalWarps + warp; qd < nquad; qd += gridDim.x * kEvalWarps) {
        const int q = qd * CPW + g;
        const bool live = q < S.bc;
        int j, dc;
        bool up;
        long long s;
        bin_column<G>(d, q, live, sub, j, up, s, dc);
        if (sub == 0 && live) {
            S.kS[q] = s;
            S.kD[q] = dc;
        }
    }
}

// Violated normalised rows per block of kSrBlk physical rows, and the control
// words of the search.
__global__ void __launch_bounds__(kSrBlk) k_keep_rows(Dev d, Search S)
{
    const int i = blockIdx.x * kSrBlk + threadIdx.x;
    int v1 = 0, v2 = 0;
    if (i < d.m) {
        const RowState s = d.rs[i];
        const bool integ = d.row_int[i] != 0;
        v1 = integ ? s.r > 0 : dneg(s.m1);
        v2 = s.w2 >= 0 && (integ ? s.r < 0 : dneg(s.m2));
    }
    const int n1 = __syncthreads_count(v1), n2 = __syncthreads_count(v2);
    if (threadIdx.x == 0) {
        S.vcnt[blockIdx.x] = n1 + n2;
        if (blockIdx.x == 0) *S.sc = SrCtl{};
    }
}

// ------------------------------------------------------------------- walk

// Flip terms of one entry (coefficient bits a) of a row in one state.
template <bool FP>
__device__ __forceinline__ void sr_flip(long long rb, double eps, int w1, int w2, long long a, bool up, long long &s,
                                        int &dc)
{
    if (!FP) {
        blk_int(rb, make_int2(w1, w2), up ? (int)a : -(int)a, s, dc);
    } else {
        const double r = __longlong_as_double(rb), ad = up ? __longlong_as_double(a) : dflip(__longlong_as_double(a));
        const long long m2 = __double_as_longlong(__dadd_rn(eps, r));
        blk_fp(__dsub_rn(eps, r), &m2, make_int2(w1, w2), ad, s, dc);
    }
}

// Chunk `part` of a record's row by the calling warp.  The moved column's own
// sums are not walked: the flip back changes every half's penalty by exactly
// the opposite amount, so they change sign.
template <bool FP>
__device__ __forceinline__ void sr_walk_entries(const Dev &d, const Search &S, const SrTeam *T, const SrLocal &L,
                                                const SrRec &r, int part, int moved)
{
    constexpr int PER = kSrChunk / 32;
    const int lane = threadIdx.x & 31;
    const long long e0 = r.p0 + (long long)part * kSrChunk;
    const int n = min(kSrChunk, r.len - part * kSrChunk);
    int q[PER];
    long long a[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int o = 32 * k + lane;
        q[k] = INT_MAX;
        a[k] = 0;
        if (32 * k < n && o < n) {
            q[k] = __ldg(S.epos + e0 + o);
            a[k] = __ldg(S.eval + e0 + o);
        }
    }
    bool up[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) up[k] = q[k] < S.bc ? sr_up(d, L, q[k]) : false;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        if (32 * k >= n) break;
        if (q[k] >= S.bc || q[k] == moved) continue;
        long long s0 = 0, s1 = 0;
        int d0 = 0, d1 = 0;
        sr_flip<FP>(r.r0, r.eps, r.w1, r.w2, a[k], up[k], s0, d0);
        sr_flip<FP>(r.r1, r.eps, r.w1 + (r.inc & 1), r.w2 + ((r.inc >> 1) & 1), a[k], up[k], s1, d1);
        s1 -= s0;
        d1 -= d0;
        if (s1 != 0) {
            atomicAdd(reinterpret_cast<unsigned long long *>(S.kS + q[k]), (unsigned long long)s1);
            // a fall of a score that is not its block's best leaves the best
            // as it is (only looked up where the summary is this CTA's own)
            if (s1 > 0 || !T || T->nct > 1 || L.tops[q[k] / kSrBlk].q == q[k]) sr_mark(S, T, L, q[k]);
        }
        if (d1 != 0) atomicAdd(S.kD + q[k], d1);
    }
}

__device__ __forceinline__ void sr_walk_chunk(const Dev &d, const Search &S, const SrTeam *T, const SrLocal &L,
                                              const SrRec &r, int part, int moved)
{
    if (r.integral) sr_walk_entries<false>(d, S, T, L, r, part, moved);
    else sr_walk_entries<true>(d, S, T, L, r, part, moved);
}

// Chunks first, first + stride, ... of the records listed in global memory.
__device__ __forceinline__ void sr_walk_listed(const Dev &d, const Search &S, const SrTeam *T, const SrLocal &L,
                                               unsigned nchunks, unsigned first, unsigned stride, int moved)
{
    for (unsigned c = first; c < nchunks; c += stride) {
        const int2 ch = __ldcg(S.chunk + c);
        const int4 *p = reinterpret_cast<const int4 *>(S.rec + ch.x);
        const int4 a0 = __ldcg(p), a1 = __ldcg(p + 1), a2 = __ldcg(p + 2), a3 = __ldcg(p + 3);
        SrRec r;
        r.r0 = row_r(a0);
        r.r1 = (long long)(((unsigned long long)(unsigned)a0.w << 32) | (unsigned)a0.z);
        r.eps = i4_double_lo(a1);
        r.p0 = (long long)(((unsigned long long)(unsigned)a1.w << 32) | (unsigned)a1.z);
        r.len = a2.x;
        r.w1 = a2.y;
        r.w2 = a2.z;
        r.inc = a2.w;
        r.integral = a3.x;
        sr_walk_chunk(d, S, T, L, r, ch.y, moved);
    }
}

// Prefix of the chunk counts of the first nrec records in shared memory
// (thread t: record t); a barrier must follow before sr_walk_local.
__device__ __forceinline__ void sr_count_chunks(SrShared &sh, int len)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = (len + kSrChunk - 1) / kSrChunk;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(FULLMASK, incl, o);
        if (lane >= o) incl += t;
    }
    sh.incl[threadIdx.x] = incl;
    if (lane == 31) sh.wtot[warp] = incl;
}

// Chunks first, first + stride, ... of the records in shared memory.
__device__ __forceinline__ void sr_walk_local(const Dev &d, const Search &S, const SrTeam &T, const SrLocal &L,
                                              int first, int stride, int moved)
{
    const SrShared &sh = *T.sh;
    const int lane = threadIdx.x & 31;
    int tot = lane < kSrWarps ? sh.wtot[lane] : 0;
#pragma unroll
    for (int o = 1; o < kSrWarps; o <<= 1) {
        const int t = __shfl_up_sync(FULLMASK, tot, o);
        if (lane >= o) tot += t;
    }
    const int all = __shfl_sync(FULLMASK, tot, kSrWarps - 1);
    for (int c = first; c < all; c += stride) {
        // the record of chunk c: first its warp's 32 records, then its lane
        const int w = __popc(__ballot_sync(FULLMASK, lane < kSrWarps && tot <= c));
        const int before = w > 0 ? __shfl_sync(FULLMASK, tot, w - 1) : 0;
        const int incl = sh.incl[32 * w + lane];
        const int k = __popc(__ballot_sync(FULLMASK, incl <= c - before));
        const int part = c - before - (k > 0 ? __shfl_sync(FULLMASK, incl, k - 1) : 0);
        sr_walk_chunk(d, S, &T, L, sh.rec[32 * w + k], part, moved);
    }
}

// A walk too long for the search's CTAs, by the whole GPU.
__global__ void __launch_bounds__(kSrThreads) k_search_walk(Dev d, Search S)
{
    if (!S.sc->pending) return;
    const unsigned warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = (gridDim.x * blockDim.x) >> 5;
    sr_walk_listed(d, S, nullptr, SrLocal{}, S.sc->nchunks, warp, nw, S.sc->moved);
}

// ------------------------------------------------------------------ search

// The best scores of N blocks of binary positions regardless of tabu (s = 0:
// none positive) by the calling warp, the loads of all of them in flight
// together.
template <int N>
__device__ __forceinline__ void sr_blocks(const Dev &d, const Search &S, const int (&b)[N], SrBest (&r)[N])
{
    constexpr int PER = kSrBlk / 32;
    const int lane = threadIdx.x & 31;
    long long s[N][PER];
    int v[N][PER];
#pragma unroll
    for (int n = 0; n < N; ++n)
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            const int q = b[n] * kSrBlk + 32 * k + lane;
            s[n][k] = q < S.bc ? __ldcg(S.kS + q) : 0;
            v[n][k] = q < S.bc ? __ldg(d.var_list + q) : kNoVar;
        }
#pragma unroll
    for (int n = 0; n < N; ++n) {
        // scores below 2^32 (all but those of huge weights) need one word
        unsigned big = 0, m = 0, lo[PER];
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            const int hi = (int)(s[n][k] >> 32);
            big |= hi > 0;
            lo[k] = hi == 0 ? (unsigned)s[n][k] : 0u;
            m = max(m, lo[k]);
        }
        if (!__any_sync(FULLMASK, big != 0)) {
            m = __reduce_max_sync(FULLMASK, m);
            int bv = INT_MAX, bk = 0;
#pragma unroll
            for (int k = 0; k < PER; ++k)
                if (lo[k] == m && v[n][k] < bv) { bv = v[n][k]; bk = k; }
            const int mv = __reduce_min_sync(FULLMASK, bv);
            const int src = __ffs(__ballot_sync(FULLMASK, bv == mv)) - 1;
            const int q = __shfl_sync(FULLMASK, b[n] * kSrBlk + 32 * bk + lane, src);
            r[n] = m > 0 ? SrBest{(long long)m, mv, q} : SrBest{0, kNoVar, -1};
        } else {
            r[n] = SrBest{0, kNoVar, -1};
#pragma unroll
            for (int k = 0; k < PER; ++k)
                if (s[n][k] > 0 && cand_better(s[n][k], v[n][k], r[n].s, r[n].var))
                    r[n] = SrBest{s[n][k], v[n][k], b[n] * kSrBlk + 32 * k + lane};
            r[n] = sr_warp_best(r[n]);
        }
    }
}

// Best admissible flip of one block into the lane's best.
__device__ __forceinline__ void sr_block_admissible(const Dev &d, const Search &S, const SrLocal &L, int b,
                                                    long long iter, long long nviol, long long bestnv, SrBest &best)
{
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int k = 0; k < kSrBlk / 32; ++k) {
        const int q = b * kSrBlk + 32 * k + lane;
        const long long s = q < S.bc ? __ldcg(S.kS + q) : 0;
        if (s <= 0 || s < best.s) continue;
        const SrBest c{s, __ldg(d.var_list + q), q};
        if (!sr_better(c, best)) continue;
        const int stamp = __ldcg((sr_up(d, L, q) ? d.tabu_inc : d.tabu_dec) + c.var);
        if (iter >= (long long)stamp || nviol + (long long)__ldcg(S.kD + q) < bestnv) best = c;
    }
}

// The state of row i (coefficient ai on an integral row, else af) after the
// move: its record and the change of its violation count.
__device__ __forceinline__ int sr_move_row(const Dev &d, int i, int ai, double af, double dl, long long di, SrRec &r,
                                           bool integral)
{
    const int4 *p = reinterpret_cast<const int4 *>(d.rs + i);
    const int4 s0 = __ldcg(p);
    const long long p0 = __ldg(d.row_ptr + i), p1 = __ldg(d.row_ptr + i + 1);
    r.r0 = row_r(s0);
    r.w1 = s0.z;
    r.w2 = s0.w;
    r.inc = 0;
    r.p0 = p0;
    r.len = (int)(p1 - p0);
    r.integral = integral;
    int ch;
    if (integral) {
        r.eps = 0.0;
        r.r1 = r.r0 + (long long)ai * di;
        ch = (int)(r.r1 > 0) - (int)(r.r0 > 0);
        if (r.w2 >= 0) ch += (int)(r.r1 < 0) - (int)(r.r0 < 0);
    } else {
        const int4 s1 = __ldcg(p + 1);
        r.eps = d.eps[i];
        const double r1 = __dadd_rn(__longlong_as_double(r.r0), __dmul_rn(af, dl));
        r.r1 = __double_as_longlong(r1);
        ch = (int)dneg(__dsub_rn(r.eps, r1)) - (int)dneg(i4_double_lo(s1));
        if (r.w2 >= 0) ch += (int)dneg(__dadd_rn(r.eps, r1)) - (int)dneg(i4_double_hi(s1));
    }
    return ch;
}

// Writes a moved row's state back, with its block's violation count.
__device__ __forceinline__ void sr_put_row(const Dev &d, const Search &S, int i, const SrRec &r, int ch)
{
    RowState *p = d.rs + i;
    p->r = r.r1;
    if (!r.integral) {
        const double r1 = __longlong_as_double(r.r1);
        p->m1 = __dsub_rn(r.eps, r1);
        p->m2 = __dadd_rn(r.eps, r1);
    }
    if (ch) atomicAdd(S.vcnt + i / kSrBlk, ch);
}

// Weight update of row i when it is violated: its record (len 0: it is not).
__device__ __forceinline__ bool sr_bump_row(const Dev &d, int i, SrRec &r)
{
    const int4 *p = reinterpret_cast<const int4 *>(d.rs + i);
    const int4 s0 = __ldcg(p), s1 = __ldcg(p + 1);
    const bool integ = __ldg(d.row_int + i) != 0;
    const bool v1 = integ ? row_r(s0) > 0 : dneg(i4_double_lo(s1));
    const bool v2 = s0.w >= 0 && (integ ? row_r(s0) < 0 : dneg(i4_double_hi(s1)));
    r.inc = (int)v1 | ((int)v2 << 1);
    if (!r.inc) return false;
    r.r0 = r.r1 = row_r(s0);
    r.eps = integ ? 0.0 : d.eps[i];
    r.p0 = __ldg(d.row_ptr + i);
    r.len = (int)(__ldg(d.row_ptr + i + 1) - r.p0);
    r.w1 = s0.z;
    r.w2 = s0.w;
    r.integral = integ;
    return true;
}

__device__ __forceinline__ void sr_put_weights(const Dev &d, int i, const SrRec &r)
{
    if (r.inc & 1) d.rs[i].w1 = r.w1 + 1;
    if (r.inc & 2) d.rs[i].w2 = r.w2 + 1;
}

// The chunks of a record's row listed in global memory, by the whole warp (len 0: none).
__device__ __forceinline__ void sr_list_chunks(const Search &S, int rec, int len)
{
    const int lane = threadIdx.x & 31;
    const int n = (len + kSrChunk - 1) / kSrChunk;
    int incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(FULLMASK, incl, o);
        if (lane >= o) incl += t;
    }
    const int tot = __shfl_sync(FULLMASK, incl, 31);
    if (tot == 0) return;
    unsigned base = 0;
    if (lane == 0) base = atomicAdd(&S.sc->nchunks, (unsigned)tot);
    base = __shfl_sync(FULLMASK, base, 0) + (unsigned)(incl - n);
    for (int k = 0; k < n; ++k) S.chunk[base + k] = make_int2(rec, k);
}

// Weight update of this CTA's row blocks, records in shared memory: batches of
// up to kSrRows violated rows, each walked before the next is collected.
__device__ __forceinline__ void sr_bump_local(const Dev &d, const Search &S, const SrTeam &T, const SrLocal &L)
{
    SrShared &sh = *T.sh;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int step = T.nct * kSrWarps;        // this warp's row blocks: b0 + l * step for lane l
    int b0 = T.rank + warp * T.nct, k = 0;
    unsigned mask = 0;
    bool fetched = false;
    for (;;) {
        if (threadIdx.x == 0) sh.nrec = 0;
        sh.rec[threadIdx.x].len = 0;
        __syncthreads();
        bool full = false;
        while (!full) {
            if (!fetched) {
                if (b0 >= S.nvb) break;
                const int mine = b0 + lane * step;
                mask = __ballot_sync(FULLMASK, mine < S.nvb && __ldcg(S.vcnt + mine) > 0);
                fetched = true;
            }
            if (!mask) {
                fetched = false;
                b0 += 32 * step;
                continue;
            }
            const int b = b0 + (__ffs(mask) - 1) * step;
            for (; k < kSrBlk / 32; ++k) {
                const int i = b * kSrBlk + 32 * k + lane;
                SrRec r;
                const bool v = i < d.m && sr_bump_row(d, i, r);
                const unsigned bal = __ballot_sync(FULLMASK, v);
                if (!bal) continue;
                int base = 0;
                if (lane == 0) base = atomicAdd(&sh.nrec, __popc(bal));
                base = __shfl_sync(FULLMASK, base, 0);
                // a reservation past the end is never used: the used records
                // are the ones before the first that did not fit
                if (base + __popc(bal) > kSrRows) { full = true; break; }
                if (v) {
                    sh.rec[base + __popc(bal & ((1u << lane) - 1u))] = r;
                    sr_put_weights(d, i, r);
                }
            }
            if (!full) {
                k = 0;
                mask &= mask - 1;
            }
        }
        const bool more = __syncthreads_or(full);
        sr_count_chunks(sh, sh.rec[threadIdx.x].len);
        __syncthreads();
        sr_walk_local(d, S, T, L, warp, kSrWarps, -1);
        if (!more) return;
        __syncthreads();
    }
}

// Up to max_launch iterations of the search by one CTA or one cluster.  What
// bounds it: the chain of dependent L2 loads of an iteration (stale blocks ->
// column -> row states -> entries -> sums, about 900 cycles each on sums that
// were just updated), not bytes or operations: hence one CTA where a move
// changes few entries (no barrier beyond the CTA), lists and summaries in
// shared memory, reductions by redux.  Set cover of 200k variables, 8 nonzeros
// a row: 5.0 us an iteration against 18.7 us for a full pass, apply and
// weight update as three graph nodes; of 2k variables: 4.0 us against 11.
__global__ void __launch_bounds__(kSrThreads, 1) k_search(Dev d, Search S, int nct, int max_launch)
{
    extern __shared__ __align__(16) unsigned char sr_smem[];
    SrShared &sh = *reinterpret_cast<SrShared *>(sr_smem);
    SrTeam T{nct, nct == 1 ? 0 : (int)cooperative_groups::this_cluster().block_rank(), 0, __ffs(nct) - 1, &sh};
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nw = nct * kSrWarps;
    const int gw = warp * nct + T.rank;   // neighbouring work items go to different SMs
    SrLocal L;
    L.nl = (S.nblk + nct - 1) / nct;
    L.tops = reinterpret_cast<SrBest *>(sr_smem + sizeof(SrShared));
    L.up = S.flip_words ? reinterpret_cast<unsigned *>(L.tops + L.nl) : nullptr;
    L.list = reinterpret_cast<int *>(L.tops + L.nl) + S.flip_words;
    L.stale = sr_smem + sr_stale_offset(L.nl, S.flip_words);
    Ctl *c = d.ctl;
    long long iter = __ldcg(&c->iter), nviol = __ldcg(&c->nviol), bestnv = __ldcg(&c->best_nviol);
    long long feas = __ldcg(&c->feasible_iter), moves = __ldcg(&c->moves), bumps = __ldcg(&c->bumps);
    const long long max_iter = __ldcg(&c->max_iter);
    const int stop = __ldcg(&c->stop_at_feasible);
    int done = __ldcg(&c->done);
    if (done) return;   // the same for every CTA: written only at the end of a launch
    unsigned long long t_feas = 0;
    int last_dc = 0;
    bool last_up = false;
    SrBest b{0, kNoVar, 0};
    bool pending = false;
    for (int l = threadIdx.x; l < L.nl; l += kSrThreads) {
        const int g = l * nct + T.rank;
        SrBest t{0, kNoVar, 0};
        bool st = false;
        if (g < S.nblk) {
            const int2 vq = S.bV[g];
            t = SrBest{S.bS[g], vq.x, vq.y};
            st = S.bdirty[g] != 0;
        }
        L.tops[l] = t;
        L.stale[l] = st;
    }
    if (threadIdx.x < 2) sh.nlist[threadIdx.x] = 0;
    for (int w0 = warp * 32; w0 < S.flip_words; w0 += kSrThreads) {
        // 32 words by a warp: lane k's ballots give word w0 + k
        for (int k = 0; k < 32 && w0 + k < S.flip_words; ++k) {
            const int q = 32 * (w0 + k) + lane;
            const unsigned word = __ballot_sync(FULLMASK, q < S.bc && d.bup[q] != 0);
            if (lane == 0) L.up[w0 + k] = word;
        }
    }
    T.sync();   // every CTA has read the control words before they are written
    if (T.rank == 0 && threadIdx.x == 0) {
        S.sc->pending = 0;
        S.sc->nchunks = 0;
        S.sc->nrec = 0;
    }
    for (int it = 0; it < max_launch && !done && !pending; ++it) {
        // ---- select: the stale blocks are listed and summarised again by the
        // warps in turn, two at a time
        for (int l0 = 32 * warp; l0 < L.nl; l0 += kSrThreads) {
            const bool st = l0 + lane < L.nl && L.stale[l0 + lane];
            const unsigned m = __ballot_sync(FULLMASK, st);
            if (!m) continue;
            int at = 0;
            if (lane == 0) at = atomicAdd(&sh.nlist[it & 1], __popc(m));
            at = __shfl_sync(FULLMASK, at, 0);
            if (st) L.list[at + __popc(m & ((1u << lane) - 1u))] = l0 + lane;
        }
        b = SrBest{0, kNoVar, 0};
        for (int l = threadIdx.x; l < L.nl; l += kSrThreads) {
            const SrBest t = L.tops[l];
            if (t.s > 0 && sr_better(t, b) && !L.stale[l]) b = t;
        }
        __syncthreads();
        const int nlist = sh.nlist[it & 1];
        if (threadIdx.x == 0) sh.nlist[(it + 1) & 1] = 0;
        for (int l0 = warp; l0 < nlist; l0 += 2 * kSrWarps) {
            const int l1 = L.list[l0];
            if (l0 + kSrWarps < nlist) {
                const int l2 = L.list[l0 + kSrWarps];
                SrBest r[2];
                sr_blocks<2>(d, S, {l1 * nct + T.rank, l2 * nct + T.rank}, r);
                if (lane == 0) {
                    L.tops[l1] = r[0];
                    L.tops[l2] = r[1];
                    L.stale[l1] = L.stale[l2] = 0;
                }
                if (r[0].s > 0 && sr_better(r[0], b)) b = r[0];
                if (r[1].s > 0 && sr_better(r[1], b)) b = r[1];
            } else {
                SrBest r[1];
                sr_blocks<1>(d, S, {l1 * nct + T.rank}, r);
                if (lane == 0) {
                    L.tops[l1] = r[0];
                    L.stale[l1] = 0;
                }
                if (r[0].s > 0 && sr_better(r[0], b)) b = r[0];
            }
        }
        b = T.best(b);
        // everything that depends only on the position is loaded at once
        int dc = 0, e0 = 0, e1 = 0, f0 = 0, f1 = 0;
        int2 head = make_int2(0, 0);   // this thread's entry of the column's integral part
        bool up = false;
        if (b.s > 0) {
            up = sr_up(d, L, b.q);
            dc = __ldcg(S.kD + b.q);
            const int ti = __ldcg(d.tabu_inc + b.var), td = __ldcg(d.tabu_dec + b.var);
            e0 = __ldg(d.ci_ptr + b.q); e1 = __ldg(d.ci_ptr + b.q + 1);
            f0 = __ldg(d.cf_ptr + b.q); f1 = __ldg(d.cf_ptr + b.q + 1);
            if (threadIdx.x < kSrHead) head = __ldg(S.head + (size_t)b.q * kSrHead + threadIdx.x);
            if (!(iter >= (long long)(up ? ti : td) || nviol + (long long)dc < bestnv)) {
                // the best flip is tabu: scan the blocks that can hold the
                // best admissible one
                SrBest a{0, kNoVar, 0};
                for (int l = warp; l < L.nl; l += kSrWarps) {
                    const long long top = L.tops[l].s;
                    if (top > 0 && __any_sync(FULLMASK, top >= a.s))
                        sr_block_admissible(d, S, L, l * nct + T.rank, iter, nviol, bestnv, a);
                }
                b = T.best(a);
                if (b.s > 0) {
                    up = sr_up(d, L, b.q);
                    dc = __ldcg(S.kD + b.q);
                    e0 = __ldg(d.ci_ptr + b.q); e1 = __ldg(d.ci_ptr + b.q + 1);
                    f0 = __ldg(d.cf_ptr + b.q); f1 = __ldg(d.cf_ptr + b.q + 1);
                    if (threadIdx.x < kSrHead) head = __ldg(S.head + (size_t)b.q * kSrHead + threadIdx.x);
                }
            }
        }
        // ---- apply the move, or the weight update
        const bool move = b.s > 0;
        const int nI = e1 - e0, len = nI + (f1 - f0);
        const bool local = move ? len <= kSrRows : nviol <= 4LL * kSrRows * nct;
        const double dl = up ? 1.0 : -1.0;
        const long long di = up ? 1 : -1;
        const int moved = move ? b.q : -1;
        last_up = up;
        last_dc = dc;
        SrRec rec;
        int row = -1, ch = 0;
        long long dnv = 0;
        unsigned nch = 0;
        if (move && local) {
            rec.len = 0;
            if ((int)threadIdx.x < len) {
                const bool integ = (int)threadIdx.x < nI;
                const int e = integ ? e0 + (int)threadIdx.x : f0 + ((int)threadIdx.x - nI);
                if (integ && threadIdx.x < kSrHead) {
                    row = head.x;
                    ch = sr_move_row(d, row, head.y, 0.0, dl, di, rec, true);
                } else {
                    row = integ ? __ldg(d.ci_row + e) : __ldg(d.cf_row + e);
                    ch = sr_move_row(d, row, integ ? __ldg(d.ci_val + e) : 0, integ ? 0.0 : __ldg(d.cf_val + e), dl,
                                     di, rec, integ);
                }
                sh.rec[threadIdx.x] = rec;
            }
            sr_count_chunks(sh, rec.len);
            dnv = T.add_cta(ch);
        } else if (move) {
            int t = 0;
            for (int v0 = 32 * gw; v0 < len; v0 += 32 * nw) {
                const int v = v0 + lane;
                int rl = 0;
                if (v < len) {
                    const bool integ = v < nI;
                    const int e = integ ? e0 + v : f0 + (v - nI);
                    const int i = integ ? __ldg(d.ci_row + e) : __ldg(d.cf_row + e);
                    SrRec r;
                    const int h = sr_move_row(d, i, integ ? __ldg(d.ci_val + e) : 0, integ ? 0.0 : __ldg(d.cf_val + e),
                                              dl, di, r, integ);
                    sr_put_row(d, S, i, r, h);
                    S.rec[v] = r;
                    rl = r.len;
                    t += h;
                }
                sr_list_chunks(S, v, rl);
            }
            dnv = T.add(t);
            nch = __ldcg(&S.sc->nchunks);
        } else if (!local) {
            for (int i0 = 32 * gw; i0 < d.m; i0 += 32 * nw) {
                const int i = i0 + lane;
                SrRec r;
                r.len = 0;
                const bool v = i < d.m && sr_bump_row(d, i, r);
                const unsigned bal = __ballot_sync(FULLMASK, v);
                if (!bal) continue;
                int base = 0;
                if (lane == 0) base = (int)atomicAdd(&S.sc->nrec, (unsigned)__popc(bal));
                const int k = __shfl_sync(FULLMASK, base, 0) + __popc(bal & ((1u << lane) - 1u));
                if (v) {
                    sr_put_weights(d, i, r);
                    S.rec[k] = r;
                }
                sr_list_chunks(S, k, v ? r.len : 0);
            }
            T.sync();
            nch = __ldcg(&S.sc->nchunks);
        }
        nviol += dnv;
        iter += 1;
        if (move) moves += 1;
        else bumps += 1;
        if (nviol < bestnv) bestnv = nviol;
        if (nviol == 0 && feas < 0) {
            feas = iter;
            t_feas = global_ns();
        }
        done = (stop && nviol == 0) || iter >= max_iter;
        // ---- walk the changed rows
        if (!move && local) sr_bump_local(d, S, T, L);
        pending = nch > (unsigned)(kSrBigWalk * nw);
        if (!done) {
            if (nch) {
                if (!pending) sr_walk_listed(d, S, &T, L, nch, (unsigned)gw, (unsigned)nw, moved);
            } else if (move) {
                sr_walk_local(d, S, T, L, gw, nw, moved);
            }
        }
        T.sync();
        // every CTA has read the old row states: the new ones are written
        // (read again only after the next selection's barrier)
        if (row >= 0 && ((int)threadIdx.x & (nct - 1)) == T.rank) sr_put_row(d, S, row, rec, ch);
        if (threadIdx.x == kSrThreads - 1 && move) {
            if (L.up) L.up[b.q >> 5] ^= 1u << (b.q & 31);
            const int bb = b.q / kSrBlk;
            if ((bb & (nct - 1)) == T.rank) L.stale[bb >> T.lg] = 1;
            if (T.rank == 0) {
                S.kS[b.q] = -b.s;
                S.kD[b.q] = -dc;
                d.x[b.var] = up ? 1.0 : 0.0;
                d.bup[b.q] = up ? 0 : 1;
                (up ? d.tabu_dec : d.tabu_inc)[b.var] = (int)(iter + d.tenure);
            }
        }
        if (T.rank == 0 && threadIdx.x == 0 && nch && !pending) {
            S.sc->nchunks = 0;
            S.sc->nrec = 0;
        }
    }
    for (int l = threadIdx.x; l < L.nl; l += kSrThreads) {
        const int g = l * nct + T.rank;
        if (g < S.nblk) {
            const SrBest t = L.tops[l];
            S.bS[g] = t.s;
            S.bV[g] = make_int2(t.var, t.q);
            S.bdirty[g] = L.stale[l];
        }
    }
    if (T.rank == 0 && threadIdx.x == 0) {
        c->iter = iter;
        c->nviol = nviol;
        c->best_nviol = bestnv;
        c->moves = moves;
        c->bumps = bumps;
        if (t_feas != 0) {
            c->feasible_iter = feas;
            c->t_feas_ns = t_feas;
        }
        c->done = done;
        const bool move = b.s > 0;
        c->mv_var = move ? b.var : -1;
        c->mv_s = move ? b.s : 0;
        c->mv_dc = move ? last_dc : 0;
        c->mv_new = move ? (last_up ? 1.0 : 0.0) : 0.0;
        c->mv_old = move ? (last_up ? 0.0 : 1.0) : 0.0;
        S.sc->moved = move ? b.q : -1;
        S.sc->pending = pending && !done;
    }
}
