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
//    entry is the move when tabu and aspiration admit it; otherwise the blocks
//    that can hold the best admissible one are scanned.
//  * A short non-binary column keeps its best shift while none of its halves
//    change, and else an upper bound of its score (of every value's: a later
//    change of a row moves candidates to values that were none); it is evaluated
//    again (Algorithm 1, one warp) only when that bound reaches the best score
//    found.
//    A counting-sorted column keeps its bins.
//  * Apply: one thread per row of the moved column computes the row state
//    after the move into a shared-memory record (every CTA all of them, so
//    that no list crosses CTAs; the row states are written back after the
//    walk).  A weight update records the violated rows of each CTA's blocks
//    of rows, found through a count per kSrBlk rows.
//  * Walk: a row's entries are stored binary columns first; the records' rows
//    are cut into chunks of entries of one kind, one warp per chunk.  A row
//    whose residual lies farther from 0, before and after, than any entry of
//    a kind can move it changes no sum of that kind and is not walked.
//  * A column of more than kSrRows rows, a walk of more than kSrBigWalk chunks
//    per warp or a weight update of many rows leaves the launch and is done by
//    the whole GPU (k_search_big, k_search_put).

constexpr int kSrThreads = kSrMaxRows;
constexpr int kSrWarps = kSrThreads / 32;
constexpr int kSrBlk = kSrBlkPos;   // positions of one summary block, rows of one violation count
constexpr int kSrChunkB = 256;   // binary entries of one walk chunk (8 per lane)
constexpr int kSrChunkN = 128;   // other entries of one (4 per lane: each brings its 16-byte context)
constexpr int kSrBigWalk = 6;    // chunks per warp above which the whole GPU walks
constexpr int kSrBigThreads = 256;
constexpr int kSrMaxCluster = 16;
constexpr int kSrRows = kSrThreads;     // rows of a move, or of a batch of a weight update, recorded in shared memory
constexpr int kSrFlipWords = 16384;     // words of the flip bits in shared memory (524,288 positions; more: in global memory)
constexpr int kSrMaxTops = 4096;        // summary blocks one CTA owns at most
constexpr int kSrMaxHist = 512;         // counting-sorted columns at most (their contexts sit in shared memory)

// Result of a CTA or of the cluster: larger s wins, then lower var.
struct __align__(16) SrBest {
    long long s;
    int var, q;
};

// A move of any column: SrBest with the new value and the violation change.
struct __align__(16) SrMove {
    long long s;
    int var, q;
    double xh;
    int dc, pad;
};

struct SrShared {
    SrMove mwslot[kSrWarps];
    SrMove mslot[kSrMaxCluster];
    SrMovedCtx mc;                      // contexts of the moved non-binary column before and after
    int ncand;                          // non-binary columns to evaluate
    long long found;                    // best score their evaluation has found
    SrBest wslot[2][kSrWarps];
    SrBest slot[2][kSrMaxCluster];
    unsigned wu[2][kSrWarps];           // largest bounds, saturated to 32 bits
    unsigned su[2][kSrMaxCluster];
    int wsum[2][kSrWarps];
    int wtot[kSrWarps];                 // chunks of each warp's records
    int incl[kSrRows];                  // chunks up to and with each record, inside its warp
    int nrec;
    int nlist[2];                       // stale blocks of the iteration
    long long rev;                      // the flip back of the moved binary column against the opposite of the
    int revc;                           // move: score and violation change (0 but for rounding)
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

__device__ __forceinline__ SrMove sr_warp_move(SrMove m)
{
    const int lane = threadIdx.x & 31;
    const SrBest b = sr_warp_best(SrBest{m.s, m.var, lane});   // q: the lane it comes from
    m.s = b.s;
    m.var = b.var;
    m.q = __shfl_sync(FULLMASK, m.q, b.q);
    m.xh = __shfl_sync(FULLMASK, m.xh, b.q);
    m.dc = __shfl_sync(FULLMASK, m.dc, b.q);
    return m;
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
    // Best of all threads of the team and the largest u, in every thread; a
    // team barrier.
    __device__ __forceinline__ SrBest best(SrBest b, unsigned &u)
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        b = sr_warp_best(b);
        u = __reduce_max_sync(FULLMASK, u);
        if (lane == 0) {
            sh->wslot[par][warp] = b;
            sh->wu[par][warp] = u;
        }
        __syncthreads();
        if (nct > 1) {
            if (warp == 0) {
                b = sr_warp_best(sh->wslot[par][lane & (kSrWarps - 1)]);
                u = __reduce_max_sync(FULLMASK, sh->wu[par][lane & (kSrWarps - 1)]);
                if (lane < nct) {
                    *cooperative_groups::this_cluster().map_shared_rank(&sh->slot[par][rank], lane) = b;
                    *cooperative_groups::this_cluster().map_shared_rank(&sh->su[par][rank], lane) = u;
                }
            }
            sync();
            b = sh->slot[par][lane & (nct - 1)];
            u = sh->su[par][lane & (nct - 1)];
        } else {
            b = sh->wslot[par][lane & (kSrWarps - 1)];
            u = sh->wu[par][lane & (kSrWarps - 1)];
        }
        par ^= 1;
        u = __reduce_max_sync(FULLMASK, u);
        return sr_warp_best(b);
    }
    // The same for moves of any column (one call between two uses of best()).
    __device__ __forceinline__ SrMove best(const SrMove &m)
    {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        SrMove r = sr_warp_move(m);
        if (lane == 0) sh->mwslot[warp] = r;
        __syncthreads();
        if (nct > 1) {
            if (warp == 0) {
                r = sr_warp_move(sh->mwslot[lane & (kSrWarps - 1)]);
                if (lane < nct) *cooperative_groups::this_cluster().map_shared_rank(&sh->mslot[rank], lane) = r;
            }
            sync();
            r = sh->mslot[lane & (nct - 1)];
        } else {
            r = sh->mwslot[lane & (kSrWarps - 1)];
        }
        return sr_warp_move(r);
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
    // short non-binary columns: per owned block the best kept result, the
    // largest bound of the others (saturated) and a stale mark; the columns to
    // evaluate with their bounds; the warps' entry lists
    SrBest *ntops;
    unsigned *nbound;
    unsigned char *nstale;
    unsigned short *cand;
    unsigned *candu;
    SEnt *stage;
    SrBest *htops;       // kept results of the owned counting-sorted columns (column k: CTA k % nct, place k / nct)
    KeepCtx *hc;         // contexts of the counting-sorted columns
    int nnl;
};

// Layout of the dynamic shared memory (pointers when base is given): SrShared,
// then by decreasing alignment.  Returns its size.
__host__ __device__ inline int sr_layout(const Search &S, int nct, unsigned char *base, SrLocal &L)
{
    L.nl = (S.nblk + nct - 1) / nct;
    L.nnl = (S.nnblk + nct - 1) / nct;
    int at = (int)sizeof(SrShared);
    auto take = [&](int bytes) { const int o = at; at += bytes; return base ? base + o : nullptr; };
    L.hc = reinterpret_cast<KeepCtx *>(take(S.nhist * (int)sizeof(KeepCtx)));
    L.stage = reinterpret_cast<SEnt *>(take(S.mix ? kSrWarps * kWarpListMax * (int)sizeof(SEnt) : 0));
    L.tops = reinterpret_cast<SrBest *>(take(L.nl * (int)sizeof(SrBest)));
    L.ntops = reinterpret_cast<SrBest *>(take(L.nnl * (int)sizeof(SrBest)));
    L.htops = reinterpret_cast<SrBest *>(take((S.nhist + nct - 1) / nct * (int)sizeof(SrBest)));
    L.nbound = reinterpret_cast<unsigned *>(take(L.nnl * 4));
    L.candu = reinterpret_cast<unsigned *>(take(L.nnl * kSrBlk * 4));
    L.up = reinterpret_cast<unsigned *>(take(S.flip_words * 4));
    if (!S.flip_words) L.up = nullptr;
    L.list = reinterpret_cast<int *>(take(L.nl * 4));
    L.cand = reinterpret_cast<unsigned short *>(take(L.nnl * kSrBlk * 2));
    L.stale = take(L.nl);
    L.nstale = take(L.nnl);
    return at;
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

// The same for the short non-binary column at place p (outside k_search
// nothing: a launch takes all their summaries again).
__device__ __forceinline__ void sr_nmark(const SrTeam *T, const SrLocal &L, int p)
{
    const int b = p / kSrBlk;
    if (!T) return;
    if (T->nct == 1) L.nstale[b] = 1;
    else *cooperative_groups::this_cluster().map_shared_rank(&L.nstale[b >> T->lg], b & (T->nct - 1)) = 1;
}

// --------------------------------------------- bounds of non-binary columns
//
// A short non-binary column keeps, instead of its score, an upper bound of the
// score of every value left of xbar and of every value right of it: the sum
// over its halves of the largest penalty change the half can give on that
// side.  A half that is violated improves towards one side, by 2w when its
// breakpoint can lie inside the bounds, else by w, and loses w on the other;
// a satisfied half gives 0 on one side and on the other 0, or -2w when every
// step violates it.  "Can" is decided by float products with a relative
// margin of 1e-5 (and the rounding of a continuous breakpoint), on the safe
// side.  Only a column whose bound reaches the best score found is evaluated.
//
// A half whose breakpoint is certainly outside the bounds, or certainly at
// the first step, has the same penalty change at every candidate of a side
// (decided); a change of its residual that leaves it so leaves the column's
// scores as they are.  On a continuous column the candidate of a satisfied row,
// its tight point, lies eps / |a| before its breakpoint: it has to be outside
// too, or it moves.

struct SrTerm {
    int l, r;       // largest penalty change left and right of xbar, in weights
    bool decided;
};

// Half with magnitude |m| of its margin (m = eps - r; |r| on an integral row),
// violated V, coefficient sign P (a > 0) and magnitude |a|; tf: of a satisfied
// half, at most |m| and, where it has a tight point, |r|; ok: the magnitudes are
// usable floats.
__device__ __forceinline__ SrTerm sr_term(bool V, bool P, float mf, float tf, float af, bool ok, const NbCtx &c)
{
    const float to = V == P ? c.dl : c.dh;        // distance to the bound the breakpoint lies towards
    const float reach = af * to * 1.00001f + c.tol * af, lo = (V ? mf : tf) * 0.99999f;
    const bool outside = ok && reach < lo;        // the breakpoint is past that bound
    SrTerm t;
    if (V) {
        const int up = outside ? 1 : 2;
        t.l = P ? up : -1;
        t.r = P ? -1 : up;
        t.decided = outside;
    } else {
        const bool first = c.isint && ok && mf * 1.00001f < af * 0.99999f;
        const int h = first ? -2 : 0;
        t.l = P ? 0 : h;
        t.r = P ? h : 0;
        t.decided = outside || first;
    }
    return t;
}

// Both halves' terms of one entry of a row in one state.
struct SrTerms {
    long long l, r;          // weighted bounds left and right
    bool v1, v2, decided;
};

template <bool FP>
__device__ __forceinline__ SrTerms sr_terms(long long rb, double eps, int w1, int w2, long long a, const NbCtx &c)
{
    SrTerms o;
    bool ok = true, P;
    float m1, m2, af;
    if (!FP) {
        o.v1 = rb > 0;
        o.v2 = rb < 0;
        P = a > 0;
        m1 = m2 = fabsf((float)rb);
        af = fabsf((float)(int)a);
    } else {
        const double rr = __longlong_as_double(rb), b1 = __dsub_rn(eps, rr), b2 = __dadd_rn(eps, rr);
        o.v1 = dneg(b1);
        o.v2 = dneg(b2);
        P = a >= 0;   // the sign bit
        m1 = fabsf(approx_f(b1, ok));
        m2 = fabsf(approx_f(b2, ok));
        af = fabsf(approx_f(__longlong_as_double(a), ok));
    }
    // |r| - eps, where a satisfied half has a tight point: nearer than it and than its margin
    const float tf = fminf(m1, m2);
    const SrTerm t = sr_term(o.v1, P, m1, tf, af, ok, c);
    o.l = (long long)t.l * w1;
    o.r = (long long)t.r * w1;
    o.decided = t.decided;
    if (w2 < 0) return o;
    const SrTerm u = sr_term(o.v2, !P, m2, tf, af, ok, c);
    o.l += (long long)u.l * w2;
    o.r += (long long)u.r * w2;
    o.decided = o.decided && u.decided;
    return o;
}

// Largest rise, over all values, of a half's penalty change when its row goes
// from violated v0 to v1 (weight w, raised by inc; falls: its residual fell):
// a violated half gives 2w or w on the side that improves it and -w on the
// other, a satisfied one 0 or -2w on the side that hurts it.
__device__ __forceinline__ long long sr_rise(bool v0, bool v1, bool falls, int w, int inc)
{
    if (v0) return v1 ? (long long)(falls ? w : 0) + 2 * inc : (long long)w;
    return v1 ? 2LL * w : (falls ? 2LL * w : 0);
}

// Context of a column at value x with bounds [lb, ub].
__device__ __forceinline__ NbCtx sr_nbctx(double x, double lb, double ub, bool isint)
{
    NbCtx c;
    bool ok = true;
    const double a = __dsub_rn(x, lb), b = __dsub_rn(ub, x);
    c.dl = dfinite(a) ? approx_f(a, ok) : INFINITY;
    c.dh = dfinite(b) ? approx_f(b, ok) : INFINITY;
    bool okx = true;
    const float xa = fabsf(approx_f(x, okx));
    if (!ok) c.dl = c.dh = INFINITY;   // outside the floats: no half is decided by its distance
    c.tol = isint ? 0.0f : (okx ? xa * 1.0e-10f : INFINITY);
    c.isint = isint ? 1 : 0;
    return c;
}

__device__ __forceinline__ KeepCtx sr_histctx(double x, double lb, double ub)
{
    const long long xi = dbl_int(x);
    return KeepCtx{dbl_int(lb) - xi, dbl_int(ub) - xi, xi, 0};
}

// ------------------------------------------------------------- kept values

// Row entries with the position of their column and the coefficient as int64
// (integral rows) or double bits (others), binary columns first, columns that
// are not evaluated left out; per row the counts of both kinds and how far an
// entry of each kind can move the row's residual (rounded up).  One warp per
// row, once per handle.
__global__ void k_keep_entries(Dev d, Search S)
{
    const int lane = threadIdx.x & 31;
    const int end = S.bc + S.nnb + S.nhist;
    for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < d.m; i += (gridDim.x * blockDim.x) >> 5) {
        const bool integ = d.row_int[i] != 0;
        const long long p0 = d.row_ptr[i], p1 = d.row_ptr[i + 1];
        int nb = 0, no = 0;
        float rb = 0.0f, ro = 0.0f;
        for (long long e = p0 + lane; e < p1; e += 32) {
            const int j = d.col_idx[e], q = d.vpos[j];
            if (q >= end) continue;
            bool ok = true;
            const float a = fabsf(approx_f(d.row_val[e], ok)) * 1.0001f;
            if (q < S.bc) {
                nb += 1;
                rb = fmaxf(rb, ok ? a : INFINITY);
            } else {
                const double lb = d.lb[j], ub = d.ub[j];
                no += 1;
                float w = INFINITY;
                if (ok && dfinite(lb) && dfinite(ub)) {
                    w = (float)(ub - lb) + 1.0f + 1.0e-9f * (float)fmax(fabs(lb), fabs(ub));
                    w = a * (w * 1.0001f);
                }
                ro = fmaxf(ro, w);
            }
        }
        nb = __reduce_add_sync(FULLMASK, nb);
        no = __reduce_add_sync(FULLMASK, no);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            rb = fmaxf(rb, __shfl_xor_sync(FULLMASK, rb, o));
            ro = fmaxf(ro, __shfl_xor_sync(FULLMASK, ro, o));
        }
        if (lane == 0) S.rowinfo[i] = SrRow{p0, nb, no, rb, ro, 0, 0};
        long long ab = p0, ao = p0 + nb;
        for (long long e0 = p0; e0 < p1; e0 += 32) {
            const long long e = e0 + lane;
            const int q = e < p1 ? d.vpos[d.col_idx[e]] : INT_MAX;
            const unsigned mb = __ballot_sync(FULLMASK, q < S.bc), mo = __ballot_sync(FULLMASK, q >= S.bc && q < end);
            const unsigned below = (1u << lane) - 1u;
            if (q < end) {
                const long long at = q < S.bc ? ab + __popc(mb & below) : ao + __popc(mo & below);
                const double a = d.row_val[e];
                S.epos[at] = q;
                S.eval[at] = integ ? dbl_int(a) : __double_as_longlong(a);
            }
            ab += __popc(mb);
            ao += __popc(mo);
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
__device__ __forceinline__ void keep_bin(const Dev &d, const Search &S)
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

template <int G>
__global__ void __launch_bounds__(kEvalThreads) k_keep_bin(Dev d, Search S)
{
    keep_bin<G>(d, S);
}

constexpr long long kSrNoBound = kNoScore;   // kU of a column never evaluated
constexpr long long kSrStale = -1;           // cS of a column whose kept result no longer holds

// Contexts and bounds of the short non-binary columns: 8 lanes per column.
__global__ void __launch_bounds__(kEvalThreads) k_keep_nb(Dev d, Search S)
{
    const int lane = threadIdx.x & 31, sub = lane & 7;
    for (int p0 = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 4; p0 < S.nnb; p0 += ((gridDim.x * blockDim.x) >> 5) * 4) {
        const int p = p0 + (lane >> 3);
        const bool live = p < S.nnb;
        const int q = S.bc + (live ? p : 0);
        const int j = __ldg(d.var_list + q);
        const double x = d.x[j], lb = __ldg(d.lb + j), ub = __ldg(d.ub + j);
        const NbCtx c = sr_nbctx(x, lb, ub, __ldg(d.vtype + j) != kVarCont);
        long long l = 0, r = 0;
        const int e0 = __ldg(d.ci_ptr + q), e1 = live ? __ldg(d.ci_ptr + q + 1) : e0;
        for (int e = e0 + sub; e < e1; e += 8) {
            const int4 s0 = ld_row16(d.rs + __ldg(d.ci_row + e));
            const SrTerms t = sr_terms<false>(row_r(s0), 0.0, s0.z, s0.w, (long long)__ldg(d.ci_val + e), c);
            l += t.l;
            r += t.r;
        }
        const int f0 = __ldg(d.cf_ptr + q), f1 = live ? __ldg(d.cf_ptr + q + 1) : f0;
        for (int e = f0 + sub; e < f1; e += 8) {
            const int i = __ldg(d.cf_row + e);
            const int4 s0 = ld_row16(d.rs + i);
            const SrTerms t = sr_terms<true>(row_r(s0), d.eps[i], s0.z, s0.w, __double_as_longlong(__ldg(d.cf_val + e)), c);
            l += t.l;
            r += t.r;
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            l += __shfl_xor_sync(FULLMASK, l, o);
            r += __shfl_xor_sync(FULLMASK, r, o);
        }
        if (sub == 0 && live) {
            S.kL[p] = l;
            S.kR[p] = r;
            S.kU[p] = kSrNoBound;
            S.nctx[p] = c;
            S.side[p] = (x > lb ? 1 : 0) | (x < ub ? 2 : 0);
            S.cS[p] = kSrStale;
        }
    }
}

// Contexts and bins of the counting-sorted columns: one chunk of a column's
// nonzeros per CTA, as k_eval_hist bins them (bins and accumulators zeroed
// before).
__global__ void __launch_bounds__(kHistThreads) k_keep_hist(Dev d, Search S, const Tile *tiles)
{
    extern __shared__ __align__(16) unsigned char smem[];
    HBin *sb = reinterpret_cast<HBin *>(smem);
    const Tile tl = tiles[blockIdx.x];
    const HistCol hc = d.hcols[tl.begin];
    const ColCtx c = make_col(d, hc.pos, 0);
    const long long lo = ikey_val(c.kl);
    const int D = (int)(ikey_val(c.ku) - lo) + 1;
    for (int b = threadIdx.x; b < D; b += blockDim.x) sb[b] = HBin{0, 0, 0, 0};
    __syncthreads();
    const int v0 = tl.aux * kHistChunk, v1 = min(hc.e_end, v0 + kHistChunk);
    Acc acc{0, 0, 0, 0};
    for (int v = v0 + threadIdx.x; v < v1; v += blockDim.x) {
        Half h[2];
        gen_entry(d, c, v, acc, h[0], h[1]);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            if (h[k].type == 0) continue;
            HBin *p = sb + (int)(ikey_val(h[k].key) - lo);
            atomicAdd(reinterpret_cast<unsigned long long *>(h[k].type == 1 ? &p->spre : &p->spost), (unsigned long long)h[k].D);
            atomicAdd(h[k].type == 1 ? &p->n1 : &p->n2, 1);
        }
    }
    warp_allreduce_acc(acc);
    HistAcc *ha = S.ha + tl.begin;
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(reinterpret_cast<unsigned long long *>(&ha->beta), (unsigned long long)acc.beta);
        atomicAdd(reinterpret_cast<unsigned long long *>(&ha->alpha), (unsigned long long)acc.alpha);
        atomicAdd(&ha->beta_c, acc.beta_c);
        atomicAdd(&ha->alpha_c, acc.alpha_c);
    }
    __syncthreads();
    HBin *gb = S.hb + S.hoff[tl.begin];
    for (int b = threadIdx.x; b < D; b += blockDim.x) {
        const HBin t = sb[b];
        if (t.spre) atomicAdd(reinterpret_cast<unsigned long long *>(&gb[b].spre), (unsigned long long)t.spre);
        if (t.spost) atomicAdd(reinterpret_cast<unsigned long long *>(&gb[b].spost), (unsigned long long)t.spost);
        if (t.n1) atomicAdd(&gb[b].n1, t.n1);
        if (t.n2) atomicAdd(&gb[b].n2, t.n2);
    }
    if (tl.aux == 0 && threadIdx.x == 0) {
        S.hctx[tl.begin] = sr_histctx(c.xb, __ldg(d.lb + c.j), __ldg(d.ub + c.j));
        S.cS[S.nnb + tl.begin] = kSrStale;
    }
}

// Violated normalised rows per block of kSrBlk physical rows, and the control
// words of the search.
__device__ __forceinline__ void keep_rows(const Dev &d, const Search &S, int b)
{
    const int i = b * kSrBlk + threadIdx.x;
    int v1 = 0, v2 = 0;
    if (i < d.m) {
        const RowState s = d.rs[i];
        const bool integ = d.row_int[i] != 0;
        v1 = integ ? s.r > 0 : dneg(s.m1);
        v2 = s.w2 >= 0 && (integ ? s.r < 0 : dneg(s.m2));
    }
    const int n1 = __syncthreads_count(v1), n2 = __syncthreads_count(v2);
    if (threadIdx.x == 0) {
        S.vcnt[b] = n1 + n2;
        if (b == 0) *S.sc = SrCtl{};
    }
}

__global__ void __launch_bounds__(kSrBlk) k_keep_rows(Dev d, Search S) { keep_rows(d, S, blockIdx.x); }

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

// What a walk knows beside the records: the moved column (position, -1: a
// weight update), its contexts before and after when it is not binary, the
// counting-sorted columns' contexts.
struct SrWalk {
    int moved;
    const SrMovedCtx *mc;
    const KeepCtx *hc;
    HistAcc *ha;             // their scalars (in global memory, or a CTA's share of the changes)
};

// Changes of the moved non-binary column's own sums, per thread over a walk
// (every changed row has an entry of it: one atomic per warp instead).
struct SrOwn {
    long long a, b;
    int ac, bc;
};

__device__ __forceinline__ NbCtx sr_ctx(const Search &S, int p)
{
    const int4 v = __ldcg(reinterpret_cast<const int4 *>(S.nctx + p));
    return NbCtx{__int_as_float(v.x), __int_as_float(v.y), __int_as_float(v.z), v.w};
}

// A breakpoint entry into (sign 1) or out of (sign -1) the bins of a column.
__device__ __forceinline__ void sr_bin(HBin *bins, long long lo, const Half &h, int sign)
{
    HBin *p = bins + (int)(ikey_val(h.key) - lo);
    const long long D = sign * h.D;
    atomicAdd(reinterpret_cast<unsigned long long *>(h.type == 1 ? &p->spre : &p->spost), (unsigned long long)D);
    atomicAdd(h.type == 1 ? &p->n1 : &p->n2, sign);
}

// The halves of one entry of a counting-sorted column in one state.
template <bool FP>
__device__ __forceinline__ void sr_hist_halves(long long rb, double eps, int w1, int w2, long long a, const KeepCtx &k,
                                               Acc &acc, Half &h1, Half &h2)
{
    ColCtx c;
    c.isint = true;
    c.xbi = k.xbi;
    c.lo = k.lo;
    c.hi = k.hi;
    c.kl = ikey(k.xbi + k.lo);
    c.ku = ikey(k.xbi + k.hi);
    c.lof = k.lo > -(1LL << 22) ? small_int_f(k.lo) : -INFINITY;
    c.hif = k.hi < (1LL << 22) ? small_int_f(k.hi) : INFINITY;
    h1.type = 0;
    h2.type = 0;
    if (!FP) {
        int_half(rb, a, w1, c, acc, h1);
        if (w2 >= 0) int_half(-rb, -a, w2, c, acc, h2);
    } else {
        const double r = __longlong_as_double(rb), av = __longlong_as_double(a);
        const double m1 = __dsub_rn(eps, r), m2 = __dadd_rn(eps, r);
        fp_half(r, av, m1, m2, w1, c, acc, h1);
        if (w2 >= 0) fp_half(dflip(r), dflip(av), m2, m1, w2, c, acc, h2);
    }
}

// One entry of a counting-sorted column: bins and scalars from the row's state
// before to the one after; sums of the moved column go to own.
template <bool FP>
__device__ __noinline__ void sr_entry_hist(const Search &S, const SrRec &r, int q, long long a, const SrWalk &W,
                                           SrOwn &own)
{
    const int k = q - S.bc - S.nnb;
    const bool moved = q == W.moved;
    const KeepCtx c0 = moved ? W.mc->h[0] : W.hc[k];
    const KeepCtx c1 = moved ? W.mc->h[1] : c0;
    Half o1, o2, n1, n2;
    Acc ao{0, 0, 0, 0}, an{0, 0, 0, 0};
    sr_hist_halves<FP>(r.r0, r.eps, r.w1, r.w2, a, c0, ao, o1, o2);
    sr_hist_halves<FP>(r.r1, r.eps, r.w1 + (r.inc & 1), r.w2 + (r.inc >> 1), a, c1, an, n1, n2);
    HBin *bins = S.hb + S.hoff[k];
    const long long lo = c0.xbi + c0.lo;
    bool ch = false;
    if (o1.type != n1.type || (n1.type && (o1.key != n1.key || o1.D != n1.D))) {
        ch = true;
        if (o1.type) sr_bin(bins, lo, o1, -1);
        if (n1.type) sr_bin(bins, lo, n1, 1);
    }
    if (o2.type != n2.type || (n2.type && (o2.key != n2.key || o2.D != n2.D))) {
        ch = true;
        if (o2.type) sr_bin(bins, lo, o2, -1);
        if (n2.type) sr_bin(bins, lo, n2, 1);
    }
    an.beta -= ao.beta;
    an.alpha -= ao.alpha;
    an.beta_c -= ao.beta_c;
    an.alpha_c -= ao.alpha_c;
    if (moved) {
        own.a += an.beta;
        own.b += an.alpha;
        own.ac += an.beta_c;
        own.bc += an.alpha_c;
        return;
    }
    HistAcc *ha = W.ha + k;
    if (an.beta) atomicAdd(reinterpret_cast<unsigned long long *>(&ha->beta), (unsigned long long)an.beta);
    if (an.alpha) atomicAdd(reinterpret_cast<unsigned long long *>(&ha->alpha), (unsigned long long)an.alpha);
    if (an.beta_c) atomicAdd(&ha->beta_c, an.beta_c);
    if (an.alpha_c) atomicAdd(&ha->alpha_c, an.alpha_c);
    if (ch || an.beta || an.alpha || an.beta_c || an.alpha_c) S.cS[S.nnb + k] = kSrStale;
}

__device__ __forceinline__ void sr_own_add(const Search &S, const SrWalk &W, SrOwn &own)
{
    if (W.moved < S.bc) return;
    if (!__any_sync(FULLMASK, own.a != 0 || own.b != 0 || own.ac != 0 || own.bc != 0)) return;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        own.a += __shfl_xor_sync(FULLMASK, own.a, o);
        own.b += __shfl_xor_sync(FULLMASK, own.b, o);
    }
    own.ac = __reduce_add_sync(FULLMASK, own.ac);
    own.bc = __reduce_add_sync(FULLMASK, own.bc);
    if ((threadIdx.x & 31) != 0) return;
    const int p = W.moved - S.bc;
    if (p < S.nnb) {
        atomicAdd(reinterpret_cast<unsigned long long *>(S.kL + p), (unsigned long long)own.a);
        atomicAdd(reinterpret_cast<unsigned long long *>(S.kR + p), (unsigned long long)own.b);
    } else {
        HistAcc *ha = W.ha + (p - S.nnb);
        atomicAdd(reinterpret_cast<unsigned long long *>(&ha->beta), (unsigned long long)own.a);
        atomicAdd(reinterpret_cast<unsigned long long *>(&ha->alpha), (unsigned long long)own.b);
        atomicAdd(&ha->beta_c, own.ac);
        atomicAdd(&ha->alpha_c, own.bc);
    }
}

// What the flip back over a non-integral row gives beside the opposite of the
// move (up: of the move) over it.  On an integral row, and but for rounding on
// any, nothing: the flip back changes every half's penalty by the opposite
// amount.  But the moved residual is rounded, and from it the flip back can
// meet another side of the tolerance than the one the move started from (a
// coefficient whose last place exceeds the residual's distance to it).
__device__ __forceinline__ void sr_reverse(const SrRec &r, double a, bool up, long long &s, int &dc)
{
    sr_flip<true>(r.r0, r.eps, r.w1, r.w2, __double_as_longlong(a), up, s, dc);
    sr_flip<true>(r.r1, r.eps, r.w1, r.w2, __double_as_longlong(a), !up, s, dc);
}

// One entry of a binary column.  The moved column's own sums are not walked:
// they become the opposite of the move's, with sr_reverse on non-integral rows.
template <bool FP>
__device__ __forceinline__ void sr_entry_bin(const Search &S, const SrTeam *T, const SrLocal &L, const SrRec &r, int q,
                                             long long a, bool up, int moved)
{
    if (q == moved) return;
    long long s0 = 0, s1 = 0;
    int d0 = 0, d1 = 0;
    sr_flip<FP>(r.r0, r.eps, r.w1, r.w2, a, up, s0, d0);
    sr_flip<FP>(r.r1, r.eps, r.w1 + (r.inc & 1), r.w2 + (r.inc >> 1), a, up, s1, d1);
    s1 -= s0;
    d1 -= d0;
    if (s1 != 0) {
        atomicAdd(reinterpret_cast<unsigned long long *>(S.kS + q), (unsigned long long)s1);
        // a fall of a score that is not its block's best leaves the best as it
        // is (only looked up where the summary is this CTA's own)
        if (s1 > 0 || !T || T->nct > 1 || L.tops[q / kSrBlk].q == q) sr_mark(S, T, L, q);
    }
    if (d1 != 0) atomicAdd(S.kD + q, d1);
}

// One entry of a short non-binary column with context c.
template <bool FP>
__device__ __forceinline__ void sr_entry_nb(const Search &S, const SrTeam *T, const SrLocal &L, const SrRec &r, int q,
                                            long long a, const NbCtx &c, const SrWalk &W, SrOwn &own)
{
    const int p = q - S.bc;
    const bool mine = q == W.moved;
    const int i1 = r.inc & 1, i2 = r.inc >> 1;
    const SrTerms o = sr_terms<FP>(r.r0, r.eps, r.w1, r.w2, a, mine ? W.mc->n[0] : c);
    const SrTerms n = sr_terms<FP>(r.r1, r.eps, r.w1 + i1, r.w2 + i2, a, mine ? W.mc->n[1] : c);
    if (mine) {
        own.a += n.l - o.l;
        own.b += n.r - o.r;
        return;
    }
    if (o.decided && n.decided && o.l == n.l && o.r == n.r) return;   // the same at every value
    if (n.l != o.l) atomicAdd(reinterpret_cast<unsigned long long *>(S.kL + p), (unsigned long long)(n.l - o.l));
    if (n.r != o.r) atomicAdd(reinterpret_cast<unsigned long long *>(S.kR + p), (unsigned long long)(n.r - o.r));
    const bool falls = FP ? dgt(__longlong_as_double(r.r0), __longlong_as_double(r.r1)) : r.r0 > r.r1;
    const bool rises = FP ? dgt(__longlong_as_double(r.r1), __longlong_as_double(r.r0)) : r.r1 > r.r0;
    long long up = sr_rise(o.v1, n.v1, falls, r.w1, i1);
    if (r.w2 >= 0) up += sr_rise(o.v2, n.v2, rises, r.w2, i2);
    if (up) atomicAdd(reinterpret_cast<unsigned long long *>(S.kU + p), (unsigned long long)up);
    S.cS[p] = kSrStale;
    sr_nmark(T, L, p);
}

// Binary chunk `part` of a record's row by the calling warp.  The loops are
// not unrolled (the next two rounds' entries are loaded ahead instead): the
// search runs few warps, and the fetch of unrolled code costs it more than
// the loads.
template <bool FP>
__device__ __forceinline__ void sr_walk_bin(const Dev &d, const Search &S, const SrTeam &T, const SrLocal &L,
                                            const SrRec &r, int part, int moved)
{
    const int lane = threadIdx.x & 31;
    const int n = min(kSrChunkB, r.lenB - part * kSrChunkB);
    const int *ep = S.epos + r.p0 + (long long)part * kSrChunkB;
    const long long *ev = S.eval + r.p0 + (long long)part * kSrChunkB;
    int q0 = -1, q1 = -1;
    long long a0 = 0, a1 = 0;
    if (lane < n) { q0 = __ldg(ep + lane); a0 = __ldg(ev + lane); }
    if (lane + 32 < n) { q1 = __ldg(ep + lane + 32); a1 = __ldg(ev + lane + 32); }
#pragma unroll 1
    for (int o = lane; o - lane < n; o += 32) {
        int q2 = -1;
        long long a2 = 0;
        if (o + 64 < n) { q2 = __ldg(ep + o + 64); a2 = __ldg(ev + o + 64); }
        if (q0 >= 0) sr_entry_bin<FP>(S, &T, L, r, q0, a0, sr_up(d, L, q0), moved);
        q0 = q1; a0 = a1;
        q1 = q2; a1 = a2;
    }
}

// Chunk `part` of the other entries of a record's row.
template <bool FP>
__device__ __forceinline__ void sr_walk_other(const Search &S, const SrTeam &T, const SrLocal &L, const SrRec &r,
                                              int part, const SrWalk &W, SrOwn &own)
{
    const int lane = threadIdx.x & 31;
    const int n = min(kSrChunkN, r.lenN - part * kSrChunkN);
    const int *ep = S.epos + r.p0 + r.offN + (long long)part * kSrChunkN;
    const long long *ev = S.eval + r.p0 + r.offN + (long long)part * kSrChunkN;
    int q0 = -1, q1 = -1;
    long long a0 = 0, a1 = 0;
    NbCtx c0{};
    if (lane < n) { q0 = __ldg(ep + lane); a0 = __ldg(ev + lane); }
    if (lane + 32 < n) { q1 = __ldg(ep + lane + 32); a1 = __ldg(ev + lane + 32); }
    if (q0 >= 0 && q0 - S.bc < S.nnb) c0 = sr_ctx(S, q0 - S.bc);
#pragma unroll 1
    for (int o = lane; o - lane < n; o += 32) {
        int q2 = -1;
        long long a2 = 0;
        NbCtx c1{};
        if (q1 >= 0 && q1 - S.bc < S.nnb) c1 = sr_ctx(S, q1 - S.bc);
        if (o + 64 < n) { q2 = __ldg(ep + o + 64); a2 = __ldg(ev + o + 64); }
        if (q0 >= 0) {
            if (q0 - S.bc < S.nnb) sr_entry_nb<FP>(S, &T, L, r, q0, a0, c0, W, own);
            else sr_entry_hist<FP>(S, r, q0, a0, W, own);
        }
        q0 = q1; a0 = a1; c0 = c1;
        q1 = q2; a1 = a2;
    }
}

__device__ __forceinline__ int sr_chunks(const SrRec &r)
{
    return (r.lenB + kSrChunkB - 1) / kSrChunkB + (r.lenN + kSrChunkN - 1) / kSrChunkN;
}

// Prefix of the chunk counts of the records in shared memory (thread t: record
// t of n chunks); a barrier must follow before sr_walk_local.
__device__ __forceinline__ void sr_count_chunks(SrShared &sh, int n)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(FULLMASK, incl, o);
        if (lane >= o) incl += t;
    }
    sh.incl[threadIdx.x] = incl;
    if (lane == 31) sh.wtot[warp] = incl;
}

// Inclusive prefix of the warps' chunk counts in the first kSrWarps lanes, and
// the total.
__device__ __forceinline__ int sr_total_chunks(const SrShared &sh, int &tot)
{
    const int lane = threadIdx.x & 31;
    tot = lane < kSrWarps ? sh.wtot[lane] : 0;
#pragma unroll
    for (int o = 1; o < kSrWarps; o <<= 1) {
        const int t = __shfl_up_sync(FULLMASK, tot, o);
        if (lane >= o) tot += t;
    }
    return __shfl_sync(FULLMASK, tot, kSrWarps - 1);
}

// Chunks first, first + stride, ... of the records in shared memory.
template <bool MIX>
__device__ __forceinline__ void sr_walk_local(const Dev &d, const Search &S, const SrTeam &T, const SrLocal &L,
                                              int first, int stride, const SrWalk &W)
{
    const SrShared &sh = *T.sh;
    const int lane = threadIdx.x & 31;
    int tot;
    const int all = sr_total_chunks(sh, tot);
    SrOwn own{0, 0, 0, 0};
    for (int c = first; c < all; c += stride) {
        // the record of chunk c: first its warp's 32 records, then its lane
        const int g = __popc(__ballot_sync(FULLMASK, lane < kSrWarps && tot <= c));
        const int before = g > 0 ? __shfl_sync(FULLMASK, tot, g - 1) : 0;
        const int incl = sh.incl[32 * g + lane];
        const int k = __popc(__ballot_sync(FULLMASK, incl <= c - before));
        const int part = c - before - (k > 0 ? __shfl_sync(FULLMASK, incl, k - 1) : 0);
        const SrRec &r = sh.rec[32 * g + k];
        const int nb = (r.lenB + kSrChunkB - 1) / kSrChunkB;
        if (!MIX || part < nb) {
            if (r.integral) sr_walk_bin<false>(d, S, T, L, r, part, W.moved);
            else sr_walk_bin<true>(d, S, T, L, r, part, W.moved);
        } else {
            if (r.integral) sr_walk_other<false>(S, T, L, r, part - nb, W, own);
            else sr_walk_other<true>(S, T, L, r, part - nb, W, own);
        }
    }
    if (MIX) sr_own_add(S, W, own);
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
__device__ __noinline__ void sr_block_admissible(const Dev &d, const Search &S, const SrLocal &L, int b,
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

// Where a record's row has its entries, and how many of each kind a walk must
// visit: none of a kind when the row keeps its violations and its margins lie
// farther from 0 than any entry of the kind moves the residual (every half of
// those entries then gives the same penalty change before and after).
__device__ __forceinline__ void sr_extent(const Search &S, int i, SrRec &r)
{
    const int4 *p = reinterpret_cast<const int4 *>(S.rowinfo + i);
    const int4 a = __ldg(p), b = __ldg(p + 1);
    r.p0 = row_r(a);
    r.lenB = r.offN = a.z;
    r.lenN = a.w;
    if (r.inc) return;
    float far;
    bool ok = true, same;
    if (r.integral) {
        same = (r.r0 > 0) == (r.r1 > 0) && (r.r0 < 0) == (r.r1 < 0);
        far = fminf(fabsf((float)r.r0), fabsf((float)r.r1));
    } else {
        const double x = __longlong_as_double(r.r0), y = __longlong_as_double(r.r1);
        const double a1 = __dsub_rn(r.eps, x), b1 = __dsub_rn(r.eps, y), a2 = __dadd_rn(r.eps, x), b2 = __dadd_rn(r.eps, y);
        same = dneg(a1) == dneg(b1) && dneg(a2) == dneg(b2);
        far = fminf(fminf(fabsf(approx_f(a1, ok)), fabsf(approx_f(b1, ok))),
                    fminf(fabsf(approx_f(a2, ok)), fabsf(approx_f(b2, ok))));
    }
    far *= 0.999f;
    if (!(ok && same && far < 1.0e37f)) return;
    if (far > __int_as_float(b.x)) r.lenB = 0;
    if (far > __int_as_float(b.y)) r.lenN = 0;
}

// The state of row i (coefficient ai on an integral row, else af) after the
// move: its record and the change of its violation count.
__device__ __forceinline__ int sr_move_row(const Dev &d, const Search &S, int i, int ai, double af, double dl,
                                           long long di, SrRec &r, bool integral)
{
    const int4 *p = reinterpret_cast<const int4 *>(d.rs + i);
    const int4 s0 = __ldcg(p);
    r.r0 = row_r(s0);
    r.w1 = s0.z;
    r.w2 = s0.w;
    r.inc = 0;
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
    sr_extent(S, i, r);
    return ch;
}

// Row and coefficient v of the column at e0 / f0 (nI integral entries first).
__device__ __forceinline__ int sr_col_entry(const Dev &d, int e0, int f0, int nI, int v, int &ai, double &af)
{
    if (v < nI) {
        ai = __ldg(d.ci_val + e0 + v);
        return __ldg(d.ci_row + e0 + v);
    }
    af = __ldg(d.cf_val + f0 + (v - nI));
    return __ldg(d.cf_row + f0 + (v - nI));
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

// Weight update of row i when it is violated: its record.
__device__ __forceinline__ bool sr_bump_row(const Dev &d, const Search &S, int i, SrRec &r)
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
    r.w1 = s0.z;
    r.w2 = s0.w;
    r.integral = integ;
    sr_extent(S, i, r);
    return true;
}

__device__ __forceinline__ void sr_put_weights(const Dev &d, int i, const SrRec &r)
{
    if (r.inc & 1) d.rs[i].w1 = r.w1 + 1;
    if (r.inc & 2) d.rs[i].w2 = r.w2 + 1;
}

// Weight update of this CTA's row blocks, records in shared memory: batches of
// up to kSrRows violated rows, each walked before the next is collected.
template <bool MIX>
__device__ __noinline__ void sr_bump_local(const Dev &d, const Search &S, const SrTeam &T, const SrLocal &L)
{
    SrShared &sh = *T.sh;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int step = T.nct * kSrWarps;        // this warp's row blocks: b0 + l * step for lane l
    int b0 = T.rank + warp * T.nct, k = 0;
    unsigned mask = 0;
    bool fetched = false;
    for (;;) {
        if (threadIdx.x == 0) sh.nrec = 0;
        sh.rec[threadIdx.x].lenB = sh.rec[threadIdx.x].lenN = 0;
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
                const bool v = i < d.m && sr_bump_row(d, S, i, r);
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
        sr_count_chunks(sh, sr_chunks(sh.rec[threadIdx.x]));
        __syncthreads();
        sr_walk_local<MIX>(d, S, T, L, warp, kSrWarps, SrWalk{-1, nullptr, L.hc, S.ha});
        if (!more) return;
        __syncthreads();
    }
}

// Best shift of the counting-sorted column k from its kept bins under the tabu
// state of c, by the warp: every lane scans a run of neighbouring bins, read
// as 16-byte pieces (two bins in three).
__device__ __noinline__ VCand sr_hist_eval(const Search &S, int k, const ColCtx &c, long long nviol, long long bestnv)
{
    constexpr int U = 4;   // pairs of bins in flight per lane
    const int lane = threadIdx.x & 31;
    const long long lo = ikey_val(c.kl);
    const int D = (int)(ikey_val(c.ku) - lo) + 1;
    const int4 *gb = reinterpret_cast<const int4 *>(S.hb + S.hoff[k]);
    const HistAcc *ha = S.ha + k;
    const long long beta = __ldcg(&ha->beta), alpha = __ldcg(&ha->alpha);
    const int bc = __ldcg(&ha->beta_c), ac = __ldcg(&ha->alpha_c);
    const int pairs = (D + 1) >> 1, per = (pairs + 31) >> 5;   // an even number of bins is stored, the last one zero
    const int p0 = lane * per, p1 = min(pairs, p0 + per);
    long long P = 0;
    int Pc = 0;
    for (int p = p0; p < p1; p += U) {
        int4 v[U][3];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int w = 0; w < 3; ++w) v[u][w] = p + u < p1 ? __ldcg(gb + 3 * (p + u) + w) : make_int4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            // bins: {spre, spost}, {n1, n2, spre'}, {spost', n1', n2'}
            P += row_r(v[u][0]) + (long long)(((unsigned long long)(unsigned)v[u][0].w << 32) | (unsigned)v[u][0].z);
            P += (long long)(((unsigned long long)(unsigned)v[u][1].w << 32) | (unsigned)v[u][1].z) + row_r(v[u][2]);
            Pc += v[u][1].y - v[u][1].x + v[u][2].w - v[u][2].z;
        }
    }
    const long long mine = P;
    const int minec = Pc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long t = __shfl_up_sync(FULLMASK, P, o);
        const int tc = __shfl_up_sync(FULLMASK, Pc, o);
        if (lane >= o) { P += t; Pc += tc; }
    }
    P -= mine;
    Pc -= minec;
    VCand vb{0, 0ull, 0, 0};
    auto bin = [&](int b, long long spre, long long spost, int n1, int n2) {
        if (b < D && ((n1 | n2) != 0 || b == 0 || b == D - 1)) {
            const unsigned long long key = ikey(lo + b);
            const bool right = key > c.kxb;
            consider(vb, c, key, beta + P + spre + (right ? alpha : 0), bc + Pc - n1 + (right ? ac : 0), nviol, bestnv);
        }
        P += spre + spost;
        Pc += n2 - n1;
    };
    for (int p = p0; p < p1; p += U) {
        int4 v[U][3];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int w = 0; w < 3; ++w) v[u][w] = p + u < p1 ? __ldcg(gb + 3 * (p + u) + w) : make_int4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (p + u >= p1) break;
            bin(2 * (p + u), row_r(v[u][0]), (long long)(((unsigned long long)(unsigned)v[u][0].w << 32) | (unsigned)v[u][0].z),
                v[u][1].x, v[u][1].y);
            bin(2 * (p + u) + 1, (long long)(((unsigned long long)(unsigned)v[u][1].w << 32) | (unsigned)v[u][1].z),
                row_r(v[u][2]), v[u][2].z, v[u][2].w);
        }
    }
    warp_reduce_vc(vb, c);
    return vb;
}

// The best shift of the column at place p by the warp: with free = true
// regardless of tabu (kept), else of the admissible ones.  top: of a short
// column, the largest score of any of its values.
__device__ __forceinline__ VCand sr_eval_column(const Dev &d, const Search &S, const SrLocal &L, int p, bool free,
                                                long long iter, long long nviol, long long bestnv, double &xh,
                                                long long &top)
{
    const int warp = threadIdx.x >> 5;
    const int q = S.bc + p;
    const long long it = free ? LLONG_MAX : iter;
    VCand vb;
    top = 0;
    if (p < S.nnb) {
        vb = column_best(d, q, L.stage + warp * kWarpListMax, it, nviol, bestnv, xh, top);
    } else {
        const ColCtx c = make_col(d, q, it);
        vb = sr_hist_eval(S, p - S.nnb, c, nviol, bestnv);
        xh = vb.valid ? key_value(c, vb.key) : c.xb;
    }
    return vb;
}

// Whether a shift of variable j to xh with violation change dc is admissible.
__device__ __forceinline__ bool sr_admissible(const Dev &d, int j, double xh, int dc, long long iter, long long nviol,
                                              long long bestnv)
{
    const int stamp = __ldcg((xh > __ldcg(d.x + j) ? d.tabu_inc : d.tabu_dec) + j);
    return iter >= (long long)stamp || nviol + (long long)dc < bestnv;
}

__device__ __forceinline__ void sr_take(SrMove &m, long long s, int var, int q, double xh, int dc)
{
    if (s > 0 && cand_better(s, var, m.s, m.var)) m = SrMove{s, var, q, xh, dc, 0};
}

// Evaluates the column at place p: its best shift regardless of tabu is kept;
// the best admissible one is folded into lane 0's m.
__device__ __forceinline__ void sr_refresh(const Dev &d, const Search &S, const SrLocal &L, int p, long long iter,
                                           long long nviol, long long bestnv, SrMove &m)
{
    const int lane = threadIdx.x & 31, q = S.bc + p;
    const int j = __ldg(d.var_list + q);
    double xh;
    long long top;
    VCand v = sr_eval_column(d, S, L, p, true, iter, nviol, bestnv, xh, top);
    if (lane == 0) {
        S.cS[p] = v.valid && v.s > 0 ? v.s : 0;
        if (p < S.nnb) S.kU[p] = top;
        S.cX[p] = xh;
        S.cD[p] = v.dc;
    }
    bool ok = v.valid && v.s > 0;
    if (!ok) return;
    if (!sr_admissible(d, j, xh, v.dc, iter, nviol, bestnv)) {
        v = sr_eval_column(d, S, L, p, false, iter, nviol, bestnv, xh, top);
        ok = v.valid && v.s > 0;
    }
    if (ok && lane == 0) sr_take(m, v.s, j, q, xh, v.dc);
}

__device__ __forceinline__ unsigned sr_sat(long long u)
{
    return u <= 0 ? 0u : (u >> 32) ? 0xffffffffu : (unsigned)u;
}

// The columns of one block of short non-binary columns: kept score (0 unless
// kept and positive), saturated bound of the others, by the calling warp.
struct SrNbBlock {
    long long s[kSrBlk / 32];
    unsigned u[kSrBlk / 32];
};

__device__ __forceinline__ void sr_load_nb(const Search &S, int gb, SrNbBlock &B)
{
    constexpr int PER = kSrBlk / 32;
    const int lane = threadIdx.x & 31;
    long long kl[PER], kr[PER], ku[PER], cs[PER];
    int sd[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int p = gb * kSrBlk + 32 * k + lane;
        kl[k] = kr[k] = ku[k] = cs[k] = 0;
        sd[k] = 0;
        if (p < S.nnb) {
            kl[k] = __ldcg(S.kL + p);
            kr[k] = __ldcg(S.kR + p);
            ku[k] = __ldcg(S.kU + p);
            cs[k] = __ldcg(S.cS + p);
            sd[k] = __ldcg(S.side + p);
        }
    }
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const long long a = (sd[k] & 1) ? kl[k] : 0, b = (sd[k] & 2) ? kr[k] : 0;
        B.s[k] = max(cs[k], 0LL);
        B.u[k] = cs[k] >= 0 ? 0u : sr_sat(min(max(a, b), ku[k]));
    }
}

// Summary of owned block l: its best kept result, the largest bound of the
// columns without one.
__device__ __noinline__ void sr_summarise_nb(const Dev &d, const Search &S, const SrTeam &T, const SrLocal &L, int l)
{
    constexpr int PER = kSrBlk / 32;
    const int lane = threadIdx.x & 31, gb = (l << T.lg) + T.rank;
    SrNbBlock B;
    sr_load_nb(S, gb, B);
    SrBest r{0, kNoVar, 0};
    unsigned u = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        u = max(u, B.u[k]);
        if (B.s[k] > 0 && B.s[k] >= r.s) {
            const int q = S.bc + gb * kSrBlk + 32 * k + lane, v = __ldg(d.var_list + q);
            if (cand_better(B.s[k], v, r.s, r.var)) r = SrBest{B.s[k], v, q};
        }
    }
    r = sr_warp_best(r);
    u = __reduce_max_sync(FULLMASK, u);
    if (lane == 0) {
        L.ntops[l] = r;
        L.nbound[l] = u;
        L.nstale[l] = 0;
    }
}

// Evaluates the CTA's short columns without a kept result whose bound reaches
// thr; the best admissible results go to the lanes' m.  all: kept results are
// taken too (those whose shift is not admissible evaluated again), of the
// counting-sorted columns as well.
__device__ __noinline__ void sr_evaluate(const Dev &d, const Search &S, const SrTeam &T, const SrLocal &L,
                                            long long iter, long long nviol, long long bestnv, long long thr, bool all,
                                            SrMove &m)
{
    constexpr int PER = kSrBlk / 32;
    SrShared &sh = *T.sh;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned uthr = sr_sat(thr);
    // kept results that are admissible (lane by lane); false: to be evaluated
    auto kept = [&](int p, long long s) {
        const int q = S.bc + p, j = __ldg(d.var_list + q);
        const double xh = __ldcg(S.cX + p);
        const int dc = __ldcg(S.cD + p);
        if (!sr_admissible(d, j, xh, dc, iter, nviol, bestnv)) return false;
        sr_take(m, s, j, q, xh, dc);
        return true;
    };
    if (threadIdx.x == 0) sh.found = thr;
    for (int l = warp; l < L.nnl; l += kSrWarps) {
        if (L.nbound[l] < uthr && !(all && L.ntops[l].s >= thr)) continue;
        SrNbBlock B;
        sr_load_nb(S, (l << T.lg) + T.rank, B);
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            bool want = B.u[k] >= uthr && B.u[k] > 0;
            const bool res = all && B.s[k] >= thr;
            if (!__any_sync(FULLMASK, want || res)) continue;
            if (res && !kept(((l << T.lg) + T.rank) * kSrBlk + 32 * k + lane, B.s[k])) want = true;
            const unsigned bal = __ballot_sync(FULLMASK, want);
            if (!bal) continue;
            int at = 0;
            if (lane == 0) at = atomicAdd(&sh.ncand, __popc(bal));
            at = __shfl_sync(FULLMASK, at, 0) + __popc(bal & ((1u << lane) - 1u));
            if (want) {
                L.cand[at] = (unsigned short)(l * kSrBlk + 32 * k + lane);
                L.candu[at] = B.u[k] ? B.u[k] : 0xffffffffu;
            }
        }
    }
    if (all) {
        for (int kk = warp; kk * T.nct + T.rank < S.nhist; kk += kSrWarps) {
            if (L.htops[kk].s < thr) continue;
            const int p = S.nnb + kk * T.nct + T.rank;
            bool ok = false;
            if (lane == 0) ok = kept(p, L.htops[kk].s);
            if (!__shfl_sync(FULLMASK, (int)ok, 0)) sr_refresh(d, S, L, p, iter, nviol, bestnv, m);
        }
    }
    __syncthreads();
    const int n = sh.ncand;
    for (int i = warp; i < n; i += kSrWarps) {
        // one lane reads the bound other warps raise: the warp stays together
        unsigned f = 0;
        if (lane == 0) f = sr_sat(*reinterpret_cast<volatile long long *>(&sh.found));
        if (L.candu[i] < __shfl_sync(FULLMASK, f, 0)) continue;
        const int at = L.cand[i], l = at / kSrBlk;
        sr_refresh(d, S, L, ((l << T.lg) + T.rank) * kSrBlk + (at & (kSrBlk - 1)), iter, nviol, bestnv, m);
        if (lane == 0) {
            L.nstale[l] = 1;   // its bound is its score now
            if (m.s > 0) atomicMax(&sh.found, m.s);
        }
        __syncwarp();
    }
}

// Up to max_launch iterations of the search by one CTA or one cluster (MIX:
// there are non-binary columns).  What bounds it: the chain of dependent L2
// loads of an iteration (stale blocks -> column -> row states -> entries ->
// sums, about 900 cycles each on sums that were just updated) and the barriers
// between, not bytes or operations: hence one CTA where a move changes few
// entries, lists and summaries in shared memory, reductions by redux.  Measured
// per iteration, against a full pass, apply and weight update as graph nodes:
// set cover of 2k / 200k variables 4.2 / 6 us against 11 / 18.7 (one CTA);
// general MIP of 200k variables 38 us against 142, of 21k variables near a
// feasible point 26 to 43 us (by instance) against 110 to 140, 2M skewed columns
// with 50 dense ones (every move a dense one, done by the whole GPU) 155 us against
// 410 (16 CTAs).
// FPROWS: there may be non-integral rows.
template <bool MIX, bool FPROWS>
__device__ __forceinline__ void search_body(const Dev &d, const Search &S, int nct, int max_launch,
                                            unsigned char *sr_smem)
{
    SrShared &sh = *reinterpret_cast<SrShared *>(sr_smem);
    SrTeam T{nct, nct == 1 ? 0 : (int)cooperative_groups::this_cluster().block_rank(), 0, __ffs(nct) - 1, &sh};
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nw = nct * kSrWarps;
    const int gw = warp * nct + T.rank;   // neighbouring work items go to different SMs
    SrLocal L;
    sr_layout(S, nct, sr_smem, L);
    Ctl *c = d.ctl;
    if (__ldcg(&c->done)) return;   // the same for every CTA: written only at the end of a launch
    long long iter = __ldcg(&c->iter), nviol = __ldcg(&c->nviol), bestnv = __ldcg(&c->best_nviol);
    long long feas = __ldcg(&c->feasible_iter), moves = __ldcg(&c->moves), bumps = __ldcg(&c->bumps);
    const long long max_iter = __ldcg(&c->max_iter);
    const int stop = __ldcg(&c->stop_at_feasible);
    bool done = false, pending = false;
    unsigned long long t_feas = 0;
    SrBest b{0, kNoVar, 0};
    int dc = 0;
    double xnew = 0.0, xold = 0.0;
    // end of an iteration: counters, feasibility, stop conditions
    auto finish = [&](bool move, long long dnv) {
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
    };
    const bool resume = __ldcg(&S.sc->pending) != 0;   // the whole GPU applied the last launch's iteration
    if (resume) {
        finish(__ldcg(&S.sc->moved) >= 0, __ldcg(&S.sc->dnv));
        // the record of the last move, for the control block
        b = SrBest{__ldcg(&c->mv_s), __ldcg(&c->mv_var), __ldcg(&S.sc->moved)};
        dc = __ldcg(&c->mv_dc);
        xnew = __ldcg(&c->mv_new);
        xold = __ldcg(&c->mv_old);
        if (b.var < 0) b = SrBest{0, kNoVar, 0};
    }
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
    if (threadIdx.x == 0) {
        sh.rev = 0;
        sh.revc = 0;
    }
    if (MIX) {
        // the summaries of the non-binary columns are all taken again
        for (int l = threadIdx.x; l < L.nnl; l += kSrThreads) {
            L.ntops[l] = SrBest{0, kNoVar, 0};
            L.nbound[l] = 0;
            L.nstale[l] = l * nct + T.rank < S.nnblk;
        }
        for (int h = threadIdx.x; h < S.nhist; h += kSrThreads) L.hc[h] = S.hctx[h];
        for (int kk = threadIdx.x; kk * nct + T.rank < S.nhist; kk += kSrThreads) {
            const int p = S.nnb + kk * nct + T.rank;
            const long long s = S.cS[p];
            L.htops[kk] = s > 0 ? SrBest{s, d.var_list[S.bc + p], S.bc + p} : SrBest{0, kNoVar, 0};
        }
        if (threadIdx.x == 0) sh.ncand = 0;
    }
    for (int w0 = warp * 32; w0 < S.flip_words; w0 += kSrThreads) {
        // 32 words by a warp: the ballot of step k is word w0 + k
        for (int k = 0; k < 32 && w0 + k < S.flip_words; ++k) {
            const int q = 32 * (w0 + k) + lane;
            const unsigned word = __ballot_sync(FULLMASK, q < S.bc && d.bup[q] != 0);
            if (lane == 0) L.up[w0 + k] = word;
        }
    }
    T.sync();   // every CTA has read the control words before they are written
    if (T.rank == 0 && threadIdx.x == 0) S.sc->pending = 0;
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
        unsigned u = 0;
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
        if (MIX) {
            for (int l = kSrWarps - 1 - warp; l < L.nnl; l += kSrWarps) {
                if (L.nstale[l]) sr_summarise_nb(d, S, T, L, l);
                __syncwarp();
                const SrBest t = L.ntops[l];
                u = max(u, L.nbound[l]);
                if (t.s > 0 && sr_better(t, b)) b = t;
            }
            for (int kk = warp; kk * nct + T.rank < S.nhist; kk += kSrWarps) {
                const int p = S.nnb + kk * nct + T.rank;
                if (__ldcg(S.cS + p) < 0) {
                    double xh;
                    long long top;
                    const VCand v = sr_eval_column(d, S, L, p, true, iter, nviol, bestnv, xh, top);
                    if (lane == 0) {
                        S.cS[p] = v.valid && v.s > 0 ? v.s : 0;
                        S.cX[p] = xh;
                        S.cD[p] = v.dc;
                        L.htops[kk] = v.valid && v.s > 0 ? SrBest{v.s, __ldg(d.var_list + S.bc + p), S.bc + p}
                                                         : SrBest{0, kNoVar, 0};
                    }
                    __syncwarp();
                }
                const SrBest t = L.htops[kk];
                if (t.s > 0 && sr_better(t, b)) b = t;
            }
        }
        b = T.best(b, u);
        // everything that depends only on the position is loaded at once
        int e0 = 0, e1 = 0, f0 = 0, f1 = 0;
        int2 head = make_int2(0, 0);   // this thread's entry of a binary column's integral part
        bool up = false;
        auto meta = [&]() {
            e0 = __ldg(d.ci_ptr + b.q); e1 = __ldg(d.ci_ptr + b.q + 1);
            f0 = __ldg(d.cf_ptr + b.q); f1 = __ldg(d.cf_ptr + b.q + 1);
            if (!MIX || b.q < S.bc) {
                if (threadIdx.x < kSrHead) head = __ldg(S.head + (size_t)b.q * kSrHead + threadIdx.x);
                dc = __ldcg(S.kD + b.q);
                up = sr_up(d, L, b.q);
                xnew = up ? 1.0 : 0.0;
                xold = up ? 0.0 : 1.0;
            } else {
                xold = __ldcg(d.x + b.var);
            }
        };
        dc = 0;
        bool free = true;
        if (b.s > 0) {
            const int ti = __ldcg(d.tabu_inc + b.var), td = __ldcg(d.tabu_dec + b.var);
            if (MIX && b.q >= S.bc) {
                dc = __ldcg(S.cD + (b.q - S.bc));
                xnew = __ldcg(S.cX + (b.q - S.bc));
            }
            meta();
            free = iter >= (long long)(xnew > xold ? ti : td) || nviol + (long long)dc < bestnv;
        }
        if (!free) {
            // the best entry is tabu: scan what can hold the best admissible one
            SrBest a{0, kNoVar, 0};
            for (int l = warp; l < L.nl; l += kSrWarps) {
                const long long top = L.tops[l].s;
                if (top > 0 && __any_sync(FULLMASK, top >= a.s))
                    sr_block_admissible(d, S, L, l * nct + T.rank, iter, nviol, bestnv, a);
            }
            unsigned none = 0;
            b = T.best(a, none);
            if (b.s > 0) meta();
        }
        if (MIX && (!free || (u > 0 && u >= sr_sat(b.s)))) {
            SrMove m{b.s, b.var, b.q, xnew, dc, 0};
            sr_evaluate(d, S, T, L, iter, nviol, bestnv, b.s > 1 ? b.s : 1, !free, m);
            m = T.best(m);
            if (m.q != b.q || m.s != b.s) {
                b = SrBest{m.s, m.var, m.q};
                dc = m.dc;
                xnew = m.xh;
                meta();
            }
            if (threadIdx.x == 0) sh.ncand = 0;
        }
        // ---- apply the move, or the weight update
        const bool move = b.s > 0;
        if (MIX && move && b.q >= S.bc && threadIdx.x == 0) {
            const double lb = __ldg(d.lb + b.var), ub = __ldg(d.ub + b.var);
            const bool isint = __ldg(d.vtype + b.var) != kVarCont;
            sh.mc.n[0] = sr_nbctx(xold, lb, ub, isint);
            sh.mc.n[1] = sr_nbctx(xnew, lb, ub, isint);
            if (b.q - S.bc >= S.nnb) {
                sh.mc.h[0] = sr_histctx(xold, lb, ub);
                sh.mc.h[1] = sr_histctx(xnew, lb, ub);
            }
        }
        const int nI = e1 - e0, len = move ? nI + (f1 - f0) : 0;
        pending = move ? len > kSrRows : nviol > S.big_viol;
        const double dl = __dsub_rn(xnew, xold);
        const long long di = (long long)dl;
        const long long stamp = iter + 1 + d.tenure;
        const SrWalk W{move ? b.q : -1, &sh.mc, L.hc, S.ha};
        SrRec rec;
        int row = -1, ch = 0;
        if (move && !pending) {
            int n = 0;
            if ((int)threadIdx.x < len) {
                int ai = head.y;
                double af = 0.0;
                const bool integ = (int)threadIdx.x < nI;
                row = integ && threadIdx.x < kSrHead && (!MIX || b.q < S.bc)
                          ? head.x : sr_col_entry(d, e0, f0, nI, threadIdx.x, ai, af);
                ch = sr_move_row(d, S, row, ai, af, dl, di, rec, integ);
                sh.rec[threadIdx.x] = rec;
                n = sr_chunks(rec);
                if (FPROWS && !integ && (!MIX || b.q < S.bc)) {
                    long long rs = 0;
                    int rd = 0;
                    sr_reverse(rec, af, up, rs, rd);
                    if (rs) atomicAdd(reinterpret_cast<unsigned long long *>(&sh.rev), (unsigned long long)rs);
                    if (rd) atomicAdd(&sh.revc, rd);
                }
            }
            sr_count_chunks(sh, n);
            const int dnv = T.add_cta(ch);
            int tot;
            pending = sr_total_chunks(sh, tot) > S.big_chunks;
            if (!pending) {
                finish(true, dnv);
                if (!done) sr_walk_local<MIX>(d, S, T, L, gw, nw, W);
            }
        } else if (!move && !pending) {
            finish(false, 0);
            sr_bump_local<MIX>(d, S, T, L);
        }
        // the moved column's block is stale and its flip bit or context changes
        // (nothing of these is read before the barrier: the walk passes the
        // moved column by)
        const int place = MIX && b.q >= S.bc ? b.q - S.bc : 0;
        const bool hist = MIX && b.q >= S.bc && place >= S.nnb;
        const int own = (hist ? place - S.nnb : MIX && b.q >= S.bc ? place / kSrBlk : b.q / kSrBlk);
        const bool mine = (own & (nct - 1)) == T.rank;   // this CTA summarises the moved column
        if (threadIdx.x == kSrThreads - 1 && move && !pending) {
            if (!MIX || b.q < S.bc) {
                if (L.up) L.up[b.q >> 5] ^= 1u << (b.q & 31);
                if (mine) L.stale[own >> T.lg] = 1;
            } else if (hist) {
                L.hc[place - S.nnb] = sh.mc.h[1];
            } else if (mine) {
                L.nstale[own >> T.lg] = 1;
            }
        }
        T.sync();
        // every CTA has read the old state of the rows and of the column: the
        // new one is written (by the CTA that reads it before the next team
        // barrier, its own CTA barrier between)
        if (row >= 0 && !pending && ((int)threadIdx.x & (nct - 1)) == T.rank) sr_put_row(d, S, row, rec, ch);
        if (threadIdx.x == kSrThreads - 1 && move && mine) {
            d.x[b.var] = xnew;
            (xnew > xold ? d.tabu_dec : d.tabu_inc)[b.var] = (int)stamp;
            if (!MIX || b.q < S.bc) {
                // (the whole GPU adds a pending move's own in k_search_put)
                S.kS[b.q] = (FPROWS && !pending ? sh.rev : 0) - b.s;
                S.kD[b.q] = (FPROWS && !pending ? sh.revc : 0) - dc;
                d.bup[b.q] = up ? 0 : 1;
                if (pending) L.stale[own >> T.lg] = 1;
            } else {
                S.cS[place] = kSrStale;
                if (hist) {
                    S.hctx[place - S.nnb] = sh.mc.h[1];
                } else {
                    S.nctx[place] = sh.mc.n[1];
                    S.kU[place] = kSrNoBound;
                    S.side[place] = (xnew > __ldg(d.lb + b.var) ? 1 : 0) | (xnew < __ldg(d.ub + b.var) ? 2 : 0);
                }
            }
        }
        if (FPROWS && threadIdx.x == kSrThreads - 1) {
            sh.rev = 0;
            sh.revc = 0;
        }
    }
    __syncthreads();
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
        c->mv_dc = move ? dc : 0;
        c->mv_new = move ? xnew : 0.0;
        c->mv_old = move ? xold : 0.0;
        S.sc->moved = move ? b.q : -1;
        S.sc->dnv = 0;
        if (MIX) S.sc->mc = sh.mc;
        S.sc->pending = pending;
    }
}

template <bool MIX>
__global__ void __launch_bounds__(kSrThreads, 1) k_search(Dev d, Search S, int nct, int max_launch)
{
    extern __shared__ __align__(16) unsigned char sr_smem[];
    search_body<MIX, true>(d, S, nct, max_launch, sr_smem);
}

// Many independent searches (the chains of a batch), one CTA each: no barrier
// crosses a CTA, so a chain's iteration costs what a single search's does and
// the chains fill the GPU: 64 chains over 16 set covers of 1k to 50k variables,
// 1,000 iterations each, 7.5 ms against 76 ms with every iteration of all
// chains as three grid-wide phases (autotuned).  Their columns hold at most kSrRows entries and no
// iteration is left to the whole GPU.
__global__ void __launch_bounds__(kSrThreads, 1) k_search_chains(const ChainSearch *chains, int max_launch)
{
    extern __shared__ __align__(16) unsigned char sr_smem[];
    __shared__ ChainSearch c;
    const int *src = reinterpret_cast<const int *>(chains + blockIdx.x);
    for (int i = threadIdx.x; i < (int)(sizeof(ChainSearch) / sizeof(int)); i += kSrThreads)
        reinterpret_cast<int *>(&c)[i] = src[i];
    __syncthreads();
    search_body<false, false>(c.d, c.S, 1, max_launch, sr_smem);
}

// Kept values of every chain that is not done (grid.y strides over the chains).
template <int G>
__global__ void __launch_bounds__(kEvalThreads) k_keep_chains(const ChainSearch *chains, int n)
{
    for (int k = blockIdx.y; k < n; k += gridDim.y) {
        const ChainSearch &c = chains[k];
        if (c.d.ctl->done) continue;
        if (c.S.nvb == 0 && blockIdx.x == 0 && threadIdx.x == 0) *c.S.sc = SrCtl{};   // keep_rows does it where there are rows
        keep_bin<G>(c.d, c.S);
        for (int b = blockIdx.x; b < c.S.nvb; b += gridDim.x) keep_rows(c.d, c.S, b);
        for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < c.S.nblk; b += gridDim.x * blockDim.x) c.S.bdirty[b] = 1;
    }
}

// ------------------------------------- an iteration applied by the whole GPU

// Record v of the pending iteration: row v of the moved column, or physical
// row v of a weight update; false when there is nothing to change.
__device__ __forceinline__ bool sr_big_record(const Dev &d, const Search &S, int q, int e0, int f0, int nI, int rows,
                                              double dl, int v, SrRec &r, int &row, int &ch, double &af)
{
    if (v >= rows) return false;
    ch = 0;
    af = 0.0;
    if (q < 0) {
        row = v;
        return sr_bump_row(d, S, v, r);
    }
    int ai = 0;
    row = sr_col_entry(d, e0, f0, nI, v, ai, af);
    ch = sr_move_row(d, S, row, ai, af, dl, (long long)dl, r, v < nI);
    return true;
}

// The walk of a pending iteration over the old row states.  A unit is a slice
// of the entries of 32 rows (as many slices as there are warps for); the
// entries are taken 128 at a time whatever row they belong to, so short rows
// fill the lanes.  The counting-sorted columns' scalars are summed per CTA.
template <bool MIX>
__global__ void __launch_bounds__(kSrBigThreads) k_search_big(Dev d, Search S)
{
    if (!S.sc->pending) return;
    extern __shared__ __align__(16) unsigned char big_smem[];
    HistAcc *acc = reinterpret_cast<HistAcc *>(big_smem);
    __shared__ SrRec recs[kSrBigThreads / 32][32];
    __shared__ int incls[kSrBigThreads / 32][32];
    __shared__ SrMovedCtx mc;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (MIX) {
        for (int k = threadIdx.x; k < S.nhist; k += blockDim.x) acc[k] = HistAcc{0, 0, 0, 0, 0u, 0};
        if (threadIdx.x == 0) mc = S.sc->mc;
        __syncthreads();
    }
    const int q = S.sc->moved;
    int e0 = 0, f0 = 0, nI = 0, rows = d.m;
    double dl = 0.0;
    if (q >= 0) {
        e0 = d.ci_ptr[q];
        f0 = d.cf_ptr[q];
        nI = d.ci_ptr[q + 1] - e0;
        rows = nI + d.cf_ptr[q + 1] - f0;
        dl = __dsub_rn(d.ctl->mv_new, d.ctl->mv_old);
    }
    const SrWalk W{q, &mc, S.hctx, acc};
    const SrLocal L{};
    SrOwn own{0, 0, 0, 0};
    const int nw = gridDim.x * (kSrBigThreads / 32), gw = blockIdx.x * (kSrBigThreads / 32) + warp;
    const int ng = (rows + 31) / 32, sl = max(1, nw / max(ng, 1));
    SrRec *rec = recs[warp];
    int *incl = incls[warp];
    for (long long un = gw; un < (long long)ng * sl; un += nw) {
        const int g = (int)(un / sl), s = (int)(un % sl);
        SrRec r;
        int row, ch, t = 0;
        double af;
        if (sr_big_record(d, S, q, e0, f0, nI, rows, dl, 32 * g + lane, r, row, ch, af)) {
            t = r.lenB + r.lenN;
            rec[lane] = r;
        }
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(FULLMASK, t, o);
            if (lane >= o) t += v;
        }
        incl[lane] = t;
        __syncwarp();
        const long long tot = __shfl_sync(FULLMASK, t, 31);
        const int a = (int)(tot * s / sl), z = (int)(tot * (s + 1) / sl);
        constexpr int U = 4;
        for (int b0 = a; b0 < z; b0 += 32 * U) {
            int qq[U], rr[U];
            long long av[U];
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const int e = b0 + 32 * k + lane;
                qq[k] = -1;
                rr[k] = 0;
                av[k] = 0;
                if (e < z) {
                    int lo = 0;   // the first record whose prefix exceeds e
#pragma unroll
                    for (int st = 16; st > 0; st >>= 1)
                        if (incl[lo + st - 1] <= e) lo += st;
                    const SrRec &x = rec[lo];
                    int off = e - (lo > 0 ? incl[lo - 1] : 0);
                    if (off >= x.lenB) off += x.offN - x.lenB;
                    rr[k] = lo;
                    qq[k] = __ldg(S.epos + x.p0 + off);
                    av[k] = __ldg(S.eval + x.p0 + off);
                }
            }
            NbCtx ctx[U];
            bool up[U];
#pragma unroll
            for (int k = 0; k < U; ++k) {
                up[k] = qq[k] >= 0 && qq[k] < S.bc && __ldcg(d.bup + qq[k]) != 0;
                if (MIX && qq[k] >= S.bc && qq[k] - S.bc < S.nnb) ctx[k] = sr_ctx(S, qq[k] - S.bc);
            }
#pragma unroll
            for (int k = 0; k < U; ++k) {
                if (qq[k] < 0) continue;
                const SrRec &x = rec[rr[k]];
                if (qq[k] < S.bc) {
                    if (x.integral) sr_entry_bin<false>(S, nullptr, L, x, qq[k], av[k], up[k], q);
                    else sr_entry_bin<true>(S, nullptr, L, x, qq[k], av[k], up[k], q);
                } else if (MIX) {
                    if (qq[k] - S.bc < S.nnb) {
                        if (x.integral) sr_entry_nb<false>(S, nullptr, L, x, qq[k], av[k], ctx[k], W, own);
                        else sr_entry_nb<true>(S, nullptr, L, x, qq[k], av[k], ctx[k], W, own);
                    } else {
                        if (x.integral) sr_entry_hist<false>(S, x, qq[k], av[k], W, own);
                        else sr_entry_hist<true>(S, x, qq[k], av[k], W, own);
                    }
                }
            }
        }
        __syncwarp();
    }
    if (!MIX) return;
    sr_own_add(S, W, own);
    __syncthreads();
    for (int k = threadIdx.x; k < S.nhist; k += blockDim.x) {
        const HistAcc h = acc[k];
        if (h.beta) atomicAdd(reinterpret_cast<unsigned long long *>(&S.ha[k].beta), (unsigned long long)h.beta);
        if (h.alpha) atomicAdd(reinterpret_cast<unsigned long long *>(&S.ha[k].alpha), (unsigned long long)h.alpha);
        if (h.beta_c) atomicAdd(&S.ha[k].beta_c, h.beta_c);
        if (h.alpha_c) atomicAdd(&S.ha[k].alpha_c, h.alpha_c);
    }
}

// Writes the row states of a pending iteration, after its walk, and what a
// moved binary column's own sums lack for its flip back.
__global__ void __launch_bounds__(kSrBigThreads) k_search_put(Dev d, Search S)
{
    if (!S.sc->pending) return;
    const int q = S.sc->moved;
    int e0 = 0, f0 = 0, nI = 0, rows = d.m;
    double dl = 0.0;
    if (q >= 0) {
        e0 = d.ci_ptr[q];
        f0 = d.cf_ptr[q];
        nI = d.ci_ptr[q + 1] - e0;
        rows = nI + d.cf_ptr[q + 1] - f0;
        dl = __dsub_rn(d.ctl->mv_new, d.ctl->mv_old);
    }
    int sum = 0, rd = 0;
    long long rs = 0;
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < rows; v += gridDim.x * blockDim.x) {
        SrRec r;
        int row, ch;
        double af;
        if (!sr_big_record(d, S, q, e0, f0, nI, rows, dl, v, r, row, ch, af)) continue;
        if (q < 0) sr_put_weights(d, row, r);
        else sr_put_row(d, S, row, r, ch);
        if (q >= 0 && q < S.bc && !r.integral) sr_reverse(r, af, dl > 0.0, rs, rd);
        sum += ch;
    }
    if (rs) atomicAdd(reinterpret_cast<unsigned long long *>(S.kS + q), (unsigned long long)rs);
    if (rd) atomicAdd(S.kD + q, rd);
    sum = __reduce_add_sync(FULLMASK, sum);
    if ((threadIdx.x & 31) == 0 && sum) atomicAdd(reinterpret_cast<unsigned long long *>(&S.sc->dnv), (unsigned long long)(long long)sum);
}
