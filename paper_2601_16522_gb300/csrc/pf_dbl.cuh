// pf_dbl.cuh -- the FP64 stage pass.
//
// GB300 issues FP64 at two lanes per clock and SM (about 1/64 of the FP32
// rate), so an FP64 warp instruction costs the same 16 issue cycles whether
// one lane or 32 are active, and a pass with one cell per thread, whose
// interface cells sit in every other warp a few lanes at a time, keeps that
// pipe busy with mostly empty instructions (128^3 x 32 grains, forward Euler:
// 4.09 ms, 82 % of the FP64 pipe, for 0.2 ms of arithmetic).  This pass
//  - classifies every cell with integer tests on the FP64 encodings: a cell
//    whose stencil and pointwise inputs hold one phase at exactly 1 and +0
//    otherwise (the bulk of a grain) has the closed result "the same", which
//    is written without any arithmetic;
//  - compacts the other cells of the block (in cell order, so sums stay
//    deterministic) and gives each of them to one thread: the FP64
//    instructions of the phases then run with full warps;
//  - evaluates the grand potential and the mobility of a cell once, in shared
//    memory, instead of once per face that reads it (2D: one division and 6
//    multiply-adds a cell where it had 5 and 30);
//  - replaces repeated divisions by one divisor (dx^2, N_z, the simplex sum,
//    15) by a correctly rounded reciprocal and Markstein's correction
//    (div_by), which returns the quotient's bits in 3 instructions.
// The phases' arithmetic and its order are those of cell_core, so phase
// results are the same bits; the concentration uses fused multiply-adds.
#pragma once
#include "pf_vec.cuh"

namespace pfk {

constexpr int DBL_TX = 32;           // cells along x: a warp is one row
constexpr int DBL_CAP = 8;           // nontrivial phases in a thread's shared-memory list

// a / b for a divisor used more than once, rb = 1 / b correctly rounded: the
// quotient estimate a * rb and one correction by its exact remainder (P.
// Markstein, IBM J. Res. Dev. 34 (1990), theorem 8.5 of his 2000 book: the
// result is the correctly rounded quotient while nothing over- or underflows).
__device__ __forceinline__ double div_by(double a, double b, double rb)
{
    const double q = a * rb;
    return __fma_rn(__fma_rn(-q, b, a), rb, q);
}

// Rows of a block: 8, or 2 where 8 would leave most SMs without a block (a
// 64^2 grid has 16 blocks of 8 rows; its FP64 work then queues on 16 of the
// 152 SMs).
__host__ __device__ inline int dbl_rows(const Geom &g)
{
    const long long b8 = (long long)((g.nx + DBL_TX - 1) / DBL_TX) * ((g.ny + 7) / 8) * g.nz;
    return b8 < 2 * 152 ? 2 : 8;
}
__host__ __device__ inline long long dbl_tiles(const Geom &g)
{
    const int r = dbl_rows(g);
    return (long long)((g.nx + DBL_TX - 1) / DBL_TX) * ((g.ny + r - 1) / r);
}

template <int ROWS>
struct DblSmem {
    static constexpr int T = DBL_TX * ROWS;
    double lap[DBL_CAP][T];    // Laplacian, later the RHS of the listed phase
    double cen[DBL_CAP][T];    // phi at the cell
    double dl[DBL_CAP][T];     // variational derivative
    double mu[ROWS + 2][DBL_TX + 2], M[ROWS + 2][DBL_TX + 2];   // of the tile and its face neighbours
    unsigned vis[ROWS][4];     // phases the row visits
    unsigned oldo[ROWS][4], oldr[ROWS][4];   // output / stored-RHS words before the pass
    unsigned occ[ROWS][SEG_KINDS][4];        // output words of the row's segment
    unsigned lst[ROWS][4];     // phases listed in a cell of the row
    unsigned short queue[T];   // nontrivial cells, in cell order
    int wcnt[ROWS];
    unsigned char id[DBL_CAP][T];
};

template <int ROWS>
struct DblList {
    static constexpr int CAP = DBL_CAP;
    DblSmem<ROWS> *S;
    int tid;
    __device__ __forceinline__ unsigned char &id(int k) { return S->id[k][tid]; }
    __device__ __forceinline__ double &lap(int k) { return S->lap[k][tid]; }
    __device__ __forceinline__ double &cen(int k) { return S->cen[k][tid]; }
    __device__ __forceinline__ double &dl(int k) { return S->dl[k][tid]; }
};

// Where a cell's nonzero outputs are noted (shared memory of its row); any is
// null without segment words.
struct DblWords {
    unsigned *any, *first, *last, *lst;   // first / last: null unless the cell is that one
    __device__ __forceinline__ void out(int a) const
    {
        if (!any) return;
        const unsigned m = 1u << (a & 31);
        atomicOr(any + (a >> 5), m);
        if (first) atomicOr(first + (a >> 5), m);
        if (last) atomicOr(last + (a >> 5), m);
    }
    __device__ __forceinline__ void rhs(int a) const
    {
        if (any) atomicOr(lst + (a >> 5), 1u << (a & 31));
    }
};

// The phases of one cell: RHS, stage combination, projection, first-stage
// fix, SSP(10)4 accumulators and error terms, with the options read from P.
// vis: the phases to visit (all others are +0 in every input).  Returns
// false, having written nothing, when more than LST::CAP are nontrivial.
template <int DIM, int KC, class LST>
__device__ __forceinline__ bool dbl_phases(const Geom &g, const Pass<double> &P, LST &S, const double *__restrict__ tabA,
                                           const double *__restrict__ tabB, const double *__restrict__ tabL,
                                           const signed char *__restrict__ ptype, int x, int y, int z,
                                           const unsigned *vis, double mu, const DblWords &words, double &esum,
                                           long long &ecnt)
{
    typedef double T;
    constexpr int NFACE = 2 * DIM;
    const int N = g.N, nw = seg_words(N);
    const long long Vs = g.Vs;
    const long long i = ((long long)z * g.ny + y) * g.nx + x;
    long long off[6];
    int ghost[6];
    face_offsets(g, x, y, z, off, ghost);
#pragma unroll
    for (int f = 0; f < 6; ++f)
        if (ghost[f]) off[f] = 0;      // a zero-gradient ghost of phi is the cell itself
#define PF_VISITED(a_)                                               \
    for (int w_ = 0; w_ < nw; ++w_)                                  \
        for (unsigned m_ = vis[w_], a_ = 0; m_ && ((a_ = 32u * w_ + __ffs(m_) - 1u), true); m_ &= m_ - 1u)

    // ---- activity and Laplacians --------------------------------------------
    int nz = 0;
    PF_VISITED(a)
    {
        const T *fp = P.in + (long long)a * Vs + i;
        const T v0 = ldg(fp);
        T nb[NFACE];
#pragma unroll
        for (int f = 0; f < NFACE; ++f) nb[f] = ldg(fp + off[f]);
        if (!nontrivial<NFACE>(v0, nb)) continue;
        T l = (T)0;
#pragma unroll
        for (int f = 0; f < NFACE; ++f) l = l + (nb[f] - v0);
        if (nz < LST::CAP) {
            S.id(nz) = (unsigned char)a;
            S.lap(nz) = div_by(l, g.dx2, g.idx2);
            S.cen(nz) = v0;
        }
        nz++;
    }
    if (nz > LST::CAP) return false;

    // ---- variational derivative and pairwise sum over the list -------------
    for (int k = 0; k < nz; ++k) {
        const int a = S.id(k);
        const T *Aa = tabA + a * N, *Ba = tabB + a * N;
        T d = (T)0;
        for (int k2 = 0; k2 < nz; ++k2) {
            if (k2 == k) continue;
            const int b = S.id(k2);
            d = d + (ldg(Aa + b) * S.lap(k2) + ldg(Ba + b) * S.cen(k2));
        }
        T psi = (T)0;
        if (KC) {
            const int t = ptype[a];
            psi = -(mu * mu) / ((T)2 * g.k[t]) - mu * g.c0[t];
        }
        S.dl(k) = d + psi;
    }
    const T rnz = (T)1 / (T)(nz > 0 ? nz : 1);
    for (int k = 0; k < nz; ++k) {
        T rk = (T)0;
        if (nz > 1) {
            const int a = S.id(k);
            const T *La = tabL + a * N;
            const T dk = S.dl(k);
            T s = (T)0;
            for (int k2 = 0; k2 < nz; ++k2) {
                if (k2 == k) continue;
                s = s + ldg(La + S.id(k2)) * (dk - S.dl(k2));
            }
            rk = -div_by(s, (T)nz, rnz);
        }
        S.lap(k) = rk;                  // the list now holds the RHS
    }

    // list cursor: phases are visited in ascending order
    int kk = 0;
    int curid = nz > 0 ? S.id(0) : -1;
    auto next_rhs = [&](int a) -> T {
        if (a != curid) return (T)0;
        const T r = S.lap(kk);
        kk++;
        curid = kk < nz ? S.id(kk) : -1;
        return r;
    };

    if (P.mode == MODE_RHS) {
        if (P.rhs_pm)
            for (int a = 0; a < N; ++a) P.rhs_pm[(long long)a * g.V + i] = next_rhs(a);
        if (P.nz_out) P.nz_out[i] = (unsigned char)nz;
        return true;
    }
    if (P.mode == MODE_ERR) {
        // STS error sweep (Sec. 3.3): in = u^{n+1}, p0 = u^n, r0in = F^n
        const T dt = P.c.dt, rph = P.c.r_phi, aph = P.c.a_phi, r15 = (T)1 / (T)15;
        int nc = 0;
        PF_VISITED(a)
        {
            const long long o = (long long)a * Vs + i;
            const T r1 = next_rhs((int)a);
            if (P.r0out) {                       // F(u^{n+1}) kept for reuse
                P.r0out[o] = r1;
                if (!zbits(r1)) words.rhs((int)a);
            }
            const T un = ldg(P.p0 + o), un1 = ldg(P.in + o), rn = ldg(P.r0in + o);
            // no change and no RHS: e is exactly zero (skipped like any zero e)
            if (same_bits(un, un1) && zbits(rn) && zbits(r1)) continue;
            const T sr = rn + r1;
            T e = div_by((T)12 * (un - un1) + ((T)6 * dt) * sr, (T)15, r15);
            const T trial = un + (dt / (T)2) * sr;
            if (trial < (T)0 || trial > (T)1) e = (T)0;
            if (e != (T)0) {
                const T au = tabs(un), av = tabs(un1);
                const T w = rph * (au > av ? au : av) + aph;
                const T q = e / w;
                esum += q * q;
                nc++;
            }
        }
        ecnt += (nc > 0 ? nc : 2);
        return true;
    }
    // ---- stage combination (Eq. sts / Alg. ssp2 / SSP(10)4) -----------------
    const bool project = P.project != 0;
    const T a0c = P.c.a0, a2c = P.c.a2, b1c = P.c.b1, b0c = P.c.b0, bzc = P.c.bz;
    bool changed = false;
    T best = (T)-1, ssum = (T)0;
    int bestid = -1, nnz = 0;
    PF_VISITED(a)
    {
        const long long o = (long long)a * Vs + i;
        const T r = next_rhs((int)a);
        const T v = ldg(P.in + o);
        const T p0v = P.p0 ? ldg(P.p0 + o) : (T)0, p2v = P.p2 ? ldg(P.p2 + o) : (T)0;
        const T r0v = P.r0in ? ldg(P.r0in + o) : (T)0;
        T acc = v;
        // every input +0: the combination is exactly 0 (no arithmetic)
        if (!(zbits(v) && zbits(p0v) && zbits(p2v) && zbits(r0v) && zbits(r))) {
            if (P.p0) acc = acc + a0c * (p0v - v);
            if (P.p2) acc = acc + a2c * (p2v - v);
            acc = acc + b1c * r;
            if (P.r0in) acc = acc + b0c * r0v;
        }
        if (P.r0out) {                           // replaced below where S acts (RKL2)
            P.r0out[o] = r;
            if (!zbits(r)) words.rhs((int)a);
        }
        if (P.zout) P.zout[o] = P.zin[o] + bzc * r;   // zin may alias zout
        if (!zbits(acc)) {
            if (project) {
                // S step 1: clamp negatives; step 2 candidate: largest >= 1;
                // the sum for step 3 in ascending order (+0 entries add nothing)
                if (acc < (T)0) { acc = (T)0; changed = true; }
                if (acc >= (T)1 && acc > best) { best = acc; bestid = (int)a; }
                ssum = ssum + acc;
                if (acc != (T)0) nnz++;
            }
            if (!zbits(acc)) words.out((int)a);
        }
        P.out[o] = acc;
    }
    if (project) {
        if (bestid >= 0) {
            // the >= 1 rule: the winner becomes 1, the others 0; the sum is then
            // exactly 1 (with up to 16 phases "S acted" only if that changed a
            // value, as the shared-memory form of cell_core decides it)
            if (N > Smem<T>::NV || best != (T)1 || nnz > 1) changed = true;
            ssum = (T)1;
        }
        if (!(ssum > (T)0)) raise_flag(P.flag, FLAG_SIMPLEX);
    }
    const bool fix = P.r0out && P.fix_first && changed;
    const bool emb = P.embedded_err != 0, has_out2 = P.out2 != nullptr;
    int nc = 0;
    // values that are final as written are not swept again
    if (!(bestid < 0 && (!project || ssum == (T)1) && !fix && !emb && !has_out2)) {
        const bool plain = !(ssum > 1e-200 && ssum < 1e200);   // outside div_by's range
        const T rs = plain ? (T)0 : (T)1 / ssum;
        PF_VISITED(a)
        {
            const long long o = (long long)a * Vs + i;
            T w = P.out[o];
            if (project) {
                if (bestid >= 0) w = ((int)a == bestid) ? (T)1 : (T)0;
                else if (ssum > (T)0 && ssum != (T)1 && !zbits(w)) w = plain ? w / ssum : div_by(w, ssum, rs);
            }
            if (fix) {
                const T r = (w - ldg(P.in + o)) / b1c;
                P.r0out[o] = r;
                if (!zbits(r)) words.rhs((int)a);
            }
            if (emb) {
                const T zv = P.zout[o];
                T e = w - zv;
                if (zv < (T)0 || zv > (T)1) e = (T)0;
                if (e != (T)0) {
                    const T au = tabs(ldg(P.uw + o)), av = tabs(w);
                    const T wt = P.c.r_phi * (au > av ? au : av) + P.c.a_phi;
                    const T q = e / wt;
                    esum += q * q;
                    nc++;
                }
            }
            if (has_out2) {
                const T q2 = w + P.c.m25 * (ldg(P.q2in + o) - w);
                P.out2[o] = q2;
                const T u = w + P.c.m15 * (q2 - w);
                P.out[o] = u;
                if (!zbits(u)) words.out((int)a);
            } else {
                P.out[o] = w;
            }
        }
    }
    if (emb) ecnt += (nc > 0 ? nc : 2);
    return true;
#undef PF_VISITED
}

// A cell with more than DBL_CAP nontrivial phases: the same with a
// WIDEACT-entry list in local memory (out of line: only the rare threads that
// take it touch its arrays).
template <int DIM, int KC>
__device__ __noinline__ void dbl_wide(const Geom *g, const Pass<double> *P, const double *tabA, const double *tabB,
                                      const double *tabL, const signed char *ptype, int x, int y, int z,
                                      const unsigned *vis, double mu, const DblWords *words, double *esum,
                                      long long *ecnt)
{
    WideList<double> L;
    double es = 0.0;
    long long ec = 0;
    if (!dbl_phases<DIM, KC, WideList<double>>(*g, *P, L, tabA, tabB, tabL, ptype, x, y, z, vis, mu, *words, es, ec)) {
        raise_flag(P->flag, FLAG_NZ_OVERFLOW);
        return;
    }
    *esum += es;
    *ecnt += ec;
}

template <int DIM, int KC, int ROWS>
__device__ __forceinline__ void dbl_body(const Geom &g, const Pass<double> &P, const double *__restrict__ tabA,
                                         const double *__restrict__ tabB, const double *__restrict__ tabL,
                                         const signed char *__restrict__ ptype)
{
    typedef double T;
    constexpr int NFACE = 2 * DIM;
    constexpr unsigned ALL = 0xffffffffu;
    constexpr long long ONE = 0x3ff0000000000000LL;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    if (pass_skipped(P.flag)) return;
    DblSmem<ROWS> &S = *reinterpret_cast<DblSmem<ROWS> *>(smem_raw);
    const int tid = threadIdx.x, lane = tid & 31, ty = tid >> 5;
    const int bid = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
    const int x0 = blockIdx.x * DBL_TX, y0 = blockIdx.y * ROWS, z = blockIdx.z;
    const int x = x0 + lane, y = y0 + ty;
    const int N = g.N, nw = seg_words(N);
    const long long Vs = g.Vs;
    const bool rowok = y < g.ny;                 // warp-uniform
    const bool here = rowok && x < g.nx;
    const int row = z * g.ny + (rowok ? y : g.ny - 1);
    const long long i = (long long)row * g.nx + (x < g.nx ? x : g.nx - 1);   // in bounds for every lane
    const int lastlane = (g.nx - x0 < DBL_TX ? g.nx - x0 : DBL_TX) - 1;
    const bool seg = g.seg != 0;
    const int tx = gridDim.x;
    const int q0 = row * tx + blockIdx.x;        // the row's segment (32 cells in FP64)
    double esum = 0.0;
    long long ecnt = 0;

    // ---- the phases the row visits --------------------------------------------
    {
        const int yy = rowok ? y : g.ny - 1;
        const int qym = q0 + (yy > 0 ? -tx : (g.bc_phi[2] == BC_PERIODIC ? (g.ny - 1) * tx : 0));
        const int qyp = q0 + (yy < g.ny - 1 ? tx : (g.bc_phi[3] == BC_PERIODIC ? -(g.ny - 1) * tx : 0));
        const int pl = tx * g.ny;
        const int qzm = q0 + (z > 0 ? -pl : (g.bc_phi[4] == BC_PERIODIC ? (g.nz - 1) * pl : 0));
        const int qzp = q0 + (z < g.nz - 1 ? pl : (g.bc_phi[5] == BC_PERIODIC ? -(g.nz - 1) * pl : 0));
        const int ql = blockIdx.x > 0 ? q0 - 1 : (g.bc_phi[0] == BC_PERIODIC ? q0 + tx - 1 : -1);
        const int qr = (int)blockIdx.x < tx - 1 ? q0 + 1 : (g.bc_phi[1] == BC_PERIODIC ? q0 - (tx - 1) : -1);
        for (int w = 0; w < nw; ++w) {
            const unsigned full = word_bits(N, w);
            unsigned U = full, mo = full, mr = full;
            if (seg) {
                auto word = [&](const T *v, int q, int kind) { return seg_at(g, v, q, kind)[w]; };
                U = word(P.in, q0, SEG_ANY) | word(P.in, qym, SEG_ANY) | word(P.in, qyp, SEG_ANY);
                if (DIM == 3) U |= word(P.in, qzm, SEG_ANY) | word(P.in, qzp, SEG_ANY);
                if (ql >= 0) U |= word(P.in, ql, SEG_LAST);
                if (qr >= 0) U |= word(P.in, qr, SEG_FIRST);
                if (P.p0) U |= word(P.p0, q0, SEG_ANY);
                if (P.p2) U |= word(P.p2, q0, SEG_ANY);
                if (P.r0in) U |= word(P.r0in, q0, SEG_ANY);
                if (P.zin) U |= word(P.zin, q0, SEG_ANY);
                if (P.q2in) U |= word(P.q2in, q0, SEG_ANY);
                U &= full;
                if (P.mode == MODE_STAGE) mo = word(P.out, q0, SEG_ANY) & full;
                if (P.r0out) mr = word(P.r0out, q0, SEG_ANY) & full;
                // phases not visited: +0, stored where an output holds another value
                if (here) {
                    auto clear = [&](T *v, unsigned old) {
                        for (unsigned m = old & full & ~U; m; m &= m - 1u)
                            v[(long long)(32 * w + __ffs(m) - 1) * Vs + i] = (T)0;
                    };
                    if (P.mode == MODE_STAGE) clear(P.out, mo);
                    if (P.r0out) clear(P.r0out, mr);
                    if (P.zout) clear(P.zout, word(P.zout, q0, SEG_ANY));
                    if (P.out2) clear(P.out2, word(P.out2, q0, SEG_ANY));
                }
            }
            if (lane == 0) {
                S.vis[ty][w] = U;
                S.oldo[ty][w] = mo;
                S.oldr[ty][w] = mr;
                S.lst[ty][w] = 0u;
                for (int k = 0; k < SEG_KINDS; ++k) S.occ[ty][k][w] = 0u;
            }
        }
        __syncwarp();
    }

    // ---- every cell: class, and the sums of its chemistry ---------------------
    long long off[6];
    int ghost[6];
    face_offsets(g, x < g.nx ? x : g.nx - 1, rowok ? y : g.ny - 1, z, off, ghost);
#pragma unroll
    for (int f = 0; f < 6; ++f)
        if (ghost[f]) off[f] = 0;
    // SSP(10)4 registers change bulk cells too; a pass without projection has
    // no closed bulk result
    bool trivial = !(P.zout || P.out2 || P.embedded_err || (P.mode == MODE_STAGE && !P.project));
    int bulk = -1;
    T num = (T)0, den = (T)0, M = (T)0, cc = (T)0, numz[2] = {0, 0}, denz[2] = {0, 0}, Mz[2] = {0, 0};
    if (KC) {
        const T *cf = P.in + (long long)N * Vs + i;
        cc = ldg(cf);
        num = cc;
        if (DIM == 3)
#pragma unroll
            for (int f = 0; f < 2; ++f) {
                numz[f] = ldg(cf + off[4 + f]);
                if (ghost[4 + f] && g.bc_c[4 + f] == BC_DIRICHLET) numz[f] = (T)2 * g.cdir[4 + f] - cc;
            }
    }
    for (int w = 0; w < nw; ++w)
#pragma unroll 2
        for (unsigned m = S.vis[ty][w]; m; m &= m - 1u) {
            const int a = 32 * w + __ffs(m) - 1;
            const long long o = (long long)a * Vs + i;
            const T *fp = P.in + o;
            const T v = ldg(fp);
            T nb[NFACE];
            long long orb = __double_as_longlong(v), andb = orb;
#pragma unroll
            for (int f = 0; f < NFACE; ++f) {
                nb[f] = ldg(fp + off[f]);
                orb |= __double_as_longlong(nb[f]);
                andb &= __double_as_longlong(nb[f]);
            }
            if (P.p0) { const long long b = __double_as_longlong(ldg(P.p0 + o)); orb |= b; andb &= b; }
            if (P.p2) { const long long b = __double_as_longlong(ldg(P.p2 + o)); orb |= b; andb &= b; }
            const long long r0b = P.r0in ? __double_as_longlong(ldg(P.r0in + o)) : 0LL;
            // all +0: nothing; all exactly 1 and no stored RHS: bulk of a
            if ((orb | r0b) != 0) {
                if (orb == ONE && andb == ONE && r0b == 0 && bulk < 0) bulk = a;
                else trivial = false;
            }
            if (KC) {
                const int t = ptype[a];
                const T c0t = g.c0[t], ikt = g.invk[t], dkt = g.Dk[t];
                num = __fma_rn(-v, c0t, num);
                den = __fma_rn(v, ikt, den);
                M = __fma_rn(v, dkt, M);
                if (DIM == 3)
#pragma unroll
                    for (int f = 0; f < 2; ++f) {
                        numz[f] = __fma_rn(-nb[4 % NFACE + f], c0t, numz[f]);
                        denz[f] = __fma_rn(nb[4 % NFACE + f], ikt, denz[f]);
                        Mz[f] = __fma_rn(nb[4 % NFACE + f], dkt, Mz[f]);
                    }
            }
        }
    if (bulk < 0) trivial = false;               // no phase at all: the projection reports it

    // ---- concentration: mu and mobility of the tile and around it -------------
    T mu = (T)0, rc = (T)0;
    if (KC) {
        const int cols = g.nx - x0 < DBL_TX ? g.nx - x0 : DBL_TX, rows = g.ny - y0 < ROWS ? g.ny - y0 : ROWS;
        mu = num / den;
        if (here) {
            S.mu[ty + 1][lane + 1] = mu;
            S.M[ty + 1][lane + 1] = M;
        }
        // the face neighbours outside the tile: rows above and below, then the
        // columns left and right (a domain face's ghost holds the cell's own
        // phases and, for c, the cell's value or the Dirichlet ghost)
        for (int h = tid; h < 2 * DBL_TX + 2 * ROWS; h += DBL_TX * ROWS) {
            int lx, ly, f;
            if (h < 2 * DBL_TX) {
                lx = h % DBL_TX;
                f = h < DBL_TX ? 2 : 3;
                ly = f == 2 ? -1 : rows;
                if (lx >= cols) continue;
            } else {
                const int k = h - 2 * DBL_TX;
                ly = k % ROWS;
                f = k < ROWS ? 0 : 1;
                lx = f == 0 ? -1 : cols;
                if (ly >= rows) continue;
            }
            int hx = x0 + lx, hy = y0 + ly;
            bool gh = false;
            if (hx < 0 || hx >= g.nx) {
                if (g.bc_phi[f] == BC_PERIODIC) hx = hx < 0 ? g.nx - 1 : 0;
                else { hx = hx < 0 ? 0 : g.nx - 1; gh = true; }
            }
            if (hy < 0 || hy >= g.ny) {
                if (g.bc_phi[f] == BC_PERIODIC) hy = hy < 0 ? g.ny - 1 : 0;
                else { hy = hy < 0 ? 0 : g.ny - 1; gh = true; }
            }
            const int hrow = z * g.ny + hy;
            const long long j = (long long)hrow * g.nx + hx;
            T cv = ldg(P.in + (long long)N * Vs + j);
            if (gh && g.bc_c[f] == BC_DIRICHLET) cv = (T)2 * g.cdir[f] - cv;
            T dn = (T)0, Mn = (T)0;
            for (int w = 0; w < nw; ++w) {
                unsigned m = word_bits(N, w);
                if (seg) m &= seg_at(g, P.in, hrow * tx + hx / DBL_TX, SEG_ANY)[w];
                for (; m; m &= m - 1u) {
                    const int a = 32 * w + __ffs(m) - 1, t = ptype[a];
                    const T v = ldg(P.in + (long long)a * Vs + j);
                    cv = __fma_rn(-v, g.c0[t], cv);
                    dn = __fma_rn(v, g.invk[t], dn);
                    Mn = __fma_rn(v, g.Dk[t], Mn);
                }
            }
            S.mu[ly + 1][lx + 1] = cv / dn;
            S.M[ly + 1][lx + 1] = Mn;
        }
    }

    // ---- nontrivial cells into the block's queue, in cell order ---------------
    const unsigned ball = __ballot_sync(ALL, here && !trivial);
    if (lane == 0) S.wcnt[ty] = __popc(ball);
    __syncthreads();
    int base = 0, cnt = 0;
#pragma unroll
    for (int k = 0; k < ROWS; ++k) {
        const int c = S.wcnt[k];
        if (k < ty) base += c;
        cnt += c;
    }
    if (here && !trivial) S.queue[base + __popc(ball & ((1u << lane) - 1u))] = (unsigned short)tid;

    // ---- bulk cells: the closed result ----------------------------------------
    if (here && trivial) {
        if (P.mode == MODE_RHS) {
            if (P.rhs_pm)
                for (int a = 0; a < N; ++a) P.rhs_pm[(long long)a * g.V + i] = (T)0;
            if (P.nz_out) P.nz_out[i] = 0;
        } else if (P.mode == MODE_ERR) {
            ecnt += 2;
        }
    }
    if (rowok && (P.mode == MODE_STAGE || P.r0out)) {
        const bool st = P.mode == MODE_STAGE;
        for (int w = 0; w < nw; ++w) {
            const unsigned mo = S.oldo[ty][w], mr = S.oldr[ty][w];
            if (here && trivial)
                for (unsigned m = S.vis[ty][w]; m; m &= m - 1u) {
                    const int b = __ffs(m) - 1, a = 32 * w + b;
                    const long long o = (long long)a * Vs + i;
                    if (st && (a == bulk || ((mo >> b) & 1u))) P.out[o] = a == bulk ? (T)1 : (T)0;
                    if (P.r0out && ((mr >> b) & 1u)) P.r0out[o] = (T)0;
                }
            if (seg && st) {
                const unsigned mine = here && trivial && (bulk >> 5) == w ? 1u << (bulk & 31) : 0u;
                const unsigned r = __reduce_or_sync(ALL, mine);
                if (lane == 0 && r) atomicOr(&S.occ[ty][SEG_ANY][w], r);
                if (lane == 0 && mine) atomicOr(&S.occ[ty][SEG_FIRST][w], mine);
                if (lane == lastlane && mine) atomicOr(&S.occ[ty][SEG_LAST][w], mine);
            }
        }
    }

    // ---- concentration of every cell ------------------------------------------
    if (KC && here) {
        T acc = (T)0;
        auto face = [&](T mun, T Mn) { acc = __fma_rn((T)0.5 * (M + Mn), mun - mu, acc); };
        face(S.mu[ty + 1][lane], S.M[ty + 1][lane]);
        face(S.mu[ty + 1][lane + 2], S.M[ty + 1][lane + 2]);
        face(S.mu[ty][lane + 1], S.M[ty][lane + 1]);
        face(S.mu[ty + 2][lane + 1], S.M[ty + 2][lane + 1]);
        if (DIM == 3)
#pragma unroll
            for (int f = 0; f < 2; ++f) face(numz[f] / denz[f], Mz[f]);
        rc = div_by(acc, g.dx2, g.idx2);
        const long long o = (long long)N * Vs + i;
        if (P.mode == MODE_RHS) {
            if (P.rhs_pm) P.rhs_pm[(long long)N * g.V + i] = rc;
        } else if (P.mode == MODE_ERR) {
            if (P.r0out) P.r0out[o] = rc;
            const T un = ldg(P.p0 + o), rn = ldg(P.r0in + o);
            const T e = ((T)12 * (un - cc) + ((T)6 * P.c.dt) * (rn + rc)) / (T)15;
            const T au = tabs(un + g.cref), av = tabs(cc + g.cref);
            const T q = e / (P.c.r_c * (au > av ? au : av) + P.c.a_c);
            esum += q * q;
            ecnt += 1;
        } else {
            // the small increments are summed first: c is rounded once per stage
            T d = P.c.b1 * rc;
            if (P.r0in) d = d + P.c.b0 * ldg(P.r0in + o);
            if (P.p0) d = d + P.c.a0 * (ldg(P.p0 + o) - cc);
            if (P.p2) d = d + P.c.a2 * (ldg(P.p2 + o) - cc);
            const T u = cc + d;
            if (!isfinite(u)) raise_flag(P.flag, FLAG_NONFINITE);
            if (P.r0out) P.r0out[o] = rc;
            if (P.zout) {
                const T zv = P.zin[o] + P.c.bz * rc;
                P.zout[o] = zv;
                if (P.embedded_err) {
                    const T au = tabs(ldg(P.uw + o) + g.cref), av = tabs(u + g.cref);
                    const T q = (u - zv) / (P.c.r_c * (au > av ? au : av) + P.c.a_c);
                    esum += q * q;
                    ecnt += 1;
                }
            }
            if (P.out2) {
                const T q2 = u + P.c.m25 * (ldg(P.q2in + o) - u);
                P.out2[o] = q2;
                P.out[o] = u + P.c.m15 * (q2 - u);
            } else {
                P.out[o] = u;
            }
        }
    }
    __syncthreads();

    // ---- the queued cells, one per thread -------------------------------------
    if (tid < cnt) {
        const int t = S.queue[tid], lx = t & 31, ly = t >> 5;
        DblWords words;
        words.any = seg ? S.occ[ly][SEG_ANY] : nullptr;
        words.first = lx == 0 ? S.occ[ly][SEG_FIRST] : nullptr;
        words.last = lx == lastlane ? S.occ[ly][SEG_LAST] : nullptr;
        words.lst = S.lst[ly];
        const T muq = KC ? S.mu[ly + 1][lx + 1] : (T)0;
        DblList<ROWS> L{&S, tid};
        double es = 0.0;
        long long ec = 0;
        if (!dbl_phases<DIM, KC, DblList<ROWS>>(g, P, L, tabA, tabB, tabL, ptype, x0 + lx, y0 + ly, z, S.vis[ly], muq,
                                                words, es, ec))
            dbl_wide<DIM, KC>(&g, &P, tabA, tabB, tabL, ptype, x0 + lx, y0 + ly, z, S.vis[ly], muq, &words, &es, &ec);
        esum += es;
        ecnt += ec;
    }
    if (seg && (P.mode == MODE_STAGE || P.r0out)) {
        __syncthreads();
        if (rowok && lane < nw) {
            if (P.mode == MODE_STAGE)
#pragma unroll
                for (int k = 0; k < SEG_KINDS; ++k) seg_at(g, P.out, q0, k)[lane] = S.occ[ty][k][lane];
            // the other outputs are read at their own cells only: their edge
            // words need not be sharp
#pragma unroll
            for (int k = 0; k < SEG_KINDS; ++k) {
                if (P.r0out) seg_at(g, P.r0out, q0, k)[lane] = S.lst[ty][lane];
                if (P.zout) seg_at(g, P.zout, q0, k)[lane] = S.vis[ty][lane];
                if (P.out2) seg_at(g, P.out2, q0, k)[lane] = S.vis[ty][lane];
            }
        }
    }
    if (P.mode == MODE_ERR || P.embedded_err != 0) block_partials(esum, ecnt, P.part_sum, P.part_cnt, bid, P.part_n);
    if (P.count_step) count_step_done(P.flag);
}

template <int DIM, int KC, int ROWS>
__global__ void __launch_bounds__(DBL_TX *ROWS, ROWS == 8 ? 3 : 8)
dbl_kernel(const __grid_constant__ Geom g, const __grid_constant__ Pass<double> P, const double *__restrict__ tabA,
           const double *__restrict__ tabB, const double *__restrict__ tabL, const signed char *__restrict__ ptype)
{
    pass_begin();
    dbl_body<DIM, KC, ROWS>(g, P, tabA, tabB, tabL, ptype);
}

// The same pass with its description read from device memory (device-driven
// adaptive steps; see cell_kernel_d).
template <int DIM, int KC, int ROWS>
__global__ void __launch_bounds__(DBL_TX *ROWS, ROWS == 8 ? 3 : 8)
dbl_kernel_d(const __grid_constant__ Geom g, const Pass<double> *__restrict__ Pd, const double *__restrict__ tabA,
             const double *__restrict__ tabB, const double *__restrict__ tabL, const signed char *__restrict__ ptype)
{
    __shared__ Pass<double> Ps;
    block_copy(Ps, *Pd);
    __syncthreads();
    dbl_body<DIM, KC, ROWS>(g, Ps, tabA, tabB, tabL, ptype);
}

}  // namespace pfk
