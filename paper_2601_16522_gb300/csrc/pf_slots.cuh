// pf_slots.cuh -- FP32 stage passes on per-cell phase slots (Sec. 3.1).
//
// Slot storage keeps, per cell, at most NSLOT phase values with their phase
// ids (Sec. 3.1: N_p values and N_p integers per cell, N_p = 12 in the
// paper's final benchmark), so a state of N phases costs NSLOT * 6 bytes
// per cell whatever N is: 256^3 cells with 2000 grains take 1.3 GB per state
// vector where dense planes would take 134 GB.  Layout of one state vector
// (Vs = V rounded up to 64): the slots of a cell in groups of four, group q of
// cell i at element 4 (q Vs + i) of the value planes (float) and of the id
// planes (uint16, at float offset NSLOT * Vs; SLOT_EMPTY where unused), then
// the concentration plane (float) when K = 1, at float offset
// SLOT_C_PLANES * Vs.  A cell's used slots come first, in ascending id order;
// the values of a group without a used slot are not written and never read.
// Inside a group the two ids of a 32-bit word are swapped (slot k sits at
// k ^ 1), so the next id of a list is the high half of its word.
//
// Why groups: a list's next four ids arrive with one 8-byte load, so the merge
// below runs on registers instead of waiting for the next id of every list it
// advances (one plane per slot: 62 % of the issue slots busy, the rest waits
// on that chain), and a cell of up to four phases, the usual one, is written
// with one 16-byte and three 8-byte stores instead of 24.
//
// A pass merges the sorted slot lists of the stencil input at the cell and
// its 2d face neighbours and of the pointwise inputs (ascending ids, one
// cursor per list), which visits the phases nonzero anywhere in them in
// ascending order -- the order in which the masked and dense one-cell passes
// visit them -- and applies the same arithmetic as those passes (a phase that
// is zero in every list contributes exactly nothing there), so results equal
// the dense ones bit for bit as long as no cell needs more than NSLOT slots.
// A projected cell with more nonzero values keeps the NSLOT largest (equal
// values: the lower id), the rest become zero and the kept ones are divided
// by their sum (ascending ids): the paper gives no rule for it; this is the
// reading the oracle restates.  "S acted" (the RKL2 first-stage fix) then
// includes that step.  The stored RHS F(u^n) of the STS schemes keeps, in a
// cell with more than NSLOT nonzero entries, the NSLOT largest in magnitude
// (equal magnitudes: the lower id): the same kind of reading.
#pragma once
#include "pf_kernels.cuh"

namespace pfk {

constexpr int NSLOT = 12;                              // slots per cell (N_p)
constexpr int SLOT_C_PLANES = NSLOT + NSLOT / 2;       // float planes before c
constexpr unsigned SLOT_EMPTY = 0xffffu;
constexpr int SLOT_MAXN = 32768;                       // largest phase count (N^2 tables)

// Floats per cell-plane of one slot state vector.
__host__ __device__ constexpr int slot_planes(int K) { return SLOT_C_PLANES + K; }

__device__ __forceinline__ const unsigned short *slot_ids(const float *base, int Vs)
{
    return reinterpret_cast<const unsigned short *>(base + (long long)NSLOT * Vs);
}

// Element of slot k of cell i in the value planes; its id is at slot_at ^ 1.
__device__ __forceinline__ int slot_at(int k, int Vs, int i) { return (k & ~3) * Vs + 4 * i + (k & 3); }

// The list of a crowded cell (slot_wide), in local memory.
struct SlotListW {
    static constexpr int CAP = WIDEACT;
    unsigned short id_[WIDEACT];
    float lap_[WIDEACT], cen_[WIDEACT], dl_[WIDEACT];
    __device__ __forceinline__ unsigned short &id(int k) { return id_[k]; }
    __device__ __forceinline__ float &lap(int k) { return lap_[k]; }
    __device__ __forceinline__ float &cen(int k) { return cen_[k]; }
    __device__ __forceinline__ float &dl(int k) { return dl_[k]; }
};

// Cursor over one sorted slot list: the rest of the current group of ids in
// (x, y), the next one in the high half of x, zeros shifted in behind them.
// Ids ascend strictly, so x is zero exactly when the group is used up (the
// fourth id of a group is at least 3; a broken list only ends earlier).
struct SlotCursor {
    int at;                      // element of the next slot
    unsigned x, y;
    __device__ __forceinline__ void start(const unsigned short *ids, int cell)
    {
        at = 4 * cell;
        const uint2 w = __ldg(reinterpret_cast<const uint2 *>(ids + at));
        x = w.x;
        y = w.y;
    }
    // The next group of a used-up one; past the last, an end mark.
    __device__ __forceinline__ void next(const float *base, int Vs)
    {
        if (x != 0u) return;
        at = ((at - 1) & ~3) + 4 * Vs;
        x = 0xffffffffu;
        if (at >= NSLOT * Vs) return;
        const uint2 w = __ldg(reinterpret_cast<const uint2 *>(slot_ids(base, Vs) + at));
        x = w.x;
        y = w.y;
    }
    // The value of phase a (given as a << 16) if it is the next one (advancing
    // past it), else 0.
    __device__ __forceinline__ float take(unsigned a16, const float *base)
    {
        // without a branch: the lanes of a warp merge different lists
        const bool hit = (x ^ a16) < 0x10000u;
        float v;
        asm("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\tmov.f32 %0, 0f00000000;\n\t"
            "@p ld.global.nc.f32 %0, [%1];\n\t}"
            : "=&f"(v) : "l"(base + at), "r"((unsigned)hit));
        const int sh = hit ? 16 : 0;
        x = __funnelshift_l(y, x, sh);
        y <<= sh;
        at += hit ? 1 : 0;
        return v;
    }
};

// The slots of one output cell, appended in ascending id order and written a
// group at a time.
struct SlotWriter {
    float b0, b1, b2, b3;
    unsigned x, y;
    int n;
    __device__ __forceinline__ void store(float *base, int Vs, int i)
    {
        const int at = (n & ~3) * Vs + 4 * i;
        *reinterpret_cast<float4 *>(base + at) = make_float4(b0, b1, b2, b3);
        *reinterpret_cast<uint2 *>(const_cast<unsigned short *>(slot_ids(base, Vs)) + at) = make_uint2(x, y);
    }
    __device__ __forceinline__ void clear()
    {
        b0 = b1 = b2 = b3 = 0.0f;
        x = y = 0xffffffffu;
    }
    __device__ __forceinline__ void start() { n = 0; clear(); }
    __device__ __forceinline__ void push(float v, unsigned a, float *base, int Vs, int i)
    {
        const int q = n & 3;
        const unsigned m = (q & 1) ? 0xffff0000u : 0x0000ffffu, w = (q & 1) ? a : a << 16;
        if (q < 2) x = (x & m) | w;
        else y = (y & m) | w;
        if (q == 0) b0 = v;
        if (q == 1) b1 = v;
        if (q == 2) b2 = v;
        if (q == 3) {
            b3 = v;
            store(base, Vs, i);
            clear();
        }
        n++;
    }
    // Writes the last group and marks the groups behind it empty.
    __device__ __forceinline__ void finish(float *base, int Vs, int i)
    {
        if (n & 3) store(base, Vs, i);
        unsigned short *ids = const_cast<unsigned short *>(slot_ids(base, Vs));
        for (int k = (n + 3) & ~3; k < NSLOT; k += 4)
            *reinterpret_cast<uint2 *>(ids + k * Vs + 4 * i) = make_uint2(0xffffffffu, 0xffffffffu);
    }
};

// Union capacity: every slot of every list a pass merges.
template <int DIM>
__host__ __device__ constexpr int slot_ucap() { return (1 + 2 * DIM + 3) * NSLOT; }

// The smallest next id (<< 16) of the lists of a pass.
template <int NFACE, bool HP0, bool HP2, bool HR0>
__device__ __forceinline__ unsigned slot_min(const SlotCursor &cin, const SlotCursor *cnb, const SlotCursor &cp0,
                                             const SlotCursor &cp2, const SlotCursor &cr0)
{
    unsigned m = cin.x;
#pragma unroll
    for (int f = 0; f < NFACE; ++f) m = min(m, cnb[f].x);
    if (HP0) m = min(m, cp0.x);
    if (HP2) m = min(m, cp2.x);
    if (HR0) m = min(m, cr0.x);
    return m;
}

// Per-cell body of a slot pass for a crowded cell (slot_wide): any number of
// visited phases, lists in local memory; returns false, having written
// nothing, when more than LST::CAP phases are nontrivial at the cell.  The
// arithmetic and its order are those of masked_cell (see the file comment).
template <int DIM, int KC, unsigned SIG, class LST>
__device__ __forceinline__ bool slot_cell(const Geom &g, const Pass<float> &P, LST &S, int i, const int *off,
                                          const int *ghost, const float *__restrict__ tabA,
                                          const float *__restrict__ tabB, const float *__restrict__ tabL,
                                          const signed char *__restrict__ ptype, double &esum, long long &ecnt)
{
    typedef float T;
    constexpr int NFACE = 2 * DIM;
    constexpr int UCAP = slot_ucap<DIM>();
    constexpr bool RHS = (SIG & SIG_RHS) != 0;
    constexpr bool ERR = (SIG & SIG_ERR) != 0;
    constexpr bool HP0 = (SIG & SIG_P0) != 0 || ERR;
    constexpr bool HP2 = (SIG & SIG_P2) != 0;
    constexpr bool HR0 = (SIG & SIG_R0IN) != 0 || ERR;
    constexpr bool R0OUT = (SIG & SIG_R0OUT) != 0;
    constexpr bool PROJ = (SIG & SIG_PROJECT) != 0;
    const int N = g.N;
    const int Vs = (int)g.Vs;
    const long long co = (long long)SLOT_C_PLANES * Vs;   // concentration plane
    const GeomConst<T> &gc = geom_const<T>(g);
    const T idx2 = gc.idx2;
    const T a0c = P.c.a0, a2c = P.c.a2, b1c = P.c.b1, b0c = P.c.b0;
    const T ib1 = P.c.ib1;   // first-stage fix: F <- (S(u1) - u^n) / (mu~_1 dt)
    const T dt = P.c.dt, rph = P.c.r_phi, aph = P.c.a_phi;

    // concentration
    T cc = (T)0, num_c = (T)0, den_c = (T)0, num_n[NFACE], den_n[NFACE], mf[NFACE];
#pragma unroll
    for (int f = 0; f < NFACE; ++f) { num_n[f] = (T)0; den_n[f] = (T)0; mf[f] = (T)0; }
    if (KC) {
        const T *cf = P.in + co + i;
        cc = ldg(cf);
        num_c = cc;
#pragma unroll
        for (int f = 0; f < NFACE; ++f) {
            T v = ldg(cf + off[f]);
            if (ghost[f] && g.bc_c[f] == BC_DIRICHLET) v = (T)2 * gc.cdir[f] - cc;
            num_n[f] = v;
        }
    }

    // cursors: the stencil input at the cell and its face neighbours, then
    // the pointwise inputs
    SlotCursor cin, cnb[NFACE], cp0, cp2, cr0;
    cin.start(slot_ids(P.in, Vs), i);
#pragma unroll
    for (int f = 0; f < NFACE; ++f) cnb[f].start(slot_ids(P.in, Vs), i + off[f]);
    if (HP0) cp0.start(slot_ids(P.p0, Vs), i);
    if (HP2) cp2.start(slot_ids(P.p2, Vs), i);
    if (HR0) cr0.start(slot_ids(P.r0in, Vs), i);

    // the visited phases (ascending ids) with their stage values, input
    // values (first-stage fix) and list positions
    unsigned short uid[UCAP];
    T uv[UCAP], uin[R0OUT ? UCAP : 1];
    signed char ulist[UCAP];
    T lp0[ERR ? LST::CAP : 1], lr0[ERR ? LST::CAP : 1];
    int nu = 0, nz = 0, nc = 0;
    bool changed = false;
    T best = (T)-1, ssum = (T)0;
    int bestid = -1;
    for (;;) {
        unsigned m = slot_min<NFACE, HP0, HP2, HR0>(cin, cnb, cp0, cp2, cr0);
        while (m == 0u) {      // a list's group is used up
            cin.next(P.in, Vs);
#pragma unroll
            for (int f = 0; f < NFACE; ++f) cnb[f].next(P.in, Vs);
            if (HP0) cp0.next(P.p0, Vs);
            if (HP2) cp2.next(P.p2, Vs);
            if (HR0) cr0.next(P.r0in, Vs);
            m = slot_min<NFACE, HP0, HP2, HR0>(cin, cnb, cp0, cp2, cr0);
        }
        const unsigned a = m >> 16, a16 = m & 0xffff0000u;
        if (a >= (unsigned)N) {
            // the end of every list; an id beyond the phases is a broken state
            if (a != SLOT_EMPTY) raise_flag(P.flag, FLAG_NZ_OVERFLOW);
            break;
        }
        const T v0 = cin.take(a16, P.in);
        T nb[NFACE];
#pragma unroll
        for (int f = 0; f < NFACE; ++f) nb[f] = cnb[f].take(a16, P.in);
        const T p0v = HP0 ? cp0.take(a16, P.p0) : (T)0;
        const T p2v = HP2 ? cp2.take(a16, P.p2) : (T)0;
        const T r0v = HR0 ? cr0.take(a16, P.r0in) : (T)0;
        T mx = v0, mn = v0;
#pragma unroll
        for (int f = 0; f < NFACE; ++f) {
            mx = fmaxf(mx, nb[f]);
            mn = fminf(mn, nb[f]);
        }
        if (KC) {
            const int t = ptype[a];
            const T c0t = gc.c0[t], ikt = gc.invk[t], dkt = gc.Dk[t];
            num_c = num_c - v0 * c0t;
            den_c = den_c + v0 * ikt;
#pragma unroll
            for (int f = 0; f < NFACE; ++f) {
                num_n[f] = num_n[f] - nb[f] * c0t;
                den_n[f] = den_n[f] + nb[f] * ikt;
                mf[f] = mf[f] + dkt * ((T)0.5 * (v0 + nb[f]));
            }
        }
        const bool act = mx > (T)0 && mn < (T)1;
        signed char li = -1;
        if (act) {
            if (nz >= LST::CAP) return false;
            T l = (T)0;
#pragma unroll
            for (int f = 0; f < NFACE; ++f) l = l + (nb[f] - v0);
            S.id(nz) = (unsigned short)a;
            S.lap(nz) = l * idx2;
            S.cen(nz) = v0;
            if (ERR) { lp0[nz] = p0v; lr0[nz] = r0v; }
            li = (signed char)nz;
            nz++;
        }
        if (ERR) {
            if (!act) {
                T e = ((T)12 * (p0v - v0) + ((T)6 * dt) * r0v) * ((T)1 / (T)15);
                const T trial = p0v + (dt * (T)0.5) * r0v;
                if (trial < (T)0 || trial > (T)1) e = (T)0;
                if (e != (T)0) {
                    const T wt = rph * fmaxf(fabsf(p0v), fabsf(v0)) + aph;
                    const T q = e / wt;
                    esum += (double)(q * q);
                    nc++;
                }
            }
        } else if (!RHS) {
            T acc = affine<HP0, HP2>(v0, p0v, p2v, a0c, a2c);
            if (HR0) acc = acc + b0c * r0v;
            if (!act && PROJ) {
                if (acc < (T)0) { acc = (T)0; changed = true; }
                if (acc >= (T)1 && acc > best) { best = acc; bestid = (int)a; }
                ssum = ssum + acc;
            }
            uid[nu] = (unsigned short)a;
            uv[nu] = acc;
            ulist[nu] = li;
            if (R0OUT) uin[nu] = v0;
            nu++;
        }
    }

    T mu = (T)0, rc = (T)0;
    if (KC) {
        mu = num_c / den_c;
        T acc = (T)0;
#pragma unroll
        for (int f = 0; f < NFACE; ++f) acc = acc + mf[f] * (num_n[f] / den_n[f] - mu);
        rc = acc * idx2;
    }
    // variational derivative and pairwise sum over the listed phases (with
    // uniform tables the coefficients come from the constants: same values)
    const bool uni = g.uni != 0;
    for (int k = 0; k < nz; ++k) {
        const long long a = S.id(k);
        const T *Aa = tabA + a * N, *Ba = tabB + a * N;
        T d = (T)0;
        for (int k2 = 0; k2 < nz; ++k2) {
            if (k2 == k) continue;
            const int b = S.id(k2);
            const T Aab = uni ? g.uA : ldg(Aa + b), Bab = uni ? g.uB : ldg(Ba + b);
            d = d + (Aab * S.lap(k2) + Bab * S.cen(k2));
        }
        if (KC) {
            const int t = ptype[a];
            d = d + (-(mu * mu) / ((T)2 * gc.k[t]) - mu * gc.c0[t]);
        }
        S.dl(k) = d;
    }
    const T inz = nz > 1 ? (T)1 / (T)nz : (T)0;
    for (int k = 0; k < nz; ++k) {
        T rk = (T)0;
        if (nz > 1) {
            const T *La = tabL + (long long)S.id(k) * N;
            const T dk = S.dl(k);
            T s = (T)0;
            for (int k2 = 0; k2 < nz; ++k2) {
                if (k2 == k) continue;
                const T Lab = uni ? g.uL : ldg(La + S.id(k2));
                s = s + Lab * (dk - S.dl(k2));
            }
            rk = -(s * inz);
        }
        S.lap(k) = rk;                 // the list now holds the RHS
        if (ERR) {
            const T p0v = lp0[k], v0 = S.cen(k), r0v = lr0[k];
            const T sr = r0v + rk;
            T e = ((T)12 * (p0v - v0) + ((T)6 * dt) * sr) * ((T)1 / (T)15);
            const T trial = p0v + (dt * (T)0.5) * sr;
            if (trial < (T)0 || trial > (T)1) e = (T)0;
            if (e != (T)0) {
                const T wt = rph * fmaxf(fabsf(p0v), fabsf(v0)) + aph;
                const T q = e / wt;
                esum += (double)(q * q);
                nc++;
            }
        }
    }
    if constexpr (RHS) {
        // pf_rhs: the listed phases' RHS into the zeroed FP64 output
        if (P.rhs_pm) {
            for (int k = 0; k < nz; ++k) P.rhs_pm[(long long)S.id(k) * g.V + i] = (double)S.lap(k);
            if (KC) P.rhs_pm[(long long)N * g.V + i] = (double)rc;
        }
        if (P.nz_out) P.nz_out[i] = (unsigned char)(nz < 255 ? nz : 255);
        return true;
    } else if constexpr (ERR) {
        ecnt += (nc > 0 ? nc : 2);
        if (KC) {
            const T un = ldg(P.p0 + co + i), un1 = cc, rn = ldg(P.r0in + co + i);
            const T e = ((T)12 * (un - un1) + ((T)6 * dt) * (rn + rc)) * ((T)1 / (T)15);
            const T wt = P.c.r_c * fmaxf(fabsf(un + gc.cref), fabsf(un1 + gc.cref)) + P.c.a_c;
            const T q = e / wt;
            esum += (double)(q * q);
            ecnt += 1;
        }
        return true;
    } else {
    // listed phases (ascending ids): add the RHS term, clamp, >= 1 candidates, sum
    for (int j = 0; j < nu; ++j) {
        if (ulist[j] < 0) continue;
        const int a = uid[j];
        T acc = uv[j] + b1c * S.lap(ulist[j]);
        if (PROJ) {
            if (acc < (T)0) { acc = (T)0; changed = true; }
            if (acc >= (T)1 && (acc > best || (acc == best && a < bestid))) { best = acc; bestid = a; }
            ssum = ssum + acc;
        }
        uv[j] = acc;
    }
    if (PROJ) {
        if (bestid >= 0) {
            for (int j = 0; j < nu; ++j)
                if (uv[j] != (((int)uid[j] == bestid) ? (T)1 : (T)0)) changed = true;
            ssum = (T)1;
        }
        if (!(ssum > (T)0)) raise_flag(P.flag, FLAG_SIMPLEX);
    }
    const T inv = (ssum > (T)0) ? (T)1 / ssum : (T)1;
    // projected values; then the slot rule where more than NSLOT are nonzero
    int cnt = 0;
    for (int j = 0; j < nu; ++j) {
        T wv = uv[j];
        if (PROJ) wv = (bestid >= 0) ? (((int)uid[j] == bestid) ? (T)1 : (T)0) : wv * inv;
        uv[j] = wv;
        if (wv != (T)0) cnt++;
    }
    if (cnt > NSLOT) {
        // keep the NSLOT largest (equal values: the lower id), renormalise
        bool keep[UCAP];
        for (int j = 0; j < nu; ++j) {
            keep[j] = false;
            if (uv[j] == (T)0) continue;
            int rank = 0;
            for (int m = 0; m < nu; ++m)
                if (m != j && uv[m] != (T)0 && (uv[m] > uv[j] || (uv[m] == uv[j] && uid[m] < uid[j]))) rank++;
            keep[j] = rank < NSLOT;
        }
        T sk = (T)0;
        for (int j = 0; j < nu; ++j)
            if (keep[j]) sk = sk + uv[j];
        for (int j = 0; j < nu; ++j) uv[j] = keep[j] ? uv[j] / sk : (T)0;
        changed = true;
    }
    const bool fix = R0OUT && P.fix_first && changed;
    // the stored RHS F(u^n) (stage 1): its nonzero entries; more than NSLOT
    // keep the NSLOT largest in magnitude (equal magnitudes: the lower id)
    if constexpr (R0OUT) {
        T ur[UCAP];
        int nr = 0;
        SlotWriter W;
        W.start();
        for (int j = 0; j < nu; ++j) {
            T r = ulist[j] >= 0 ? S.lap(ulist[j]) : (T)0;
            if (fix) r = (uv[j] - uin[j]) * ib1;
            ur[j] = r;
            if (r != (T)0) nr++;
        }
        for (int j = 0; j < nu; ++j) {
            if (ur[j] == (T)0) continue;
            if (nr > NSLOT) {
                int rank = 0;
                for (int m = 0; m < nu; ++m)
                    if (m != j && ur[m] != (T)0 &&
                        (fabsf(ur[m]) > fabsf(ur[j]) || (fabsf(ur[m]) == fabsf(ur[j]) && uid[m] < uid[j])))
                        rank++;
                if (rank >= NSLOT) continue;
            }
            if (W.n < NSLOT) W.push(ur[j], uid[j], P.r0out, Vs, i);   // (more only with non-finite values)
        }
        W.finish(P.r0out, Vs, i);
    }
    // outputs: the nonzero entries in ascending id order
    SlotWriter W;
    W.start();
    for (int j = 0; j < nu; ++j)
        if (uv[j] != (T)0 && W.n < NSLOT) W.push(uv[j], uid[j], P.out, Vs, i);   // (more: non-finite values, flagged)
    W.finish(P.out, Vs, i);
    if (KC) {
        // the small increments are summed first: c is rounded once per stage
        T d = b1c * rc;
        if (HR0) d = d + b0c * ldg(P.r0in + co + i);
        if (HP0) d = d + a0c * (ldg(P.p0 + co + i) - cc);
        if (HP2) d = d + a2c * (ldg(P.p2 + co + i) - cc);
        const T acc = cc + d;
        if (!isfinite(acc)) raise_flag(P.flag, FLAG_NONFINITE);
        if (R0OUT) P.r0out[co + i] = rc;
        P.out[co + i] = acc;
    }
    return true;
    }
}

// A cell that visits more than NSLOT phases, with the lists in local memory
// (out of line: only the rare threads that need it touch its local arrays);
// beyond WIDEACT nontrivial phases the pass raises FLAG_NZ_OVERFLOW.
template <int DIM, int KC, unsigned SIG>
__device__ __noinline__ void slot_wide(const Geom *g, const Pass<float> *P, int i, const int *off, const int *ghost,
                                       const float *tabA, const float *tabB, const float *tabL,
                                       const signed char *ptype, double *esum, long long *ecnt)
{
    SlotListW L;
    double es = 0.0;
    long long ec = 0;
    if (!slot_cell<DIM, KC, SIG, SlotListW>(*g, *P, L, i, off, ghost, tabA, tabB, tabL, ptype, es, ec)) {
        raise_flag(P->flag, FLAG_NZ_OVERFLOW);
        return;
    }
    *esum += es;
    *ecnt += ec;
}

// Shared-memory list of the visited phases of a block's cells: the nontrivial
// ones from entry 0 up in ascending id order, the others (rare outside bulk
// cells) from entry NSLOT - 1 down.  UNI: the problem's pairwise coefficients
// are uniform (Geom::uni), a phase's contribution A lap + B phi to the other
// phases' variational derivatives does not depend on them, and one array holds
// it and later the derivative (30 KB a block instead of 43, the rest is L1).
template <bool UNI, unsigned SIG>
struct SlotSmem {
    static constexpr bool STAGE = (SIG & (SIG_ERR | SIG_RHS)) == 0;
    static constexpr bool CEN = !UNI || !STAGE || (SIG & SIG_R0OUT) != 0;
    unsigned short id[NSLOT][BLOCK];
    float lap[NSLOT][BLOCK];                     // UNI: the contribution; else the Laplacian, later the RHS
    float cen[CEN ? NSLOT : 1][BLOCK];           // phi at the cell
    float dl[UNI ? 1 : NSLOT][BLOCK];            // dF/dphi
    float val[UNI && STAGE ? NSLOT : 1][BLOCK];  // stage value
};

// One cell of a slot pass that visits at most NSLOT phases; returns false,
// having written nothing, when there are more (slot_wide redoes the cell).
// The arithmetic and its order are those of slot_cell.
//
// Bound by instruction issue and divergence (a cell merges 8 to 10 lists; lanes
// of a warp hold different phases), so the merge keeps the ids in registers
// and takes values without branches, a warp covers 16 x 2 cells, the pairwise
// sums run unrolled in registers (uniform coefficients), and no per-thread
// array of the merged phases is kept in local memory.  256^3 x 2000 grains,
// RKL2, three attempts with the state in and out: 72 ms for slot planes merged
// from memory, 60 with ids in registers, 55 without branches, 46 with
// the lanes meeting after the merge, 40 with the sums of all 12 phases in
// registers (42 with 8 of them).
template <int DIM, int KC, unsigned SIG, bool UNI>
__device__ __forceinline__ bool slot_fast(const Geom &g, const Pass<float> &P, SlotSmem<UNI, SIG> &S, int tid, int i,
                                          const int *off, const int *ghost, const float *__restrict__ tabA,
                                          const float *__restrict__ tabB, const float *__restrict__ tabL,
                                          const signed char *__restrict__ ptype, double &esum, long long &ecnt,
                                          unsigned am)
{
    typedef float T;
    constexpr int NFACE = 2 * DIM;
    constexpr bool RHS = (SIG & SIG_RHS) != 0;
    constexpr bool ERR = (SIG & SIG_ERR) != 0;
    constexpr bool STAGE = !RHS && !ERR;
    constexpr bool HP0 = (SIG & SIG_P0) != 0 || ERR;
    constexpr bool HP2 = (SIG & SIG_P2) != 0;
    constexpr bool HR0 = (SIG & SIG_R0IN) != 0 || ERR;
    constexpr bool R0OUT = (SIG & SIG_R0OUT) != 0;
    constexpr bool PROJ = (SIG & SIG_PROJECT) != 0;
    const int N = g.N;
    const int Vs = (int)g.Vs;
    const long long co = (long long)SLOT_C_PLANES * Vs;   // concentration plane
    const GeomConst<T> &gc = geom_const<T>(g);
    const T idx2 = gc.idx2;
    const T a0c = P.c.a0, a2c = P.c.a2, b1c = P.c.b1, b0c = P.c.b0;
    const T ib1 = P.c.ib1;   // first-stage fix: F <- (S(u1) - u^n) / (mu~_1 dt)
    const T dt = P.c.dt, rph = P.c.r_phi, aph = P.c.a_phi;

    // concentration
    T cc = (T)0, num_c = (T)0, den_c = (T)0, num_n[NFACE], den_n[NFACE], mf[NFACE];
#pragma unroll
    for (int f = 0; f < NFACE; ++f) { num_n[f] = (T)0; den_n[f] = (T)0; mf[f] = (T)0; }
    if (KC) {
        const T *cf = P.in + co + i;
        cc = ldg(cf);
        num_c = cc;
#pragma unroll
        for (int f = 0; f < NFACE; ++f) {
            T v = ldg(cf + off[f]);
            if (ghost[f] && g.bc_c[f] == BC_DIRICHLET) v = (T)2 * gc.cdir[f] - cc;
            num_n[f] = v;
        }
    }

    SlotCursor cin, cnb[NFACE], cp0, cp2, cr0;
    cin.start(slot_ids(P.in, Vs), i);
#pragma unroll
    for (int f = 0; f < NFACE; ++f) cnb[f].start(slot_ids(P.in, Vs), i + off[f]);
    if (HP0) cp0.start(slot_ids(P.p0, Vs), i);
    if (HP2) cp2.start(slot_ids(P.p2, Vs), i);
    if (HR0) cr0.start(slot_ids(P.r0in, Vs), i);

    // stage values (!UNI), pointwise inputs (ERR) and RHS (UNI, stage 1) of the list
    T lval[STAGE && !UNI ? NSLOT : 1], lp0[ERR ? NSLOT : 1], lr0[ERR ? NSLOT : 1], lrk[UNI && R0OUT ? NSLOT : 1];
    auto val = [&](int k) -> T & { return UNI ? S.val[k][tid] : lval[STAGE && !UNI ? k : 0]; };
    int nz = 0, ne = 0, nc = 0;      // listed phases, others, error entries
    bool changed = false, crowd = false;
    T best = (T)-1, ssum = (T)0;
    int bestid = -1;
    for (;;) {
        unsigned m = slot_min<NFACE, HP0, HP2, HR0>(cin, cnb, cp0, cp2, cr0);
        while (m == 0u) {      // a list's group is used up
            cin.next(P.in, Vs);
#pragma unroll
            for (int f = 0; f < NFACE; ++f) cnb[f].next(P.in, Vs);
            if (HP0) cp0.next(P.p0, Vs);
            if (HP2) cp2.next(P.p2, Vs);
            if (HR0) cr0.next(P.r0in, Vs);
            m = slot_min<NFACE, HP0, HP2, HR0>(cin, cnb, cp0, cp2, cr0);
        }
        const unsigned a = m >> 16, a16 = m & 0xffff0000u;
        if (a >= (unsigned)N) {
            // the end of every list; an id beyond the phases is a broken state
            if (a != SLOT_EMPTY) raise_flag(P.flag, FLAG_NZ_OVERFLOW);
            break;
        }
        const T v0 = cin.take(a16, P.in);
        T nb[NFACE];
#pragma unroll
        for (int f = 0; f < NFACE; ++f) nb[f] = cnb[f].take(a16, P.in);
        const T p0v = HP0 ? cp0.take(a16, P.p0) : (T)0;
        const T p2v = HP2 ? cp2.take(a16, P.p2) : (T)0;
        const T r0v = HR0 ? cr0.take(a16, P.r0in) : (T)0;
        T mx = v0, mn = v0;
#pragma unroll
        for (int f = 0; f < NFACE; ++f) {
            mx = fmaxf(mx, nb[f]);
            mn = fminf(mn, nb[f]);
        }
        if (KC) {
            const int t = ptype[a];
            const T c0t = gc.c0[t], ikt = gc.invk[t], dkt = gc.Dk[t];
            num_c = num_c - v0 * c0t;
            den_c = den_c + v0 * ikt;
#pragma unroll
            for (int f = 0; f < NFACE; ++f) {
                num_n[f] = num_n[f] - nb[f] * c0t;
                den_n[f] = den_n[f] + nb[f] * ikt;
                mf[f] = mf[f] + dkt * ((T)0.5 * (v0 + nb[f]));
            }
        }
        const bool act = mx > (T)0 && mn < (T)1;
        T acc = (T)0;
        if (STAGE) {
            acc = affine<HP0, HP2>(v0, p0v, p2v, a0c, a2c);
            if (HR0) acc = acc + b0c * r0v;
        }
        if (act || STAGE) {
            if (nz + ne >= NSLOT) { crowd = true; break; }
            const int k = act ? nz : NSLOT - 1 - ne;
            S.id[k][tid] = (unsigned short)a;
            if (SlotSmem<UNI, SIG>::CEN) S.cen[k][tid] = v0;
            if (act) {
                T l = (T)0;
#pragma unroll
                for (int f = 0; f < NFACE; ++f) l = l + (nb[f] - v0);
                l = l * idx2;
                S.lap[k][tid] = UNI ? g.uA * l + g.uB * v0 : l;
                if (ERR) { lp0[k] = p0v; lr0[k] = r0v; }
                nz++;
            } else {
                if (PROJ) {
                    if (acc < (T)0) { acc = (T)0; changed = true; }
                    if (acc >= (T)1 && acc > best) { best = acc; bestid = (int)a; }
                    ssum = ssum + acc;
                }
                ne++;
            }
            if (STAGE) val(k) = acc;
        } else if (ERR) {
            T e = ((T)12 * (p0v - v0) + ((T)6 * dt) * r0v) * ((T)1 / (T)15);
            const T trial = p0v + (dt * (T)0.5) * r0v;
            if (trial < (T)0 || trial > (T)1) e = (T)0;
            if (e != (T)0) {
                const T wt = rph * fmaxf(fabsf(p0v), fabsf(v0)) + aph;
                const T q = e / wt;
                esum += (double)(q * q);
                nc++;
            }
        }
    }

    // every lane leaves the merge here, the crowded ones too: a return inside the
    // loop left no point where the lanes of a warp meet again, and they went
    // through the sums and stores below a few at a time (12.6 lanes an
    // instruction on average, 16.3 so)
    __syncwarp(am);
    if (crowd) return false;

    T mu = (T)0, rc = (T)0;
    if (KC) {
        mu = num_c / den_c;
        T acc = (T)0;
#pragma unroll
        for (int f = 0; f < NFACE; ++f) acc = acc + mf[f] * (num_n[f] / den_n[f] - mu);
        rc = acc * idx2;
    }
    // chemical part of the derivative per type
    T chem[2] = {(T)0, (T)0};
    if (KC && nz > 0) {
#pragma unroll
        for (int t = 0; t < 2; ++t) chem[t] = -(mu * mu) / ((T)2 * gc.k[t]) - mu * gc.c0[t];
    }
    // the RHS rk of listed phase k: the RHS itself, the error term, or the
    // stage value with its clamp, >= 1 candidate and sum
    auto listed = [&](int k, T rk) {
        if (RHS) {
            // pf_rhs: the listed phases' RHS into the zeroed FP64 output
            if (P.rhs_pm) P.rhs_pm[(long long)S.id[k][tid] * g.V + i] = (double)rk;
        }
        if (R0OUT) {
            if (UNI) lrk[k] = rk;
            else S.lap[k][tid] = rk;
        }
        if (ERR) {
            const T p0v = lp0[k], v0 = S.cen[k][tid], r0v = lr0[k];
            const T sr = r0v + rk;
            T e = ((T)12 * (p0v - v0) + ((T)6 * dt) * sr) * ((T)1 / (T)15);
            const T trial = p0v + (dt * (T)0.5) * sr;
            if (trial < (T)0 || trial > (T)1) e = (T)0;
            if (e != (T)0) {
                const T wt = rph * fmaxf(fabsf(p0v), fabsf(v0)) + aph;
                const T q = e / wt;
                esum += (double)(q * q);
                nc++;
            }
        }
        if (STAGE) {
            T acc = val(k) + b1c * rk;
            if (PROJ) {
                const int a = S.id[k][tid];
                if (acc < (T)0) { acc = (T)0; changed = true; }
                if (acc >= (T)1 && (acc > best || (acc == best && a < bestid))) { best = acc; bestid = a; }
                ssum = ssum + acc;
            }
            val(k) = acc;
        }
    };
    // variational derivatives and pairwise sums over the listed phases
    if (UNI) {
        if (nz > 0) {
            T t[NSLOT], ch[NSLOT], rk[NSLOT];
#pragma unroll
            for (int k = 0; k < NSLOT; ++k) {
                t[k] = k < nz ? S.lap[k][tid] : (T)0;
                ch[k] = KC && k < nz ? (ptype[S.id[k][tid]] ? chem[1] : chem[0]) : (T)0;
            }
            uni_rhs<KC, NSLOT>(nz, t, ch, g.uL, rk);
#pragma unroll
            for (int k = 0; k < NSLOT; ++k)
                if (k < nz) listed(k, rk[k]);
        }
    } else {
        for (int k = 0; k < nz; ++k) {
            const long long a = S.id[k][tid];
            const T *Aa = tabA + a * N, *Ba = tabB + a * N;
            T d = (T)0;
            for (int k2 = 0; k2 < nz; ++k2) {
                if (k2 == k) continue;
                const int b = S.id[k2][tid];
                d = d + (ldg(Aa + b) * S.lap[k2][tid] + ldg(Ba + b) * S.cen[k2][tid]);
            }
            if (KC) d = d + (ptype[a] ? chem[1] : chem[0]);
            S.dl[k][tid] = d;
        }
        const T inz = nz > 1 ? (T)1 / (T)nz : (T)0;
        for (int k = 0; k < nz; ++k) {
            T rk = (T)0;
            if (nz > 1) {
                const T *La = tabL + (long long)S.id[k][tid] * N;
                const T dk = S.dl[k][tid];
                T s = (T)0;
                for (int k2 = 0; k2 < nz; ++k2) {
                    if (k2 == k) continue;
                    s = s + ldg(La + S.id[k2][tid]) * (dk - S.dl[k2][tid]);
                }
                rk = -(s * inz);
            }
            listed(k, rk);
        }
    }
    if constexpr (RHS) {
        if (KC && P.rhs_pm) P.rhs_pm[(long long)N * g.V + i] = (double)rc;
        if (P.nz_out) P.nz_out[i] = (unsigned char)(nz < 255 ? nz : 255);
    }
    if constexpr (ERR) {
        ecnt += (nc > 0 ? nc : 2);
        if (KC) {
            const T un = ldg(P.p0 + co + i), un1 = cc, rn = ldg(P.r0in + co + i);
            const T e = ((T)12 * (un - un1) + ((T)6 * dt) * (rn + rc)) * ((T)1 / (T)15);
            const T wt = P.c.r_c * fmaxf(fabsf(un + gc.cref), fabsf(un1 + gc.cref)) + P.c.a_c;
            const T q = e / wt;
            esum += (double)(q * q);
            ecnt += 1;
        }
    }
    if constexpr (STAGE) {
        if (PROJ) {
            if (bestid >= 0) {
                for (int k = 0; k < NSLOT; ++k)
                    if ((k < nz || k >= NSLOT - ne) &&
                        val(k) != (((int)S.id[k][tid] == bestid) ? (T)1 : (T)0))
                        changed = true;
                ssum = (T)1;
            }
            if (!(ssum > (T)0)) raise_flag(P.flag, FLAG_SIMPLEX);
        }
        const T inv = (ssum > (T)0) ? (T)1 / ssum : (T)1;
        const bool fix = R0OUT && P.fix_first && changed;
        // the nonzero results in ascending id order: the list merged with the others
        SlotWriter W, R;
        W.start();
        R.start();
        int k = 0, x = NSLOT - 1;
        while (k < nz || x >= NSLOT - ne) {
            const bool lst = x < NSLOT - ne || (k < nz && S.id[k][tid] < S.id[x][tid]);
            const int j = lst ? k++ : x--;
            const unsigned a = S.id[j][tid];
            T w = val(j);
            if (PROJ) w = (bestid >= 0) ? (((int)a == bestid) ? (T)1 : (T)0) : w * inv;
            if (w != (T)0) W.push(w, a, P.out, Vs, i);
            if (R0OUT) {
                T r = lst ? (UNI ? lrk[UNI && R0OUT ? j : 0] : S.lap[j][tid]) : (T)0;
                if (fix) r = (w - S.cen[SlotSmem<UNI, SIG>::CEN ? j : 0][tid]) * ib1;
                if (r != (T)0) R.push(r, a, P.r0out, Vs, i);
            }
        }
        W.finish(P.out, Vs, i);
        if (R0OUT) R.finish(P.r0out, Vs, i);
        if (KC) {
            // the small increments are summed first: c is rounded once per stage
            T d = b1c * rc;
            if (HR0) d = d + b0c * ldg(P.r0in + co + i);
            if (HP0) d = d + a0c * (ldg(P.p0 + co + i) - cc);
            if (HP2) d = d + a2c * (ldg(P.p2 + co + i) - cc);
            const T acc = cc + d;
            if (!isfinite(acc)) raise_flag(P.flag, FLAG_NONFINITE);
            if (R0OUT) P.r0out[co + i] = rc;
            P.out[co + i] = acc;
        }
    }
    return true;
}

// Resident blocks per SM (register budget), 256^3 x 2000 grains: 44.5 ms at 3,
// 42.4 at 4 and 50 at 5, where 48 registers spill; with a concentration 4 spill.
__host__ __device__ constexpr int slot_minb(int K) { return K ? 3 : 4; }

// One slot pass: one cell per thread, 32 x 8 tiles, one z plane per block.
template <int DIM, int KC, unsigned SIG, bool UNI>
__global__ void __launch_bounds__(BLOCK, slot_minb(KC))
slot_kernel(const __grid_constant__ Geom g, const __grid_constant__ Pass<float> P, const float *__restrict__ tabA,
            const float *__restrict__ tabB, const float *__restrict__ tabL, const signed char *__restrict__ ptype)
{
    pass_begin();
    __shared__ SlotSmem<UNI, SIG> S;
    if (pass_skipped(P.flag)) return;
    const int tid = threadIdx.x;
    const int bid = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
    int tx, ty;
    tile_cell<WARP_X>(tid, tx, ty);
    const int x = blockIdx.x * TX + tx;
    const int y = blockIdx.y * TY + ty;
    const int z = blockIdx.z;
    double esum = 0.0;
    long long ecnt = 0;
    const bool here = x < g.nx && y < g.ny;
    const unsigned am = __ballot_sync(0xffffffffu, here);
    if (here) {
        const int i = (int)(((long long)z * g.ny + y) * g.nx + x);
        long long off64[6];
        int ghost[6], off[6];
        face_offsets(g, x, y, z, off64, ghost);
#pragma unroll
        for (int f = 0; f < 6; ++f) off[f] = ghost[f] ? 0 : (int)off64[f];
        if (!slot_fast<DIM, KC, SIG, UNI>(g, P, S, tid, i, off, ghost, tabA, tabB, tabL, ptype, esum, ecnt, am)) {
            esum = 0.0;
            ecnt = 0;
            slot_wide<DIM, KC, SIG>(&g, &P, i, off, ghost, tabA, tabB, tabL, ptype, &esum, &ecnt);
        }
    }
    if (SIG & SIG_ERR) block_partials(esum, ecnt, P.part_sum, P.part_cnt, bid, P.part_n);
    if (P.count_step) count_step_done(P.flag);
}

}  // namespace pfk
