// One real Krylov sequence per node for all of its poles, in fixed point.
//
// H_R is real symmetric and the right-hand side e_j is real, so the COCG
// iterates of the P shifted systems (H_R - z_p) x = e_j of a node all lie in
// the same real Krylov spaces: COCG's x_k is the Galerkin solution in
// span(q_1 .. q_k), x_k = Q_k (T_k - z_p)^-1 e_1, with Q_k, T_k from the
// symmetric Lanczos process on H_R started at e_j (shift invariance;
// Frommer, Computing 70 (2003)).  One Lanczos sequence, as long as the
// slowest pole needs, therefore replaces P complex COCG solves: the node
// entry x_jp(j) = [(T_k - z_p)^-1]_11 and the residual norms come from the
// L D L^T factors of the tridiagonal T_k - z_p, P scalars per step:
//   d_k = alpha_k - z_p - beta_{k-1}^2 / d_{k-1},  zeta_{k+1} = -zeta_k beta_k / d_k,
//   x_jp(j) = sum_k zeta_k^2 / d_k,                ||r_k|| = |zeta_{k+1}|.
// The bulk configuration needs max_p 1,142 real steps per node in place of
// sum_p 4,560 complex iterations.
//
// Precision.  The recurrence must hold FP64-like accuracy over a thousand
// steps (FP32 vectors lose the density at 1e-5), and this part issues 1.7
// FP64 FMAs per clock and SM against 31 integer multiply-adds into 64 bits
// and 115 FP32 FMAs (measured).  So the vectors are 62-bit fixed point: a
// value u is hi 2^-31 + lo 2^-62 with two signed 31-bit limbs.  Of a product,
// hi hi is exact in a 64-bit integer sum; the mixed terms, 2^-31 of it, are
// 64-bit integers in FP64 calls and FP32 in most mixed ones; the lo lo term,
// below 2^-62, is dropped, except in w.w, where it adds up.  Each result is
// rounded once to 2^-62.
// Vectors are kept at norm [1/8, 1/4) by exact powers of two, so the rounding
// is ~1e-16 of the norm per step, the size of FP64's.  A = (H_R - shift) /
// scale has ||A|| < 1/2, which bounds every sum below the 64-bit range.
// ||u||^2 comes from the recurrence (see the step); where |alpha| exceeds beta
// an error of it would grow, and the norm is summed.
//
// Layout.  A thread-block cluster works on one node.  The region is cut into
// z-slabs, one per CTA; each CTA holds its slab of the current vector u and
// Q halo planes on either side in shared memory (rows Q zeros apart, so that
// x neighbours need no bounds checks).  A thread takes pairs of points along
// x.  The previous vector, the new one, V and the projector rows that cover a
// pair are touched by their own thread only, coalesced, in a per-CTA scratch
// slot that stays in L2.  Per step:
//   dot    projections on the local projector tables, summed over the cluster
//   A      w = A u - g u_prev with the nonlocal term, u.w, w.w
//          one exchange of u.w and w.w: alpha = u.w / u.u, and
//          ||w - alpha u||^2 = w.w - alpha u.w gives beta in the same one
//   B      u_new = (w - alpha u) 2^e, halo planes pushed to the neighbours
// One warp of each CTA computes no points: it sums the partials, and in
// rank 0 it runs the pole recurrences of step k-1 during step k.
//
// Bound: instruction issue and latency at 20 warps an SM (19 computing, 96
// registers): 245 instructions a point-step without projectors, 554 with them
// (integer mixed terms), 1.5 to 1.9 issued a clock.  96 nodes x 16 poles on
// 33^3 regions with projectors take 109 ms, 500 with one complex COCG per pole
// in mixed precision; 13 nodes x 16 poles on 25^3 in FP64 8.9 ms against 277.
#include <cuda_runtime.h>

#include <cfloat>
#include <cstddef>
#include <cstdint>

#include "md_krylov.h"
#include "md_operator.cuh"

namespace md {

namespace {

constexpr int kMaxThreads = 19 * 32 + 32;   // 20 warps: 96 registers a thread
constexpr int kMaxWarps = kMaxThreads / 32;
constexpr int kMaxC = 8;
constexpr int kMeasure = -1;   // KShared::stop: sum ||w - alpha u||^2 first

__device__ __forceinline__ uint32_t k_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t k_nrank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void k_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void k_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void k_sync() {
    k_arrive();
    k_wait();
}
__device__ __forceinline__ uint32_t k_map(uint32_t a, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void k_st_remote(uint32_t a, int4 v) {
    asm volatile("st.shared::cluster.v4.s32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
                 : "memory");
}
__device__ __forceinline__ void k_st_remote(uint32_t a, long long v) {
    asm volatile("st.shared::cluster.s64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}

// ---- 62-bit fixed point ----------------------------------------------------

// acc += a b, one IMAD.WIDE
__device__ __forceinline__ void madw(long long& acc, int a, int b) { acc += (long long)a * b; }
// Hides where a value comes from: the compiler keeps loop-carried operands of
// madw sign-extended and then multiplies 64 x 64 bits.
__device__ __forceinline__ int opaque(int x) {
    asm("" : "+r"(x));
    return x;
}
__device__ __forceinline__ int2 split31(long long x) {
    x += 1LL << 30;
    return make_int2(opaque((int)(x >> 31)), opaque((int)(x & 0x7fffffffLL) - (1 << 30)));
}
// A product of two 62-bit values is hi hi 2^-62 + (hi lo + lo hi) 2^-93 + ..:
// the first term exactly, in 64 bits; the mixed terms, 2^-31 of it, in one of
// two ways.
// FP32 (X = false), the form of most mixed calls.  IMAD.WIDE with distinct
// operands runs at 31 a clock and SM (measured), FFMA2 at 65 pairs, so they cost
// a quarter of what they do in integers.  But lo is as large where hi is small,
// and 24 bits of lo hi leave 2^-57 on every component: against 64-bit Jacobi
// matrices, beta is off by 5e-15 after a few steps and alpha by 1e-13 after 40
// on 17^3 regions.
// 64-bit integers (X = true), the form of FP64 calls and of mixed ones whose
// tolerance asks for it: exact but for the terms' last 8 bits.  Beta is within
// 1e-15 and alpha within 5e-15 there (FP64 arithmetic: 1e-15 and 1e-14).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack(float a, float b) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float sum2(f32x2 v) {
    float a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
    return a + b;
}
// acc += a b, elementwise
__device__ __forceinline__ void fma2(f32x2& acc, f32x2 a, f32x2 b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ float as_float(int x) { return __int_as_float(x); }
__device__ __forceinline__ int as_int(float x) { return __float_as_int(x); }
// Left operand: {(float)hi, (float)lo} or lo beside hi; right operand the same
// with {(float)lo, (float)hi}.
template <bool X>
struct Lhs {
    int h;
    f32x2 f;
    __device__ __forceinline__ Lhs(int hi, int lo) : h(hi), f(pack((float)hi, (float)lo)) {}
};
template <>
struct Lhs<true> {
    int h, l;
    __device__ __forceinline__ Lhs(int hi, int lo) : h(hi), l(lo) {}
};
template <bool X>
struct Rhs {
    int h;
    f32x2 f;
    __device__ __forceinline__ Rhs(int hi, int lo) : h(hi), f(pack((float)lo, (float)hi)) {}
    __device__ __forceinline__ Rhs(int hi, int, f32x2 lo_hi) : h(hi), f(lo_hi) {}
};
template <>
struct Rhs<true> {
    int h, l;
    __device__ __forceinline__ Rhs(int hi, int lo) : h(hi), l(lo) {}
    __device__ __forceinline__ Rhs(int hi, int lo, f32x2) : h(hi), l(lo) {}
};
// A table entry: (hi, bits of (float)lo), or (hi, lo).  A pair of floats in
// registers would have to be assembled by moves, so its mixed terms are single
// FMAs.
template <bool X>
struct TabVal {
    int h;
    float f, l;
    __device__ __forceinline__ TabVal(int hi, int lo) : h(hi), f((float)hi), l(as_float(lo)) {}
};
template <>
struct TabVal<true> {
    int h, l;
    __device__ __forceinline__ TabVal(int hi, int lo) : h(hi), l(lo) {}
};
template <bool X>
__device__ __forceinline__ int2 tab_limbs(int2 v) {
    return X ? v : make_int2(v.x, as_int((float)v.y));
}
template <bool X>
__device__ __forceinline__ int4 tab_entry(int4 v) {
    const int2 a = tab_limbs<X>(make_int2(v.x, v.y)), b = tab_limbs<X>(make_int2(v.z, v.w));
    return make_int4(a.x, a.y, b.x, b.y);
}
// a value from its limbs
template <bool X>
__device__ __forceinline__ TabVal<X> tab_of(int2 v) {
    const int2 t = tab_limbs<X>(make_int2(opaque(v.x), X ? opaque(v.y) : v.y));
    return TabVal<X>(t.x, t.y);
}
template <bool X>
struct Acc {
    long long hh = 0;
    f32x2 f = 0;      // mixed terms, units of 2^-93
    float s = 0.f;    // those of table entries
    __device__ __forceinline__ void mac(const Lhs<X>& a, const Rhs<X>& b) {
        madw(hh, a.h, b.h);
        fma2(f, a.f, b.f);
    }
    __device__ __forceinline__ void mac(const TabVal<X>& a, const TabVal<X>& b) {
        madw(hh, a.h, b.h);
        s = fmaf(a.f, b.l, fmaf(a.l, b.f, s));
    }
    // a b + c d of one projector row
    __device__ __forceinline__ void mac(const TabVal<X>& a, const TabVal<X>& b, const TabVal<X>& c, const TabVal<X>& d) {
        mac(a, b);
        mac(c, d);
    }
    // rounded to 2^-62; |mixed| < 2^62, as ||u|| < 1/4
    __device__ __forceinline__ long long fold() const { return hh + __float2int_rn((sum2(f) + s) * 0x1p-31f); }
};
template <>
struct Acc<true> {
    long long hh = 0;
    // Mixed terms, units of 2^-93, and those of projector rows, units of 2^-85.
    // |hi lo| sums to less than 2^61.9 over the stencil (the |u| of 27 points of a
    // vector of norm 1/4: 1.75), |lo hi| to 2^62 (weights: 2^30, V and g: 2^31.6).
    long long hl = 0, lh = 0, hs = 0;
    __device__ __forceinline__ void mac(const Lhs<true>& a, const Rhs<true>& b) {
        madw(hh, a.h, b.h);
        madw(hl, a.h, b.l);
        madw(lh, a.l, b.h);
    }
    __device__ __forceinline__ void mac(const TabVal<true>& a, const TabVal<true>& b) {
        madw(hh, a.h, b.h);
        madw(hl, a.h, b.l);
        madw(lh, a.l, b.h);
    }
    // (up to 16 rows meet at a point: a row's mixed terms, below 2^62.7, are
    // scaled before they are added)
    __device__ __forceinline__ void mac(const TabVal<true>& a, const TabVal<true>& b, const TabVal<true>& c,
                                        const TabVal<true>& d) {
        madw(hh, a.h, b.h);
        madw(hh, c.h, d.h);
        long long m = 0;
        madw(m, a.h, b.l);
        madw(m, a.l, b.h);
        madw(m, c.h, d.l);
        madw(m, c.l, d.h);
        hs += m >> 8;
    }
    __device__ __forceinline__ long long fold() const { return hh + ((((hl + lh) >> 8) + hs + (1LL << 22)) >> 23); }
};
// Partial sums of u.w and w.w: hi hi exact, the mixed terms in float or, 16
// points at a time, in integers; the lo lo terms (in w.w they add up, 2e-13 of
// the sum) in float.
template <bool X>
struct Dots {
    long long hh1 = 0, hh2 = 0;
    f32x2 f1 = 0, f2 = 0;
    float q1 = 0.f;
    __device__ __forceinline__ void add(const Lhs<X>& u, int2 w) {
        madw(hh1, u.h, w.x);
        madw(hh2, w.x, w.x);
        const float wh = (float)w.x, wl = (float)w.y;
        fma2(f1, u.f, pack(wl, wh));
        fma2(f2, pack(wh, wl), pack(wl, wl * 0x1p-32f));
        q1 = fmaf(__uint_as_float((uint32_t)(u.f >> 32)), wl * 0x1p-31f, q1);
    }
    __device__ __forceinline__ void flush() {}
    // mixed parts in units of 2^-83 (w.w: half of them)
    __device__ __forceinline__ long long l1() const { return __float2ll_rn((sum2(f1) + q1) * 0x1p-10f); }
    __device__ __forceinline__ long long l2() const { return __float2ll_rn(sum2(f2) * 0x1p-10f); }
};
template <>
struct Dots<true> {
    long long hh1 = 0, hh2 = 0;
    long long x1 = 0, y1 = 0, x2 = 0, s1 = 0, s2 = 0;
    float q1 = 0.f, q2 = 0.f;
    int n = 0;
    __device__ __forceinline__ void add(const Lhs<true>& u, int2 w) {
        madw(hh1, u.h, w.x);
        madw(x1, u.h, w.y);
        madw(y1, u.l, w.x);
        madw(hh2, w.x, w.x);
        madw(x2, w.x, w.y);
        const float f = (float)w.y;
        q1 = fmaf((float)u.l, f, q1);
        q2 = fmaf(f, f, q2);
    }
    // after every pair: 8 pairs of |hi| <= 2^29 times |lo| <= 2^30 stay below 2^63
    __device__ __forceinline__ void flush() {
        if ((++n & 7) == 0) {
            s1 += (x1 >> 10) + (y1 >> 10);
            s2 += x2 >> 10;
            x1 = y1 = x2 = 0;
        }
    }
    __device__ __forceinline__ long long l1() const {
        return s1 + (x1 >> 10) + (y1 >> 10) + __float2ll_rn(q1 * 0x1p-41f);
    }
    __device__ __forceinline__ long long l2() const { return s2 + (x2 >> 10) + __float2ll_rn(q2 * 0x1p-42f); }
};
__device__ __forceinline__ int2 to_limbs(double v) { return split31(__double2ll_rn(v * 0x1p62)); }

struct KRow {        // one run of a projector row inside the slab
    int voff;        // index of window slot 0 in the u buffer
    int uu;          // u0 | u1 << 8 | local atom << 16
    int2 r0, r1, r2; // g_y g_z, (d g)_y g_z, g_y (d g)_z: hi, lo (a float unless the mixed terms are integers)
};
static_assert(sizeof(KRow) == 32, "row record");

struct KChunk {      // up to kKryChunkRows rows of one atom
    int row, count, slot, tab;
};

struct KShared {
    long long part[kMaxWarps][4];
    // per rank: u.w (2), w.w (2), stop flag of rank 0, ||w - alpha u||^2 (2), defect
    // of the FP64 check (a word of its own: no barrier of the cluster lies between
    // rank 0's reads of the last step's words and the check of a CTA with little to do)
    long long mbox[kMaxC][8];
    int2 ca, cg;                  // alpha and g as limbs
    int e;                        // u_new = (w - alpha u) 2^e
    int zlo[kMaxC + 1];           // first plane of each rank's slab
    int stop;                     // 0, 1 done, 2 timeout
    int work;
    // scalar warp's state
    double s0, inv0;              // ||u||^2, 1/||u||^2
    double drift;                 // bound of the relative error of s0
    double a_hat, b2_hat;         // alpha, beta^2 of the step just taken (in units of scale)
    double scale0;                // Lanczos breakdown scale
    int e_hat;                    // its e
    int nonfinite;
};
struct VecHead {      // one pole's update of its solution vector
    double sw, sv;    // powers of two the coefficients were divided by
    double2 om, nu;
    int act, first, last;   // last: the solution is complete, no further direction
};
struct KSharedVec {
    int4 co[4 * kKryVec];         // coefficients of the pole in hand
    VecHead head;
    double2 cp[kKryMaxPoles];     // pole factors of the outputs
};
struct KSharedNl {
    int n_local, n_rows, n_chunks, n_tab, over;
    int la_id[kMaxLocalProjAtoms];
    short la_off[kMaxLocalProjAtoms][3];
};

// Elements of a row in shared memory: even (pairs are 16-byte aligned), Q
// zeros after the row's points (they also serve as the next row's left
// neighbours) and a whole pair of zeros.
__host__ __device__ __forceinline__ int kry_pitch(int q, int m0) {
    const int e = (m0 + 1) & ~1;
    return (m0 + q > e + 2 ? m0 + q + 1 : e + 3) & ~1;
}
__device__ __forceinline__ int slab_lo(int m2, int C, int r) { return r * (m2 / C) + min(r, m2 % C); }

// Projector rows of the slab: per local atom, its window rows that meet the
// slab's planes and the region, split where the window wraps; chunks of rows
// for the projections, the atoms' x tables side by side, and for every pair
// of points (2k, 2k+1) of a region row the projector rows that cover one or
// both: 1 + row id | x table entry of the first << 16, entry of the second
// (entry and row 0 are zeros: a point outside the row, an empty record).
template <bool X>
__device__ void build_rows(const KrylovParams& P, const int m[3], const int lo[3], int z0, int depth, int q,
                           int pitch, int pp, KSharedNl& S, KRow* rows, KChunk* chunks, int4* xtab, int* cnt,
                           uint2* rec) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int npx = (m[0] + 1) >> 1;
    // local atoms in ascending order, the same list in every CTA of the cluster
    if (warp == 0) {
        int count = 0;
        for (long long base = 0; base < P.n_atoms; base += 32) {
            const long long a = base + lane;
            bool hit = a < P.n_atoms;
            short off[3] = {0, 0, 0};
            if (hit) {
                for (int d = 0; d < 3; ++d) {
                    const int len = P.proj_len[3 * a + d];
                    int o = P.proj_i0[3 * a + d] - lo[d];
                    if (P.periodic[d]) {
                        o %= P.n[d];
                        if (o < 0) o += P.n[d];
                        hit = hit && (o < m[d] || o + len - 1 >= P.n[d]);
                    } else {
                        hit = hit && o < m[d] && o + len - 1 >= 0;
                    }
                    off[d] = (short)o;
                }
            }
            const unsigned mask = __ballot_sync(0xffffffffu, hit);
            if (hit) {
                const int slot = count + __popc(mask & ((1u << lane) - 1u));
                if (slot < kMaxLocalProjAtoms) {
                    S.la_id[slot] = (int)a;
                    for (int d = 0; d < 3; ++d) S.la_off[slot][d] = off[d];
                }
            }
            count += __popc(mask);
        }
        if (lane == 0) {
            S.n_local = min(count, kMaxLocalProjAtoms);
            S.over = count > kMaxLocalProjAtoms;
            S.n_rows = 0;
            S.n_chunks = 0;
            S.n_tab = 0;
        }
    }
    __syncthreads();
    for (int k = warp; k < S.n_local; k += nw) {
        const int a = S.la_id[k];
        const int lx = P.proj_len[3 * a], ly = P.proj_len[3 * a + 1], lz = P.proj_len[3 * a + 2];
        const Runs rx = axis_runs(S.la_off[k][0], lx, P.n[0], m[0], P.periodic[0]);
        const unsigned char* rw = P.proj_rows + 2LL * a * kMaxProjWin * kMaxProjWin;
        const int4* tx = P.proj_fx + 3LL * a * kMaxProjWin;
        const int4* ty = tx + kMaxProjWin;
        const int4* tz = ty + kMaxProjWin;
        int first = 0, tab = 0;
        for (int pass = 0; pass < 2; ++pass) {
            int total = 0;
            for (int t0 = 0; t0 < 2 * ly * lz; t0 += 32) {
                const int t = t0 + lane;
                const int run = t & 1, row = t >> 1;
                bool ok = t < 2 * ly * lz;
                const int ww = ok ? row / ly : 0, vv = ok ? row - ww * ly : 0;
                const int b = region_slot(S.la_off[k][1], vv, P.n[1], m[1], P.periodic[1]);
                const int c = region_slot(S.la_off[k][2], ww, P.n[2], m[2], P.periodic[2]);
                ok = ok && b >= 0 && c >= z0 && c < z0 + depth;
                const int u0 = max((int)rw[2 * (ww * kMaxProjWin + vv)], rx.lo[run]);
                const int u1 = min((int)rw[2 * (ww * kMaxProjWin + vv) + 1], rx.hi[run]);
                ok = ok && u0 <= u1;
                const unsigned mask = __ballot_sync(0xffffffffu, ok);
                if (pass == 1 && ok) {
                    const int id = first + total + __popc(mask & ((1u << lane) - 1u));
                    KRow r;
                    const int sh = rx.shift[run];
                    r.voff = (c - z0 + q) * pp + b * pitch + sh;
                    r.uu = u0 | (u1 << 8) | (k << 16);
                    const int4 y = tab_entry<X>(ty[vv]), z = tab_entry<X>(tz[ww]);
                    Acc<X> r0, r1, r2;
                    r0.mac(TabVal<X>(y.x, y.y), TabVal<X>(z.x, z.y));
                    r1.mac(TabVal<X>(y.z, y.w), TabVal<X>(z.x, z.y));
                    r2.mac(TabVal<X>(y.x, y.y), TabVal<X>(z.z, z.w));
                    r.r0 = tab_limbs<X>(split31(r0.fold()));
                    r.r1 = tab_limbs<X>(split31(r1.fold()));
                    r.r2 = tab_limbs<X>(split31(r2.fold()));
                    rows[id] = r;
                    const int item0 = ((c - z0) * m[1] + b) * npx;
                    for (int pr = (u0 + sh) >> 1; pr <= (u1 + sh) >> 1; ++pr) {
                        const int u = 2 * pr - sh;   // window slot of the pair's first point
                        const bool f0 = u >= u0 && u <= u1, f1 = u + 1 >= u0 && u + 1 <= u1;
                        const uint32_t x = 1 + tab * P.win_x + u;
                        const int pos = atomicAdd(cnt + item0 + pr, 1);
                        if (pos < 2 * P.rec_words)
                            rec[(size_t)(item0 + pr) * 2 * P.rec_words + pos] =
                                make_uint2((uint32_t)(id + 1) | (f0 ? x << 16 : 0u), (f1 ? x + 1 : 0u) | (uint32_t)k << 16);
                        else S.over = 1;
                    }
                }
                total += __popc(mask);
            }
            if (pass == 0) {
                if (total == 0) break;
                const int nch = (total + kKryChunkRows - 1) / kKryChunkRows;
                int cf = 0;
                if (lane == 0) {
                    first = atomicAdd(&S.n_rows, total);
                    cf = atomicAdd(&S.n_chunks, nch);
                    tab = atomicAdd(&S.n_tab, 1);
                }
                first = __shfl_sync(0xffffffffu, first, 0);
                cf = __shfl_sync(0xffffffffu, cf, 0);
                tab = __shfl_sync(0xffffffffu, tab, 0);
                if (first + total > P.row_cap) {
                    if (lane == 0) S.over = 1;
                    break;
                }
                for (int i = lane; i < nch; i += 32)
                    chunks[cf + i] = KChunk{first + kKryChunkRows * i, min(kKryChunkRows, total - kKryChunkRows * i), k,
                                            1 + tab * P.win_x};
                for (int u = lane; u < P.win_x; u += 32) xtab[1 + tab * P.win_x + u] = tab_entry<X>(tx[u]);
            }
        }
    }
    __syncthreads();
    // A pair's entries by atom and row, whichever warp was first: the mixed
    // terms of mixed precision are floats, whose sum depends on the order.
    // (Row ids ascend within an atom; the atom's slot rides in the second word.)
    for (int t = threadIdx.x; t < depth * m[1] * npx; t += blockDim.x) {
        uint2* r = rec + (size_t)t * 2 * P.rec_words;
        const int n = min(cnt[t], 2 * P.rec_words);
        auto key = [](uint2 e) { return (e.y & 0xffff0000u) | (e.x & 0xffffu); };
        for (int i = 1; i < n; ++i) {
            const uint2 e = r[i];
            int j = i;
            for (; j > 0 && key(r[j - 1]) > key(e); --j) r[j] = r[j - 1];
            r[j] = e;
        }
        for (int i = 0; i < n; ++i) r[i].y &= 0xffffu;
    }
    __syncthreads();
}

// Sum over the warp of four 64-bit values; lane l of the first four ends
// with value l.
__device__ __forceinline__ long long warp_sum4(long long s0, long long s1, long long s2, long long s3, int lane) {
    const bool h1 = lane & 1, h2 = lane & 2;
    long long a = h1 ? s1 : s0, b = h1 ? s3 : s2;
    a += __shfl_xor_sync(0xffffffffu, h1 ? s0 : s1, 1);
    b += __shfl_xor_sync(0xffffffffu, h1 ? s2 : s3, 1);
    long long c = h2 ? b : a;
    c += __shfl_xor_sync(0xffffffffu, h2 ? a : b, 2);
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    return c;
}

// Partial projections of u on the local atoms over this slab, added to
// acc[slot][l].  The projectors are products of x, y and z tables: a half
// warp takes one row at a time, a lane per x, and sums R u over the rows for
// the row's three y z factors R; the x tables enter once, at the end.
// (A lane per row, each walking its run with both x tables, took 21,800
// cycles a step on the bulk regions, four times the issue slots.)
template <bool X>
__device__ __forceinline__ void project(const KrylovParams& P, const int2* __restrict__ U, const KRow* rows,
                                        const KChunk* chunks, int n_chunks, int nw, const int4* xtab, int4* stage,
                                        long long* acc) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, half = lane >> 4;
    stage += warp * 2 * kKryChunkRows;
    // a lane's row of the next chunk is on its way while this one is summed
    const int4 none = make_int4(0, 0xff, 0, 0);   // an empty run
    int4 n0 = none, n1 = none;
    if (warp < n_chunks && lane < chunks[warp].count) {
        const int4* r = reinterpret_cast<const int4*>(rows + chunks[warp].row + lane);
        n0 = r[0];
        n1 = r[1];
    }
    for (int ch = warp; ch < n_chunks; ch += nw) {
        const KChunk k = chunks[ch];
        __syncwarp();
        stage[2 * lane] = n0;
        stage[2 * lane + 1] = n1;
        n0 = none;
        if (ch + nw < n_chunks && lane < chunks[ch + nw].count) {
            const int4* r = reinterpret_cast<const int4*>(rows + chunks[ch + nw].row + lane);
            n0 = r[0];
            n1 = r[1];
        }
        __syncwarp();
        long long s0 = 0, s1 = 0, s2 = 0, s3 = 0;
        for (int ub = 0; ub < P.win_x; ub += 16) {
            const int u = ub + (lane & 15);
            Acc<X> A0, A1, A2;
            const int4* st = stage + 2 * half;
            // rows past the count are empty runs, so the half warps stay together
#pragma unroll 4
            for (int i = 0; i < k.count; i += 2) {
                const int4 a = st[2 * i], b = st[2 * i + 1];
                const int u0 = a.y & 0xff, u1 = (a.y >> 8) & 0xff;
                int2 v = make_int2(0, 0);
                if (u >= u0 && u <= u1) v = U[a.x + u];
                const TabVal<X> t = tab_of<X>(v);
                A0.mac(t, TabVal<X>(a.z, a.w));
                A1.mac(t, TabVal<X>(b.x, b.y));
                A2.mac(t, TabVal<X>(b.z, b.w));
            }
            const int4 t = u < P.win_x ? xtab[k.tab + u] : make_int4(0, 0, 0, 0);
            const TabVal<X> g(t.x, t.y), dg(t.z, t.w);
            const int2 l0 = tab_limbs<X>(split31(A0.fold())), l1 = tab_limbs<X>(split31(A1.fold()));
            const int2 l2 = tab_limbs<X>(split31(A2.fold()));
            Acc<X> r0, r1, r2, r3;
            r0.mac(TabVal<X>(l0.x, l0.y), g);
            r1.mac(TabVal<X>(l0.x, l0.y), dg);
            r2.mac(TabVal<X>(l1.x, l1.y), g);
            r3.mac(TabVal<X>(l2.x, l2.y), g);
            s0 += r0.fold();
            s1 += r1.fold();
            s2 += r2.fold();
            s3 += r3.fold();
        }
        const long long s = warp_sum4(s0, s1, s2, s3, lane);
        if (lane < 4)
            atomicAdd(reinterpret_cast<unsigned long long*>(acc + 4 * k.slot + lane), (unsigned long long)s);
    }
}

// One row's factors of the apply: nonlocal(u)(i) = sum over the rows that
// cover i of g_x K1 + (d g)_x K2.
template <bool X>
__device__ __forceinline__ int4 row_factors(const KRow* row, const int2* cl) {
    const int4 a = reinterpret_cast<const int4*>(row)[0], b = reinterpret_cast<const int4*>(row)[1];
    const int4* c = reinterpret_cast<const int4*>(cl + 4 * ((a.y >> 16) & 0xff));
    const int4 c01 = c[0], c23 = c[1];
    Acc<X> k1, k2;
    k1.mac(TabVal<X>(a.z, a.w), TabVal<X>(c01.x, c01.y));
    k1.mac(TabVal<X>(b.x, b.y), TabVal<X>(c23.x, c23.y));
    k1.mac(TabVal<X>(b.z, b.w), TabVal<X>(c23.z, c23.w));
    k2.mac(TabVal<X>(a.z, a.w), TabVal<X>(c01.z, c01.w));
    const int2 x = tab_limbs<X>(split31(k1.fold())), y = tab_limbs<X>(split31(k2.fold()));
    return make_int4(x.x, x.y, y.x, y.y);
}

// A slab as pairs of points (2k, 2k+1) along x, `npc` a plane: two points a
// thread halve the shared-memory instructions of the stencil (16-byte loads)
// and give each thread two independent sums.
struct SlabArgs {
    const int2* U;
    int4* Vp;            // [depth][npc] V limbs of the pair
    longlong2* Wp;       // w
    const uint4* Rec;    // [depth][npc][rec_words]
    int m0, m1, npx, npc, n_items, pitch, pp;
    FastDiv div_pc, div_px;
};

// Nonlocal term of one record entry on both points of a pair.
template <bool X>
__device__ __forceinline__ void nl_entry(const int4* ktab, const int4* xtab, uint32_t e0, uint32_t e1,
                                         Acc<X> (&acc)[2]) {
    const int4 k = ktab[e0 & 0xffffu], t0 = xtab[e0 >> 16], t1 = xtab[e1];
    const TabVal<X> k1(k.x, k.y), k2(k.z, k.w);
    acc[0].mac(TabVal<X>(t0.x, t0.y), k1, TabVal<X>(t0.z, t0.w), k2);
    acc[1].mac(TabVal<X>(t1.x, t1.y), k1, TabVal<X>(t1.z, t1.w), k2);
}

// Sums of the stencil's off-diagonal terms on a pair at p (16-byte units);
// kInside: the rows b-Q .. b+Q all lie in the region.
template <int Q, bool kInside, bool X>
__device__ __forceinline__ void stencil(const KrylovParams& P, const SlabArgs& A, const int4* p, int4 c, int a, int b,
                                        Acc<X> (&acc)[2]) {
    constexpr int H = (Q + 1) / 2;   // loads on either side of the pair
    const int pitch = A.pitch >> 1, pp = A.pp >> 1;
    auto add = [&](int i, int h, int l, int d, int o) {
        acc[i].mac(Lhs<X>(h, l), Rhs<X>(P.wh[d][o - 1], P.wl[d][o - 1], P.wf[d][o - 1]));
    };
    {
        int2 x[2 * (2 * H + 1)];     // the row around the pair: x[2H], x[2H+1] are its points
#pragma unroll
        for (int h = 0; h <= 2 * H; ++h) {
            const int4 t = h == H ? c : p[h - H];
            x[2 * h] = make_int2(t.x, t.y);
            x[2 * h + 1] = make_int2(t.z, t.w);
        }
#pragma unroll
        for (int o = 1; o <= Q; ++o)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int2 xa = x[2 * H + i + o], xb = x[2 * H + i - o];
                add(i, xa.x + xb.x, xa.y + xb.y, 0, o);
            }
    }
    const int zero = (((A.m0 + 1) & ~1) - a) >> 1;   // two of the zeros after this row
#pragma unroll
    for (int o = 1; o <= Q; ++o) {
        const int4 ya = p[kInside || b + o < A.m1 ? o * pitch : zero], yb = p[kInside || b - o >= 0 ? -o * pitch : zero];
        add(0, ya.x + yb.x, ya.y + yb.y, 1, o);
        add(1, ya.z + yb.z, ya.w + yb.w, 1, o);
    }
#pragma unroll
    for (int o = 1; o <= Q; ++o) {
        const int4 za = p[o * pp], zb = p[-o * pp];
        add(0, za.x + zb.x, za.y + zb.y, 2, o);
        add(1, za.z + zb.z, za.w + zb.w, 2, o);
    }
}

// w = A u - g u_prev over the slab, stored to Wp, and the partial sums of
// u.w and w.w (g negated by the caller).  Every stencil value is read from
// shared memory: a column's z values kept in registers along a march save
// seven of the twenty 16-byte loads of a pair but need more than 128 registers,
// and 19 warps at 96 registers are the faster trade.
template <int Q, bool kNl, bool X>
__device__ __forceinline__ void slab_apply(const KrylovParams& P, const SlabArgs& A, const int4* ktab,
                                           const int4* xtab, const int4* u_prev, int nw, int2 g, Dots<X>& dots) {
    const Rhs<X> gr(opaque(g.x), opaque(g.y));
    // lanes past the last pair repeat it and add nothing, so that warps stay whole
    for (int i0 = threadIdx.x & ~31; i0 < A.n_items; i0 += 32 * nw) {
        const int i = i0 + (int)(threadIdx.x & 31);
        const bool act = i < A.n_items;
        const int item = act ? i : A.n_items - 1;
        const int4 v = A.Vp[item], um = u_prev[item];   // used after the stencil sums
        uint4 rc = make_uint4(0u, 0u, 0u, 0u);
        if (kNl) rc = A.Rec[(size_t)item * P.rec_words];
        const int d = (int)fdiv((uint32_t)item, A.div_pc), pc = item - d * A.npc;
        const int b = (int)fdiv((uint32_t)pc, A.div_px), a = 2 * (pc - b * A.npx);
        const int4* p = reinterpret_cast<const int4*>(A.U + (d + Q) * A.pp + b * A.pitch + a);
        const int4 c = *p;
        Acc<X> acc[2];
        if (__all_sync(0xffffffffu, b >= Q && b + Q < A.m1)) stencil<Q, true>(P, A, p, c, a, b, acc);
        else stencil<Q, false>(P, A, p, c, a, b, acc);
        const Lhs<X> c0(c.x, c.y), c1(c.z, c.w);
        acc[0].mac(c0, Rhs<X>(v.x, v.y));
        acc[1].mac(c1, Rhs<X>(v.z, v.w));
        acc[0].mac(Lhs<X>(um.x, um.y), gr);
        acc[1].mac(Lhs<X>(um.z, um.w), gr);
        if constexpr (kNl) {
            for (int q = 0; q < P.rec_words; ++q) {
                const uint4 r = q == 0 ? rc : A.Rec[(size_t)item * P.rec_words + q];
                if (!__any_sync(0xffffffffu, r.x)) break;
                nl_entry(ktab, xtab, r.x, r.y, acc);
                if (!__any_sync(0xffffffffu, r.z)) break;
                nl_entry(ktab, xtab, r.z, r.w, acc);
            }
        }
        const long long r0 = acc[0].fold();
        const long long r1 = a + 1 < A.m0 ? acc[1].fold() : 0;
        if (act) {
            A.Wp[item] = make_longlong2(r0, r1);
            dots.add(c0, split31(r0));
            dots.add(c1, split31(r1));
            dots.flush();
        }
    }
}

__device__ __forceinline__ double limbs(int hi, int lo) { return fma((double)hi, 0x1p-31, (double)lo * 0x1p-62); }

// Sum over the slab of (A u - g u_prev - w)^2, everything evaluated in FP64
// from the FP64 potential and projector values: how far the fixed-point step
// just taken is from the operator's.  c: [n_local][4] projections, zeroed here;
// xsum exchanges them over the cluster.  A CTA's share is summed in units of
// 2^-60 / sqrt(dV) (a projector has norm 1 / sqrt(dV) and ||u|| < 1/4), so that
// it does not depend on the order of the atomics.
template <int Q, bool kNl, class F>
__device__ __noinline__ double check_step(const KrylovParams& P, const SlabArgs& A, const int lo[3], int z0,
                                          const KSharedNl& S, double* c, const int4* u_prev, int2 g2,
                                          F&& xsum) {
    const double g = limbs(g2.x, g2.y);
    auto global_point = [&](int item, int& d, int& b, int& a) {
        d = item / A.npc;
        const int pc = item - d * A.npc;
        b = pc / A.npx;
        a = 2 * (pc - b * A.npx);
        return (long long)P.n[0] * (wrap_once(lo[1] + b, P.n[1]) + (long long)P.n[1] * wrap_once(lo[2] + z0 + d, P.n[2]));
    };
    auto slot_of = [&](int atom) {
        int l = 0, h = S.n_local - 1;
        while (l <= h) {
            const int m = (l + h) >> 1;
            if (S.la_id[m] == atom) return m;
            if (S.la_id[m] < atom) l = m + 1;
            else h = m - 1;
        }
        return -1;
    };
    if constexpr (kNl) {
        unsigned long long* ci = reinterpret_cast<unsigned long long*>(c);
        const double unit = sqrt(P.dV) * 0x1p60;
        for (int t = threadIdx.x; t < 4 * S.n_local; t += blockDim.x) ci[t] = 0;
        __syncthreads();
        for (int item = threadIdx.x; item < A.n_items; item += blockDim.x) {
            int d, b, a;
            const long long row = global_point(item, d, b, a);
            for (int i = 0; i < 2 && a + i < A.m0; ++i) {
                const int2 u2 = A.U[(d + Q) * A.pp + b * A.pitch + a + i];
                const double u = limbs(u2.x, u2.y);
                const long long gi = row + wrap_once(lo[0] + a + i, P.n[0]);
                for (int e = P.pl_ptr[gi]; e < P.pl_ptr[gi + 1]; ++e) {
                    const int s = slot_of(P.pl_atom[e]);
                    if (s < 0) continue;
                    const double2 p = P.pl_val64[2 * e], q = P.pl_val64[2 * e + 1];
                    const double f[4] = {p.x, p.y, q.x, q.y};
                    for (int l = 0; l < 4; ++l)
                        atomicAdd(ci + 4 * s + l, (unsigned long long)__double2ll_rn(f[l] * u * unit));
                }
            }
        }
        __syncthreads();
        for (int t = threadIdx.x; t < 4 * S.n_local; t += blockDim.x) c[t] = (double)(long long)ci[t] / unit;
        xsum();
    }
    const double inv = 1.0 / P.scale;
    double s2 = 0.0;
    for (int item = threadIdx.x; item < A.n_items; item += blockDim.x) {
        int d, b, a;
        const long long row = global_point(item, d, b, a);
        for (int i = 0; i < 2 && a + i < A.m0; ++i) {
            const int2* p = A.U + (d + Q) * A.pp + b * A.pitch + a + i;
            const long long gi = row + wrap_once(lo[0] + a + i, P.n[0]);
            double y = P.V[gi] * limbs(p->x, p->y);
            for (int o = 1; o <= Q; ++o) {
                double s = limbs(p[o].x, p[o].y) + limbs(p[-o].x, p[-o].y);
                y += P.coef[0][o - 1] * s;
                s = 0.0;
                if (b + o < A.m1) s += limbs(p[o * A.pitch].x, p[o * A.pitch].y);
                if (b - o >= 0) s += limbs(p[-o * A.pitch].x, p[-o * A.pitch].y);
                y += P.coef[1][o - 1] * s;
                y += P.coef[2][o - 1] * (limbs(p[o * A.pp].x, p[o * A.pp].y) + limbs(p[-o * A.pp].x, p[-o * A.pp].y));
            }
            if constexpr (kNl) {
                for (int e = P.pl_ptr[gi]; e < P.pl_ptr[gi + 1]; ++e) {
                    const int s = slot_of(P.pl_atom[e]);
                    if (s < 0) continue;
                    const double2 v = P.pl_val64[2 * e], q = P.pl_val64[2 * e + 1];
                    y += P.dV * (P.e_s * v.x * c[4 * s] + P.e_p * (v.y * c[4 * s + 1] + q.x * c[4 * s + 2] + q.y * c[4 * s + 3]));
                }
            }
            const int4 um = u_prev[item];
            const longlong2 w = A.Wp[item];
            const double t = y * inv - g * (i ? limbs(um.z, um.w) : limbs(um.x, um.y)) - (double)(i ? w.y : w.x) * 0x1p-62;
            s2 += t * t;
        }
    }
    return s2;
}

// The scalar recurrences of one pole (see the head of this file), in units
// of the scaled operator.
struct PoleState {
    double zr, zi;     // (z - shift) / scale
    double er, ei;     // beta^2 / d of the previous step
    double fr, fi;     // zeta^2
    double gr, gi;     // x(j) * scale
    double rn;         // ||r||
    int conv;          // step at which ||r|| <= tol
    double cr, ci;     // chi = zeta / ||u||
    double mr, mi;     // m of the last step of the chunk before
};
__device__ __forceinline__ void pole_step(PoleState& s, double a, double b2, bool sum) {
    const double dr = a - s.zr - s.er, di = -s.zi - s.ei;
    const double inv = 1.0 / (dr * dr + di * di);
    const double ir = dr * inv, ii = -di * inv;
    const double qr = s.fr * ir - s.fi * ii, qi = s.fr * ii + s.fi * ir;
    if (sum) {
        s.gr += qr;
        s.gi += qi;
    }
    s.er = b2 * ir;
    s.ei = b2 * ii;
    s.fr = qr * s.er - qi * s.ei;
    s.fi = qr * s.ei + qi * s.er;
}

// Solution vectors.  In terms of the vectors u_k as kept, COCG's directions
// and iterates of a pole are
//   p_k = u_k - m_{k-1} p_{k-1},   m_k = 2^{e_k} beta_k^2 / d_k,
//   x  += c_k p_k,                 c_k = chi_k / d_k,  chi_{k+1} = -2^{-e_k} c_k.
// kKryVec steps are applied at a time: with u_{s+1} .. u_e kept,
//   x <- x + sum_j w_j u_j + omega p_s,   w_j = c_j - m_j w_{j+1}, omega = -m_s w_{s+1},
//   p <-     sum_j v_j u_j + nu p_s,      v_j = -m_j v_{j+1},      nu = -m_s v_{s+1}.
struct VecHist {
    double2 c, m;
};

// Coefficients of a pole's update as fixed point: {hi, (float)hi, (float)lo, lo}
// of Re w, Im w, Re v, Im v for every vector, scaled to an l1 norm below 1/2
// so that no sum overflows.
__device__ void vec_coefs(const VecHist* hist, int n, int s0, PoleState& s, int pole, int4* co, VecHead* head) {
    double2 w = make_double2(0.0, 0.0), v = make_double2(1.0, 0.0);
    double nw = 0.0, nv = 0.0;
    for (int pass = 0; pass < 2; ++pass) {
        double sw = 1.0, sv = 1.0;
        if (pass == 1) {   // powers of two above twice the norms
            if (nw > 0.0) sw = __hiloint2double(((__double2hiint(nw) >> 20) + 2) << 20, 0);
            sv = __hiloint2double(((__double2hiint(nv) >> 20) + 2) << 20, 0);
        }
        for (int j = n - 1; j >= 0; --j) {
            const VecHist h = hist[(size_t)j * kKryMaxPoles + pole];
            const bool on = s.conv == 0 || s0 + 1 + j <= s.conv;   // a solution ends where its pole met tol
            const double2 c = on ? h.c : make_double2(0.0, 0.0);
            if (j == n - 1) {
                w = c;
                v = make_double2(1.0, 0.0);
            } else {
                w = make_double2(c.x - (h.m.x * w.x - h.m.y * w.y), c.y - (h.m.x * w.y + h.m.y * w.x));
                v = make_double2(-(h.m.x * v.x - h.m.y * v.y), -(h.m.x * v.y + h.m.y * v.x));
            }
            if (pass == 0) {
                nw += fabs(w.x) + fabs(w.y);
                nv += fabs(v.x) + fabs(v.y);
            } else {
                const double f[4] = {w.x / sw, w.y / sw, v.x / sv, v.y / sv};
                for (int k = 0; k < 4; ++k) {
                    const int2 l = to_limbs(f[k]);
                    co[4 * j + k] = make_int4(l.x, __float_as_int((float)l.x), __float_as_int((float)l.y), l.y);
                }
            }
        }
        if (pass == 1) {
            head->sw = sw;
            head->sv = sv;
            head->om = make_double2(-(s.mr * w.x - s.mi * w.y), -(s.mr * w.y + s.mi * w.x));
            head->nu = make_double2(-(s.mr * v.x - s.mi * v.y), -(s.mr * v.y + s.mi * v.x));
            head->act = s.conv == 0 || s.conv > s0;
            head->first = s0 == 0;
            head->last = s.conv != 0;
        }
    }
    const double2 m = hist[(size_t)(n - 1) * kKryMaxPoles + pole].m;
    s.mr = m.x;
    s.mi = m.y;
}

// x and p of one pole over the slab: fixed-point sums over the kept vectors
// (the mixed terms in float or in integers), joined in FP64.  A pair's
// first point lies at Xv[xoff(item)], the second beside it.
template <bool kLast, bool X, class F>
__device__ __forceinline__ void vec_update(const SlabArgs& A, int n, const int4* co, const VecHead& h, const int4* Ub,
                                           double2* Xv, double2* Pv, F&& xoff) {
    const double sx = h.sw * 0x1p-62, sp = h.sv * 0x1p-62;
    for (int item = threadIdx.x; item < A.n_items; item += blockDim.x) {
        long long hh[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        // (integers: the u_j of one point are entries of nearly orthogonal vectors of
        // norm 1/4, so the 32 |u_j| sum to less than sqrt(32) / 4, the |lo| terms to 2^62)
        float f[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        long long mx[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        const int4* up = Ub + item;
#pragma unroll 2
        for (int j = 0; j < n; ++j) {
            const int4 u = *up;
            up += A.n_items;
            const float a0 = (float)u.x, b0 = (float)u.y, a1 = (float)u.z, b1 = (float)u.w;
#pragma unroll
            for (int k = 0; k < (kLast ? 2 : 4); ++k) {
                const int4 c = co[4 * j + k];
                madw(hh[2 * k], u.x, c.x);
                madw(hh[2 * k + 1], u.z, c.x);
                if constexpr (X) {
                    madw(mx[2 * k], u.x, c.w);
                    madw(mx[2 * k], u.y, c.x);
                    madw(mx[2 * k + 1], u.z, c.w);
                    madw(mx[2 * k + 1], u.w, c.x);
                } else {
                    const float ch = as_float(c.y), cl = as_float(c.z);
                    f[2 * k] = fmaf(a0, cl, fmaf(b0, ch, f[2 * k]));
                    f[2 * k + 1] = fmaf(a1, cl, fmaf(b1, ch, f[2 * k + 1]));
                }
            }
        }
        double2* x = Xv + xoff(item);
        double2* p = Pv + 2 * (size_t)item;
        const int pc = item % A.npc;
        const int two = 2 * (pc % A.npx) + 1 < A.m0 ? 2 : 1;
        for (int i = 0; i < two; ++i) {
            double v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                v[k] = (double)((i ? hh[2 * k + 1] : hh[2 * k]) +
                                (X ? (i ? mx[2 * k + 1] : mx[2 * k]) >> 31
                                   : (long long)((i ? f[2 * k + 1] : f[2 * k]) * 0x1p-31f)));
            double2 xv = make_double2(v[0] * sx, v[1] * sx), pv = make_double2(v[2] * sp, v[3] * sp);
            if (!h.first) {
                const double2 po = p[i], xo = x[i];
                xv.x += xo.x + (h.om.x * po.x - h.om.y * po.y);
                xv.y += xo.y + (h.om.x * po.y + h.om.y * po.x);
                pv.x += h.nu.x * po.x - h.nu.y * po.y;
                pv.y += h.nu.x * po.y + h.nu.y * po.x;
            }
            x[i] = xv;
            if (!kLast) p[i] = pv;
        }
    }
}

template <int Q, bool kNl, bool X>
__global__ void __launch_bounds__(kMaxThreads, 1) k_krylov(const __grid_constant__ KrylovParams P) {
    extern __shared__ __align__(16) unsigned char dsm[];
    __shared__ KShared S;
    __shared__ KSharedVec SV;
    __shared__ KSharedNl SN[1];   // untouched (and dropped) without projectors
    const int C = (int)k_nrank(), rank = (int)k_rank();
    const int nwp = (int)(blockDim.x >> 5) - 1;  // warps that compute points
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool scalar_warp = warp == nwp;
    // the budget runs from the first CTA of any of the call's launches
    uint64_t t_start = 0;
    if (P.timeout_ns && rank == 0 && scalar_warp && lane == 0) {
        const uint64_t now = global_time_ns(), first = atomicCAS(P.t_start, 0ULL, (unsigned long long)now);
        t_start = first ? first : now;
    }
    auto timed_out = [&]() {   // lane 0 of rank 0's scalar warp
        if (!P.timeout_ns) return false;
        const uint64_t now = global_time_ns();
        return now > t_start && now - t_start > P.timeout_ns;
    };
    int2* U = reinterpret_cast<int2*>(dsm);
    char* slot = P.scratch + (size_t)blockIdx.x * P.cta_bytes;
    char* slot0 = P.scratch + (size_t)(blockIdx.x - rank) * P.cta_bytes;   // rank 0's slot
    int4* const Vp = reinterpret_cast<int4*>(slot);
    int4* const Up = reinterpret_cast<int4*>(slot + P.off_up);   // u_k limbs in place (k - 1) mod ring
    const int ring = P.vec ? kKryVec : 1;
    double2* const Xs = reinterpret_cast<double2*>(slot + P.off_x);
    double2* const Ps = reinterpret_cast<double2*>(slot + P.off_p);
    VecHist* const hist = reinterpret_cast<VecHist*>(slot0 + P.off_hist);
    char* const coef = slot0 + P.off_coef;   // per pole: VecHead, then kKryVec x 4 int4
    constexpr size_t kCoefBytes = 128 + sizeof(int4) * 4 * kKryVec;
    longlong2* const Wp = reinterpret_cast<longlong2*>(slot + P.off_w);
    uint4* const Rec = reinterpret_cast<uint4*>(slot + P.off_rec);
    KRow* const rows = reinterpret_cast<KRow*>(slot + P.off_rows);
    KChunk* const chunks = reinterpret_cast<KChunk*>(slot + P.off_chunk);
    long long* const cpart = reinterpret_cast<long long*>(slot + P.off_cpart);

    k_sync();   // every CTA of the cluster runs: its shared memory may be written from here on
    for (;;) {
        if (rank == 0 && tid == 0) {
            const int w = (int)atomicAdd(P.work_counter, 1u);
            for (int r = 0; r < C; ++r) {
                uint32_t a = k_map(smem_addr(&S.work), r);
                asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(a), "r"(w) : "memory");
            }
        }
        k_sync();
        if (S.work >= P.n_work) break;
        const int node = P.list[S.work];
        const NodeDesc nd = P.nodes[node];
        const int m[3] = {nd.dims[0], nd.dims[1], nd.dims[2]};
        const int lo[3] = {nd.lo[0], nd.lo[1], nd.lo[2]};
        const int m0 = m[0], m1 = m[1], m2 = m[2];
        const int npx = (m0 + 1) >> 1, npc = npx * m1, ncol = m0 * m1;
        const int pitch = kry_pitch(Q, m0), pp = pitch * m1;
        const FastDiv div_px = make_fastdiv((uint32_t)npx);
        const int z0 = slab_lo(m2, C, rank), depth = slab_lo(m2, C, rank + 1) - z0;
        const int n_items = depth * npc;
        const int src_z = nd.src / ncol, src_col = nd.src - src_z * ncol;

        // ---- set-up: zero u, V limbs, projector rows ------------------------
        for (int t = tid; t < (depth + 2 * Q) * pp; t += blockDim.x) U[t] = make_int2(0, 0);
        if (tid == 0) S.nonfinite = 0;
        if (tid <= C) S.zlo[tid] = slab_lo(m2, C, tid);
        if (kNl) {
            for (int t = tid; t < n_items; t += blockDim.x) reinterpret_cast<int*>(Wp)[t] = 0;   // record lengths
            for (int t = tid; t < n_items * P.rec_words; t += blockDim.x) Rec[t] = make_uint4(0u, 0u, 0u, 0u);
        }
        __syncthreads();
        const double vs = 0x1p62 / P.scale;
        for (int t = tid; t < n_items; t += blockDim.x) {
            const int d = t / npc, pc = t - d * npc;
            const int b = (int)fdiv((uint32_t)pc, div_px), a = 2 * (pc - b * npx);
            const int gy = wrap_once(lo[1] + b, P.n[1]), gz = wrap_once(lo[2] + z0 + d, P.n[2]);
            const double* row = P.V + (long long)P.n[0] * (gy + (long long)P.n[1] * gz);
            int2 x[2] = {make_int2(0, 0), make_int2(0, 0)};
            for (int i = 0; i < 2 && a + i < m0; ++i) {
                const double v = row[wrap_once(lo[0] + a + i, P.n[0])];
                if (!(fabs(v) < 0.5 * P.scale)) S.nonfinite = 1;
                x[i] = split31(__double2ll_rn(v * vs));
            }
            Vp[t] = make_int4(x[0].x, x[0].y, x[1].x, x[1].y);
            Up[(size_t)(ring - 1) * n_items + t] = make_int4(0, 0, 0, 0);   // u_0 = 0
        }
        long long* acc = nullptr;   // [n_local][4] partial projections
        int2* cl = nullptr;         // [n_local][4] coefficients
        double* cf = nullptr;       // [n_local][4] their factors
        int4* xtab = nullptr;       // x tables of the slab's atoms
        int4* ktab = nullptr;       // [1 + n_rows] row factors of the apply, a zero row first
        bool tab_smem = true;       // both in shared memory
        int4 *xt_s = nullptr, *kt_s = nullptr;   // where they lie in shared memory
        int4* stage = nullptr;      // rows of the chunk a warp works on
        const KChunk* chk = chunks;
        int n_loc4 = 0, n_rows = 0, n_x = 0;
        if constexpr (kNl) {
            build_rows<X>(P, m, lo, z0, depth, Q, pitch, pp, SN[0], rows, chunks,
                       reinterpret_cast<int4*>(slot + P.off_xtab), reinterpret_cast<int*>(Wp),
                       reinterpret_cast<uint2*>(Rec));
            n_loc4 = 4 * SN[0].n_local;
            n_rows = min(SN[0].n_rows, P.row_cap);
            n_x = SN[0].n_tab * P.win_x;
            const size_t off = ((size_t)(depth + 2 * Q) * pp * sizeof(int2) + 15) / 16 * 16;
            // [projections][x tables][chunks][row factors | staged rows]: the
            // rows are staged before the factors are formed
            acc = reinterpret_cast<long long*>(dsm + off);
            cl = reinterpret_cast<int2*>(acc + n_loc4);
            cf = reinterpret_cast<double*>(cl + n_loc4);
            xt_s = reinterpret_cast<int4*>(cf + n_loc4);
            int4* const xg = reinterpret_cast<int4*>(slot + P.off_xtab);
            const int n_ch = SN[0].n_chunks, n_st = (nwp + 1) * 2 * kKryChunkRows;
            kt_s = xt_s + n_x + 1 + n_ch;
            if ((size_t)((unsigned char*)kt_s - dsm) + (size_t)max(n_rows + 1, n_st) * 16 <= (size_t)P.smem_bytes) {
                xtab = xt_s;
                ktab = stage = kt_s;
                KChunk* cs = reinterpret_cast<KChunk*>(xt_s + n_x + 1);
                for (int t = tid; t <= n_x; t += blockDim.x) xtab[t] = xg[t];
                for (int t = tid; t < n_ch; t += blockDim.x) cs[t] = chunks[t];
                chk = cs;
            } else {   // slower, but any number of rows
                tab_smem = false;
                stage = reinterpret_cast<int4*>(dsm + off);
                xtab = xg;
                ktab = reinterpret_cast<int4*>(slot + P.off_ktab);
                acc = cpart + 4 * kMaxLocalProjAtoms;
                cl = reinterpret_cast<int2*>(acc + 4 * kMaxLocalProjAtoms);
                cf = reinterpret_cast<double*>(cl + 4 * kMaxLocalProjAtoms);
            }
            for (int t = tid; t < n_loc4; t += blockDim.x) {
                acc[t] = 0;
                cf[t] = P.proj_fxc[4LL * SN[0].la_id[t >> 2] + (t & 3)] / P.scale * 0x1p-62;
            }
            __syncthreads();
            if (tid == 0) xtab[0] = make_int4(0, 0, 0, 0);
        }
        const SlabArgs SA{U, Vp, Wp, Rec, m0, m1, npx, npc, n_items, pitch, pp,
                          make_fastdiv((uint32_t)npc), div_px};
        __syncthreads();
        // any CTA that cannot run the node stops the whole cluster
        if (tid == 0) {
            const long long bad = S.nonfinite ? 3 : (kNl && SN[0].over ? 1 : 0);
            for (int r = 0; r < C; ++r) k_st_remote(k_map(smem_addr(&S.mbox[rank][4]), r), bad);
        }
        k_sync();
        int bad = 0;
        for (int r = 0; r < C; ++r) bad = max(bad, (int)S.mbox[r][4]);
        // u_1 = e_j / 8, pushed to every CTA whose slab or halo holds the plane
        if (tid == 0) {
            const int b = src_col / m0, a = src_col - b * m0;
            if (src_z >= z0 - Q && src_z < z0 + depth + Q)
                U[(src_z - z0 + Q) * pp + b * pitch + a] = split31(1LL << 59);
            S.s0 = 0x1p-6;
            S.inv0 = 0x1p6;
            S.drift = 0x1p-53;
            S.cg = make_int2(0, 0);
            S.stop = 0;
            S.a_hat = 0.0;
            S.b2_hat = 0.0;
            S.scale0 = 0.0;
        }
        PoleState ps[2];
        int np = 0;
        if (scalar_warp && rank == 0 && P.K == 0) {
            for (int k = lane; k < P.P; k += 32, ++np) {
                const double2 z = P.z[k];
                ps[np] = PoleState{(z.x - P.shift) / P.scale, z.y / P.scale, 0.0, 0.0, 1.0, 0.0, 0.0, 0.0, 1.0, 0, 8.0, 0.0,
                                   0.0, 0.0};
            }
        }
        k_sync();

        // Where a pair's first point lies in a solution vector: region order in
        // a checkpoint, pair order in scratch.
        auto vec_index = [&](int item) -> long long {
            if (!P.ckpt) return 2 * (long long)item;
            const int d = (int)fdiv((uint32_t)item, SA.div_pc), pc = item - d * npc;
            const int pb = (int)fdiv((uint32_t)pc, div_px);
            return ((long long)(z0 + d) * m1 + pb) * m0 + 2 * (pc - pb * npx);
        };
        // Pole recurrences of step k (the scalar warp of rank 0); true once
        // all have met tol.  x_jp(j) sums up to the step after that, whether or
        // not vectors are kept.
        int proc = 0, g_stop = 0;
        bool all_done = false;
        auto poles = [&](int step) {
            bool all = true;
            const double p2 = __hiloint2double((1023 + S.e_hat) << 20, 0);
            for (int k = 0; k < np; ++k) {
                PoleState& s = ps[k];
                const double dr = S.a_hat - s.zr - s.er, di = -s.zi - s.ei;   // d of this step
                pole_step(s, S.a_hat, S.b2_hat, g_stop == 0 || step <= g_stop);
                if (P.vec) {
                    const double inv = 1.0 / (dr * dr + di * di);
                    VecHist h;
                    h.c = make_double2((s.cr * dr + s.ci * di) * inv, (s.ci * dr - s.cr * di) * inv);
                    h.m = make_double2(p2 * s.er, p2 * s.ei);
                    hist[(size_t)((step - 1) % kKryVec) * kKryMaxPoles + lane + 32 * k] = h;
                    s.cr = -h.c.x / p2;
                    s.ci = -h.c.y / p2;
                }
                const double rn = sqrt(sqrt(s.fr * s.fr + s.fi * s.fi));
                if (!s.conv) {
                    s.rn = rn;
                    if (rn <= P.tol_conv) s.conv = step;
                }
                all = all && s.conv;
            }
            all = __all_sync(0xffffffffu, all);
            if (all && !g_stop) g_stop = step + 1;
            proc = step;
            all_done = all;
        };
        int s0 = 0;   // steps the solution vectors hold
        int it = 0, stop = bad ? 1 : 0;
        while (!stop) {
            if constexpr (kNl) {
                // projections of the slab, their sum over the cluster, row factors
                project<X>(P, U, rows, chk, SN[0].n_chunks, nwp + 1, xtab, stage, acc);
                __syncthreads();
                for (int t = tid; t < n_loc4; t += blockDim.x) {
                    cpart[t] = acc[t];
                    acc[t] = 0;
                }
                k_sync();
                for (int t = tid; t < n_loc4; t += blockDim.x) {
                    long long s = 0;
                    for (int r = 0; r < C; ++r)
                        s += __ldcg(reinterpret_cast<const long long*>(slot0 + (size_t)r * P.cta_bytes + P.off_cpart) + t);
                    cl[t] = tab_limbs<X>(to_limbs((double)s * cf[t]));
                }
                __syncthreads();
#pragma unroll 4
                for (int t = tid; t < n_rows; t += blockDim.x) ktab[t + 1] = row_factors<X>(rows + t, cl);
                if (tid == 0) ktab[0] = make_int4(0, 0, 0, 0);
                __syncthreads();
            }
            Dots<X> dots;
            if (scalar_warp) {
                // pole recurrences of the step before, while the others compute
                if (rank == 0 && P.K == 0) {
                    if (it > proc) poles(it);
                    int flag = all_done ? 1 : 0;
                    if (lane == 0 && timed_out()) flag = 2;
                    flag = __shfl_sync(0xffffffffu, flag, 0);
                    if (lane == 0) S.stop = flag;
                } else if (rank == 0) {
                    if (lane == 0 && timed_out()) S.stop = 2;
                }
            } else {
                const int2 g = make_int2(-S.cg.x, -S.cg.y);
                const int4* up = Up + (size_t)((it - 1 + ring) % ring) * n_items;
                // (the compiler sees that these tables are in shared memory)
                if (!kNl || tab_smem) slab_apply<Q, kNl, X>(P, SA, kt_s, xt_s, up, nwp, g, dots);
                else slab_apply<Q, kNl, X>(P, SA, ktab, xtab, up, nwp, g, dots);
            }
            // ---- u.w and w.w over the cluster ------------------------------
            if (!scalar_warp) {
                const long long s = warp_sum4(dots.hh1, dots.l1(), dots.hh2, dots.l2(), lane);
                if (lane < 4) S.part[warp][lane] = s;
            }
            __syncthreads();
            if (scalar_warp) {
                const bool on = lane < nwp;
                const long long s = warp_sum4(on ? S.part[lane][0] : 0LL, on ? S.part[lane][1] : 0LL,
                                              on ? S.part[lane][2] : 0LL, on ? S.part[lane][3] : 0LL, lane);
                // lanes 4 r + k: value k to rank r (C <= 8); warp_sum4 leaves value lane mod 4 in every lane
                if ((lane >> 2) < C) k_st_remote(k_map(smem_addr(&S.mbox[rank][lane & 3]), lane >> 2), s);
                if (rank == 0 && lane < C) k_st_remote(k_map(smem_addr(&S.mbox[0][4]), lane), (long long)S.stop);
            }
            k_sync();
            ++it;
            if (scalar_warp) {
                long long t[4] = {0, 0, 0, 0};
                for (int r = 0; r < C; ++r)
                    for (int k = 0; k < 4; ++k) t[k] += S.mbox[r][k];
                const int flag = (int)S.mbox[0][4];
                // u.w = hh 2^-62 + l 2^-83, w.w = hh 2^-62 + 2 l 2^-83
                const double s1 = (double)t[0] * 0x1p-62 + (double)t[1] * 0x1p-83;
                const double s2 = (double)t[2] * 0x1p-62 + (double)t[3] * 0x1p-82;
                const double al = s1 * S.inv0;
                double n2 = s2 - s1 * al, err = 0x1p-53 * s2;
                // An error d of ||u||^2 makes one of d alpha^2 / beta^2 in the
                // next: it dies out while |alpha| < beta and grows step by step
                // where the potential dominates H.  Beyond 2^-49 the norm is
                // summed instead (one more pass over w and u; no step of the
                // usual Hamiltonians needs it).
                err += al * al * S.drift * S.s0;
                if (!flag && !(err <= 0x1p-49 * n2)) {
                    const double top = fmax(n2, 0x1p-40 * s2);
                    const int e = min(40, (-4 - (((__double2hiint(top) >> 20) & 0x7ff) - 1022)) >> 1);
                    const int2 ca = to_limbs(al);
                    __syncwarp();
                    if (lane == 0) {
                        S.ca = ca;
                        S.e = e;
                        S.stop = kMeasure;
                    }
                    __syncthreads();
                    __syncthreads();
                    const bool on = lane < nwp;
                    const long long s = warp_sum4(on ? S.part[lane][0] : 0LL, on ? S.part[lane][1] : 0LL, 0LL, 0LL, lane);
                    if ((lane & 2) == 0 && (lane >> 2) < C)
                        k_st_remote(k_map(smem_addr(&S.mbox[rank][5 + (lane & 1)]), lane >> 2), s);
                    k_sync();
                    long long hh = 0, l = 0;
                    for (int r = 0; r < C; ++r) hh += S.mbox[r][5], l += S.mbox[r][6];
                    n2 = ldexp((double)hh * 0x1p-62 + (double)l * 0x1p-82, -2 * e);
                    err = 0x1p-53 * n2;
                }
                if (!(n2 > 0.0)) n2 = 0.0;
                const double b2 = n2 * S.inv0;
                int st = flag;
                // an invariant space: the next vector would be rounding noise
                if (n2 < 0x1p-112 * S.s0) st = st ? st : 1;
                if (P.K > 0) {
                    const double a_true = al * P.scale + P.shift, b_true = sqrt(b2) * P.scale;
                    if (it == 1) S.scale0 = fabs(a_true) + b_true + 1.0;
                    __syncwarp();
                    const bool last = it >= P.K || b_true <= P.breakdown_tol * S.scale0;
                    if (rank == 0 && lane == 0) {
                        P.alpha[(long long)node * P.K + it - 1] = a_true;
                        if (!last) P.beta[(long long)node * P.K + it - 1] = b_true;
                    }
                    if (last && !st) st = 1;
                } else if (it >= P.maxit && !st) {
                    st = 1;
                }
                // ||u_new||^2 = n2 4^e in [1/64, 1/16)
                // (n2 >= 2^-116 here, or the node stops)
                const int ex = max(((__double2hiint(n2) >> 20) & 0x7ff) - 1022, -120);
                const int e = min(40, (-4 - ex) >> 1);
                const int2 ca = to_limbs(al);
                __syncwarp();
                if (lane == 0) {
                    S.ca = ca;
                    S.e = e;
                    S.stop = st;
                }
                __syncthreads();
                // the rest while the others form u_new
                const double p2 = __hiloint2double((1023 + e) << 20, 0);   // 2^e
                const double s0n = n2 * p2 * p2;
                const int2 cg = to_limbs(n2 * p2 * S.inv0);
                const double inv = 1.0 / s0n, drift = err * p2 * p2 * inv;
                __syncwarp();
                if (lane == 0) {
                    S.a_hat = al;
                    S.b2_hat = b2;
                    S.e_hat = e;
                    if (!st) {
                        S.cg = cg;
                        S.s0 = s0n;
                        S.inv0 = inv;
                        S.drift = drift;
                    }
                }
                __syncwarp();
            } else {
                __syncthreads();
                if (S.stop == kMeasure) {
                    const int2 al = S.ca;
                    const Rhs<X> ar(opaque(al.x), opaque(al.y));
                    const int e = S.e;
                    Dots<X> sq;
#pragma unroll 1
                    for (int item = tid; item < n_items; item += 32 * nwp) {
                        const int d = (int)fdiv((uint32_t)item, SA.div_pc), pc = item - d * npc;
                        const int pb = (int)fdiv((uint32_t)pc, div_px);
                        const int4 u = *reinterpret_cast<const int4*>(U + (d + Q) * pp + pb * pitch + 2 * (pc - pb * npx));
                        const longlong2 w = Wp[item];
                        Acc<X> a0, a1;
                        a0.mac(Lhs<X>(u.x, u.y), ar);
                        a1.mac(Lhs<X>(u.z, u.w), ar);
                        const long long t0 = w.x - a0.fold(), t1 = w.y - a1.fold();
                        sq.add(Lhs<X>(0, 0), split31(e >= 0 ? t0 << e : t0 >> -e));
                        sq.add(Lhs<X>(0, 0), split31(e >= 0 ? t1 << e : t1 >> -e));
                        sq.flush();
                    }
                    const long long s = warp_sum4(sq.hh2, sq.l2(), 0LL, 0LL, lane);
                    if (lane < 2) S.part[warp][lane] = s;
                    __syncthreads();
                    k_sync();
                    __syncthreads();
                }
            }
            stop = S.stop;
            if (P.vec && (stop || it % kKryVec == 0)) {
                // apply the vectors kept to the solutions
                const int n = it - s0;
                if (scalar_warp && rank == 0) {
                    if (it > proc) poles(it);
                    __syncwarp();
                    for (int k = 0; k < np; ++k) {
                        char* cb = coef + (size_t)(lane + 32 * k) * kCoefBytes;
                        vec_coefs(hist, n, s0, ps[k], lane + 32 * k, reinterpret_cast<int4*>(cb + 128),
                                  reinterpret_cast<VecHead*>(cb));
                    }
                }
                for (int item = tid; item < n_items; item += blockDim.x) {   // u_it itself
                    const int d = (int)fdiv((uint32_t)item, SA.div_pc), pc = item - d * npc;
                    const int pb = (int)fdiv((uint32_t)pc, div_px);
                    Up[(size_t)((it - 1) % ring) * n_items + item] =
                        *reinterpret_cast<const int4*>(U + (d + Q) * pp + pb * pitch + 2 * (pc - pb * npx));
                }
                k_sync();
                for (int pole = 0; pole < P.P; ++pole) {
                    const char* cb = coef + (size_t)pole * kCoefBytes;
                    if (!__ldcg(reinterpret_cast<const int*>(cb + offsetof(VecHead, act)))) continue;
                    __syncthreads();
                    for (int t = tid; t < 4 * n; t += blockDim.x)
                        SV.co[t] = __ldcg(reinterpret_cast<const int4*>(cb + 128) + t);
                    if (tid < (int)(sizeof(VecHead) / 4))
                        reinterpret_cast<int*>(&SV.head)[tid] = __ldcg(reinterpret_cast<const int*>(cb) + tid);
                    __syncthreads();
                    double2* x = P.ckpt ? P.ckpt + P.ckpt_off[(long long)node * P.P + pole]
                                        : Xs + (size_t)pole * 2 * n_items;
                    double2* pv = Ps + (size_t)pole * 2 * n_items;
                    if (SV.head.last) vec_update<true, X>(SA, n, SV.co, SV.head, Up, x, pv, vec_index);
                    else vec_update<false, X>(SA, n, SV.co, SV.head, Up, x, pv, vec_index);
                }
                s0 = it;
                k_sync();   // from here the coefficients may be written again
            }
            if (stop) break;
            if (!scalar_warp) {
                const int2 al = S.ca;
                const Rhs<X> ar(opaque(al.x), opaque(al.y));
                const int e = S.e;
                const uint32_t ubase = smem_addr(U);
                // three pairs at a time: their loads are in flight together
                constexpr int kB = 3;
                for (int i0 = tid; i0 < n_items; i0 += kB * 32 * nwp) {
                    longlong2 w[kB];
#pragma unroll
                    for (int j = 0; j < kB; ++j)
                        if (i0 + 32 * nwp * j < n_items) w[j] = Wp[i0 + 32 * nwp * j];
#pragma unroll
                    for (int j = 0; j < kB; ++j) {
                        const int item = i0 + 32 * nwp * j;
                        if (item >= n_items) break;
                        const int d = (int)fdiv((uint32_t)item, SA.div_pc), pc = item - d * npc;
                        const int pb = (int)fdiv((uint32_t)pc, div_px);
                        const int idx = pb * pitch + 2 * (pc - pb * npx);
                        int4* up = reinterpret_cast<int4*>(U + (d + Q) * pp + idx);
                        const int4 u = *up;
                        Acc<X> a0, a1;
                        a0.mac(Lhs<X>(u.x, u.y), ar);
                        a1.mac(Lhs<X>(u.z, u.w), ar);
                        const long long t0 = w[j].x - a0.fold(), t1 = w[j].y - a1.fold();
                        const int2 a = split31(e >= 0 ? t0 << e : t0 >> -e), b = split31(e >= 0 ? t1 << e : t1 >> -e);
                        const int4 nu = make_int4(a.x, a.y, b.x, b.y);
                        Up[(size_t)((it - 1) % ring) * n_items + item] = u;
                        *up = nu;
                        // the CTAs whose halo holds this plane
                        const int z = z0 + d;
                        if (d < Q)
                            for (int r = rank - 1; r >= 0 && z - S.zlo[r + 1] < Q; --r)
                                k_st_remote(k_map(ubase + (uint32_t)((z - S.zlo[r] + Q) * pp + idx) * 8u, r), nu);
                        if (d >= depth - Q)
                            for (int r = rank + 1; r < C && S.zlo[r] - z <= Q; ++r)
                                k_st_remote(k_map(ubase + (uint32_t)((z - S.zlo[r] + Q) * pp + idx) * 8u, r), nu);
                    }
                }
            }
            k_sync();
        }
        // ---- mixed precision: the last step once more, in FP64 ---------------
        double defect = 0.0;
        if (!X && P.check && !bad) {
            double* c = reinterpret_cast<double*>(acc);   // free once the steps are done
            double* part = reinterpret_cast<double*>(cpart);
            double s2 = check_step<Q, kNl>(P, SA, lo, z0, SN[0], c, Up + (size_t)((it - 2 + ring) % ring) * n_items, S.cg, [&]() {
                __syncthreads();
                for (int t = tid; t < n_loc4; t += blockDim.x) part[t] = c[t];
                k_sync();
                for (int t = tid; t < n_loc4; t += blockDim.x) {
                    double s = 0.0;
                    for (int r = 0; r < C; ++r)
                        s += __ldcg(reinterpret_cast<const double*>(slot0 + (size_t)r * P.cta_bytes + P.off_cpart) + t);
                    c[t] = s;
                }
                __syncthreads();
            });
            s2 = warp_sum(s2);
            if (lane == 0) S.part[warp][0] = __double_as_longlong(s2);
            __syncthreads();
            if (tid == 0) {
                s2 = 0.0;
                for (int k = 0; k <= nwp; ++k) s2 += __longlong_as_double(S.part[k][0]);
                k_st_remote(k_map(smem_addr(&S.mbox[rank][7]), 0), __double_as_longlong(s2));
            }
            k_sync();
            for (int r = 0; r < C; ++r) defect += __longlong_as_double(S.mbox[r][7]);   // rank 0 holds them
            defect = sqrt(defect * S.inv0) * P.scale;   // relative to ||u||, in units of H
        }
        // ---- outputs of the solution vectors ----------------------------------
        if (P.vec) {
            if (tid < P.P) {
                const double2 z = P.z[tid], w = P.w[tid];
                const double aj = P.fused_a ? P.fused_a[node] : 0.0, bj = P.fused_b ? P.fused_b[node] : 0.0;
                const double cr = 2.0 * aj / P.dV + 2.0 * bj * z.x, ci = 2.0 * bj * z.y;
                SV.cp[tid] = P.dm_rows ? w : make_double2(cr * w.x - ci * w.y, cr * w.y + ci * w.x);
            }
            __syncthreads();
            const double inv = 1.0 / P.scale, nan = __longlong_as_double(0x7ff8000000000000LL);
            for (int item = tid; item < n_items; item += blockDim.x) {
                const int d = (int)fdiv((uint32_t)item, SA.div_pc), pc = item - d * npc;
                const int pb = (int)fdiv((uint32_t)pc, div_px), a = 2 * (pc - pb * npx);
                const long long xi = vec_index(item);
                for (int i = 0; i < 2 && a + i < m0; ++i) {
                    double sum = 0.0;
                    for (int pole = 0; pole < P.P; ++pole) {
                        double2* xp = (P.ckpt ? P.ckpt + P.ckpt_off[(long long)node * P.P + pole]
                                              : Xs + (size_t)pole * 2 * n_items) + xi + i;
                        const double2 x = bad ? make_double2(nan, nan) : make_double2(xp->x * inv, xp->y * inv);
                        if (P.ckpt) *xp = x;
                        const double2 c = SV.cp[pole];
                        if (P.dm_rows) sum += c.x * x.y + c.y * x.x;
                        else sum -= c.x * (2.0 * x.x * x.y) + c.y * (x.x * x.x - x.y * x.y);
                    }
                    if (P.dm_rows) P.dm_rows[P.dm_off[node] + ((long long)(z0 + d) * m1 + pb) * m0 + a + i] = sum;
                    if (P.fused_dLdV) {
                        const int gx = wrap_once(lo[0] + a + i, P.n[0]), gy = wrap_once(lo[1] + pb, P.n[1]);
                        const int gz = wrap_once(lo[2] + z0 + d, P.n[2]);
                        atomicAdd(P.fused_dLdV + gx + (long long)P.n[0] * (gy + (long long)P.n[1] * gz), sum);
                    }
                }
            }
        }
        // ---- results ---------------------------------------------------------
        if (rank == 0 && scalar_warp) {
            if (P.K == 0 && it > proc) poles(it);
            if (P.K > 0) {
                // a potential that is not finite: so is the Jacobi matrix, and its QR fails
                if (bad == 3) {
                    const double nan = __longlong_as_double(0x7ff8000000000000LL);
                    for (int k = lane; k < P.K; k += 32) {
                        P.alpha[(long long)node * P.K + k] = nan;
                        P.beta[(long long)node * P.K + k] = nan;
                    }
                }
                if (lane == 0) {
                    P.k_used[node] = bad == 3 ? P.K : (bad ? 0 : it);
                    P.node_status[node] = bad == 1 ? 1 : (stop == 2 ? 4 : 0);
                }
            } else {
                for (int k = 0; k < np; ++k) {
                    const long long o = (long long)node * P.P + lane + 32 * k;
                    const double nan = __longlong_as_double(0x7ff8000000000000LL);
                    // the true residual: the recurrence's and, with ||x||^2 =
                    // Im x(j) / Im z, what a defect of every step would add
                    if (P.check && !bad) {
                        const double x2 = fabs(ps[k].gi / ps[k].zi) / (P.scale * P.scale);
                        ps[k].rn = sqrt(ps[k].rn * ps[k].rn + defect * defect * x2);
                        if (ps[k].rn > P.tol) ps[k].conv = 0;
                    }
                    P.x_src[o] = bad ? make_double2(nan, nan) : make_double2(ps[k].gr / P.scale, ps[k].gi / P.scale);
                    P.status[o] = bad ? bad : (ps[k].conv ? 0 : (stop == 2 ? 4 : 2));
                    P.iters[o] = ps[k].conv ? ps[k].conv : it;
                    P.resid[o] = ps[k].rn;
                    P.n_rel[o] = P.check && !bad ? 1 : 0;
                }
            }
        }
        __syncthreads();
    }
}

// Per atom: the x, y, z tables scaled to unit norm (and halved, so that a
// one-point window fits the limbs) and the coefficients that make up for it:
// E_l dV C_l^2 p p^T = (64 E_l C'^2) q q^T, q the product of three tables.
__global__ void k_proj_fixed(long long n_atoms, const int* __restrict__ len, const double* __restrict__ dtab,
                             const double* __restrict__ gtab, const double* __restrict__ C, double dV, double e_s,
                             double e_p, int4* __restrict__ fx, double* __restrict__ fxc, int* __restrict__ bad) {
    const long long a = blockIdx.x;
    __shared__ double n2[3][2];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp < 3) {
        double g2 = 0.0, d2 = 0.0;
        const long long base = (3 * a + warp) * kMaxProjWin;
        for (int u = lane; u < len[3 * a + warp]; u += 32) {
            const double g = gtab[base + u], dg = dtab[base + u] * g;
            g2 += g * g;
            d2 += dg * dg;
        }
        g2 = warp_sum(g2);
        d2 = warp_sum(d2);
        if (lane == 0) {
            n2[warp][0] = g2;
            n2[warp][1] = d2;
        }
        const double ig = 0.5 / sqrt(g2), id = 0.5 / sqrt(d2);
        for (int u = lane; u < kMaxProjWin; u += 32) {
            const bool in = u < len[3 * a + warp];
            const double g = in ? gtab[base + u] : 0.0, dg = in ? dtab[base + u] * g : 0.0;
            const int2 x = to_limbs(g * ig), y = to_limbs(dg * id);
            fx[base + u] = make_int4(x.x, x.y, y.x, y.y);
        }
    }
    __syncthreads();
    if (threadIdx.x < 4) {
        const int l = threadIdx.x;
        double c2 = dV * C[4 * a + l] * C[4 * a + l];
        for (int d = 0; d < 3; ++d) c2 *= n2[d][l == d + 1 ? 1 : 0];
        if (!(c2 > 0.0 && c2 < 16.0)) atomicExch(bad, 1);
        fxc[4 * a + l] = 64.0 * (l == 0 ? e_s : e_p) * c2;
    }
}

template <int Q, bool kNl, bool X>
int max_clusters(int csz, int block, size_t smem) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = csz;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = csz;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaFuncSetAttribute(k_krylov<Q, kNl, X>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, k_krylov<Q, kNl, X>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

template <int Q, bool kNl, bool X>
cudaError_t launch(const KrylovParams& P, int csz, int grid, int block, size_t smem, cudaStream_t stream) {
    cudaError_t e = cudaFuncSetAttribute(k_krylov<Q, kNl, X>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = csz;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_krylov<Q, kNl, X>, P);
}

}  // namespace

size_t kry_u_bytes(int q, int m0, int m1, int depth) {
    return ((size_t)(depth + 2 * q) * kry_pitch(q, m0) * m1 * sizeof(int2) + 15) / 16 * 16;
}
size_t kry_static_smem_bytes(int) { return sizeof(KShared) + sizeof(KSharedNl) + sizeof(KSharedVec) + 64; }
size_t kry_vec_bytes(int P) {
    return (size_t)kKryVec * kKryMaxPoles * sizeof(VecHist) + (size_t)P * (128 + 64 * kKryVec);
}
int kry_max_threads() { return kMaxThreads - 32; }

// (clusters of the mixed kernel and of the FP64 one are the same size)
int kry_max_clusters(int q, int nonlocal, int csz, int block, size_t smem) {
    switch (q * 2 + (nonlocal ? 1 : 0)) {
        case 2: return max_clusters<1, false, true>(csz, block, smem);
        case 3: return max_clusters<1, true, true>(csz, block, smem);
        case 4: return max_clusters<2, false, true>(csz, block, smem);
        case 5: return max_clusters<2, true, true>(csz, block, smem);
        case 6: return max_clusters<3, false, true>(csz, block, smem);
        case 7: return max_clusters<3, true, true>(csz, block, smem);
        case 8: return max_clusters<4, false, true>(csz, block, smem);
        case 9: return max_clusters<4, true, true>(csz, block, smem);
    }
    return 0;
}

cudaError_t launch_krylov(const KrylovParams& P, int q, int nonlocal, int csz, int grid, int block, size_t smem,
                          cudaStream_t stream) {
    switch ((q * 2 + (nonlocal ? 1 : 0)) * 2 + (P.exact ? 1 : 0)) {
        case 4: return launch<1, false, false>(P, csz, grid, block, smem, stream);
        case 5: return launch<1, false, true>(P, csz, grid, block, smem, stream);
        case 6: return launch<1, true, false>(P, csz, grid, block, smem, stream);
        case 7: return launch<1, true, true>(P, csz, grid, block, smem, stream);
        case 8: return launch<2, false, false>(P, csz, grid, block, smem, stream);
        case 9: return launch<2, false, true>(P, csz, grid, block, smem, stream);
        case 10: return launch<2, true, false>(P, csz, grid, block, smem, stream);
        case 11: return launch<2, true, true>(P, csz, grid, block, smem, stream);
        case 12: return launch<3, false, false>(P, csz, grid, block, smem, stream);
        case 13: return launch<3, false, true>(P, csz, grid, block, smem, stream);
        case 14: return launch<3, true, false>(P, csz, grid, block, smem, stream);
        case 15: return launch<3, true, true>(P, csz, grid, block, smem, stream);
        case 16: return launch<4, false, false>(P, csz, grid, block, smem, stream);
        case 17: return launch<4, false, true>(P, csz, grid, block, smem, stream);
        case 18: return launch<4, true, false>(P, csz, grid, block, smem, stream);
        case 19: return launch<4, true, true>(P, csz, grid, block, smem, stream);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_proj_fixed(long long n_atoms, const int* len, const double* dtab, const double* gtab,
                              const double* C, double dV, double e_s, double e_p, int4* fx, double* fxc, int* bad,
                              cudaStream_t stream) {
    k_proj_fixed<<<(unsigned)n_atoms, 128, 0, stream>>>(n_atoms, len, dtab, gtab, C, dV, e_s, e_p, fx, fxc, bad);
    return cudaGetLastError();
}

}  // namespace md
