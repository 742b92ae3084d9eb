// wavelet_bodies.cuh -- per-record work of the wavelet predictors, shared by
// the single-tree kernels (wavelet.cu) and the batched kernel (batched.cu).
// Each body is called once per node record, in post-order, with the same
// record for every thread of the CTA; see wavelet.cu for the mapping.
#pragma once

#include "df64.cuh"
#include "staging.cuh"
#include "wt_internal.cuh"

namespace wt {
namespace {

constexpr int kChunkD = 64;    // records per staging buffer (48 B each): the float64 stack leaves room for few CTAs
constexpr int kChunkDF = 128;  // double-float form (48 B each): smaller buffers, more CTAs per SM
constexpr int kChunkF = 384;   // (32 B each)
constexpr int kChunkW = kRecChunkW;   // regrouped float32 form (32 B each): its stack is small, so the
                               // staging buffers set how many CTAs fit on an SM

__device__ __forceinline__ int clamp_row(uint32_t r, int maxrow) { return min(static_cast<int>(r), maxrow); }

// ---------------------------------------------------------------- float64
// Eq. 17 in float64. A thread's stack holds xi = 4^(J-j) eta, so a node's xi
// is the plain sum of its children's and gamma^m sigma^m = a_m (H_m
// xi_children) with the scale factors already in a_m (RecD): 22 operations of
// the float64 pipe for a node of several children and 2 for an only child,
// where eta and the three sigma with their factors took 32 and 10; with the
// sine and cosine's 13 for 18, 201 600 visibilities of 1 115 leaves 16.4 ->
// 13.6 ms (12.3 with the tiles' waves evened out: fp64_resident; 11.6 with leaves
// in groups: at).
template <int NT, int VPT>
struct Eq17D {
    double u[VPT], v[VPT], w[VPT];
    double vr[VPT], vi[VPT];
    double sgn;
    double2* stk;   // shared stack + threadIdx.x; row stride VPT * NT
    int maxrow;     // 4 (J - 1) - 1

    __device__ __forceinline__ double2& slot(int row, int k) { return stk[(row * VPT + k) * NT]; }

    __device__ __forceinline__ void wave(const RecD& r, int k, double2& e) const
    {
        const double t = fma(w[k], r.c, fma(v[k], r.b, u[k] * r.a));
        sincos_turns_f64(t, e.y, e.x);
    }

    // A node of several children, one visibility.
    __device__ __forceinline__ void node(const RecD& r, bool root, int srow, int k, double2 c0, double2 c1,
                                         double2 c2, double2 c3)
    {
        const double ar = c0.x + c1.x, ai = c0.y + c1.y;   // c0 + c1
        const double br = c0.x - c1.x, bi = c0.y - c1.y;   // c0 - c1
        const double cr = c2.x + c3.x, ci = c2.y + c3.y;   // c2 + c3
        const double dr = c2.x - c3.x, di = c2.y - c3.y;   // c2 - c3
        const double er = ar + cr, ei = ai + ci;           // Eq. 9 form (times 4^(J-j))
        // Eq. 10 rows (+ - + -), (+ + - -), (+ - - +), weighted by gamma
        vr[k] = fma(r.a, br + dr, fma(r.b, ar - cr, fma(r.c, br - dr, vr[k])));
        vi[k] = fma(r.a, bi + di, fma(r.b, ai - ci, fma(r.c, bi - di, vi[k])));
        if (root) {
            vr[k] = fma(r.e, er, vr[k]);
            vi[k] = fma(r.e, ei, vi[k]);
        } else {
            slot(srow, k) = make_double2(er, ei);
        }
    }

    // One step of the sweep; returns the records it took. Two leaves in a row
    // are siblings (a last sibling is followed by its parent) and independent:
    // their chains of float64 operations run side by side, which an SM's eight
    // warps alone do not hide. Where the whole run and its parent are in the
    // chunk (the run as long as the parent has children), the waves go to the
    // parent's butterfly in registers, not through the stack. 201 563 visibilities
    // of 1 126 leaves: 12.49 ms a leaf at a time, 11.81 in pairs, 11.75 so (a
    // smaller batch, 1.58 ms before: 1.17, 1.12, 1.10).
    __device__ __forceinline__ int at(const RecD* cb, int r, int n)
    {
        const uint32_t m0 = cb[r].meta;
        if ((m0 & (kRecLeaf | kRecRoot)) == kRecLeaf && r + 1 < n && (cb[r + 1].meta & kRecLeaf)) {
            const int len = r + 2 < n && !(cb[r + 2].meta & kRecLeaf)   ? 2
                            : r + 3 < n && !(cb[r + 3].meta & kRecLeaf) ? 3
                            : r + 4 < n && !(cb[r + 4].meta & kRecLeaf) ? 4
                                                                        : 0;
            const uint32_t mask = len ? rec_mask(cb[r + len].meta) : 0u;
            if (len && __popc(mask) == len) {
                const RecD& par = cb[r + len];
                const bool root = par.meta & kRecRoot;
                const int srow = clamp_row(rec_store_row(par.meta), maxrow);
                const bool b0 = mask & 1u, b1 = mask & 2u, b2 = mask & 4u, b3 = mask & 8u;
                const int before2 = (b0 ? 1 : 0) + (b1 ? 1 : 0);
                const double2 zero = make_double2(0.0, 0.0);
#pragma unroll
                for (int k = 0; k < VPT; ++k) {
                    double2 e0, e1, e2 = zero, e3 = zero;
                    wave(cb[r], k, e0);
                    wave(cb[r + 1], k, e1);
                    if (len == 4) {
                        wave(cb[r + 2], k, e2);
                        wave(cb[r + 3], k, e3);
                        node(par, root, srow, k, e0, e1, e2, e3);
                    } else {
                        if (len == 3) wave(cb[r + 2], k, e2);
                        const double2 c0 = b0 ? e0 : zero;
                        const double2 c1 = !b1 ? zero : b0 ? e1 : e0;
                        const double2 c2 = !b2 ? zero : before2 == 2 ? e2 : before2 == 1 ? e1 : e0;
                        const double2 c3 = !b3 ? zero : len == 3 ? e2 : e1;
                        node(par, root, srow, k, c0, c1, c2, c3);
                    }
                }
                return len + 1;
            }
            const RecD& p = cb[r];
            const RecD& q = cb[r + 1];
            const int row0 = clamp_row(rec_store_row(m0), maxrow), row1 = clamp_row(rec_store_row(q.meta), maxrow);
#pragma unroll
            for (int k = 0; k < VPT; ++k) {
                double2 e0, e1;
                wave(p, k, e0);
                wave(q, k, e1);
                slot(row0, k) = e0;
                slot(row1, k) = e1;
            }
            return 2;
        }
        (*this)(cb[r]);
        return 1;
    }

    __device__ void operator()(const RecD& r)
    {
        const uint32_t meta = r.meta;
        const bool root = meta & kRecRoot;
        const int srow = clamp_row(rec_store_row(meta), maxrow);
        if (meta & kRecLeaf) {
#pragma unroll
            for (int k = 0; k < VPT; ++k) {
                double t = fma(w[k], r.c, fma(v[k], r.b, u[k] * r.a));
                double s, c;
                sincos_turns_f64(t, s, c);
                if (root) {
                    vr[k] = fma(r.d, c, vr[k]);
                    vi[k] = fma(r.d, s, vi[k]);
                } else {
                    slot(srow, k) = make_double2(c, s);
                }
            }
        } else if (meta & kRecSingle) {
            const int crow = clamp_row(rec_child_row(meta), maxrow);
#pragma unroll
            for (int k = 0; k < VPT; ++k) {
                const double2 xi = slot(crow, k);   // the node's xi is its child's
                vr[k] = fma(r.a, xi.x, vr[k]);
                vi[k] = fma(r.a, xi.y, vi[k]);
                if (root) {
                    vr[k] = fma(r.e, xi.x, vr[k]);
                    vi[k] = fma(r.e, xi.y, vi[k]);
                } else {
                    slot(srow, k) = xi;
                }
            }
        } else {
            const int crow = clamp_row(rec_child_row(meta), maxrow - 3);
            const uint32_t mask = rec_mask(meta);
#pragma unroll
            for (int k = 0; k < VPT; ++k) {
                double2 c0 = make_double2(0.0, 0.0), c1 = c0, c2 = c0, c3 = c0;
                if (mask & 1u) c0 = slot(crow, k);
                if (mask & 2u) c1 = slot(crow + 1, k);
                if (mask & 4u) c2 = slot(crow + 2, k);
                if (mask & 8u) c3 = slot(crow + 3, k);
                node(r, root, srow, k, c0, c1, c2, c3);
            }
        }
    }
};

template <int VPT>
struct Eq16D {
    double u[VPT], v[VPT], w[VPT];
    double vr[VPT], vi[VPT];
    double sgn;
    __device__ void operator()(const RecD& r)
    {
#pragma unroll
        for (int k = 0; k < VPT; ++k) {
            double t = fma(w[k], r.c, fma(v[k], r.b, u[k] * r.a));
            double s, c;
            sincos_turns_f64(t, s, c);
            vr[k] = fma(r.d, c, vr[k]);
            vi[k] = fma(r.d, s, vi[k]);
        }
    }
};

// ---------------------------------------------------------------- mixed
// Eq. 17 in the mixed forms, on packed float32 pairs. A thread's stack
// holds xi = 4^(J-j) eta (RecF): a node's xi is the plain sum of its
// children's, and gamma^m sigma^m = a_m (H_m xi_children) with the scale
// factors already in a_m. A complex value is one pair; the leaf phases of
// visibilities 2p and 2p + 1 are formed as one pair (VPT = 1 forms its one
// phase on scalars). Per visibility a four-child node costs 15 paired
// operations, Kahan included.
template <int NT, int VPT, bool FAST = false, bool GRID = false>
struct Eq17F {
    static constexpr int NP = VPT / 2;                // visibility pairs
    static constexpr bool ODD = (VPT & 1) != 0;       // a last, unpaired visibility
    F2 u[VPT], v[VPT], w[VPT];                        // set by the caller, then start()
    DF2 U[NP > 0 ? NP : 1], V[NP > 0 ? NP : 1], W[NP > 0 ? NP : 1];
    float2 Cg[NP > 0 ? NP : 1];                       // GRID: the grid constants of visibilities 2p, 2p + 1
    float Cs;                                         // GRID: that of the last, unpaired visibility
    float2 acc[VPT], comp[VPT];                       // Kahan sum of V and its compensation
    float2* stk;
    int maxrow;

    __device__ __forceinline__ float2& slot(int row, int k) { return stk[(row * VPT + k) * NT]; }

    __device__ __forceinline__ void start()
    {
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            U[p] = df2_pack(u[2 * p], u[2 * p + 1]);
            V[p] = df2_pack(v[2 * p], v[2 * p + 1]);
            W[p] = df2_pack(w[2 * p], w[2 * p + 1]);
        }
#pragma unroll
        for (int k = 0; k < VPT; ++k) {
            acc[k] = make_float2(0.f, 0.f);
            comp[k] = make_float2(0.f, 0.f);
        }
    }

    __device__ __forceinline__ float2 result(int k) const { return sub2(acc[k], comp[k]); }

    // The plane wave at a leaf's centre, every visibility.
    __device__ __forceinline__ void leaf_waves(const RecF& r, float2 (&e)[VPT]) const
    {
        const F2 su{r.a, r.b}, sv{r.c, r.d}, sw{r.e, r.f};
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            float2 h, tl;
            if constexpr (GRID) phase_turns_grid2(U[p], V[p], W[p], su, sv, sw, Cg[p], h, tl);
            else phase_turns_df2(U[p], V[p], W[p], su, sv, sw, h, tl);
            sincos_mixed2<FAST>(h, tl, e[2 * p], e[2 * p + 1]);
        }
        if constexpr (ODD) {
            constexpr int k = VPT - 1;
            float th, tl, s, c;
            if constexpr (GRID) phase_turns_grid(u[k], v[k], w[k], su, sv, sw, Cs, th, tl);
            else phase_turns_df(u[k], v[k], w[k], su, sv, sw, th, tl);
            sincos_mixed<FAST>(th, tl, s, c);
            e[k] = make_float2(c, s);
        }
    }

    // A node with a single child: its xi is the child's.
    __device__ __forceinline__ void node_single(const RecF& r, bool root, int srow, const float2 (&xi)[VPT])
    {
        const float2 a = bcast2(r.a), g = bcast2(r.g);
#pragma unroll
        for (int k = 0; k < VPT; ++k) {
            float2 x = mul2(a, xi[k]);
            if (root) x = fma2(g, xi[k], x);
            else slot(srow, k) = xi[k];
            kahan_add2(acc[k], comp[k], x);
        }
    }

    // A node of several children, one visibility.
    __device__ __forceinline__ void node(const RecF& r, bool root, int srow, int k, float2 c0, float2 c1, float2 c2,
                                         float2 c3)
    {
        const float2 ga = bcast2(r.a), gb = bcast2(r.b), gc = bcast2(r.c);
        const float2 a = add2(c0, c1), b = sub2(c0, c1);   // c0 +- c1
        const float2 c = add2(c2, c3), d = sub2(c2, c3);   // c2 +- c3
        const float2 xi = add2(a, c);                      // Eq. 9 (times 4^(J-j))
        // Eq. 10 rows (+ - + -), (+ + - -), (+ - - +), weighted by gamma
        float2 x = fma2(ga, add2(b, d), fma2(gb, sub2(a, c), mul2(gc, sub2(b, d))));
        if (root) x = fma2(bcast2(r.g), xi, x);
        else slot(srow, k) = xi;
        kahan_add2(acc[k], comp[k], x);
    }

    __device__ void operator()(const RecF& r)
    {
        const uint32_t meta = r.meta;
        const bool root = meta & kRecRoot;
        const int srow = clamp_row(rec_store_row(meta), maxrow);
        if (meta & kRecLeaf) {
            float2 e[VPT];
            leaf_waves(r, e);
#pragma unroll
            for (int k = 0; k < VPT; ++k) {
                if (root) kahan_add2(acc[k], comp[k], mul2(bcast2(r.g), e[k]));
                else slot(srow, k) = e[k];
            }
        } else if (meta & kRecSingle) {
            const int crow = clamp_row(rec_child_row(meta), maxrow);
            float2 xi[VPT];
#pragma unroll
            for (int k = 0; k < VPT; ++k) xi[k] = slot(crow, k);
            node_single(r, root, srow, xi);
        } else {
            const int crow = clamp_row(rec_child_row(meta), maxrow - 3);
            const uint32_t mask = rec_mask(meta);
#pragma unroll
            for (int k = 0; k < VPT; ++k) {
                float2 c0 = make_float2(0.f, 0.f), c1 = c0, c2 = c0, c3 = c0;
                if (mask & 1u) c0 = slot(crow, k);
                if (mask & 2u) c1 = slot(crow + 1, k);
                if (mask & 4u) c2 = slot(crow + 2, k);
                if (mask & 8u) c3 = slot(crow + 3, k);
                node(r, root, srow, k, c0, c1, c2, c3);
            }
        }
    }

    // One step of the sweep; returns the records it took. A group (a run of
    // sibling leaves and their parent, in one chunk by construction) is one
    // step: the leaves' waves go to the parent's butterfly in registers, never
    // to the stack, and the record's decoding is shared. 2 032 000 visibilities
    // of 1 530 leaves, polynomial form: 9.76 -> 8.43 ms.
    __device__ __forceinline__ int at(const RecF* cb, int r, int n)
    {
        const uint32_t meta = cb[r].meta;
        if (meta & kRecGroup) {
            const int k = static_cast<int>((meta >> kRecGroupShift) & 7u);
            if (k >= 1 && k <= 4 && r + k < n) {
                group(cb + r, k);
                return k + 1;
            }
        }
        (*this)(cb[r]);
        return 1;
    }

    __device__ __forceinline__ void group(const RecF* g, int k)
    {
        const RecF& par = g[k];
        const uint32_t meta = par.meta;
        const bool root = meta & kRecRoot;
        const int srow = clamp_row(rec_store_row(meta), maxrow);
        const uint32_t mask = rec_mask(meta);
        if (k == 1) {
            float2 e[VPT];
            leaf_waves(g[0], e);
            node_single(par, root, srow, e);
        } else if (k == 4) {
            float2 c0[VPT], c1[VPT], c2[VPT], c3[VPT];
            leaf_waves(g[0], c0);
            leaf_waves(g[1], c1);
            leaf_waves(g[2], c2);
            leaf_waves(g[3], c3);
#pragma unroll
            for (int i = 0; i < VPT; ++i) node(par, root, srow, i, c0[i], c1[i], c2[i], c3[i]);
        } else {                                       // two or three children, in slot order
            const float2 zero = make_float2(0.f, 0.f);
            float2 e0[VPT], e1[VPT], e2[VPT];
            leaf_waves(g[0], e0);
            leaf_waves(g[1], e1);
            if (k == 3) {
                leaf_waves(g[2], e2);
            } else {
#pragma unroll
                for (int i = 0; i < VPT; ++i) e2[i] = zero;
            }
            // the slot of the i-th leaf is that of the mask's i-th bit
            const bool b0 = mask & 1u, b1 = mask & 2u, b2 = mask & 4u, b3 = mask & 8u;
            const int before2 = (b0 ? 1 : 0) + (b1 ? 1 : 0);
#pragma unroll
            for (int i = 0; i < VPT; ++i) {
                const float2 c0 = b0 ? e0[i] : zero;
                const float2 c1 = !b1 ? zero : b0 ? e1[i] : e0[i];
                const float2 c2 = !b2 ? zero : before2 == 2 ? e2[i] : before2 == 1 ? e1[i] : e0[i];
                const float2 c3 = !b3 ? zero : k == 3 ? e2[i] : e1[i];
                node(par, root, srow, i, c0, c1, c2, c3);
            }
        }
    }
};

// Eq. 16 in the mixed forms on packed pairs: a thread's visibilities taken
// two at a time (their phases against one leaf as one pair of double-floats,
// each visibility's (cos, sin) its own pair), an odd last visibility of the
// thread alone; the leaf records kSumBlock at a time (their terms added by
// FMAs into a partial per visibility, the partial then into its Kahan sum:
// blockwise compensated summation). GRID: the phases with their heads on each visibility's
// grid (constants Cg / Cs, set by the caller; phase_turns_grid2), else with
// error-free sums (phase_turns_df2).
template <int VPT, bool FAST, bool GRID>
struct Eq16F2 {
    static constexpr int NP = VPT / 2;
    static constexpr bool ODD = (VPT & 1) != 0;
    DF2 U[NP > 0 ? NP : 1], V[NP > 0 ? NP : 1], W[NP > 0 ? NP : 1];
    F2 us, vs, ws;                                    // the unpaired last visibility
    float2 Cg[NP > 0 ? NP : 1];
    float Cs;
    float2 acc[VPT], comp[VPT];

    __device__ __forceinline__ void start(const F2 (&u)[VPT], const F2 (&v)[VPT], const F2 (&w)[VPT],
                                          const float (&C)[VPT])
    {
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            U[p] = df2_pack(u[2 * p], u[2 * p + 1]);
            V[p] = df2_pack(v[2 * p], v[2 * p + 1]);
            W[p] = df2_pack(w[2 * p], w[2 * p + 1]);
            Cg[p] = make_float2(C[2 * p], C[2 * p + 1]);
        }
        us = u[VPT - 1];
        vs = v[VPT - 1];
        ws = w[VPT - 1];
        Cs = C[VPT - 1];
#pragma unroll
        for (int k = 0; k < VPT; ++k) {
            acc[k] = make_float2(0.f, 0.f);
            comp[k] = make_float2(0.f, 0.f);
        }
    }

    __device__ __forceinline__ float2 result(int k) const { return sub2(acc[k], comp[k]); }

    // One leaf's terms into the partials: p[k] += Phi exp(i 2 pi phase) of
    // visibility k.
    __device__ __forceinline__ void add_terms(const RecF& r, float2 (&x)[VPT]) const
    {
        const F2 su{r.a, r.b}, sv{r.c, r.d}, sw{r.e, r.f};
        const float2 fl = bcast2(r.g);
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            float2 h, tl, e0, e1;
            if constexpr (GRID) phase_turns_grid2(U[p], V[p], W[p], su, sv, sw, Cg[p], h, tl);
            else phase_turns_df2(U[p], V[p], W[p], su, sv, sw, h, tl);
            sincos_mixed2<FAST>(h, tl, e0, e1);
            x[2 * p] = fma2(fl, e0, x[2 * p]);
            x[2 * p + 1] = fma2(fl, e1, x[2 * p + 1]);
        }
        if constexpr (ODD) {
            float th, tl, sn, cs;
            if constexpr (GRID) phase_turns_grid(us, vs, ws, su, sv, sw, Cs, th, tl);
            else phase_turns_df(us, vs, ws, su, sv, sw, th, tl);
            sincos_mixed<FAST>(th, tl, sn, cs);
            x[VPT - 1] = fma2(fl, make_float2(cs, sn), x[VPT - 1]);
        }
    }

    // One block of leaves from record r on; returns how many it took
    // (kSumBlock, or what is left of a list's last chunk).
    __device__ __forceinline__ int at(const RecF* cb, int r, int n)
    {
        float2 x[VPT];
#pragma unroll
        for (int k = 0; k < VPT; ++k) x[k] = make_float2(0.f, 0.f);
        int taken;
        if (r + kSumBlock <= n) {
#pragma unroll 2
            for (int j = 0; j < kSumBlock; ++j) add_terms(cb[r + j], x);
            taken = kSumBlock;
        } else {
            for (int j = r; j < n; ++j) add_terms(cb[j], x);
            taken = n - r;
        }
#pragma unroll
        for (int k = 0; k < VPT; ++k) kahan_add2(acc[k], comp[k], x[k]);
        return taken;
    }
};

// ---------------------------------------------------------------- regrouped Eq. 17
// V = sum_n w_n xi_n, xi = 4^(J-j) eta (see RecWD in wt_internal.cuh). Per
// level j = 1 .. J-2 a thread keeps the sum of the children's xi of the open
// level-j node in shared memory (row j - 1); that of the open level-(J-1) node
// lives in registers, so a leaf never touches shared memory. A node's xi is
// that sum (the Eq. 9 form, times 4^(J-j)); it adds w xi to V and passes xi up
// to its parent (the first child writes, the others add).
template <int NT, int VPT>
struct Eq17WD {
    double u[VPT], v[VPT], w[VPT];
    double vr[VPT], vi[VPT];
    double sr[VPT], si[VPT];
    double2* stk;   // shared stack + threadIdx.x; row stride VPT * NT
    int J;
    int maxrow;

    __device__ __forceinline__ double2& slot(int row, int k) { return stk[(row * VPT + k) * NT]; }

    __device__ void operator()(const RecWD& r)
    {
        const uint32_t meta = r.meta;
        const int lev = static_cast<int>(meta & 31u);
        const bool root = meta & kRwRoot, first = meta & kRwFirst;
        if (meta & kRwLeaf) {
#pragma unroll
            for (int k = 0; k < VPT; ++k) {
                const double t = fma(w[k], r.c, fma(v[k], r.b, u[k] * r.a));
                double s, c;
                sincos_turns_f64(t, s, c);
                vr[k] = fma(r.d, c, vr[k]);
                vi[k] = fma(r.d, s, vi[k]);
                if (first) {
                    sr[k] = c;
                    si[k] = s;
                } else {
                    sr[k] += c;
                    si[k] += s;
                }
            }
            return;
        }
        const bool in_regs = (lev == J - 1);
        const int own = clamp_row(static_cast<uint32_t>(lev - 1), maxrow);
        const int par = clamp_row(static_cast<uint32_t>(lev > 1 ? lev - 2 : 0), maxrow);
#pragma unroll
        for (int k = 0; k < VPT; ++k) {
            const double2 S = in_regs ? make_double2(sr[k], si[k]) : slot(own, k);
            vr[k] = fma(r.d, S.x, vr[k]);
            vi[k] = fma(r.d, S.y, vi[k]);
            if (root) continue;
            double2& ps = slot(par, k);
            if (first) ps = S;
            else ps = make_double2(ps.x + S.x, ps.y + S.y);
        }
    }
};

// Eq. 16 in double-float (WT_FP64_DF, RecWDF): V = sum over the leaves of
// Phi_k times the plane wave at the pixel centre, in blocks of four leaves
// (df_accumulate); internal records are passed over. VPT = 1 alone, or pairs of
// visibilities (df64.cuh).
constexpr int kBlock16 = 4;
template <int VPT>
struct Eq16DF {
    static constexpr int NP = VPT / 2;
    DF2 U[NP], V[NP], W[NP];
    DFP vr[NP], vi[NP];
    DFP br[NP], bi[NP];    // the block's
    int held;              // leaves in it
    const float4* tab;
    __device__ __forceinline__ void start(const F2 (&u)[VPT], const F2 (&v)[VPT], const F2 (&w)[VPT])
    {
        held = 0;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            U[p] = df2_pack(u[2 * p], u[2 * p + 1]);
            V[p] = df2_pack(v[2 * p], v[2 * p + 1]);
            W[p] = df2_pack(w[2 * p], w[2 * p + 1]);
            vr[p] = vi[p] = dfp_zero();
        }
    }
    __device__ __forceinline__ double2 result(int k) const
    {
        double2 v = dfp_vis(vr[k / 2], vi[k / 2], k & 1);
        if (held) {
            const double2 b = dfp_vis(br[k / 2], bi[k / 2], k & 1);
            v = make_double2(v.x + b.x, v.y + b.y);
        }
        return v;
    }
    __device__ void operator()(const RecWDF& r)
    {
        if (!(r.meta & kRwLeaf)) return;
        const F2 su{r.ah, r.al}, sv{r.bh, r.bl}, sw{r.ch, r.cl};
        const DFS phi = dfs(r.fh, r.fl);
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            float2 th, tl;
            phase_turns_dfp(U[p], V[p], W[p], su, sv, sw, th, tl);
            DFP s, c;
            sincos_turns_dfp(th, tl, tab, s, c);
            if (held == 0) {
                br[p] = dfp_product(phi, c);
                bi[p] = dfp_product(phi, s);
            } else {
                dfp_accumulate_product(br[p], phi, c);
                dfp_accumulate_product(bi[p], phi, s);
            }
        }
        if (++held < kBlock16) return;
        held = 0;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            dfp_renorm(br[p]);
            dfp_renorm(bi[p]);
            dfp_add_block(vr[p], br[p]);
            dfp_add_block(vi[p], bi[p]);
        }
    }
};

template <>
struct Eq16DF<1> {
    F2 u, v, w;
    DF vr, vi;
    DF br, bi;
    int held;
    const float4* tab;
    __device__ __forceinline__ void start(const F2 (&u1)[1], const F2 (&v1)[1], const F2 (&w1)[1])
    {
        u = u1[0];
        v = v1[0];
        w = w1[0];
        vr = vi = DF{0.f, 0.f};
        held = 0;
    }
    __device__ __forceinline__ double2 result(int) const
    {
        return make_double2(df_to_double(vr) + (held ? df_to_double(br) : 0.0),
                            df_to_double(vi) + (held ? df_to_double(bi) : 0.0));
    }
    __device__ void operator()(const RecWDF& r)
    {
        if (!(r.meta & kRwLeaf)) return;
        const DF phi{r.fh, r.fl};
        float th, tl;
        phase_turns_df(u, v, w, F2{r.ah, r.al}, F2{r.bh, r.bl}, F2{r.ch, r.cl}, th, tl);
        DF s, c;
        sincos_turns_df(th, tl, tab, s, c);
        if (held == 0) {
            br = df_product(phi, c);
            bi = df_product(phi, s);
        } else {
            df_accumulate_product(br, phi, c);
            df_accumulate_product(bi, phi, s);
        }
        if (++held < kBlock16) return;
        held = 0;
        df_renorm(br);
        df_renorm(bi);
        df_add_block(vr, br);
        df_add_block(vi, bi);
    }
};

// Regrouped Eq. 17 in double-float (WT_FP64_DF, RecWDF): V = sum_n w_n eta_n
// with every quantity a double-float on the float32 pipe. Each node adds
// its w eta to V as soon as its eta is known, in blocks (df_accumulate): a run of
// sibling leaves and what follows it, up to the next run's first leaf, where the
// block joins V beside that leaf's phase, which does not wait for it. Over random
// trees the error is 0.70e-15 of Sigma |w eta| RMS (1.0 for 50 leaves, 1.3 for
// isolated components at J = 12), 1.40 (1.36, 2.3) when every addition was
// renormalised. Per visibility a thread keeps
// the sum of the children's eta of the open level-j node (j = 1 .. J-2) in
// shared-memory row j - 1; that of the open level-(J-1) node lives in
// registers, so a leaf never touches shared memory. A node's eta is a quarter
// of its children's sum (the Eq. 9 form; exact scaling), which it passes up to
// its parent (the first child writes, the others add). Pairs of visibilities
// (slots 2 p: the pair's real parts as heads, lows; 2 p + 1: the imaginary
// ones), or VPT = 1 alone (re h, re l, im h, im l). The medium sum 6.8 -> 6.3 ms
// by pairs.
template <int NT, int VPT>
struct Eq17DF {
    static constexpr int NP = VPT / 2;
    DF2 U[NP], V[NP], W[NP];
    DFP vr[NP], vi[NP];    // V
    DFP br[NP], bi[NP];    // the block's part of V
    DFP lr[NP], li[NP];    // children's eta sum of the open level-(J-1) node
    float4* stk;           // shared stack + threadIdx.x; row stride VPT * NT
    const float4* tab;     // exp(i 2 pi k/1024), sincos_turns_dfp
    int J;
    int maxrow;

    __device__ __forceinline__ float4& slot(int row, int k) { return stk[(row * VPT + k) * NT]; }

    __device__ __forceinline__ void start(const F2 (&u)[VPT], const F2 (&v)[VPT], const F2 (&w)[VPT])
    {
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            U[p] = df2_pack(u[2 * p], u[2 * p + 1]);
            V[p] = df2_pack(v[2 * p], v[2 * p + 1]);
            W[p] = df2_pack(w[2 * p], w[2 * p + 1]);
            vr[p] = vi[p] = br[p] = bi[p] = lr[p] = li[p] = dfp_zero();
        }
    }
    __device__ __forceinline__ double2 result(int k) const
    {
        const double2 v = dfp_vis(vr[k / 2], vi[k / 2], k & 1), b = dfp_vis(br[k / 2], bi[k / 2], k & 1);
        return make_double2(v.x + b.x, v.y + b.y);
    }

    __device__ void operator()(const RecWDF& r)
    {
        const uint32_t meta = r.meta;
        const int lev = static_cast<int>(meta & 31u);
        const bool root = meta & kRwRoot, first = meta & kRwFirst;
        const DFS wgt = dfs(r.wh, r.wl);
        if (meta & kRwLeaf) {
            const F2 su{r.ah, r.al}, sv{r.bh, r.bl}, sw{r.ch, r.cl};
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                float2 th, tl;
                phase_turns_dfp(U[p], V[p], W[p], su, sv, sw, th, tl);
                DFP s, c;
                sincos_turns_dfp(th, tl, tab, s, c);
                if (first) {           // (every leaf of level 1 is one)
                    dfp_add_block(vr[p], br[p]);
                    dfp_add_block(vi[p], bi[p]);
                    br[p] = dfp_product(wgt, c);
                    bi[p] = dfp_product(wgt, s);
                    lr[p] = c;
                    li[p] = s;
                } else {
                    dfp_accumulate_product(br[p], wgt, c);
                    dfp_accumulate_product(bi[p], wgt, s);
                    dfp_accumulate(lr[p], c);
                    dfp_accumulate(li[p], s);
                }
            }
            return;
        }
        const bool in_regs = (lev == J - 1);
        const int own = clamp_row(static_cast<uint32_t>(lev > 1 ? lev - 1 : 0), maxrow);
        const int par = clamp_row(static_cast<uint32_t>(lev > 2 ? lev - 2 : 0), maxrow);
        const float2 quarter = bcast2(0.25f);
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            DFP er, ei;
            if (in_regs) {
                er = lr[p];
                ei = li[p];
            } else {
                const float4 a = slot(own, 2 * p), b = slot(own, 2 * p + 1);
                er = DFP{make_float2(a.x, a.y), make_float2(a.z, a.w)};
                ei = DFP{make_float2(b.x, b.y), make_float2(b.z, b.w)};
            }
            er = DFP{mul2(er.h, quarter), mul2(er.l, quarter)};
            ei = DFP{mul2(ei.h, quarter), mul2(ei.l, quarter)};
            dfp_accumulate_product(br[p], wgt, er);
            dfp_accumulate_product(bi[p], wgt, ei);
            if (root) continue;
            float4& A = slot(par, 2 * p);
            float4& B = slot(par, 2 * p + 1);
            if (!first) {
                const float4 a = A, b = B;
                DFP pr{make_float2(a.x, a.y), make_float2(a.z, a.w)}, pi{make_float2(b.x, b.y), make_float2(b.z, b.w)};
                dfp_accumulate(pr, er);
                dfp_accumulate(pi, ei);
                er = pr;
                ei = pi;
            }
            A = make_float4(er.h.x, er.h.y, er.l.x, er.l.y);
            B = make_float4(ei.h.x, ei.h.y, ei.l.x, ei.l.y);
        }
    }
};

template <int NT>
struct Eq17DF<NT, 1> {
    F2 u, v, w;
    DF vr, vi;
    DF br, bi;
    DF lr, li;
    float4* stk;
    const float4* tab;
    int J;
    int maxrow;

    __device__ __forceinline__ float4& slot(int row) { return stk[row * NT]; }

    __device__ __forceinline__ void start(const F2 (&u1)[1], const F2 (&v1)[1], const F2 (&w1)[1])
    {
        u = u1[0];
        v = v1[0];
        w = w1[0];
        vr = vi = br = bi = lr = li = DF{0.f, 0.f};
    }
    __device__ __forceinline__ double2 result(int) const
    {
        return make_double2(df_to_double(vr) + df_to_double(br), df_to_double(vi) + df_to_double(bi));
    }

    __device__ void operator()(const RecWDF& r)
    {
        const uint32_t meta = r.meta;
        const int lev = static_cast<int>(meta & 31u);
        const bool root = meta & kRwRoot, first = meta & kRwFirst;
        const DF wgt{r.wh, r.wl};
        if (meta & kRwLeaf) {
            // no branch (few visibilities, a warp or two per scheduler: a run's
            // later leaves add an empty block beside the phase, which costs less
            // than waiting for a branch's chain)
            const DF none{0.f, 0.f};
            df_add_block(vr, first ? br : none);
            df_add_block(vi, first ? bi : none);
            br = first ? none : br;
            bi = first ? none : bi;
            lr = first ? none : lr;
            li = first ? none : li;
            float th, tl;
            phase_turns_df(u, v, w, F2{r.ah, r.al}, F2{r.bh, r.bl}, F2{r.ch, r.cl}, th, tl);
            DF s, c;
            sincos_turns_df(th, tl, tab, s, c);
            df_accumulate_product(br, wgt, c);
            df_accumulate_product(bi, wgt, s);
            df_accumulate(lr, c.h, c.l);
            df_accumulate(li, s.h, s.l);
            return;
        }
        const int own = clamp_row(static_cast<uint32_t>(lev > 1 ? lev - 1 : 0), maxrow);
        const int par = clamp_row(static_cast<uint32_t>(lev > 2 ? lev - 2 : 0), maxrow);
        DF er, ei;
        if (lev == J - 1) {
            er = df_scale(lr, 0.25f);
            ei = df_scale(li, 0.25f);
        } else {
            const float4 S = slot(own);
            er = DF{0.25f * S.x, 0.25f * S.y};
            ei = DF{0.25f * S.z, 0.25f * S.w};
        }
        df_accumulate_product(br, wgt, er);
        df_accumulate_product(bi, wgt, ei);
        if (root) return;
        float4& P = slot(par);
        if (first) {
            P = make_float4(er.h, er.l, ei.h, ei.l);
        } else {
            DF pr{P.x, P.y}, pi{P.z, P.w};
            df_accumulate(pr, er.h, er.l);
            df_accumulate(pi, ei.h, ei.l);
            P = make_float4(pr.h, pr.l, pi.h, pi.l);
        }
    }
};

// Regrouped Eq. 17 in the mixed forms: V = sum_n w_n xi_n over every node,
// xi = 4^(J-j) eta and w_n scaled to match by the build (RecWF). Per
// visibility a thread keeps one pair per level: the xi sum of the open
// level-j node (j = 1 .. J-3) in shared-memory row j - 1 (layout
// [row][thread][vis]: a thread's visibilities side by side, one 16-byte
// access per row at two visibilities per thread); those of the open
// level-(J-1) and level-(J-2) nodes live in registers, with the plain
// float32 sums of their children's terms (w xi, at most four each), so
// leaves and level-(J-1) nodes touch neither shared memory nor the
// compensated sum. Any other internal node reads its xi, adds w xi (plus,
// at level J-2, its children's terms) to V with compensation and passes xi
// up (the first child writes its parent's sum, the others add).
// Packed pairs as in Eq17F. GRID: the leaf phases with their heads on the
// common grid of each visibility's constant C (phase_turns_grid2; the
// caller sets Cg and Cs and guarantees that the grid is valid), else with
// error-free sums (phase_turns_df2). GROUPS: the fast form takes a group
// (a run of sibling leaves and their level-(J-1) parent) in one step of a
// variable-stride sweep, else every record in a fixed-stride sweep, the
// second leaf of a pair skipped (measured: groups faster in the single-tree
// predictor, slower in the batched one).
template <int NT, int VPT, bool FAST = false, bool GRID = false, bool GROUPS = true>
struct Eq17WF {
    static constexpr int NP = VPT / 2;
    static constexpr bool ODD = (VPT & 1) != 0;
    F2 u[VPT], v[VPT], w[VPT];                        // set by the caller, then start()
    DF2 U[NP > 0 ? NP : 1], V[NP > 0 ? NP : 1], W[NP > 0 ? NP : 1];
    float2 Cg[NP > 0 ? NP : 1];                       // GRID: the grid constants of visibilities 2p, 2p + 1
    float Cs;                                         // GRID: that of the last, unpaired visibility
    float2 acc[VPT], comp[VPT];                       // Kahan sum of V and its compensation
    float2 low[VPT];                                  // xi sum of the open level-(J-1) node
    float2 lowx[VPT];                                 // w xi sum of its leaves
    float2 mid[VPT];                                  // xi sum of the open level-(J-2) node
    float2 midx[VPT];                                 // plain sum of the terms of its children
                                                      // (at most 4)
    float2* stk;                                      // shared stack + threadIdx.x * VPT
    int J;
    int maxrow;

    __device__ __forceinline__ float2* row_ptr(int row) { return stk + row * (NT * VPT); }

    __device__ __forceinline__ void load_row(int row, float2 (&x)[VPT])
    {
        const float2* p = row_ptr(row);
        if constexpr (VPT % 2 == 0) {
#pragma unroll
            for (int k = 0; k < VPT; k += 2) {
                const float4 q = *reinterpret_cast<const float4*>(p + k);
                x[k] = make_float2(q.x, q.y);
                x[k + 1] = make_float2(q.z, q.w);
            }
        } else {
#pragma unroll
            for (int k = 0; k < VPT; ++k) x[k] = p[k];
        }
    }

    __device__ __forceinline__ void store_row(int row, const float2 (&x)[VPT])
    {
        float2* p = row_ptr(row);
        if constexpr (VPT % 2 == 0) {
#pragma unroll
            for (int k = 0; k < VPT; k += 2)
                *reinterpret_cast<float4*>(p + k) = make_float4(x[k].x, x[k].y, x[k + 1].x, x[k + 1].y);
        } else {
#pragma unroll
            for (int k = 0; k < VPT; ++k) p[k] = x[k];
        }
    }

    __device__ __forceinline__ void start()
    {
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            U[p] = df2_pack(u[2 * p], u[2 * p + 1]);
            V[p] = df2_pack(v[2 * p], v[2 * p + 1]);
            W[p] = df2_pack(w[2 * p], w[2 * p + 1]);
        }
#pragma unroll
        for (int k = 0; k < VPT; ++k) {
            acc[k] = make_float2(0.f, 0.f);
            comp[k] = make_float2(0.f, 0.f);
            low[k] = make_float2(0.f, 0.f);
            lowx[k] = make_float2(0.f, 0.f);
            mid[k] = make_float2(0.f, 0.f);
            midx[k] = make_float2(0.f, 0.f);
        }
    }

    __device__ __forceinline__ float2 result(int k) const { return sub2(acc[k], comp[k]); }

    __device__ __forceinline__ void phase2(int p, F2 su, F2 sv, F2 sw, float2& h, float2& tl) const
    {
        if constexpr (GRID) phase_turns_grid2(U[p], V[p], W[p], su, sv, sw, Cg[p], h, tl);
        else phase_turns_df2(U[p], V[p], W[p], su, sv, sw, h, tl);
    }

    __device__ __forceinline__ void phase1(F2 su, F2 sv, F2 sw, float& th, float& tl) const
    {
        constexpr int k = VPT - 1;
        if constexpr (GRID) phase_turns_grid(u[k], v[k], w[k], su, sv, sw, Cs, th, tl);
        else phase_turns_df(u[k], v[k], w[k], su, sv, sw, th, tl);
    }

    // A leaf's sums start from zero: its parent clears them after reading.
    __device__ __forceinline__ void leaf_up(int k, float2 xi, float2 wv, bool root)
    {
        if (root) {                                   // J = 1: the leaf is a level-1 pixel
            kahan_add2(acc[k], comp[k], mul2(wv, xi));
            return;
        }
        low[k] = add2(low[k], xi);
        lowx[k] = fma2(wv, xi, lowx[k]);
    }

    // Two sibling leaves together: four independent phase chains per thread
    // (two visibilities x two leaves), one dispatch.
    __device__ __forceinline__ void leaf_pair(const RecWF& a, const RecWF& b)
    {
        const F2 su0{a.a, a.b}, sv0{a.c, a.d}, sw0{a.e, a.f};
        const F2 su1{b.a, b.b}, sv1{b.c, b.d}, sw1{b.e, b.f};
        const float2 w0 = bcast2(a.g), w1 = bcast2(b.g);
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            float2 h0, tl0, h1, tl1, e00, e01, e10, e11;
            phase2(p, su0, sv0, sw0, h0, tl0);
            phase2(p, su1, sv1, sw1, h1, tl1);
            sincos_mixed2<FAST>(h0, tl0, e00, e01);
            sincos_mixed2<FAST>(h1, tl1, e10, e11);
            low[2 * p] = add2(low[2 * p], add2(e00, e10));
            low[2 * p + 1] = add2(low[2 * p + 1], add2(e01, e11));
            lowx[2 * p] = fma2(w1, e10, fma2(w0, e00, lowx[2 * p]));
            lowx[2 * p + 1] = fma2(w1, e11, fma2(w0, e01, lowx[2 * p + 1]));
        }
        if constexpr (ODD) {
            constexpr int k = VPT - 1;
            float th0, tl0, s0, c0, th1, tl1, s1, c1;
            phase1(su0, sv0, sw0, th0, tl0);
            phase1(su1, sv1, sw1, th1, tl1);
            sincos_mixed<FAST>(th0, tl0, s0, c0);
            sincos_mixed<FAST>(th1, tl1, s1, c1);
            const float2 e0 = make_float2(c0, s0), e1 = make_float2(c1, s1);
            low[k] = add2(low[k], add2(e0, e1));
            lowx[k] = fma2(w1, e1, fma2(w0, e0, lowx[k]));
        }
    }

    // One step of the fast form's grouped sweep; returns the records it took.
    // A group (in one chunk by construction) is one step: its leaves in
    // pairs, then the parent; a leaf marked as the first of a pair takes its
    // sibling with it.
    __device__ __forceinline__ int at_grouped(const RecWF* cb, int r, int n)
    {
        const RecWF& a = cb[r];
        const uint32_t meta = a.meta;
        if (meta & kRwGroup) {
            const int k = static_cast<int>((meta >> kRwGroupShift) & 7u);
            if (k >= 1 && k <= 4 && r + k < n) {
                group(cb + r, k);
                return k + 1;
            }
        } else if ((meta & kRwPairFirst) && r + 1 < n) {
            leaf_pair(a, cb[r + 1]);
            return 2;
        }
        (*this)(a);
        return 1;
    }

    // One record of a fixed-stride sweep: the fast form's first leaf of a
    // pair takes its sibling, the second is skipped. The polynomial form
    // takes every record alone: its four chains need more registers than the
    // pairing saves (measured 2 % slower).
    __device__ __forceinline__ void at_single(const RecWF* cb, int r, int n)
    {
        const RecWF& a = cb[r];
        if constexpr (FAST) {
            if (a.meta & (kRwPairFirst | kRwPairSecond)) {
                if (a.meta & kRwPairFirst) leaf_pair(a, cb[r + 1 < n ? r + 1 : r]);
                return;
            }
        }
        (*this)(a);
    }

    // The polynomial form takes every record alone: a fixed stride.
    __device__ __forceinline__ auto at(const RecWF* cb, int r, int n)
    {
        if constexpr (GROUPS && FAST) return at_grouped(cb, r, n);
        else at_single(cb, r, n);
    }

    // A group of k sibling leaves g[0 .. k-1] and their parent g[k].
    __device__ __forceinline__ void group(const RecWF* g, int k)
    {
        if (k >= 2) leaf_pair(g[0], g[1]);
        else leaf(g[0], false);
        if (k == 4) leaf_pair(g[2], g[3]);
        else if (k == 3) leaf(g[2], false);
        low_levels(g[k], g[k].meta);
    }

    // Parent's xi sum: the first child writes it, the others add (a select,
    // not a branch: internal nodes are most records of deep, sparse trees).
    __device__ __forceinline__ void pass_up(int par, bool first, const float2 (&xi)[VPT])
    {
        float2 ps[VPT];
        load_row(par, ps);
#pragma unroll
        for (int k = 0; k < VPT; ++k) ps[k] = first ? xi[k] : add2(ps[k], xi[k]);
        store_row(par, ps);
    }

    // Nodes at levels J - 1 and J - 2, whose sums are in registers.
    __device__ __forceinline__ void low_levels(const RecWF& r, uint32_t meta)
    {
        const bool root = meta & kRwRoot, first = meta & kRwFirst;
        const float2 wv = bcast2(r.g);
        float2 xi[VPT];
        if (meta & kRwLowSum) {                        // level J - 1: registers only
#pragma unroll
            for (int k = 0; k < VPT; ++k) {
                xi[k] = low[k];
                const float2 x = fma2(wv, xi[k], lowx[k]);
                low[k] = make_float2(0.f, 0.f);
                lowx[k] = make_float2(0.f, 0.f);
                if (root) {
                    kahan_add2(acc[k], comp[k], x);
                } else {                               // the parent (level J - 2) takes both
                    midx[k] = add2(midx[k], x);
                    mid[k] = add2(mid[k], xi[k]);
                }
            }
            return;
        }
#pragma unroll
        for (int k = 0; k < VPT; ++k) {                // level J - 2
            xi[k] = mid[k];
            kahan_add2(acc[k], comp[k], fma2(wv, xi[k], midx[k]));
            mid[k] = make_float2(0.f, 0.f);
            midx[k] = make_float2(0.f, 0.f);
        }
        if (!root) pass_up(clamp_row(__float_as_uint(r.b), maxrow), first, xi);
    }

    // One leaf alone (root: a level-1 pixel, J = 1).
    __device__ __forceinline__ void leaf(const RecWF& r, bool root)
    {
        const float2 wv = bcast2(r.g);
        const F2 su{r.a, r.b}, sv{r.c, r.d}, sw{r.e, r.f};
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            float2 h, tl, e0, e1;
            phase2(p, su, sv, sw, h, tl);
            sincos_mixed2<FAST>(h, tl, e0, e1);
            leaf_up(2 * p, e0, wv, root);
            leaf_up(2 * p + 1, e1, wv, root);
        }
        if constexpr (ODD) {
            constexpr int k = VPT - 1;
            float th, tl, s, c;
            phase1(su, sv, sw, th, tl);
            sincos_mixed<FAST>(th, tl, s, c);
            leaf_up(k, make_float2(c, s), wv, root);
        }
    }

    __device__ void operator()(const RecWF& r)
    {
        const uint32_t meta = r.meta;
        const float2 wv = bcast2(r.g);
        if (meta & kRwLeaf) {
            leaf(r, (meta & kRwRoot) != 0);
            return;
        }
        if (meta & (kRwLowSum | kRwMidSum)) {
            low_levels(r, meta);
            return;
        }
        // any other internal node (level <= J - 3): rows pre-decoded by the
        // build (own: lev - 1, parent's: lev - 2), clamped to the stack. A
        // level-1 node (a root, always a first child) writes its xi back into
        // its own row 0, which the next level-1 node's first child overwrites.
        const int own = clamp_row(__float_as_uint(r.a), maxrow);
        const int par = clamp_row(__float_as_uint(r.b), maxrow);
        float2 xi[VPT];
        load_row(own, xi);
#pragma unroll
        for (int k = 0; k < VPT; ++k) kahan_add2(acc[k], comp[k], mul2(wv, xi[k]));
        pass_up(par, (meta & kRwFirst) != 0, xi);
    }
};

// The regrouped Eq. 17 in a mixed form runs in a grid pass and an exact
// pass (the tile helpers in wt_internal.cuh: tile_grid_constants,
// tile_deferred, mark_deferred).

// One tile's sweep of the regrouped Eq. 17 (GRID: on the head grid of the
// constants C, else with error-free sums; GROUPS as Eq17WF). Returns false
// (CTA-wide) if a staging copy did not arrive; res receives V of each
// visibility.
template <int NT, int VPT, bool FAST, bool GRID, bool GROUPS = true>
__device__ __forceinline__ bool sweep_regrouped_mixed(Stager<RecWF>& st, const F2 (&u)[VPT], const F2 (&v)[VPT],
                                      const F2 (&w)[VPT], const float (&C)[VPT], float2* stk, int J, int maxrow,
                                      float2 (&res)[VPT])
{
    Eq17WF<NT, VPT, FAST, GRID, GROUPS> b;
#pragma unroll
    for (int k = 0; k < VPT; ++k) { b.u[k] = u[k]; b.v[k] = v[k]; b.w[k] = w[k]; }
    if constexpr (GRID) {
#pragma unroll
        for (int p = 0; p < VPT / 2; ++p) b.Cg[p] = make_float2(C[2 * p], C[2 * p + 1]);
        b.Cs = C[VPT - 1];
    }
    b.start();
    b.stk = stk;
    b.J = J;
    b.maxrow = maxrow;
    const bool good = st.sweep_at(b);
#pragma unroll
    for (int k = 0; k < VPT; ++k) res[k] = b.result(k);
    return good;
}


}  // namespace
}  // namespace wt
