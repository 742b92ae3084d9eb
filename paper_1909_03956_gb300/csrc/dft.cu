// dft.cu -- dft_predict_vis: the direct sum over the clean-component list
// (Sec. 3.3, Eq. 12; the "more accurate alternative" of Sec. 2.2):
//   V_n = sum_m C_m exp(sign i 2 pi [u_n l_m + v_n m_m + w_n (n_m - 1)]).
//
// A prologue kernel packs each component once into a 32-byte record in a
// scratch buffer: (l, m, n - 1, C) in float64 for WT_FP64, or double-float
// halves of l, m, n - 1 and C for the other forms (the mixed forms use C's
// high half only), and reduces the bounds max |l|, |m|, |n - 1| of the
// float32 heads into a 16-byte block after the records. The main kernel gives
// each thread one visibility (float64) or two (mixed, on packed float32
// pairs) and streams the records through shared memory (bulk copies,
// double-buffered, broadcast reads), like the wavelet kernels. The mixed
// forms run a grid pass and an exact pass, as the regrouped wavelet sum does
// (wt_internal.cuh): the phase heads on each visibility's common grid where
// the bounds allow, else error-free sums.
#include "df64.cuh"
#include "staging.cuh"
#include "wt_internal.cuh"

namespace wt {

// dft_tc.cu: the tensor-core form (WT_MIXED_TC)
size_t dft_tc_scratch_bytes(int64_t n_comp);
int dft_tc_launch(const double* l, const double* m, const double* flux, int64_t n_comp, const void* recs,
                  const uint32_t* bound, void* tc, const TermParts& tp, const double* uvw, int64_t n_vis, void* vis,
                  int sign, int* status, cudaStream_t s);
int64_t dft_tc_tiles(int64_t n_vis, int64_t n_comp);

namespace {

constexpr int kChunk = 512;

struct CompD {
    double l, m, nm1, flux;
};
static_assert(sizeof(CompD) == 32, "component record layout");

// n - 1 = -(l^2 + m^2) / (1 + sqrt(1 - l^2 - m^2)), free of cancellation.
// bound (float records only; zeroed before the launch, its fourth word the
// flag of deferred tiles): the largest |l|, |m|, |n - 1| of the float32 heads as float bit patterns (non-negative
// floats order as their bits), reduced per warp, then by atomicMax; a
// component that fails the range check adds nothing.
__global__ void k_pack_components(const double* __restrict__ l, const double* __restrict__ m,
                                  const double* __restrict__ flux, int64_t n, CompD* __restrict__ outd,
                                  CompF* __restrict__ outf, uint32_t* __restrict__ bound, int* status)
{
    const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    uint32_t bl = 0, bm = 0, bn = 0;
    if (i < n) {
        const double li = l[i], mi = m[i], fi = flux[i];
        const double r2 = li * li + mi * mi;
        double nm1 = 0.0;
        const bool good = r2 < 1.0 && isfinite(li) && isfinite(mi) && isfinite(fi);
        if (!good) record_status(status, WT_ERR_RANGE);
        else nm1 = -r2 / (1.0 + sqrt(1.0 - r2));
        if (outd) outd[i] = CompD{li, mi, nm1, fi};
        if (outf) {
            const F2 a = split_f64(li), b = split_f64(mi), c = split_f64(nm1), f = split_f64(fi);
            outf[i] = CompF{a.hi, a.lo, b.hi, b.lo, c.hi, c.lo, f.hi, f.lo};
            if (good) {
                bl = __float_as_uint(fabsf(a.hi));
                bm = __float_as_uint(fabsf(b.hi));
                bn = __float_as_uint(fabsf(c.hi));
            }
        }
    }
    if (!bound) return;
    bl = __reduce_max_sync(0xffffffffu, bl);
    bm = __reduce_max_sync(0xffffffffu, bm);
    bn = __reduce_max_sync(0xffffffffu, bn);
    if ((threadIdx.x & 31) == 0) {
        if (bl) atomicMax(&bound[0], bl);
        if (bm) atomicMax(&bound[1], bm);
        if (bn) atomicMax(&bound[2], bn);
    }
}

struct BodyD {
    double u, v, w, sgn, vr, vi;
    __device__ void operator()(const CompD& c)
    {
        double t = fma(w, c.nm1, fma(v, c.m, u * c.l));
        double s, co;
        sincos_turns_f64(t, s, co);
        vr = fma(c.flux, co, vr);
        vi = fma(c.flux, s, vi);
    }
};

// Mixed forms on packed float32 pairs: a thread owns two visibilities
// (n and n + NT of its tile). The phases of the two visibilities against one
// component form one pair of double-floats; each visibility's (cos, sin)
// comes out as its own pair. The components are taken kSumBlock at a time:
// their terms added by FMAs into a partial per visibility, the partial then
// into its Kahan sum (blockwise compensated summation).
// GRID: the phases with their heads on the grids of Cg (phase_turns_grid2),
// else with error-free sums (phase_turns_df2).
template <bool FAST, bool GRID>
struct BodyF2 {
    DF2 U, V, W;
    float2 Cg;
    float2 acc[2], comp[2];

    // p0 += flux (cos, sin) of visibility 0, p1 of visibility 1
    __device__ __forceinline__ void add_term(const CompF& c, float2& p0, float2& p1) const
    {
        float2 h, tl, e0, e1;
        if constexpr (GRID) phase_turns_grid2(U, V, W, F2{c.lh, c.ll}, F2{c.mh, c.ml}, F2{c.nh, c.nl}, Cg, h, tl);
        else phase_turns_df2(U, V, W, F2{c.lh, c.ll}, F2{c.mh, c.ml}, F2{c.nh, c.nl}, h, tl);
        sincos_mixed2<FAST>(h, tl, e0, e1);
        const float2 f = bcast2(c.flux);
        p0 = fma2(f, e0, p0);
        p1 = fma2(f, e1, p1);
    }

    // One block of components from record r on; returns how many it took
    // (kSumBlock, or what is left of a list's last chunk).
    __device__ __forceinline__ int at(const CompF* cb, int r, int n)
    {
        float2 p0 = make_float2(0.f, 0.f), p1 = p0;
        int taken;
        if (r + kSumBlock <= n) {
#pragma unroll 2
            for (int j = 0; j < kSumBlock; ++j) add_term(cb[r + j], p0, p1);
            taken = kSumBlock;
        } else {
            for (int j = r; j < n; ++j) add_term(cb[j], p0, p1);
            taken = n - r;
        }
        kahan_add2(acc[0], comp[0], p0);
        kahan_add2(acc[1], comp[1], p1);
        return taken;
    }
};

// The float64-class double-float form: two visibilities per thread (n and n +
// NT of its tile) as a pair, every step in double-float (df64.cuh).
struct BodyDF {
    DF2 U, V, W;
    DFP vr, vi;
    const float4* tab;
    // a block's terms (df_accumulate): kBlock, or fewer
    static constexpr int kBlock = 4;
    template <bool FIRST>
    __device__ __forceinline__ void term(const CompF& c, DFP& br, DFP& bi) const
    {
        float2 th, tl;
        phase_turns_dfp(U, V, W, F2{c.lh, c.ll}, F2{c.mh, c.ml}, F2{c.nh, c.nl}, th, tl);
        DFP s, co;
        sincos_turns_dfp(th, tl, tab, s, co);
        const DFS f = dfs(c.flux, c.flux_lo);
        if constexpr (FIRST) {
            br = dfp_product(f, co);
            bi = dfp_product(f, s);
        } else {
            dfp_accumulate_product(br, f, co);
            dfp_accumulate_product(bi, f, s);
        }
    }
    // Two blocks side by side, or one of what is left of a chunk, into the sums;
    // returns how many components.
    __device__ __forceinline__ int at(const CompF* cb, int r, int n)
    {
        DFP br, bi;
        int taken = 2 * kBlock;
        term<true>(cb[r], br, bi);
        if (r + 2 * kBlock <= n) {
            DFP cr, ci;
            term<true>(cb[r + kBlock], cr, ci);
#pragma unroll
            for (int j = 1; j < kBlock; ++j) {
                term<false>(cb[r + j], br, bi);
                term<false>(cb[r + kBlock + j], cr, ci);
            }
            dfp_renorm(br);
            dfp_renorm(bi);
            dfp_renorm(cr);
            dfp_renorm(ci);
            dfp_accumulate(br, cr);
            dfp_accumulate(bi, ci);
        } else {
            taken = n - r < kBlock ? n - r : kBlock;
            for (int j = 1; j < taken; ++j) term<false>(cb[r + j], br, bi);
            dfp_renorm(br);
            dfp_renorm(bi);
        }
        dfp_add_block(vr, br);
        dfp_add_block(vi, bi);
        return taken;
    }
};
constexpr int kChunkDirDF = 128;   // records per staging buffer beside the 16 KB table

// Few visibilities. A CTA per tile of visibilities leaves most SMs idle when
// there are fewer tiles than SMs (one integration of 128 antennas, 8 128
// visibilities: 64 float64 tiles on 152 SMs, 4.06 ms for 5 000 components), so
// the terms are then cut into parts, a CTA per (tile, part) on grid.y, each
// writing its sum to its own row of a workspace, and k_sum_parts adds the rows
// in order (in float64): 1.46 ms. 780 visibilities x 3 760 components on the
// special-function unit: 377 -> 40 us. CUT: the kernel takes its part of the
// list; a list that is not cut runs the kernel without this (20 components, 3.9 M
// visibilities: 2.5 % of the double-float form, 1.2 of the polynomial mixed one).
template <bool CUT, class Rec, class C>
__device__ __forceinline__ void take_part(const Rec* __restrict__& recs, int64_t& n_terms, int64_t per_part,
                                          C* __restrict__& vis, int64_t n_vis)
{
    if constexpr (CUT) {
        const int64_t from = static_cast<int64_t>(blockIdx.y) * per_part;
        recs += from;
        n_terms = max(n_terms - from, int64_t(0));
        if (blockIdx.y + 1 < gridDim.y) n_terms = min(n_terms, per_part);   // the last takes the rest
        vis += blockIdx.y * n_vis;
    }
}

// vis[i] = sum over p of partial[p][i], in order, in float64.
template <class C>
__global__ void k_sum_parts(const double2* __restrict__ partial, int parts, int64_t n_vis, C* __restrict__ vis)
{
    const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= n_vis) return;
    double2 a = make_double2(0.0, 0.0);
#pragma unroll 4
    for (int p = 0; p < parts; ++p) {
        const double2 x = partial[p * n_vis + i];
        a.x += x.x;
        a.y += x.y;
    }
    vis[i].x = static_cast<decltype(vis[i].x)>(a.x);
    vis[i].y = static_cast<decltype(vis[i].y)>(a.y);
}

template <int NT, bool CUT>
__global__ void __launch_bounds__(NT) k_dft_df(const CompF* __restrict__ comps, int64_t n_comp, int64_t per_part,
                                               const double* __restrict__ uvw, int64_t n_vis,
                                               double2* __restrict__ vis, double sgn, int* status)
{
    extern __shared__ __align__(16) unsigned char smem[];
    take_part<CUT>(comps, n_comp, per_part, vis, n_vis);
    Stager<CompF> st;
    stager_setup(st, smem, comps, n_comp, kChunkDirDF);
    float4* tab = reinterpret_cast<float4*>(smem + stager_bytes<CompF>(kChunkDirDF));
    load_sincos_table_df(tab);
    __syncthreads();
    const int64_t ntiles = (n_vis + 2 * NT - 1) / (2 * NT);
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t n0 = tile * 2 * NT + threadIdx.x, n1 = n0 + NT;
        const bool ok0 = n0 < n_vis, ok1 = n1 < n_vis;
        auto pair = [&](int c) {   // sign folded into the baseline (exact)
            return df2_pack(split_f64(ok0 ? sgn * uvw[3 * n0 + c] : 0.0), split_f64(ok1 ? sgn * uvw[3 * n1 + c] : 0.0));
        };
        BodyDF b;
        b.U = pair(0);
        b.V = pair(1);
        b.W = pair(2);
        b.vr = b.vi = dfp_zero();
        b.tab = tab;
        if (!st.sweep_at(b)) {
            if (threadIdx.x == 0) record_status(status, WT_ERR_TIMEOUT);
            return;
        }
        if (ok0) vis[n0] = dfp_vis(b.vr, b.vi, 0);
        if (ok1) vis[n1] = dfp_vis(b.vr, b.vi, 1);
    }
}

template <int NT, bool CUT>
__global__ void __launch_bounds__(NT) k_dft_fp64(const CompD* __restrict__ comps, int64_t n_comp, int64_t per_part,
                                                 const double* __restrict__ uvw, int64_t n_vis,
                                                 double2* __restrict__ vis, double sgn, int* status)
{
    extern __shared__ __align__(16) unsigned char smem[];
    take_part<CUT>(comps, n_comp, per_part, vis, n_vis);
    Stager<CompD> st;
    stager_setup(st, smem, comps, n_comp, kChunk);
    const int64_t ntiles = (n_vis + NT - 1) / NT;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t n = tile * NT + threadIdx.x;
        const bool valid = n < n_vis;
        // the sign is folded into the baseline: exp(-i 2 pi t) = exp(i 2 pi (-t)), exact
        BodyD b{valid ? sgn * uvw[3 * n] : 0.0, valid ? sgn * uvw[3 * n + 1] : 0.0,
                valid ? sgn * uvw[3 * n + 2] : 0.0, sgn, 0.0, 0.0};
        if (!st.sweep(b)) {
            if (threadIdx.x == 0) record_status(status, WT_ERR_TIMEOUT);
            return;
        }
        if (valid) vis[n] = make_double2(b.vr, b.vi);
    }
}

// GRIDPASS: the grid pass (every tile; a tile whose phases do not all fit
// the head grid is swept too, its results discarded, and marked for the
// exact pass); else the exact pass (only the marked tiles). bound: the
// records' coordinate bounds (k_pack_components).
template <int NT, bool FAST, bool GRIDPASS, bool CUT>
__global__ void __launch_bounds__(NT) k_dft_mixed(const CompF* __restrict__ comps, int64_t n_comp, int64_t per_part,
                                                  const uint32_t* __restrict__ bound,
                                                  const double* __restrict__ uvw, int64_t n_vis,
                                                  MixedOut<CUT>* __restrict__ vis, float sgn, int* status)
{
    extern __shared__ __align__(16) unsigned char smem[];
    if constexpr (!GRIDPASS) {
        if (!any_deferred(reinterpret_cast<const float*>(bound))) return;
    }
    take_part<CUT>(comps, n_comp, per_part, vis, n_vis);
    Stager<CompF> st;
    stager_setup(st, smem, comps, n_comp, kChunk);
    const int64_t ntiles = (n_vis + 2 * NT - 1) / (2 * NT);
    const double sg = static_cast<double>(sgn);       // sign folded into the baseline (exact)
    float smax[3] = {0.f, 0.f, 0.f};
    if constexpr (GRIDPASS) {
        smax[0] = __uint_as_float(bound[0]);
        smax[1] = __uint_as_float(bound[1]);
        smax[2] = __uint_as_float(bound[2]);
    }
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        float2* first_vis = reinterpret_cast<float2*>(vis + tile * 2 * NT);
        if constexpr (!GRIDPASS) {
            if (!tile_deferred(first_vis)) continue;   // done by the grid pass
        }
        const int64_t n0 = tile * 2 * NT + threadIdx.x, n1 = n0 + NT;
        const bool ok0 = n0 < n_vis, ok1 = n1 < n_vis;
        const F2 u[2] = {split_f64(ok0 ? sg * uvw[3 * n0] : 0.0), split_f64(ok1 ? sg * uvw[3 * n1] : 0.0)};
        const F2 v[2] = {split_f64(ok0 ? sg * uvw[3 * n0 + 1] : 0.0), split_f64(ok1 ? sg * uvw[3 * n1 + 1] : 0.0)};
        const F2 w[2] = {split_f64(ok0 ? sg * uvw[3 * n0 + 2] : 0.0), split_f64(ok1 ? sg * uvw[3 * n1 + 2] : 0.0)};
        BodyF2<FAST, GRIDPASS> b;
        bool defer = false;
        if constexpr (GRIDPASS) {
            float C[2];
            defer = !tile_grid_constants<2>(u, v, w, smax, C);   // a CTA-wide decision
            b.Cg = make_float2(C[0], C[1]);
        }
        b.U = df2_pack(u[0], u[1]);
        b.V = df2_pack(v[0], v[1]);
        b.W = df2_pack(w[0], w[1]);
        b.acc[0] = b.acc[1] = b.comp[0] = b.comp[1] = make_float2(0.f, 0.f);
        if (!st.sweep_at(b)) {
            if (threadIdx.x == 0) record_status(status, WT_ERR_TIMEOUT);
            return;
        }
        if (defer) {
            mark_deferred(first_vis, reinterpret_cast<const float*>(bound));
            continue;
        }
        if (ok0) store_sum(vis[n0], b.acc[0], b.comp[0]);
        if (ok1) store_sum(vis[n1], b.acc[1], b.comp[1]);
    }
}

template <class K>
int grid_for(K kernel, int threads, int nt, size_t smem, int64_t n_vis, dim3& grid)
{
    const int rc = allow_dynamic_smem(reinterpret_cast<const void*>(kernel), smem);
    if (rc) return rc;
    int per_sm = 0;
    WT_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem));
    if (per_sm < 1) return set_error(WT_ERR_UNSUPPORTED, "dft kernel does not fit on an SM");
    // one CTA per tile (nt visibilities), so that the hardware balances the
    // SMs as CTAs finish; the kernels stride only if the grid is capped
    const int64_t ntiles = (n_vis + nt - 1) / nt;
    grid = dim3(static_cast<unsigned>(ntiles < 0x7fffffff ? ntiles : 0x7fffffff));
    return WT_OK;
}

}  // namespace

// The cut of a sum of n_terms over `tiles` tiles of visibilities, `fill` CTAs
// filling an SM's pipes. Not cut while the tiles alone do that: beyond, the
// hardware balances them as they finish. Else into equal parts (in blocks of
// kPartTerms terms), all resident together, so that an SM's time goes with its
// CTAs times a part's length, half a block added for a CTA's set-up: the cut,
// up to ten CTAs per SM, that comes nearest to an even load of all SMs. 8 128
// visibilities x 5 000 components in float64: 64 tiles, 14 parts.
TermParts term_parts(int64_t tiles, int64_t n_terms, int fill)
{
    const int64_t sms = num_sms(), blocks = n_terms > 0 ? (n_terms + kPartTerms - 1) / kPartTerms : 1;
    TermParts tp{1, blocks * kPartTerms};
    if (tiles < 1 || tiles >= fill * sms) return tp;
    double best = 1e300;
    for (int64_t p = 1; p <= blocks && (p == 1 || p * tiles <= 10 * sms); ++p) {
        const int64_t per = (blocks + p - 1) / p, parts = (blocks + per - 1) / per;
        const int64_t busiest = (tiles * parts + sms - 1) / sms;
        const double time = (static_cast<double>(per) + 0.5) * static_cast<double>(busiest < fill ? fill : busiest);
        if (time < best) {
            best = time;
            tp = TermParts{parts, per * kPartTerms};
        }
    }
    return tp;
}

namespace {
// The cut of a form's sum by the tiles of its main kernel: CTAs of 128 threads
// (160 on the tensor cores), four to fill an SM; of 256 (mixed), two; of 64
// (double-float), eight.
TermParts dft_parts(int mode, int64_t n_vis, int64_t n_comp)
{
    if (mode == WT_MIXED || mode == WT_MIXED_FAST) return term_parts((n_vis + 511) / 512, n_comp, 2);
    return term_parts(mode == WT_MIXED_TC ? dft_tc_tiles(n_vis, n_comp) : (n_vis + 127) / 128, n_comp,
                      mode == WT_FP64_DF ? 8 : 4);
}
}  // namespace

int sum_parts(const void* partial, const TermParts& tp, int64_t n_vis, void* vis, bool c128, cudaStream_t s)
{
    const unsigned blocks = static_cast<unsigned>((n_vis + 127) / 128);
    const int parts = static_cast<int>(tp.parts);
    const double2* x = static_cast<const double2*>(partial);
    if (c128) k_sum_parts<<<blocks, 128, 0, s>>>(x, parts, n_vis, static_cast<double2*>(vis));
    else k_sum_parts<<<blocks, 128, 0, s>>>(x, parts, n_vis, static_cast<float2*>(vis));
    WT_CUDA_TRY(cudaGetLastError());
    return WT_OK;
}

// Launch the DFT on component records already packed in `scratch`
// (n_comp records of 32 bytes, 256-byte aligned) with their coordinate
// bounds at `bound` (mixed forms); errors go to `status`. vis: the
// visibilities, or the parts' sums [tp.parts][n_vis], complex128 in every mode.
int dft_launch_packed(const void* scratch, const uint32_t* bound, int64_t n_comp, const TermParts& tp,
                      const double* uvw, int64_t n_vis, void* vis, int mode, int sign, int* status, cudaStream_t s)
{
    dim3 grid;
    if (mode == WT_FP64) {
        constexpr int NT = 128;
        const size_t smem = static_cast<size_t>(stager_bytes<CompD>(kChunk));
        auto k = tp.parts > 1 ? k_dft_fp64<NT, true> : k_dft_fp64<NT, false>;
        int rc = grid_for(k, NT, NT, smem, n_vis, grid);
        if (rc) return rc;
        grid.y = static_cast<unsigned>(tp.parts);
        k<<<grid, NT, smem, s>>>(static_cast<const CompD*>(scratch), n_comp, tp.per_part, uvw, n_vis,
                                 static_cast<double2*>(vis), static_cast<double>(sign), status);
    } else if (mode == WT_FP64_DF) {
        constexpr int NT = 64;
        const size_t smem = static_cast<size_t>(stager_bytes<CompF>(kChunkDirDF)) + kDfTableEntries * sizeof(float4);
        auto k = tp.parts > 1 ? k_dft_df<NT, true> : k_dft_df<NT, false>;
        int rc = grid_for(k, NT, 2 * NT, smem, n_vis, grid);
        if (rc) return rc;
        grid.y = static_cast<unsigned>(tp.parts);
        k<<<grid, NT, smem, s>>>(static_cast<const CompF*>(scratch), n_comp, tp.per_part, uvw, n_vis,
                                 static_cast<double2*>(vis), static_cast<double>(sign), status);
    } else {
        // the grid pass, then the exact pass over the tiles it left marked
        constexpr int NT = 256;
        const size_t smem = static_cast<size_t>(stager_bytes<CompF>(kChunk));
        const CompF* recs = static_cast<const CompF*>(scratch);
        auto both = [&](auto kg, auto ke, auto* out) {
            dim3 grid_e;
            int rc = grid_for(kg, NT, 2 * NT, smem, n_vis, grid);   // two visibilities per thread
            if (!rc) rc = grid_for(ke, NT, 2 * NT, smem, n_vis, grid_e);
            if (rc) return rc;
            grid.y = grid_e.y = static_cast<unsigned>(tp.parts);
            kg<<<grid, NT, smem, s>>>(recs, n_comp, tp.per_part, bound, uvw, n_vis, out, static_cast<float>(sign),
                                      status);
            WT_CUDA_TRY(cudaGetLastError());
            ke<<<exact_grid(grid_e), NT, smem, s>>>(recs, n_comp, tp.per_part, bound, uvw, n_vis, out,
                                                    static_cast<float>(sign), status);
            return static_cast<int>(WT_OK);
        };
        const bool fast = mode == WT_MIXED_FAST;
        auto* sums = static_cast<double2*>(vis);
        auto* out = static_cast<float2*>(vis);
        const int rc =
            tp.parts > 1 ? fast ? both(k_dft_mixed<NT, true, true, true>, k_dft_mixed<NT, true, false, true>, sums)
                                : both(k_dft_mixed<NT, false, true, true>, k_dft_mixed<NT, false, false, true>, sums)
            : fast ? both(k_dft_mixed<NT, true, true, false>, k_dft_mixed<NT, true, false, false>, out)
                   : both(k_dft_mixed<NT, false, true, false>, k_dft_mixed<NT, false, false, false>, out);
        if (rc) return rc;
    }
    WT_CUDA_TRY(cudaGetLastError());
    return WT_OK;
}

// The exact pass of the mixed fast direct sum over 128-visibility tiles
// (64 threads, two visibilities each): only the tiles whose first
// visibility carries kDeferredMark are evaluated (the tensor-core form's
// tiles beyond its range). vis: as dft_launch_packed.
int dft_exact_pass_128(const void* recs, const uint32_t* bound, int64_t n_comp, const TermParts& tp, const double* uvw,
                       int64_t n_vis, void* vis, int sign, int* status, cudaStream_t s)
{
    constexpr int NT = 64;
    const size_t smem = static_cast<size_t>(stager_bytes<CompF>(kChunk));
    auto exact = [&](auto ke, auto* out) {
        dim3 grid;
        const int rc = grid_for(ke, NT, 2 * NT, smem, n_vis, grid);
        if (rc) return rc;
        grid.y = static_cast<unsigned>(tp.parts);
        ke<<<exact_grid(grid), NT, smem, s>>>(static_cast<const CompF*>(recs), n_comp, tp.per_part, bound, uvw, n_vis,
                                              out, static_cast<float>(sign), status);
        return static_cast<int>(WT_OK);
    };
    const int rc = tp.parts > 1 ? exact(k_dft_mixed<NT, true, false, true>, static_cast<double2*>(vis))
                                : exact(k_dft_mixed<NT, true, false, false>, static_cast<float2*>(vis));
    if (rc) return rc;
    WT_CUDA_TRY(cudaGetLastError());
    return WT_OK;
}

// Pack the components into `scratch` and, for the float forms, zero and
// reduce their coordinate bounds at `bound` (16 bytes, 16-byte aligned).
int dft_pack(const double* l, const double* m, const double* flux, int64_t n_comp, void* scratch, uint32_t* bound,
             int mode, int* status, cudaStream_t s)
{
    const bool f64 = mode == WT_FP64;
    if (!f64) WT_CUDA_TRY(cudaMemsetAsync(bound, 0, 4 * sizeof(uint32_t), s));
    if (n_comp == 0) return WT_OK;
    const int tb = 256;
    k_pack_components<<<static_cast<unsigned>((n_comp + tb - 1) / tb), tb, 0, s>>>(
        l, m, flux, n_comp, f64 ? static_cast<CompD*>(scratch) : nullptr, f64 ? nullptr : static_cast<CompF*>(scratch),
        f64 ? nullptr : bound, status);
    WT_CUDA_TRY(cudaGetLastError());
    return WT_OK;
}

int predict_dft(const double* l, const double* m, const double* flux, int64_t n_comp, const double* uvw,
                int64_t n_vis, void* vis, int mode, int sign, cudaStream_t s)
{
    if (n_vis == 0) return WT_OK;
    // 32-byte records (a 16-byte multiple, as the bulk copies need), then
    // the 16-byte block of coordinate bounds; the tensor-core form's slices
    // after them; then the parts' sums, where the terms are cut
    const bool tc = mode == WT_MIXED_TC;
    const bool c128 = mode == WT_FP64 || mode == WT_FP64_DF;
    TermParts tp = dft_parts(mode, n_vis, n_comp);
    const size_t rec_bytes = ((static_cast<size_t>(n_comp > 0 ? n_comp : 1) * 32 + 255) / 256) * 256;
    const size_t tc_bytes = tc ? (dft_tc_scratch_bytes(n_comp) + 255) / 256 * 256 : 0;
    const size_t base_bytes = rec_bytes + 256 + tc_bytes;
    const size_t part_bytes =
        tp.parts > 1 ? static_cast<size_t>(tp.parts) * static_cast<size_t>(n_vis) * sizeof(double2) : 0;
    void* scratch = nullptr;
    cudaError_t e = cudaMallocAsync(&scratch, base_bytes + part_bytes, s);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return set_error(WT_ERR_NOMEM, "dft_predict_vis: scratch allocation of %zu bytes failed: %s",
                         base_bytes + part_bytes, cudaGetErrorString(e));
    }
    uint32_t* bound = reinterpret_cast<uint32_t*>(static_cast<unsigned char*>(scratch) + rec_bytes);
    void* out = tp.parts > 1 ? static_cast<void*>(static_cast<unsigned char*>(scratch) + base_bytes) : vis;
    int* status = device_status_word();
    if (!status) {
        cudaFreeAsync(scratch, s);
        return set_error(WT_ERR_CUDA, "dft_predict_vis: no device status word");
    }
    int rc = dft_pack(l, m, flux, n_comp, scratch, bound, tc ? WT_MIXED_FAST : mode, status, s);
    if (rc == WT_OK) {
        if (tc)
            rc = dft_tc_launch(l, m, flux, n_comp, scratch, bound, static_cast<unsigned char*>(scratch) + rec_bytes + 256,
                               tp, uvw, n_vis, out, sign, status, s);
        else
            rc = dft_launch_packed(scratch, bound, n_comp, tp, uvw, n_vis, out, mode, sign, status, s);
    }
    if (rc == WT_OK && tp.parts > 1) rc = sum_parts(out, tp, n_vis, vis, c128, s);
    cudaError_t ef = cudaFreeAsync(scratch, s);
    if (rc != WT_OK) return rc;
    if (ef != cudaSuccess) return cuda_error(ef, "cudaFreeAsync");
    return WT_OK;
}

}  // namespace wt

#include <mutex>

// ===========================================================================
// dft_predict_vis_noalloc -- the direct sum without any device allocation.
//
// For callers that must not allocate device memory once they are running:
// an application that reserves its whole device-memory budget up front and
// forbids allocation in its steady state (an allocation there could fail, or
// stall behind the allocator's synchronisation), or a host framework that
// owns every device allocation itself. dft_predict_vis allocates a scratch
// buffer for the packed component records on each call; this variant packs
// them instead into the fixed array below, which lives in the library's
// device image. The paper has no counterpart: it is plumbing, not method.
//
// Every GPU that loads the library holds the array (2 MiB) until the
// process exits. All calls on a device share it and it keeps the previous
// call's records, so two calls whose work overlaps on the GPU (different
// streams, no ordering between them) race on it and give wrong results.
// Nothing in it has to start at zero: each call overwrites the records it
// reads.
// ===========================================================================
namespace wt {
namespace {

constexpr int64_t kNoAllocMaxComponents = 65536;   // 32-byte records: 2 MiB
static_assert(sizeof(CompD) == 32 && sizeof(CompF) == 32, "record size assumed below");

static __device__ __align__(256) unsigned char g_noalloc_records[kNoAllocMaxComponents * 32];
// The records' coordinate bounds (the mixed forms' grid pass).
static __device__ __align__(16) uint32_t g_noalloc_bound[4];
// Where the kernels record errors when the caller passes no status word.
static __device__ int g_noalloc_status_sink;

std::mutex g_noalloc_mu;
void* g_noalloc_addr[64] = {nullptr};
uint32_t* g_noalloc_bnd[64] = {nullptr};
int* g_noalloc_sink[64] = {nullptr};
uint64_t g_noalloc_ctx[64] = {0};   // context ID the addresses belong to

// Device addresses of the three arrays above on the current device. The first
// call on a device looks them up (cudaGetSymbolAddress, with that device
// current), and so does the first call in a new context on it (after
// cudaDeviceReset, say: the module is loaded again and the arrays may move);
// in host code the names are only host-side stand-ins and must never be
// handed to a kernel.
int noalloc_addresses(void** records, uint32_t** bound, int** sink)
{
    int dev = 0;
    WT_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return set_error(WT_ERR_CUDA, "device ordinal %d out of range", dev);
    const uint64_t ctx = current_context_id();
    if (ctx == 0) return set_error(WT_ERR_CUDA, "dft_predict_vis_noalloc: no current CUDA context");
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_addr[dev] || g_noalloc_ctx[dev] != ctx) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_records);
        if (e != cudaSuccess) return cuda_error(e, "cudaGetSymbolAddress(g_noalloc_records)");
        void* q = nullptr;
        e = cudaGetSymbolAddress(&q, g_noalloc_status_sink);
        if (e != cudaSuccess) return cuda_error(e, "cudaGetSymbolAddress(g_noalloc_status_sink)");
        void* b = nullptr;
        e = cudaGetSymbolAddress(&b, g_noalloc_bound);
        if (e != cudaSuccess) return cuda_error(e, "cudaGetSymbolAddress(g_noalloc_bound)");
        if (!p || !q || !b) return set_error(WT_ERR_CUDA, "cudaGetSymbolAddress returned a null address");
        g_noalloc_addr[dev] = p;
        g_noalloc_bnd[dev] = static_cast<uint32_t*>(b);
        g_noalloc_sink[dev] = static_cast<int*>(q);
        g_noalloc_ctx[dev] = ctx;
    }
    *records = g_noalloc_addr[dev];
    *bound = g_noalloc_bnd[dev];
    *sink = g_noalloc_sink[dev];
    return WT_OK;
}

}  // namespace

}  // namespace wt

extern "C" int dft_predict_vis_noalloc(const double* l, const double* m, const double* flux, int64_t n_comp,
                                       const double* uvw, int64_t n_vis, void* vis_out, int mode, int sign,
                                       int* status, void* stream)
{
    using namespace wt;
    const char* fn = "dft_predict_vis_noalloc";
    if (n_comp < 0 || n_vis < 0) return set_error(WT_ERR_ARG, "%s: negative size", fn);
    if (n_comp > kNoAllocMaxComponents)
        return set_error(WT_ERR_RANGE, "%s: %lld components exceed the fixed capacity of %lld", fn,
                         static_cast<long long>(n_comp), static_cast<long long>(kNoAllocMaxComponents));
    if (sign != 1 && sign != -1) return set_error(WT_ERR_ARG, "%s: sign must be +1 or -1", fn);
    if (mode != WT_FP64 && mode != WT_FP64_DF && mode != WT_MIXED && mode != WT_MIXED_FAST)
        return set_error(WT_ERR_ARG, "%s: bad mode %d", fn, mode);
    const bool c128 = mode == WT_FP64 || mode == WT_FP64_DF;
    const size_t nb = static_cast<size_t>(n_comp) * 8;
    const size_t ob = static_cast<size_t>(n_vis) * (c128 ? 16 : 8);
    int rc;
    if ((rc = check_device_buffer(l, nb, fn, "l", 8)) || (rc = check_device_buffer(m, nb, fn, "m", 8)) ||
        (rc = check_device_buffer(flux, nb, fn, "flux", 8)) ||
        (rc = check_device_buffer(uvw, static_cast<size_t>(n_vis) * 24, fn, "uvw", 8)) ||
        (rc = check_device_buffer(vis_out, ob, fn, "vis_out", vis_align(mode))) ||
        (status && (rc = check_device_buffer(status, sizeof(int), fn, "status", 4))))
        return rc;
    void* records = nullptr;
    uint32_t* bound = nullptr;
    int* sink = nullptr;
    if ((rc = noalloc_addresses(&records, &bound, &sink))) return rc;
    if (!status) status = sink;
    if (n_vis == 0) return WT_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if ((rc = dft_pack(l, m, flux, n_comp, records, bound, mode, status, s))) return rc;
    // no workspace for parts: the terms are not cut
    return dft_launch_packed(records, bound, n_comp, TermParts{1, kNoAllocMaxComponents}, uvw, n_vis, vis_out, mode,
                             sign, status, s);
}

// ===========================================================================
// wt_selftest_context_reset -- the per-context caches across a context reset.
//
// One component of flux 3 at the phase centre (so that V = 3 exactly for
// every baseline in float64) through dft_predict_vis_noalloc with no status
// word (the library's sink) and a read of the device status word; then
// cudaDeviceReset, which ends this process's context on the device and with
// it every device allocation; then the same again in the new context, with
// buffers allocated afresh. Both rounds must give V = 3 + 0i and a clear
// status word, which they can only if the array addresses and the status
// word were looked up again for the new context.
// ===========================================================================
namespace wt {
namespace {

int noalloc_round(cudaStream_t s)
{
    // one allocation: l, m, flux at d[0..2], uvw at d[3..8], the two
    // complex128 outputs at d[10..13] (16-byte aligned, as the kernel's
    // stores need)
    const double l = 0.0, m = 0.0, flux = 3.0;
    const double uvw[6] = {1234.5, -987.25, 12.5, -3.0e4, 2.0e4, -150.0};
    double* d = nullptr;
    WT_CUDA_TRY(cudaMalloc(&d, sizeof(double) * 14));
    double out[4] = {0, 0, 0, 0};
    int rc = WT_OK;
    cudaError_t e = cudaMemcpy(d, &l, sizeof(double), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(d + 1, &m, sizeof(double), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(d + 2, &flux, sizeof(double), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(d + 3, uvw, sizeof(uvw), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) rc = cuda_error(e, "wt_selftest_context_reset: upload");
    if (rc == WT_OK)
        rc = dft_predict_vis_noalloc(d, d + 1, d + 2, 1, d + 3, 2, d + 10, WT_FP64, 1, nullptr, s);
    if (rc == WT_OK) {
        e = cudaMemcpyAsync(out, d + 10, sizeof(out), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) rc = cuda_error(e, "wt_selftest_context_reset: download");
    }
    cudaFree(d);
    if (rc != WT_OK) return rc;
    if (out[0] != 3.0 || out[1] != 0.0 || out[2] != 3.0 || out[3] != 0.0)
        return set_error(WT_ERR_CORRUPT, "wt_selftest_context_reset: V = (%g, %g), (%g, %g), expected (3, 0)", out[0],
                         out[1], out[2], out[3]);
    return wt_device_status(s);
}

}  // namespace
}  // namespace wt

extern "C" int wt_selftest_context_reset(void)
{
    using namespace wt;
    int rc = noalloc_round(nullptr);
    if (rc != WT_OK) return rc;
    WT_CUDA_TRY(cudaDeviceReset());
    return noalloc_round(nullptr);
}
