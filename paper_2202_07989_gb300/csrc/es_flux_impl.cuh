// Flux + divergence kernel of the semi-discrete scheme, one launch per direction k
// (Eqs. (semi_U), (semi_J)), with the SSP-RK3 stage update fused into the last
// direction; the per-node, per-pair and per-interface arithmetic is in es_flux_core.cuh.
//
// Tile: (S + 6) x WT nodes staged in shared memory (3 halo nodes per side along
// k), one thread per interface ((S + 1) x WT = 256), one thread per node in the
// load and store phases (coalesced along the contiguous dimension).
#pragma once

#include "es_flux_core.cuh"

namespace es {

template <int S, int WT>
struct Tile {
    static constexpr int NN = (S + 6) * WT;   // staged nodes (3 halo nodes per side)
    static constexpr int NI = (S + 1) * WT;   // interfaces
    static constexpr int NP = (3 * S + 6) * WT;   // distinct node pairs (j, j+m), m = 1..3
};
// The 3D FP64 tiles (S = WT = 0 here) get their extent with the launch: any S and WT <=
// FLUX_WT_MAX with (S + 1) WT <= 256, in arrays of the capacity of the widest.  The mixed form
// keeps its extents at compile time: with run-time ones its 3D launches took 3-5% longer
template <>
struct Tile<0, 0> {
    static constexpr int NN = FLUX_TPB + 5 * FLUX_WT_MAX;
    static constexpr int NI = FLUX_TPB;
    static constexpr int NP = 3 * FLUX_TPB + 3 * FLUX_WT_MAX;
};

// rows of the staging buffer: JU (n_c), J and the metric row of direction k (d + 1); a 2D
// stage's Md rows (metrics M + s dt Md) are read directly in phase 1 (staging them too cost
// the RK launch of the batched form a quarter of its speed)
template <int D, int NS>
__host__ __device__ constexpr int stage_rows() { return NS + 2 * D + 3; }

// whether tiles of this case stage the next tile's inputs (not in 3D, whose tiles run 4 CTAs per SM)
template <int D, int NS>
__host__ __device__ constexpr bool stages_inputs() { return D != 3; }

// byte offset of the staging buffer behind the compute-type arrays of a flux tile (16-byte aligned)
template <int D, int NS, typename R, int S, int WT>
__host__ __device__ constexpr size_t stage_offset()
{
    using Y = Lay<D, NS>;
    using TL = Tile<S, WT>;
    return (sizeof(double) * (TL::NI + TL::NN) +
            sizeof(R) * (Y::NF * TL::NN + Y::NC * TL::NP + (NS + 1) * TL::NI + Y::NC * TL::NI) + 15) / 16 * 16;
}

// asynchronous 8-byte global -> shared copies (cp.async), one group per tile
__device__ __forceinline__ void cp_async8(double* smem, const double* gmem)
{
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Issue the raw FP64 node inputs of tile `wi` into the staging buffer stg[stage_rows][NN]:
// JU and J of the node the boundary map of direction k reaches (nothing for an inflow
// ghost, whose state is a constant) and the metric row of direction k at the node.
template <int D, int NS, int S, int WT>
__device__ __forceinline__ void flux_stage(const FluxLaunch& L, int k, int wi, double* stg)
{
    using TL = Tile<S, WT>;
    constexpr int NC = NS + D + 1, NN = TL::NN;
    const int adim = k == 0 ? 1 : 0, bdim = k == 2 ? 1 : 2;
    const int2 it = L.work[wi];
    const Inst& I = L.insts[it.x];
    const double* JU = L.ptrs ? L.ptrs[it.x].JU : L.single.JU;
    const double* J = L.ptrs ? L.ptrs[it.x].J : L.single.J;
    const double* M = L.ptrs ? L.ptrs[it.x].M : L.single.M;
    const int nk = I.n[k], na = I.n[adim];
    const int ns = (nk + S - 1) / S, nat = (na + WT - 1) / WT;
    const int s0 = (it.y % ns) * S, a0 = ((it.y / ns) % nat) * WT, tb = it.y / (ns * nat);
    const long long ncell = I.ncell, np = I.npad;
    for (int t = threadIdx.x; t < NN; t += blockDim.x) {
        int s, w;
        if (k == 0) { s = t % (S + 6); w = t / (S + 6); }
        else { w = t % WT; s = t / WT; }
        const int node = w * (S + 6) + s;
        const int g = s0 - 3 + s, a = a0 + w;
        if (a >= na || g > nk + 2) continue;
        int idx[3] = { 0, 0, 0 };
        idx[k] = g;
        idx[adim] = a;
        if (bdim < D) idx[bdim] = tb;
        int gi, side;
        if (map_line(I, k, g, gi, side) != 2) {
            int src[3] = { idx[0], idx[1], idx[2] };
            src[k] = gi;
            const long long id = lin(I, src[0], src[1], src[2]);
#pragma unroll
            for (int q = 0; q < NC; ++q) cp_async8(stg + q * NN + node, JU + q * ncell + id);
            cp_async8(stg + NC * NN + node, J + id);
        }
        const long long pid = plin(I, idx[0], idx[1], idx[2]);
#pragma unroll
        for (int c = 0; c <= D; ++c) cp_async8(stg + (NC + 1 + c) * NN + node, M + (long long)(k * (D + 1) + c) * np + pid);
    }
    cp_async_commit();
}

// t / n for 0 <= t < 2^21 and any n >= 1, given r = 1/n in binary32: (t + 1/2) r, with two roundings of
// 2^-24, is off (t + 1/2) / n by less than 1 / (4n), and that lies at least 1 / (2n) from an integer,
// so its integer part is t / n.  (The FP64 3D tiles divide by up to 3 * 255 + 6 = 771.)
__device__ __forceinline__ int div_small(int t, float r) { return (int)(((float)t + 0.5f) * r); }

// Phases of one tile: (1) node states, entropy variables and metrics into shared memory;
// (2) every distinct two-point flux F(U_j, U_{j+m}) (m = 1, 2, 3) of the tile, once; (3)
// per interface the 2w-order EC flux as sum_m alpha_m sum_s of the stored pairs, the GCL
// flux of J xi_k/t and the ES dissipation; (4) divergence and output / RK stage.
// FP32 tiles: 3 CTAs per SM in 2D (<= 85 registers), 4 in 3D (<= 64 registers: the compact 3D
// node layout and no staging buffer leave room for 4, measured 3-10% faster than 3 with the
// staging buffer, spills included); FP64 tiles: 1 (FP64-pipe bound)
template <int D, int NS, typename R, int S_, int WT_, int WK>
__global__ void __launch_bounds__(FLUX_TPB, (sizeof(R) == 4 ? (D == 3 ? 4 : 3) : 1)) flux_kernel(FluxLaunch L)
{
    pdl_entry();
    using Y = Lay<D, NS>;
    using TL = Tile<S_, WT_>;
    constexpr int NC = Y::NC, NN = TL::NN, NI = TL::NI, NF = Y::NF, NP = TL::NP;
    constexpr bool PRIM = D == 3 && std::is_same<R, float>::value;
    static_assert(NP < (1 << 21) && NN < (1 << 21), "div_small");
    const int S = S_ > 0 ? S_ : L.S, WT = S_ > 0 ? WT_ : L.WT, NPL = 3 * S + 6;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double* gt = reinterpret_cast<double*>(smem_raw);           // [NI] GCL flux of J xi_k/t
    double* mt64 = gt + NI;                                      // [NN] J xi_k/t at the nodes
    R* nr = reinterpret_cast<R*>(mt64 + NN);                     // [NF][NN] node data
    R* pf = nr + NF * NN;                                        // [NC][NP] pair fluxes
    R* cm = pf + NC * NP;                                        // [NS + 1][NI] centre-pair means
    R* fl = cm + (NS + 1) * NI;                                  // [NC][NI] interface fluxes
    double* stg = reinterpret_cast<double*>(smem_raw + stage_offset<D, NS, R, S_, WT_>());   // [NC + D + 2][NN]
    const int k = L.k;
    const int adim = k == 0 ? 1 : 0, bdim = k == 2 ? 1 : 2;

    // When a CTA has several tiles, their node inputs go through the staging buffer: the
    // first tile's now, each later tile's once the previous tile's phase 1 has consumed the
    // buffer, so their loads overlap phases 2-4.  With one tile per CTA there is nothing to
    // overlap, and phase 1 loads directly.
    const bool staged = stages_inputs<D, NS>() && L.nwork > (int)gridDim.x;
    if constexpr (stages_inputs<D, NS>())
        if (staged && blockIdx.x < L.nwork) flux_stage<D, NS, S_, WT_>(L, k, blockIdx.x, stg);
    for (int wi = blockIdx.x; wi < L.nwork; wi += gridDim.x) {
        const int2 it = L.work[wi];
        const Inst& I = L.insts[it.x];
        const StagePtrs P = L.ptrs ? L.ptrs[it.x] : L.single;
        const int nk = I.n[k], na = I.n[adim];
        const int ns = (nk + S - 1) / S, nat = (na + WT - 1) / WT;
        const int ts = it.y % ns, ta = (it.y / ns) % nat, tb = it.y / (ns * nat);
        const int s0 = ts * S, a0 = ta * WT;
        const long long ncell = I.ncell;
        // the tile's own extent: its items are numbered over the nodes it has, so that the last,
        // partial tile of a line or of the plane costs what it holds
        const int sE = min(S, nk - s0), wE = min(WT, na - a0);
        const float rN = 1.0f / (float)(sE + 6), rW = 1.0f / (float)wE, rP = 1.0f / (float)(3 * sE + 6),
                    rI = 1.0f / (float)(sE + 1), rS = 1.0f / (float)sE;
        // 2D stage metrics M + s Md with s = mcoef dt (the stage mesh is x^n + s xdot)
        const double sM = (D == 2 && L.mcoef != 0.0) ? L.mcoef * *P.dt : 0.0;

        // ---------------- phase 1: node states, entropy variables, metrics ----------------
        if (staged) {
            cp_async_wait_all();
            __syncthreads();
        }
        for (int t = threadIdx.x; t < (sE + 6) * wE; t += blockDim.x) {
            int s, w;
            if (k == 0) { w = div_small(t, rN); s = t - w * (sE + 6); }
            else { s = div_small(t, rW); w = t - s * wE; }
            const int node = w * (S + 6) + s;
            const int g = s0 - 3 + s, a = a0 + w;
            int idx[3] = { 0, 0, 0 };
            idx[k] = g;
            idx[adim] = a;
            if (bdim < D) idx[bdim] = tb;
            // the node's fields, from the conserved point state of the staged or loaded JU, J; the
            // boundary map of direction k negates the normal momentum (reflect) or gives the fixed
            // state (inflow).  The 3D mixed form reads the fields that prim3d_kernel formed
            const long long pid = plin(I, idx[0], idx[1], idx[2]);
            {
                int gi, side;
                const int tmap = map_line(I, k, g, gi, side);
                R U[MAXC];
                if (tmap == 2) {
                    for (int q = 0; q < NC; ++q) U[q] = to_r<R>(I.inflow[k][side][q]);
                    node_fields<D, NS, R>(I, U, nr, NN, node, L.status);
                } else {
                    int src[3] = { idx[0], idx[1], idx[2] };
                    src[k] = gi;
                    const long long id = staged ? 0 : lin(I, src[0], src[1], src[2]);
                    if constexpr (PRIM) {
                        float f[Y::MR];
#pragma unroll
                        for (int q = 0; q < Y::MR; ++q) f[q] = P.prim[q * ncell + id];
                        // a reflection negates the normal velocity and its entropy variable
#pragma unroll
                        for (int q = 0; q < D; ++q)
                            if (tmap == 1 && q == k) {
                                f[Y::V + q] = -f[Y::V + q];
                                f[Y::VV + NS + q] = -f[Y::VV + NS + q];
                            }
#pragma unroll
                        for (int q = 0; q < Y::MR; ++q) nr[q * NN + node] = f[q];
                    } else {
                    const R inv = Ar<R>::rcp(to_r<R>(staged ? stg[NC * NN + node] : P.J[id]));
#pragma unroll
                    for (int q = 0; q < NC; ++q) U[q] = mulr(to_r<R>(staged ? stg[q * NN + node] : P.JU[q * ncell + id]), inv);
                    if (tmap == 1) U[NS + k] = -U[NS + k];
                    node_fields<D, NS, R>(I, U, nr, NN, node, L.status);
                    }
                }
            }
            // metrics of direction k at this node from the metrics kernel (padded buffer covering
            // g in [-3, n + 3))
            {
                const long long mrow = (long long)(k * (D + 1)) * I.npad + pid;
                double mv[D + 1];
#pragma unroll
                for (int c = 0; c <= D; ++c) mv[c] = staged ? stg[(NC + 1 + c) * NN + node] : P.M[mrow + c * I.npad];
                if (D == 2 && sM != 0.0) {
#pragma unroll
                    for (int c = 0; c <= D; ++c)
                        mv[c] = fma(sM, P.Md[mrow + c * I.npad], mv[c]);
                }
                mt64[node] = mv[0];
                nr[Y::MR * NN + node] = to_r<R>(mv[0]);
#pragma unroll
                for (int j = 0; j < D; ++j) nr[(Y::MR + 1 + j) * NN + node] = to_r<R>(mv[1 + j]);
            }
        }
        __syncthreads();
        if constexpr (stages_inputs<D, NS>())
            if (staged && wi + (int)gridDim.x < L.nwork) flux_stage<D, NS, S_, WT_>(L, k, wi + (int)gridDim.x, stg);

        // ---------------- phase 2: distinct two-point EC fluxes ----------------
        for (int t = threadIdx.x; t < (3 * sE + 6) * wE; t += blockDim.x) {
            const int w = div_small(t, rP), r_ = t - w * (3 * sE + 6);
            // the pair's kind m, its left node Ln and its place among the line's NPL pairs
            int m, Ln, pl;
            if (r_ < sE + 1) { m = 1; Ln = r_ + 2; pl = r_; }
            else if (r_ < 2 * sE + 3) { m = 2; Ln = r_ - (sE + 1) + 1; pl = r_ - sE + S; }
            else { m = 3; Ln = r_ - (2 * sE + 3); pl = r_ - 2 * sE + 2 * S; }
            const int l = w * (S + 6) + Ln;
            pair_flux<D, NS, R>(I, nr, NN, Y::MR, l, l + m, pf, NP, w * NPL + pl, cm, NI, m == 1 ? w * (S + 1) + (Ln - 2) : -1);
        }
        __syncthreads();

        // ---------------- phase 3: interface fluxes ----------------
        for (int t = threadIdx.x; t < (sE + 1) * wE; t += blockDim.x) {
            const int w = div_small(t, rI), s = t - w * (sE + 1);     // interface s0 - 1 + s + 1/2
            const int f = w * (S + 1) + s;
            const int base = w * (S + 6) + s;   // node gi - 2
            const int p1 = w * NPL + s, p2 = w * NPL + (S + 1) + s, p3 = w * NPL + (2 * S + 3) + s;
            iface_flux<D, NS, R, WK>(I, nr + base, NN, 1, Y::MR, mt64 + base, 1, pf, NP, p1, p2, p3, 1, cm, NI, f, fl, gt);
        }
        __syncthreads();

        // ---------------- phase 4: divergence and output ----------------
        const double dt = L.mode == MODE_RK ? *P.dt : 0.0;
        for (int t = threadIdx.x; t < sE * wE; t += blockDim.x) {
            int s, w;
            if (k == 0) { w = div_small(t, rS); s = t - w * sE; }
            else { s = div_small(t, rW); w = t - s * wE; }
            const int g = s0 + s, a = a0 + w;
            int idx[3] = { 0, 0, 0 };
            idx[k] = g;
            idx[adim] = a;
            if (bdim < D) idx[bdim] = tb;
            const long long id = lin(I, idx[0], idx[1], idx[2]);
            const int fr = w * (S + 1) + s + 1, fL = fr - 1;
            double r[NC + 1];
            node_div<NC, R>(I, fl, NI, gt, fr, fL, k, r);
            if (L.mode == MODE_WRITE) {
#pragma unroll
                for (int q = 0; q < NC; ++q) P.accU[q * ncell + id] = r[q];
                P.accJ[id] = r[NC];
            } else if (L.mode == MODE_ACC) {
#pragma unroll
                for (int q = 0; q < NC; ++q) P.accU[q * ncell + id] += r[q];
                P.accJ[id] += r[NC];
            } else {
#pragma unroll
                for (int q = 0; q < NC; ++q)
                    P.JUo[q * ncell + id] = rk_stage(L, P.JU[q * ncell + id], P.JU0 + q * ncell + id, dt, P.accU[q * ncell + id] + r[q]);
                P.Jo[id] = rk_stage(L, P.J[id], P.J0 + id, dt, P.accJ[id] + r[NC]);
                if (P.xo) {    // null on a fixed mesh; xdot is constant over the step: x^n + xc dt xdot
                    const double cdt = L.xc * dt;
#pragma unroll
                    for (int j = 0; j < D; ++j) P.xo[j * ncell + id] = fma(cdt, P.xdot[j * ncell + id], P.x0[j * ncell + id]);
                }
            }
        }
        __syncthreads();
    }
}

template <int D, int NS, typename R, int S, int WT>
static size_t smem_of()
{
    return stage_offset<D, NS, R, S, WT>() + (stages_inputs<D, NS>() ? sizeof(double) * stage_rows<D, NS>() * Tile<S, WT>::NN : 0);
}

// one case per tile shape of the table in es_kernels.cuh; 3D FP64: the run-time extent
#define ES_FLUX_SHAPES(X) X(0) X(1) X(2) X(3) X(4) X(5)
static_assert(NSHAPE == 6, "ES_FLUX_SHAPES lists every tile shape");

template <int D, typename R>
__host__ __device__ constexpr bool fits_tiles() { return D == 3 && std::is_same<R, double>::value; }

template <int D, int NS, typename R, int S, int WT, int WK>
static void prepare_shape()
{
    cudaFuncSetAttribute(flux_kernel<D, NS, R, S, WT, WK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)smem_of<D, NS, R, S, WT>());
}

template <int D, int NS, typename R, int WK>
void prepare_flux()
{
    if constexpr (fits_tiles<D, R>()) {
        prepare_shape<D, NS, R, 0, 0, WK>();
    } else {
#define ES_PREP(SH) prepare_shape<D, NS, R, SHAPE_S[SH], SHAPE_WT[SH], WK>();
        ES_FLUX_SHAPES(ES_PREP)
#undef ES_PREP
    }
}

template <int D, int NS, typename R, int S, int WT, int WK>
static int shape_blocks()
{
    int nb = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, flux_kernel<D, NS, R, S, WT, WK>, FLUX_TPB, smem_of<D, NS, R, S, WT>());
    return nb > 0 ? nb : 1;
}

template <int D, int NS, typename R, int WK>
int flux_blocks_per_sm(int shape)
{
    if constexpr (fits_tiles<D, R>()) {
        (void)shape;
        return shape_blocks<D, NS, R, 0, 0, WK>();
    } else {
#define ES_OCC(SH) if (shape == SH) return shape_blocks<D, NS, R, SHAPE_S[SH], SHAPE_WT[SH], WK>();
        ES_FLUX_SHAPES(ES_OCC)
#undef ES_OCC
        return 1;
    }
}

template <int D, int NS, typename R, int S, int WT, int WK>
static void launch_shape(const FluxLaunch& L, int grid, cudaStream_t st)
{
    // the staging buffer only when a CTA has several tiles (the kernel's own test)
    const bool staged = stages_inputs<D, NS>() && L.nwork > grid;
    pdl_launch(flux_kernel<D, NS, R, S, WT, WK>, grid, FLUX_TPB,
               staged ? smem_of<D, NS, R, S, WT>() : stage_offset<D, NS, R, S, WT>(), st, L);
}

template <int D, int NS, typename R, int WK>
void launch_flux(const FluxLaunch& L, int shape, int grid, cudaStream_t st)
{
    if constexpr (fits_tiles<D, R>()) {
        (void)shape;
        launch_shape<D, NS, R, 0, 0, WK>(L, grid, st);
    } else {
#define ES_LAUNCH(SH) if (shape == SH) launch_shape<D, NS, R, SHAPE_S[SH], SHAPE_WT[SH], WK>(L, grid, st);
        ES_FLUX_SHAPES(ES_LAUNCH)
#undef ES_LAUNCH
    }
}

// explicit instantiation of one (dimension, species, reconstruction) case in both compute types
#define ES_FLUX_INSTANTIATE(D, NS, WK)                                                        \
    template void prepare_flux<D, NS, double, WK>();                                          \
    template void prepare_flux<D, NS, float, WK>();                                           \
    template int flux_blocks_per_sm<D, NS, double, WK>(int);                                  \
    template int flux_blocks_per_sm<D, NS, float, WK>(int);                                   \
    template void launch_flux<D, NS, double, WK>(const FluxLaunch&, int, int, cudaStream_t);  \
    template void launch_flux<D, NS, float, WK>(const FluxLaunch&, int, int, cudaStream_t);

}  // namespace es
