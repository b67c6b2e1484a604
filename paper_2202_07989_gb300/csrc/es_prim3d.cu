// Node fields of the 3D mixed form, once per node and stage: species densities, velocity and
// entropy variables (phase 1 of the flux kernels, es_flux_core.cuh) from the stage input, in
// binary32, field-major on the grid's nodes.  The three per-direction flux launches of a stage
// read them instead of forming them again from the FP64 state.
#include "es_flux_core.cuh"

namespace es {

// Why: a node's fields take about 400 instructions, two or three logarithms, four reciprocals and
// six to seven FP64 -> FP32 conversions among them, and the tiles of the three directions formed
// them 1.2 times each; here they cost one pass of 84 to 100 bytes per node.  Steps: Riemann 128^3
// 6074 -> 5856 us, 3D shock-bubble 128 x 64 x 64 2083 -> 1989, Example 5.11 400 x 80 x 80 4917 -> 4523.
template <int NS>
__global__ void __launch_bounds__(NODE_TPB) prim3d_kernel(const Inst* __restrict__ insts, StagePtrs single,
                                                           const StagePtrs* __restrict__ table,
                                                           const int2* __restrict__ work, int nwork, int* status)
{
    pdl_entry();
    using Y = Lay<3, NS>;
    constexpr int NP = prim_fields<NS>();
    static_assert(Y::COMPACT && Y::MR == NP, "the fields before the metrics");
    for (int wi = blockIdx.x; wi < nwork; wi += gridDim.x) {
        const int2 it = work[wi];
        const Inst& I = insts[it.x];
        ES_PTRS(P);
        int i0, i1, i2;
        if (!tile_node(I, it.y, 0, i0, i1, i2)) continue;
        const long long id = lin(I, i0, i1, i2), n = I.ncell;
        float U[MAXC], f[NP];
        const float inv = Ar<float>::rcp(f64_to_f32(P.J[id]));
#pragma unroll
        for (int q = 0; q < Y::NC; ++q) U[q] = __fmul_rn(f64_to_f32(P.JU[q * n + id]), inv);    // rounded: not fused into the sums below
        node_fields<3, NS, float>(I, U, f, 1, 0, status);
#pragma unroll
        for (int q = 0; q < NP; ++q) P.prim[q * n + id] = f[q];
    }
}

void launch_prim3d(int N, int grid, cudaStream_t st, const Inst* insts, const StagePtrs& single, const StagePtrs* table,
                   const int2* work, int nwork, int* status)
{
    if (N == 1) pdl_launch(prim3d_kernel<1>, grid, NODE_TPB, 0, st, insts, single, table, work, nwork, status);
    else pdl_launch(prim3d_kernel<2>, grid, NODE_TPB, 0, st, insts, single, table, work, nwork, status);
}

}  // namespace es
