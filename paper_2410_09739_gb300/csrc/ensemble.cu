// ensemble.cu -- many independent periodic boxes of uneven sizes and
// viscosities advanced by ONE persistent launch per time step.
//
// Every box keeps its own SoA population block (27 slot rows of stride_b
// elements, AA pattern, see cell.cuh).  The cells of all boxes are cut into
// tiles of `block` cells (a box's last tile is ragged); tile t belongs to box
// tile_box[t].  A persistent grid of SMs x resident-blocks strides over the
// tile list; each tile runs the same per-cell update as a single box, with
// the box's own geometry and shear rate 1/tau_b.  Boxes never exchange data.
#include <cstring>
#include <type_traits>
#include <vector>

#include "rtalloc.h"
#include "cell.cuh"
#include "handle.h"

namespace fpc {

template <typename R>
__device__ __forceinline__ R both(float v)
{
    if constexpr (std::is_same<R, f2>::value) return f2(v, v);
    else return v;
}

// One shear rate for all five of a box (the same values as Rates::keep and Rates::unit of a single
// box with that rate, so both advance a box bit for bit alike when both run one cell per thread or both two).
template <int FORCE, int MODE, typename R>
__device__ __forceinline__ Shear<R> box_shear(const EnsBox& B)
{
    if constexpr (scaled_shear(FORCE, MODE)) {
        const R k4 = both<R>(__ldg(&B.keep4)), k6 = both<R>(__ldg(&B.keep6));
        return {k4, k4, k4, k6, k6};
    } else {
        const R k = both<R>(__ldg(&B.keep));
        return {k, k, k, k, k};
    }
}

template <bool ODD, int FORCE, int MODE, int MINB>
__global__ void __launch_bounds__(256, MINB) k_ens_step(const EnsArgs a)
{
    float* __restrict__ base = static_cast<float*>(a.buf);
    chain_wait();
    for (unsigned t = blockIdx.x; t < a.ntiles; t += gridDim.x) {
        const unsigned b = __ldg(a.tile_box + t);
        const EnsBox& B = a.boxes[b];
        const unsigned first = (t - __ldg(&B.tile0)) * a.tile_cells;
        const unsigned ncells = __ldg(&B.ncells);
        CellGeom G;
        G.stride = __ldg(&B.stride);
        G.nx = __ldg(&B.nx);
        G.ny = __ldg(&B.ny);
        G.nz = __ldg(&B.nz);
        G.div_nx.d = __ldg(&B.div_nx.d);
        G.div_nx.m = __ldg(&B.div_nx.m);
        G.div_nx.s = __ldg(&B.div_nx.s);
        G.div_nxny.d = __ldg(&B.div_nxny.d);
        G.div_nxny.m = __ldg(&B.div_nxny.m);
        G.div_nxny.s = __ldg(&B.div_nxny.s);
        const Shear<float> sh = box_shear<FORCE, MODE, float>(B);
        float* buf = base + __ldg(&B.off);
        for (unsigned c = threadIdx.x; c < a.tile_cells; c += blockDim.x) {
            const unsigned cell = first + c;
            if (cell >= ncells) break;
            update_cell<float, float, ODD, BC_PERIODIC, FORCE, MODE>(buf, G, cell, a.rates, a.Fx, a.Fy, a.Fz,
                                                               sh, nullptr, a.flag);
        }
    }
}

// Paired variant (pair.cuh): neighbouring cells 2t, 2t + 1 of a tile share a
// thread (one vector access per slot where the pair's values are adjacent; see
// update_pair_even and update_pair_odd_adj), except on the odd step of a box
// with odd nx, where cells t and t + tile/2 do.
template <bool ODD, int FORCE, int MODE, int MINB>
__global__ void __launch_bounds__(128, MINB) k_ens_pair(const EnsArgs a)
{
    float* __restrict__ base = static_cast<float*>(a.buf);
    const unsigned half = a.tile_cells / 2;
    chain_wait();
    for (unsigned t = blockIdx.x; t < a.ntiles; t += gridDim.x) {
        const unsigned b = __ldg(a.tile_box + t);
        const EnsBox& B = a.boxes[b];
        const unsigned first = (t - __ldg(&B.tile0)) * a.tile_cells;
        const unsigned ncells = __ldg(&B.ncells);
        CellGeom G;
        G.stride = __ldg(&B.stride);
        G.nx = __ldg(&B.nx);
        G.ny = __ldg(&B.ny);
        G.nz = __ldg(&B.nz);
        G.div_nx.d = __ldg(&B.div_nx.d);
        G.div_nx.m = __ldg(&B.div_nx.m);
        G.div_nx.s = __ldg(&B.div_nx.s);
        G.div_nxny.d = __ldg(&B.div_nxny.d);
        G.div_nxny.m = __ldg(&B.div_nxny.m);
        G.div_nxny.s = __ldg(&B.div_nxny.s);
        const Shear<f2> sh = box_shear<FORCE, MODE, f2>(B);
        float* buf = base + __ldg(&B.off);
        for (unsigned c = threadIdx.x; c < half; c += blockDim.x) {
            if (ODD && (G.nx & 1) == 0) {  // even nx: neighbouring cells, shared neighbour table
                if (first + 2 * c >= ncells) break;
                update_pair_odd_adj<float, BC_PERIODIC, FORCE, MODE>(buf, G, first / 2 + c, a.rates2, a.Fx2, a.Fy2,
                                                                     a.Fz2, sh, a.flag);
            } else if (ODD) {
                const unsigned c1 = first + c;
                if (c1 >= ncells) break;
                update_pair<float, ODD, BC_PERIODIC, FORCE, MODE>(buf, G, c1, half, ncells, a.rates2, a.Fx2, a.Fy2,
                                                                  a.Fz2, sh, a.flag);
            } else {  // neighbouring cells first + 2c, first + 2c + 1 (tiles and box blocks are even-aligned)
                if (first + 2 * c >= ncells) break;
                update_pair_even<float, BC_PERIODIC, FORCE, MODE>(buf, G, first / 2 + c, ncells, a.rates2, a.Fx2,
                                                                  a.Fy2, a.Fz2, sh, a.flag);
            }
        }
    }
}

// Resident blocks of 128 threads per SM of the even-step paired kernel with a given cap.
template <int FORCE, int MODE, int MINB>
static int occ_even_pair()
{
    static int n = 0;  // benign race: every thread computes the same value
    if (n == 0) {
        int v = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, k_ens_pair<false, FORCE, MODE, MINB>, 128, 0) !=
                cudaSuccess ||
            v < 1) {
            cudaGetLastError();
            v = 1;
        }
        n = v;
    }
    return n;
}

template <bool ODD, int FORCE, int MODE>
static cudaError_t go(const EnsArgs& a, int block, int minb, int grid, int variant, cudaStream_t st)
{
    if (variant == 2) {
        if (block != 128 || a.tile_cells % (2 * block) != 0) return cudaErrorInvalidValue;
        if constexpr (!ODD && !FORCE && r1_mode(MODE)) {
            // the unit-rate even step without force (vector accesses, no neighbour table, no source
            // terms) fits 5 blocks per SM without spilling;
            // the persistent grid, sized by the tuner for the capped kernel, is scaled to match
            const int o = minb == 3 ? occ_even_pair<FORCE, MODE, 3>() : occ_even_pair<FORCE, MODE, 4>();
            const long long g5 = (long long)grid * occ_even_pair<FORCE, MODE, 5>() / o;
            return launch_chained(k_ens_pair<false, FORCE, MODE, 5>, (unsigned)(g5 > 0 ? g5 : 1), (unsigned)block, 0, st, a);
        }
        return launch_chained(minb == 3 ? k_ens_pair<ODD, FORCE, MODE, 3> : k_ens_pair<ODD, FORCE, MODE, 4>,
                              (unsigned)grid, (unsigned)block, 0, st, a);
    }
    return launch_chained(minb == 3 ? k_ens_step<ODD, FORCE, MODE, 3> : k_ens_step<ODD, FORCE, MODE, 2>, (unsigned)grid,
                          (unsigned)block, 0, st, a);
}

template <int MODE>
static cudaError_t go_mode(int odd, int force, const EnsArgs& a, int block, int minb, int grid, int variant,
                           cudaStream_t st)
{
#define FPC_ENS_GO(O, F) go<O, F, MODE>(a, block, minb, grid, variant, st)
    if constexpr (r1_mode(MODE)) {
        if (force == FORCE_X) return odd ? FPC_ENS_GO(true, FORCE_X) : FPC_ENS_GO(false, FORCE_X);
    }
    if (odd) return force ? FPC_ENS_GO(true, FORCE_ANY) : FPC_ENS_GO(true, FORCE_NONE);
    return force ? FPC_ENS_GO(false, FORCE_ANY) : FPC_ENS_GO(false, FORCE_NONE);
#undef FPC_ENS_GO
}

cudaError_t launch_ens_step(int odd, int force, int mode, const EnsArgs& a, int block, int minb, int grid,
                            int variant, cudaStream_t st)
{
    if (grid <= 0 || block <= 0 || block > 256 || a.tile_cells % block != 0) return cudaErrorInvalidValue;
    switch (mode) {
        case MODE_FP: return go_mode<MODE_FP>(odd, force, a, block, minb, grid, variant, st);
        case MODE_EQ: return go_mode<MODE_EQ>(odd, force, a, block, minb, grid, variant, st);
        case MODE_FP_R1: return go_mode<MODE_FP_R1>(odd, force, a, block, minb, grid, variant, st);
        case MODE_EQ_R1: return go_mode<MODE_EQ_R1>(odd, force, a, block, minb, grid, variant, st);
    }
    return cudaErrorInvalidValue;
}

// Resident blocks per SM of the even-step kernel of the variant that launch_ens_step runs.
template <int MODE>
static int ens_occupancy(int block, int minb, int variant)
{
    int n = 0;
    cudaError_t e;
    if (variant == 2)
        e = minb == 3 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_ens_pair<false, FORCE_NONE, MODE, 3>, block, 0)
                      : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_ens_pair<false, FORCE_NONE, MODE, 4>, block, 0);
    else
        e = minb == 3 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_ens_step<false, FORCE_NONE, MODE, 3>, block, 0)
                      : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_ens_step<false, FORCE_NONE, MODE, 2>, block, 0);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return n > 0 ? n : 1;
}

int ens_max_blocks_per_sm(int block, int minb, int mode, int variant)
{
    switch (mode) {
        case MODE_EQ: return ens_occupancy<MODE_EQ>(block, minb, variant);
        case MODE_FP_R1: return ens_occupancy<MODE_FP_R1>(block, minb, variant);
        case MODE_EQ_R1: return ens_occupancy<MODE_EQ_R1>(block, minb, variant);
    }
    return ens_occupancy<MODE_FP>(block, minb, variant);
}

}  // namespace fpc

using namespace fpc;

extern "C" int fpclbm_create_ensemble(fpclbm_t* out, int n_boxes, const int* dims, const double* tau, int precision,
                                      void* cuda_stream)
{
    g_create_error.clear();
    if (!out) {
        g_create_error = "out is NULL";
        return FPCLBM_ERR_ARG;
    }
    *out = nullptr;
    if (n_boxes < 1 || !dims || !tau) {
        g_create_error = "need n_boxes >= 1, dims and tau";
        return FPCLBM_ERR_ARG;
    }
    if (precision != FPCLBM_FP32) {
        g_create_error = "ensembles support FPCLBM_FP32 only";
        return FPCLBM_ERR_ARG;
    }
    fpclbm* h = new (std::nothrow) fpclbm();
    if (!h) {
        g_create_error = "host allocation failed";
        return FPCLBM_ERR_ALLOC;
    }
    h->ensemble = true;
    h->precision = precision;
    h->bc = FPCLBM_BC_PERIODIC;
    h->stream = static_cast<cudaStream_t>(cuda_stream);
    rates_from_params(1.0, 0.0, h->omega);
    unsigned long long off = 0, cells = 0;
    const int tile = 256;  // cells per tile = the largest block size the tuner may pick
    unsigned tiles = 0;
    for (int b = 0; b < n_boxes; ++b) {
        const int nx = dims[3 * b], ny = dims[3 * b + 1], nz = dims[3 * b + 2];
        if (nx < 1 || ny < 1 || nz < 1) {
            g_create_error = "box dimensions must be >= 1";
            delete h;
            return FPCLBM_ERR_ARG;
        }
        const double w = 1.0 / tau[b];
        if (!(w > 0.0 && w < 2.0)) {
            g_create_error = "box " + std::to_string(b) + ": 1/tau outside (0, 2)";
            delete h;
            return FPCLBM_ERR_PARAM;
        }
        Box bx;
        bx.nx = nx;
        bx.ny = ny;
        bx.nz = nz;
        const unsigned long long n = (unsigned long long)nx * ny * nz;
        bx.ncells = (unsigned)n;
        bx.stride = (unsigned)((n + 63) / 64 * 64);
        bx.off = off;
        bx.cell0 = (unsigned)cells;
        bx.tau = tau[b];
        bx.tile0 = tiles;
        bx.ntiles = (unsigned)((n + tile - 1) / tile);
        off += 27ull * bx.stride;
        cells += n;
        tiles += bx.ntiles;
        if (n >= (1ull << 31) || 27ull * bx.stride >= (1ull << 32) || cells >= (1ull << 32)) {
            g_create_error = "ensemble too large";
            delete h;
            return FPCLBM_ERR_ARG;
        }
        h->boxes.push_back(bx);
    }
    h->total_cells = cells;
    h->ntiles = tiles;
    h->tile_cells = tile;
    int rc = alloc_common(h);
    cudaError_t e = cudaSuccess;
    if (rc == FPCLBM_OK) {
        e = rt_malloc(&h->d_pop, off * elem_size(precision));
        if (e == cudaSuccess) e = rt_malloc(&h->d_ens_boxes, sizeof(EnsBox) * n_boxes);
        if (e == cudaSuccess) e = rt_malloc(&h->d_tile_box, sizeof(unsigned) * tiles);
        if (e == cudaSuccess) {
            std::vector<EnsBox> tab(n_boxes);
            std::vector<unsigned> tb(tiles);
            for (int b = 0; b < n_boxes; ++b) {
                const Box& bx = h->boxes[b];
                EnsBox& E = tab[b];
                std::memset(&E, 0, sizeof E);
                E.off = bx.off;
                E.stride = bx.stride;
                E.ncells = bx.ncells;
                E.nx = bx.nx;
                E.ny = bx.ny;
                E.nz = bx.nz;
                E.div_nx = make_fastdiv((unsigned)bx.nx);
                E.div_nxny = make_fastdiv((unsigned)(bx.nx * bx.ny));
                const double keep = 1.0 - 1.0 / bx.tau;
                E.keep = (float)keep;
                E.keep4 = (float)(keep / 4);
                E.keep6 = (float)(keep / 6);
                E.tile0 = bx.tile0;
                E.cell0 = bx.cell0;
                for (unsigned t = 0; t < bx.ntiles; ++t) tb[bx.tile0 + t] = (unsigned)b;
            }
            e = cudaMemcpyAsync(h->d_ens_boxes, tab.data(), sizeof(EnsBox) * n_boxes, cudaMemcpyHostToDevice,
                                h->stream);
            if (e == cudaSuccess)
                e = cudaMemcpyAsync(h->d_tile_box, tb.data(), sizeof(unsigned) * tiles, cudaMemcpyHostToDevice,
                                    h->stream);
            if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
        }
        if (e != cudaSuccess) {
            g_create_error = std::string("CUDA: ") + cudaGetErrorString(e);
            rc = e == cudaErrorMemoryAllocation ? FPCLBM_ERR_ALLOC : FPCLBM_ERR_CUDA;
        }
    }
    if (rc != FPCLBM_OK) {
        fpclbm_destroy(h);
        return rc;
    }
    h->block = tile;
    h->minb = 2;
    h->grid = h->sm_count * ens_max_blocks_per_sm(tile, 2, MODE_FP, 0);
    *out = h;
    return FPCLBM_OK;
}
