// closure_train.cu -- training data and training kernels of the learned closure.
//
// The learned closure (no counterpart in the paper, whose channel flow uses a
// Smagorinsky LES) is a per-cell MLP 9 -> 64 -> 64 -> 1 that corrects the shear
// relaxation rate of a coarse-grid FPC-LBM (inference: closure.cuh).
//
// fpclbm_closure_sample: box filter of a fine run onto r^3 blocks, features
//   and labels per block (definitions in include/fpclbm.h).
// fpclbm_closure_train:  Adam on the mean squared error, mini-batches, bf16
//   weights in the forward and backward kernels, fp32 accumulation and
//   gradients, fp64 loss accumulation, fp32 master weights.
// fpclbm_closure_grad:   one loss/gradient evaluation, for checking.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <string>
#include <vector>

#include "rtalloc.h"
#include "aux.cuh"
#include "closure.cuh"
#include "field_math.cuh"
#include "handle.h"

namespace fpc {
namespace {

constexpr double kCs2 = 1.0 / 3.0;

// ---------------------------------------------------------------------------
// Training data: filter, strain rate, eddy viscosity, labels
// ---------------------------------------------------------------------------

struct FilterArgs {
    BoxGeom b;
    int parity, r;
    int cx, cy, cz;  // coarse dimensions
    int group;       // coarse cells per block: as many as have columns for the block's threads, at least 1
    int has_force;   // any of the force is not zero
    double Fx, Fy, Fz;
    double* acc;     // [10][Nc]: rho, ux, uy, uz, uxx, uyy, uzz, uxy, uxz, uyz
};

// Density and half-force velocity of a cell for the filter: fp64 storage in fp64; fp32 and 16-bit
// storage from compensated fp32 sums (aux.cuh), as k_moments does.
template <typename S>
__device__ __forceinline__ void filter_fields(const FilterArgs& a, unsigned cell, double& r, double& u, double& v,
                                              double& w)
{
    if constexpr (!std::is_same<S, double>::value) {
        float g[27];
        load_cell<S>(a.b, a.parity, cell, g);
        float ds = 0.f, dc = 0.f, xs = 0.f, xc = 0.f, ys = 0.f, yc = 0.f, zs = 0.f, zc = 0.f;
#pragma unroll
        for (int s = 0; s < 27; ++s) {
            const int ex = s % 3 - 1, ey = (s / 3) % 3 - 1, ez = s / 9 - 1;
            sum2_add(ds, dc, g[s]);
            if (ex != 0) sum2_add(xs, xc, ex > 0 ? g[s] : -g[s]);
            if (ey != 0) sum2_add(ys, yc, ey > 0 ? g[s] : -g[s]);
            if (ez != 0) sum2_add(zs, zc, ez > 0 ? g[s] : -g[s]);
        }
        // sums that left fp32 (infinite, NaN or far beyond a density) take the fp64 form
        if (fabsf(ds) + fabsf(xs) + fabsf(ys) + fabsf(zs) < 1e30f) {
            r = 1.0 + (widen(ds) + widen(dc));
            const double inv = 1.0 / r;
            u = widen(xs) + widen(xc);
            v = widen(ys) + widen(yc);
            w = widen(zs) + widen(zc);
            if (a.has_force) {
                u += 0.5 * a.Fx;
                v += 0.5 * a.Fy;
                w += 0.5 * a.Fz;
            }
            u *= inv;
            v *= inv;
            w *= inv;
            return;
        }
    }
    double g[27];
    load_cell<S>(a.b, a.parity, cell, g);
    fields_of(g, a.Fx, a.Fy, a.Fz, r, u, v, w);
}

// Box filter.  A block takes `group` consecutive coarse cells, over the ends of rows, a thread one column of
// fine cells along y and z, so a warp reads consecutive fine cells of each slot row; the columns of a
// coarse cell are then summed through shared memory.  (One thread per coarse cell, all in fp64, read
// every r-th cell and kept the fp64 pipe busy with about 180 operations per fine cell: 5.48 ms for 256^3
// fp32 cells, r = 4, against 0.91 ms.  Blocks that ended with the row left most threads idle in short rows; whole
// calls, fp32 / fp64 storage: 8x256x256, r = 2, 0.45 -> 0.17 / 1.30 -> 0.32 ms; 4x512x512, r = 4, 1.05 -> 0.09 /
// 4.33 -> 0.36; 96^3, r = 4, 0.12 -> 0.08 / 0.28.)
constexpr int kFilterThreads = 256;

template <typename S>
__global__ void __launch_bounds__(kFilterThreads) k_cl_filter(FilterArgs a)
{
    extern __shared__ double cl_sums[];  // [10][threads]
    const unsigned nc = (unsigned)a.cx * a.cy * a.cz, r = (unsigned)a.r, tid = threadIdx.x, nt = blockDim.x;
    const unsigned first = blockIdx.x * a.group, cells = min((unsigned)a.group, nc - first);
    double s[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (unsigned c = tid; c < cells * r; c += nt) {  // more than one column only if group == 1
        const unsigned lc = c / r, row = (first + lc) / a.cx, Z = row / a.cy;
        const unsigned x = (first + lc - row * a.cx) * r + (c - lc * r), y0 = (row - Z * a.cy) * r, z0 = Z * r;
        for (unsigned k = 0; k < r; ++k)
            for (unsigned j = 0; j < r; ++j) {
                double rho, u, v, w;
                filter_fields<S>(a, x + (unsigned)a.b.nx * (y0 + j + (unsigned)a.b.ny * (z0 + k)), rho, u, v, w);
                s[0] += rho;
                s[1] += u;
                s[2] += v;
                s[3] += w;
                s[4] += u * u;
                s[5] += v * v;
                s[6] += w * w;
                s[7] += u * v;
                s[8] += u * w;
                s[9] += v * w;
            }
    }
    for (int q = 0; q < 10; ++q) cl_sums[q * nt + tid] = s[q];
    __syncthreads();
    const unsigned per = min(r, nt);
    const double inv = 1.0 / ((double)a.r * a.r * a.r);
    for (unsigned i = tid; i < 10 * cells; i += nt) {
        const unsigned q = i / cells, c = i - q * cells;
        const double* p = cl_sums + q * nt + c * per;
        double t = p[0];
        for (unsigned m = 1; m < per; ++m) t += p[m];
        a.acc[(size_t)q * nc + first + c] = t * inv;
    }
}

// Strain rate of the filtered velocity (central differences in coarse cells,
// periodic in x and z, periodic in y or, at y walls, through the no-slip wall
// value), eddy viscosity from the sub-filter stress, label and features.
__global__ void k_cl_label(const double* __restrict__ acc, int cx, int cy, int cz, int walls, double tau_c,
                           float* X, float* T)
{
    const unsigned nc = (unsigned)cx * cy * cz;
    const unsigned c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nc) return;
    const int x = c % cx, y = (c / cx) % cy, z = c / (cx * cy);
    auto at = [&](int q, int xx, int yy, int zz) {
        return acc[(size_t)q * nc + (unsigned)(xx + cx * (yy + cy * zz))];
    };
    // d u_i / d x_j, i = 0..2 (u, v, w), j = 0..2 (x, y, z)
    double gr[3][3];
    for (int i = 0; i < 3; ++i) {
        const int q = 1 + i;
        gr[i][0] = 0.5 * (at(q, (x + 1) % cx, y, z) - at(q, (x - 1 + cx) % cx, y, z));
        gr[i][2] = 0.5 * (at(q, x, y, (z + 1) % cz) - at(q, x, y, (z - 1 + cz) % cz));
        // next to a no-slip wall (y = -1/2 or cy - 1/2) the derivative of the quadratic through the
        // wall value 0 and the two nearest rows
        if (!walls)
            gr[i][1] = 0.5 * (at(q, x, (y + 1) % cy, z) - at(q, x, (y - 1 + cy) % cy, z));
        else if (y == 0)
            gr[i][1] = at(q, x, 0, z) + at(q, x, 1, z) / 3.0;
        else if (y == cy - 1)
            gr[i][1] = -(at(q, x, cy - 1, z) + at(q, x, cy - 2, z) / 3.0);
        else
            gr[i][1] = 0.5 * (at(q, x, y + 1, z) - at(q, x, y - 1, z));
    }
    double S[3][3];
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) S[i][j] = 0.5 * (gr[i][j] + gr[j][i]);
    const double u[3] = {at(1, x, y, z), at(2, x, y, z), at(3, x, y, z)};
    const double rho = at(0, x, y, z);
    // <u_i u_j>: q = 4 uu, 5 vv, 6 ww, 7 uv, 8 uw, 9 vw
    const int uq[3][3] = {{4, 7, 8}, {7, 5, 9}, {8, 9, 6}};
    double tau[3][3];
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) tau[i][j] = at(uq[i][j], x, y, z) - u[i] * u[j];
    const double tr = (tau[0][0] + tau[1][1] + tau[2][2]) / 3.0;
    double num = 0, den = 0;
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) {
            const double td = tau[i][j] - (i == j ? tr : 0.0);
            num += td * S[i][j];
            den += S[i][j] * S[i][j];
        }
    double nut = den > 0 ? -num / (2.0 * den) : 0.0;
    if (!(nut > 0)) nut = 0.0;
    const double nu = kCs2 * (tau_c - 0.5);
    const double label = 1.0 / ((nu + nut) / kCs2 + 0.5) - 1.0 / (nu / kCs2 + 0.5);
    const double f = -2.0 * rho * kCs2 * tau_c;
    float* xo = X + (size_t)9 * c;
    xo[0] = (float)(f * S[0][0]);
    xo[1] = (float)(f * S[1][1]);
    xo[2] = (float)(f * S[2][2]);
    xo[3] = (float)(f * S[0][1]);
    xo[4] = (float)(f * S[0][2]);
    xo[5] = (float)(f * S[1][2]);
    xo[6] = (float)u[0];
    xo[7] = (float)u[1];
    xo[8] = (float)u[2];
    T[c] = (float)label;
}

// ---------------------------------------------------------------------------
// Network forward/backward on mini-batches
// ---------------------------------------------------------------------------

// Mini-batch forward and backward on the tensor cores.  A block takes a tile of kMB = 128 samples,
// 16 per warp.  Every contraction is an mma.sync.m16n8k16 bf16 x bf16 -> fp32 product:
//   forward   Z1 = [x, 1] [W1 | b1]^T (K = 16: 9 inputs, the bias input 1, zeros),
//             Z2 = H1 W2^T (K = 64), H = tanh(Z) in fp32, y = w3 . H2 + b3 in fp32;
//   backward  G2 = gy w3 (1 - H2^2), G1 = (G2 W2) (1 - H1^2)  (K = 64);
//   weights   dW2 = G2^T [H1, 1] and dW1 = G1^T [x, 1] over the tile's samples
//             (K = 128); the column of ones gives the bias gradients db2, db1;
//             dw3 = sum gy H2 and db3 = sum gy in fp32.
// The operands x, H1, G2, G1 are rounded to bf16 (the weights are bf16 already);
// products accumulate in fp32.  The fp32 accumulator fragments of one product
// are the A-operand fragments of the next (row g / g+8, columns 2t, 2t+1), so
// H1 and G2 stay in registers; for the weight gradients, whose K runs over the
// samples, H1, G2, G1 and x are also written to shared memory, sample-major, and read back as
// transposed fragments (ldmatrix.trans).  Row pitches spread eight rows over all banks.
//
// What bounds it is the chain of one tile (a batch of 1,024 samples is eight tiles on 152 SMs), so
// eight warps share a tile and nothing is transposed with scalar stores.  Four warps of two row
// tiles each, scalar transposes and 8-way bank conflicts took 17.2 us for it.
//
// Two kernels run the tiles:
//   k_cl_epoch  batches of up to kMaxCluster tiles: one cluster of blocks runs up to kEpochBatches
//               batches in a launch, a tile per block.  The gradients go straight into the shared memory of the
//               block that owns the parameter, which sums them in block order, applies Adam to its
//               fp32 master weights there and writes the new bf16 weight into every block's copy;
//               two cluster barriers per batch, no launch and no global memory but the samples
//               (10.1 us a batch of 1,024 against 20 us and a launch gap of two kernels);
//   k_cl_mma    larger batches and the gradient entry point: a block per tile writes its gradient
//               (4865 fp32) and its loss (fp64) to its own slot of a scratch array;
//               k_cl_reduce_adam / k_cl_reduce_grad sum the slots.
// Both sum the tiles in the same fixed order: training is deterministic and does not depend on
// which of the two runs.

constexpr int kMB = 128;          // samples per tile
constexpr int kTrainThreads = 256;
constexpr int kMaxCluster = 16;   // blocks of a cluster (above 8 they need the non-portable size)

struct NetArgs {
    const float* X;             // [n][9]
    const float* T;             // [n]
    unsigned long long n;       // samples in the data set
    unsigned long long first;   // first position of this batch in the epoch order
    unsigned long long count;   // samples in this batch
    unsigned long long perm_a, perm_c;  // epoch order: sample(i) = (a i + c) mod n
    float mu[10], inv_sd[10];   // standardisation of the 9 inputs and the target
    float scale;                // dL/dy factor 2 / batch
    const __nv_bfloat16* W;     // bf16 weights (closure layout)
    float* part;                // per-block gradients [blocks][4865]
    double* part_loss;          // per-block sums of squared errors [blocks]
};

struct __align__(16) TrainSmem {
    __nv_bfloat16 W1p[64][24];  // [j][i]: W1, then b1 in column 9, zeros to column 15
    __nv_bfloat16 W2s[64][72];  // W2[j][k]
    __nv_bfloat16 XS[kMB][24];  // [m][i] inputs of the tile's samples, 1 in column 9, zeros to column 15
    __nv_bfloat16 H1[kMB][88];  // [m][k], column 64 = 1, columns 65..71 = 0
    __nv_bfloat16 G2[kMB][72];  // [m][j]
    __nv_bfloat16 G1[kMB][72];  // [m][j]
    double carry_loss[4][32];
    double loss[4];
    float carry[4][32][17];     // dw3 and db3 of a pair's first row tile, per lane
    float b2[64], w3[64], tgt[kMB], vld[kMB], dw3[4][64];
    float b3, db3[4];
};

__device__ __forceinline__ uint32_t lds32(const __nv_bfloat16* p) { return *reinterpret_cast<const uint32_t*>(p); }
__device__ __forceinline__ void sts32(__nv_bfloat16* p, uint32_t v) { *reinterpret_cast<uint32_t*>(p) = v; }

// Four 8x8 bf16 matrices, transposed: lane l gives the row address of matrix l / 8, row l % 8, and
// receives of each matrix the elements (row 2t, col g) and (row 2t + 1, col g).
__device__ __forceinline__ void ldsm_x4_trans(uint32_t (&r)[4], const __nv_bfloat16* p)
{
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(a)
                 : "memory");
}

// Weight p of the closure layout into the tile's copy of the weights.
__device__ __forceinline__ __nv_bfloat16* weight_slot(TrainSmem& S, int p)
{
    if (p < CL_B1) return &S.W1p[p / 9][p % 9];
    if (p < CL_W2) return &S.W1p[p - CL_B1][9];
    return &S.W2s[(p - CL_W2) >> 6][(p - CL_W2) & 63];  // p < CL_B2
}
__device__ __forceinline__ float* weight_slot_f(TrainSmem& S, int p)
{
    return p < CL_W3 ? &S.b2[p - CL_B2] : p < CL_B3 ? &S.w3[p - CL_W3] : &S.b3;
}

// Constant parts of the tables and the weights (closure layout) into shared memory.
__device__ __forceinline__ void train_setup(TrainSmem& S, const __nv_bfloat16* W)
{
    const int tid = threadIdx.x;
    const __nv_bfloat16 zero = __float2bfloat16_rn(0.f), one = __float2bfloat16_rn(1.f);
    for (int i = tid; i < 64 * 8; i += kTrainThreads) S.W1p[i >> 3][8 + (i & 7)] = zero;
    for (int i = tid; i < kMB * 8; i += kTrainThreads) S.H1[i >> 3][64 + (i & 7)] = (i & 7) ? zero : one;
    __syncthreads();
    for (int p = tid; p < CL_N; p += kTrainThreads) {
        if (p < CL_B2) *weight_slot(S, p) = W[p];
        else *weight_slot_f(S, p) = __bfloat162float(W[p]);
    }
}

// One sample, standardised.
struct Sample {
    float x[9], t;
    bool valid;
};

__device__ __forceinline__ Sample load_sample(const NetArgs& a, unsigned long long pos, unsigned long long end)
{
    Sample s;
    s.valid = pos < end;
    s.t = 0.f;
#pragma unroll
    for (int i = 0; i < 9; ++i) s.x[i] = 0.f;
    if (s.valid) {
        const unsigned long long idx = (a.perm_a * pos + a.perm_c) % a.n;
#pragma unroll
        for (int i = 0; i < 9; ++i) s.x[i] = (a.X[idx * 9 + i] - a.mu[i]) * a.inv_sd[i];
        s.t = (a.T[idx] - a.mu[9]) * a.inv_sd[9];
    }
    return s;
}

__device__ __forceinline__ void put_sample(TrainSmem& S, int m, const Sample& s)
{
#pragma unroll
    for (int i = 0; i < 8; i += 2) sts32(&S.XS[m][i], pack_bf16x2(s.x[i], s.x[i + 1]));
    sts32(&S.XS[m][8], pack_bf16x2(s.x[8], 1.f));
#pragma unroll
    for (int i = 10; i < 16; i += 2) sts32(&S.XS[m][i], 0u);
    S.tgt[m] = s.t;
    S.vld[m] = s.valid ? 1.f : 0.f;  // padding rows of a short batch: no error, no gradient
}

// Forward and backward of the tile in S (all threads of the block; the samples and weights are in
// place and synchronised).  put(p, v): gradient of parameter p; the loss goes to put_loss(v).
template <typename Put, typename PutLoss>
__device__ __forceinline__ void tile_gradient(TrainSmem& S, float scale, Put put, PutLoss put_loss)
{
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, g = lane >> 2, t = lane & 3;
    const int r0 = 16 * w + g, r1 = r0 + 8, pair = w >> 1;
    // rows of the transposed fragments' matrices: lanes 0-7 and 8-15 give the first eight rows of two
    // column blocks, lanes 16-31 the next eight (A operand); for the B operand of two n-tiles the
    // middle two are swapped
    const int arow = (lane & 7) + ((lane >> 4) << 3), acol = ((lane >> 3) & 1) << 3;
    const int brow = (lane & 7) + (((lane >> 3) & 1) << 3), bcol = (lane >> 4) << 3;

    // ---- layer 1: Z1 = [x, 1] [W1 | b1]^T, H1 = tanh(Z1)
    const uint32_t xa0 = lds32(&S.XS[r0][2 * t]), xa1 = lds32(&S.XS[r1][2 * t]);
    const uint32_t xa2 = lds32(&S.XS[r0][2 * t + 8]), xa3 = lds32(&S.XS[r1][2 * t + 8]);
    float h1[8][4];
    uint32_t A2[4][4];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
        float c[4] = {0.f, 0.f, 0.f, 0.f};
        mma_bf16_16816(c, xa0, xa1, xa2, xa3, lds32(&S.W1p[8 * nt + g][2 * t]), lds32(&S.W1p[8 * nt + g][2 * t + 8]));
#pragma unroll
        for (int q = 0; q < 4; ++q) h1[nt][q] = tanhf(c[q]);
        const uint32_t lo = pack_bf16x2(h1[nt][0], h1[nt][1]), hi = pack_bf16x2(h1[nt][2], h1[nt][3]);
        A2[nt >> 1][(nt & 1) * 2] = lo;
        A2[nt >> 1][(nt & 1) * 2 + 1] = hi;
        sts32(&S.H1[r0][8 * nt + 2 * t], lo);
        sts32(&S.H1[r1][8 * nt + 2 * t], hi);
        // the backward pass needs 1 - H1^2 of the bf16 operand's source value
#pragma unroll
        for (int q = 0; q < 4; ++q) h1[nt][q] = 1.f - h1[nt][q] * h1[nt][q];
    }
    // ---- layer 2 and output: Z2 = H1 W2^T + b2, H2 = tanh(Z2), y = w3 . H2 + b3
    float h2[8][4];
    float y0 = 0.f, y1 = 0.f;
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
        float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int kt = 0; kt < 4; ++kt)
            mma_bf16_16816(c, A2[kt][0], A2[kt][1], A2[kt][2], A2[kt][3], lds32(&S.W2s[8 * nt + g][16 * kt + 2 * t]),
                           lds32(&S.W2s[8 * nt + g][16 * kt + 2 * t + 8]));
        const int c0 = 8 * nt + 2 * t;
        h2[nt][0] = tanhf(c[0] + S.b2[c0]);
        h2[nt][1] = tanhf(c[1] + S.b2[c0 + 1]);
        h2[nt][2] = tanhf(c[2] + S.b2[c0]);
        h2[nt][3] = tanhf(c[3] + S.b2[c0 + 1]);
        y0 = fmaf(S.w3[c0], h2[nt][0], fmaf(S.w3[c0 + 1], h2[nt][1], y0));
        y1 = fmaf(S.w3[c0], h2[nt][2], fmaf(S.w3[c0 + 1], h2[nt][3], y1));
    }
    y0 += __shfl_xor_sync(0xffffffffu, y0, 1);
    y0 += __shfl_xor_sync(0xffffffffu, y0, 2);
    y1 += __shfl_xor_sync(0xffffffffu, y1, 1);
    y1 += __shfl_xor_sync(0xffffffffu, y1, 2);
    const float e0 = S.vld[r0] * (y0 + S.b3 - S.tgt[r0]), e1 = S.vld[r1] * (y1 + S.b3 - S.tgt[r1]);
    const float gy0 = scale * e0, gy1 = scale * e1;
    // dw3, db3 and the loss of the row tiles 2 pair and 2 pair + 1 are one chain of additions: the
    // first warp of the pair hands its partial sums to the second through shared memory
    if (!(w & 1)) {
#pragma unroll
        for (int nt = 0; nt < 8; ++nt) {
            S.carry[pair][lane][2 * nt] = fmaf(gy0, h2[nt][0], fmaf(gy1, h2[nt][2], 0.f));
            S.carry[pair][lane][2 * nt + 1] = fmaf(gy0, h2[nt][1], fmaf(gy1, h2[nt][3], 0.f));
        }
        S.carry[pair][lane][16] = t == 0 ? gy0 + gy1 : 0.f;
        S.carry_loss[pair][lane] = t == 0 ? (double)e0 * e0 + (double)e1 * e1 : 0.0;
    }
    // ---- G2 = gy w3 (1 - H2^2): A operand of G2 W2 and sample-major copy for dW2
    uint32_t AG[4][4];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
        const int c0 = 8 * nt + 2 * t;
        const float wa = S.w3[c0], wb = S.w3[c0 + 1];
        const uint32_t lo = pack_bf16x2(gy0 * wa * (1.f - h2[nt][0] * h2[nt][0]), gy0 * wb * (1.f - h2[nt][1] * h2[nt][1]));
        const uint32_t hi = pack_bf16x2(gy1 * wa * (1.f - h2[nt][2] * h2[nt][2]), gy1 * wb * (1.f - h2[nt][3] * h2[nt][3]));
        AG[nt >> 1][(nt & 1) * 2] = lo;
        AG[nt >> 1][(nt & 1) * 2 + 1] = hi;
        sts32(&S.G2[r0][c0], lo);
        sts32(&S.G2[r1][c0], hi);
    }
    // ---- G1 = (G2 W2) (1 - H1^2), sample-major copy for dW1; B fragments W2[j][k], K = j, of the
    // n-tiles nt and nt + 1
#pragma unroll
    for (int nt = 0; nt < 8; nt += 2) {
        float c[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
        for (int kt = 0; kt < 4; ++kt) {
            uint32_t b[4];
            ldsm_x4_trans(b, &S.W2s[16 * kt + brow][8 * nt + bcol]);
            mma_bf16_16816(c[0], AG[kt][0], AG[kt][1], AG[kt][2], AG[kt][3], b[0], b[1]);
            mma_bf16_16816(c[1], AG[kt][0], AG[kt][1], AG[kt][2], AG[kt][3], b[2], b[3]);
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int c0 = 8 * (nt + q) + 2 * t;
            sts32(&S.G1[r0][c0], pack_bf16x2(c[q][0] * h1[nt + q][0], c[q][1] * h1[nt + q][1]));
            sts32(&S.G1[r1][c0], pack_bf16x2(c[q][2] * h1[nt + q][2], c[q][3] * h1[nt + q][3]));
        }
    }
    __syncthreads();
    if (w & 1) {  // warp sums of dw3 (over the rows, lane bits 2..4), db3 and the loss
#pragma unroll
        for (int nt = 0; nt < 8; ++nt)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                float v = fmaf(gy0, h2[nt][q], fmaf(gy1, h2[nt][2 + q], S.carry[pair][lane][2 * nt + q]));
                v += __shfl_xor_sync(0xffffffffu, v, 4);
                v += __shfl_xor_sync(0xffffffffu, v, 8);
                v += __shfl_xor_sync(0xffffffffu, v, 16);
                if (g == 0) S.dw3[pair][8 * nt + 2 * t + q] = v;
            }
        float db3a = S.carry[pair][lane][16];
        double lossa = S.carry_loss[pair][lane];
        if (t == 0) {
            db3a += gy0 + gy1;
            lossa += (double)e0 * e0 + (double)e1 * e1;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            db3a += __shfl_xor_sync(0xffffffffu, db3a, o);
            lossa += __shfl_xor_sync(0xffffffffu, lossa, o);
        }
        if (lane == 0) {
            S.db3[pair] = db3a;
            S.loss[pair] = lossa;
        }
    }

    // ---- weight gradients over the tile's samples: warps w and w + 4 own rows j = 16 (w % 4) ..;
    // the first takes the n-tiles 0..3 and 8 (the column of ones: db2) of dW2, the second 4..7 and dW1
    const int jb = 16 * (w & 3), j0 = jb + g, j1 = j0 + 8;
    const bool second = w >= 4;
    uint32_t A[kMB / 16][4];
#pragma unroll
    for (int kt = 0; kt < kMB / 16; ++kt) ldsm_x4_trans(A[kt], &S.G2[16 * kt + arow][jb + acol]);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int nt = (second ? 4 : 0) + 2 * q;
        float c[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
        for (int kt = 0; kt < kMB / 16; ++kt) {
            uint32_t b[4];
            ldsm_x4_trans(b, &S.H1[16 * kt + brow][8 * nt + bcol]);
            mma_bf16_16816(c[0], A[kt][0], A[kt][1], A[kt][2], A[kt][3], b[0], b[1]);
            mma_bf16_16816(c[1], A[kt][0], A[kt][1], A[kt][2], A[kt][3], b[2], b[3]);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int k0 = 8 * (nt + i) + 2 * t;
            put(CL_W2 + 64 * j0 + k0, c[i][0]);
            put(CL_W2 + 64 * j0 + k0 + 1, c[i][1]);
            put(CL_W2 + 64 * j1 + k0, c[i][2]);
            put(CL_W2 + 64 * j1 + k0 + 1, c[i][3]);
        }
    }
    if (!second) {
        float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int kt = 0; kt < kMB / 16; ++kt) {
            uint32_t b[4];  // columns 64..71 (the last two matrices repeat the first two)
            ldsm_x4_trans(b, &S.H1[16 * kt + brow][64]);
            mma_bf16_16816(c, A[kt][0], A[kt][1], A[kt][2], A[kt][3], b[0], b[1]);
        }
        if (t == 0) {
            put(CL_B2 + j0, c[0]);
            put(CL_B2 + j1, c[2]);
        }
    } else {
        float c[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
        for (int kt = 0; kt < kMB / 16; ++kt) {  // dW1 (i = 0..8) and db1 (i = 9)
            uint32_t a[4], b[4];
            ldsm_x4_trans(a, &S.G1[16 * kt + arow][jb + acol]);
            ldsm_x4_trans(b, &S.XS[16 * kt + brow][bcol]);
            mma_bf16_16816(c[0], a[0], a[1], a[2], a[3], b[0], b[1]);
            mma_bf16_16816(c[1], a[0], a[1], a[2], a[3], b[2], b[3]);
        }
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const int i = 8 * nt + 2 * t + q;
                if (i < 9) {
                    put(CL_W1 + 9 * j0 + i, c[nt][q]);
                    put(CL_W1 + 9 * j1 + i, c[nt][2 + q]);
                } else if (i == 9) {
                    put(CL_B1 + j0, c[nt][q]);
                    put(CL_B1 + j1, c[nt][2 + q]);
                }
            }
    }
    __syncthreads();
    if (tid < 64) put(CL_W3 + tid, (S.dw3[0][tid] + S.dw3[1][tid]) + (S.dw3[2][tid] + S.dw3[3][tid]));
    if (tid == 64) put(CL_B3, (S.db3[0] + S.db3[1]) + (S.db3[2] + S.db3[3]));
    if (tid == 65) put_loss((S.loss[0] + S.loss[1]) + (S.loss[2] + S.loss[3]));
}

__global__ void __launch_bounds__(kTrainThreads) k_cl_mma(NetArgs a)
{
    extern __shared__ __align__(16) unsigned char cl_smem[];
    TrainSmem& S = *reinterpret_cast<TrainSmem*>(cl_smem);
    const int tid = threadIdx.x;
    Sample s;
    if (tid < kMB) s = load_sample(a, a.first + (unsigned long long)blockIdx.x * kMB + tid, a.first + a.count);
    train_setup(S, a.W);
    if (tid < kMB) put_sample(S, tid, s);
    __syncthreads();
    float* part = a.part + (size_t)blockIdx.x * CL_N;
    tile_gradient(S, a.scale, [&](int p, float v) { part[p] = v; }, [&](double v) { a.part_loss[blockIdx.x] = v; });
}

// Adam (Kingma & Ba 2015) of one parameter: the new master weight; m and v in place.
__device__ __forceinline__ float adam(float w, float& m, float& v, float g, float lr, float b1, float b2, float c1,
                                      float c2, float eps)
{
    const float mm = b1 * m + (1.f - b1) * g;
    const float vv = b2 * v + (1.f - b2) * g * g;
    m = mm;
    v = vv;
    return w - lr * (mm * c1) / (sqrtf(vv * c2) + eps);
}

// Up to kEpochBatches consecutive batches of an epoch on one cluster (gridDim.x = cluster size = tiles
// of a full batch, at most kMaxCluster).  Adam's bias corrections come as kernel arguments, as
// k_cl_reduce_adam's do: they are exact host values, and no host buffer has to outlive the launch.
// 256 of them keep the arguments under 4 KB, and a launch under a few milliseconds whatever the
// number of batches (2.6 ms for 256 batches of 1,024 samples).
constexpr int kEpochBatches = 256;

struct EpochArgs {
    NetArgs net;              // X, T, n, epoch order, standardisation, W (bf16 weights before the first batch)
    long long batch, first;   // samples per batch, first batch of this launch
    int batches;              // batches of this launch, at most kEpochBatches
    float lr, b1, b2, eps;
    float *w, *m, *v;         // fp32 master weights and moments, in place
    __nv_bfloat16* wb;        // bf16 weights, out
    double* loss;             // sum of squared errors of the epoch, continued
    FastDiv chunk;            // parameters owned by a block
    float2 corr[kEpochBatches];  // Adam's bias corrections (c1, c2) of every batch
};
static_assert(sizeof(EpochArgs) <= 4096, "kernel arguments");

// Shared memory behind the tile's tables: received gradients [tiles][chunk], received losses, the
// owned parameters' master weights and moments.
__host__ __device__ constexpr size_t epoch_smem(int blocks, int chunk)
{
    return sizeof(TrainSmem) + sizeof(double) * kMaxCluster + sizeof(float) * (size_t)chunk * (blocks + 3);
}

__device__ __forceinline__ uint32_t cluster_addr(const void* p, unsigned rank)
{
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n"
                 : "=r"(a)
                 : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ void cluster_st(uint32_t a, float v)
{
    asm volatile("st.shared::cluster.f32 [%0], %1;\n" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void cluster_st(uint32_t a, double v)
{
    asm volatile("st.shared::cluster.f64 [%0], %1;\n" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_st(uint32_t a, unsigned short v)
{
    asm volatile("st.shared::cluster.u16 [%0], %1;\n" ::"r"(a), "h"(v) : "memory");
}
// All threads of the cluster; writes to any block's shared memory before it are visible after it.
__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;\n" ::: "memory");
}

__global__ void __launch_bounds__(kTrainThreads) k_cl_epoch(const __grid_constant__ EpochArgs a)
{
    extern __shared__ __align__(16) unsigned char cl_smem[];
    TrainSmem& S = *reinterpret_cast<TrainSmem*>(cl_smem);
    const int tid = threadIdx.x;
    const unsigned rank = blockIdx.x, nb = gridDim.x, chunk = a.chunk.d;
    double* recv_loss = reinterpret_cast<double*>(cl_smem + sizeof(TrainSmem));
    float* recv = reinterpret_cast<float*>(recv_loss + kMaxCluster);  // [tile][chunk]
    float *mw = recv + (size_t)nb * chunk, *mm = mw + chunk, *mv = mm + chunk;
    const int p0 = (int)(rank * chunk), owned = max(0, min((int)chunk, CL_N - p0));
    for (int i = tid; i < owned; i += kTrainThreads) {
        mw[i] = a.w[p0 + i];
        mm[i] = a.m[p0 + i];
        mv[i] = a.v[p0 + i];
    }
    train_setup(S, a.net.W);
    const unsigned long long n = a.net.n;
    auto fetch = [&](int it) {
        const unsigned long long first = (unsigned long long)((a.first + it) * a.batch);
        const unsigned long long end = min(first + (unsigned long long)a.batch, n);
        return load_sample(a.net, it < a.batches ? first + (unsigned long long)rank * kMB + tid : end, end);
    };
    Sample s;
    if (tid < kMB) s = fetch(0);
    // one chain of additions over the batches of an epoch, whatever launches it takes
    const bool sums_loss = rank == 0 && tid == kTrainThreads - 1;
    double loss = sums_loss ? *a.loss : 0.0;
    cluster_barrier();  // every block's tables are in place before another one writes to them
    for (int it = 0; it < a.batches; ++it) {
        const long long first = (a.first + it) * a.batch;
        const long long count = min((long long)n - first, a.batch);
        const unsigned tiles = (unsigned)((count + kMB - 1) / kMB);
        if (rank < tiles) {
            if (tid < kMB) put_sample(S, tid, s);
            __syncthreads();
        }
        if (tid < kMB) s = fetch(it + 1);  // in flight during this batch
        if (rank < tiles)
            tile_gradient(
                S, 2.0f / (float)count,
                [&](int p, float v) {
                    const unsigned o = fdiv((unsigned)p, a.chunk);
                    cluster_st(cluster_addr(recv + (size_t)rank * chunk + ((unsigned)p - o * chunk), o), v);
                },
                [&](double v) { cluster_st(cluster_addr(recv_loss + rank, 0), v); });
        cluster_barrier();  // the gradients have arrived at their owners
        const float2 corr = a.corr[it];
        for (int i = tid; i < owned; i += kTrainThreads) {
            float g = 0.f;
            for (unsigned b = 0; b < tiles; ++b) g += recv[(size_t)b * chunk + i];
            const float wn = adam(mw[i], mm[i], mv[i], g, a.lr, a.b1, a.b2, corr.x, corr.y, a.eps);
            mw[i] = wn;
            const __nv_bfloat16 wb = __float2bfloat16_rn(wn);
            const int p = p0 + i;
            if (p < CL_B2) {
                const __nv_bfloat16* at = weight_slot(S, p);
                for (unsigned b = 0; b < nb; ++b) cluster_st(cluster_addr(at, b), __bfloat16_as_ushort(wb));
            } else {
                const float* at = weight_slot_f(S, p);
                for (unsigned b = 0; b < nb; ++b) cluster_st(cluster_addr(at, b), __bfloat162float(wb));
            }
        }
        if (sums_loss) {
            double l = 0.0;
            for (unsigned b = 0; b < tiles; ++b) l += recv_loss[b];
            loss += l;
        }
        cluster_barrier();  // the new weights have arrived, the received gradients are used up
    }
    for (int i = tid; i < owned; i += kTrainThreads) {
        a.w[p0 + i] = mw[i];
        a.m[p0 + i] = mm[i];
        a.v[p0 + i] = mv[i];
        a.wb[p0 + i] = __float2bfloat16_rn(mw[i]);
    }
    if (sums_loss) *a.loss = loss;
}

// Second stage: sum of the block gradients in block order; the loss (fp64) is added to *loss.
__device__ __forceinline__ float sum_blocks(const float* part, int blocks, int p)
{
    float s = 0.f;
    for (int b = 0; b < blocks; ++b) s += part[(size_t)b * CL_N + p];
    return s;
}

__global__ void k_cl_reduce_grad(const float* part, const double* part_loss, int blocks, float* grad, double* loss)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < CL_N) grad[p] = sum_blocks(part, blocks, p);
    if (p == 0) {
        double l = 0.0;
        for (int b = 0; b < blocks; ++b) l += part_loss[b];
        *loss += l;
    }
}

// Adam on fp32 master weights; the gradient is the sum of the block partials.
__global__ void k_cl_reduce_adam(float* w, float* m, float* v, const float* part, const double* part_loss, int blocks,
                                 double* loss, __nv_bfloat16* wb, float lr, float b1, float b2, float c1, float c2,
                                 float eps)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p == 0) {
        double l = 0.0;
        for (int b = 0; b < blocks; ++b) l += part_loss[b];
        *loss += l;
    }
    if (p >= CL_N) return;
    const float wn = adam(w[p], m[p], v[p], sum_blocks(part, blocks, p), lr, b1, b2, c1, c2, eps);
    w[p] = wn;
    wb[p] = __float2bfloat16_rn(wn);
}

// Column sums and sums of squares of the inputs and the target (column 9): per-block partials in
// out[block][20], each block's in a fixed tree order, summed over blocks by the host in block order.
constexpr int kStatBlocks = 256, kStatThreads = 256;

__global__ void __launch_bounds__(kStatThreads) k_cl_stats(const float* X, const float* T, unsigned long long n,
                                                            double* out)
{
    __shared__ double sh[20][kStatThreads];
    double s[20];
    for (int k = 0; k < 20; ++k) s[k] = 0.0;
    for (unsigned long long i = (unsigned long long)blockIdx.x * kStatThreads + threadIdx.x; i < n;
         i += (unsigned long long)kStatBlocks * kStatThreads) {
        for (int k = 0; k < 10; ++k) {
            const double v = k < 9 ? X[i * 9 + k] : T[i];
            s[k] += v;
            s[10 + k] += v * v;
        }
    }
    for (int k = 0; k < 20; ++k) sh[k][threadIdx.x] = s[k];
    __syncthreads();
    for (int w = kStatThreads / 2; w > 0; w >>= 1) {
        if (threadIdx.x < (unsigned)w)
            for (int k = 0; k < 20; ++k) sh[k][threadIdx.x] += sh[k][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x < 20) out[blockIdx.x * 20 + threadIdx.x] = sh[threadIdx.x][0];
}

// splitmix64 (Steele, Lea & Flood 2014) for the initial weights and epoch orders
uint64_t splitmix(uint64_t& s)
{
    uint64_t z = (s += 0x9E3779B97F4A7C15ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

uint64_t gcd64(uint64_t a, uint64_t b)
{
    while (b) {
        const uint64_t t = a % b;
        a = b;
        b = t;
    }
    return a;
}

unsigned short bf16_bits(float v)
{
    const __nv_bfloat16 b = __float2bfloat16_rn(v);
    unsigned short u;
    std::memcpy(&u, &b, sizeof u);
    return u;
}

int err(int code, const std::string& m)
{
    g_create_error = m;
    return code;
}

}  // namespace
}  // namespace fpc

using namespace fpc;

#define FPC_CL_CK(call, what)                                                                   \
    do {                                                                                        \
        cudaError_t e_ = (call);                                                                \
        if (e_ != cudaSuccess)                                                                  \
            return err(e_ == cudaErrorMemoryAllocation ? FPCLBM_ERR_ALLOC : FPCLBM_ERR_CUDA,      \
                       std::string(what) + ": " + cudaGetErrorString(e_));                        \
    } while (0)

extern "C" int fpclbm_closure_sample(fpclbm_t h, int r, double tau_coarse, float* X, float* T, int on_device)
{
    if (!h) return FPCLBM_ERR_ARG;
    h->err.clear();
    if (h->ensemble) return fail(h, FPCLBM_ERR_ARG, "closure_sample needs a single box");
    if (!h->initialized) return fail(h, FPCLBM_ERR_STATE, "populations not initialised");
    const Box& B = h->boxes[0];
    if (r < 1 || B.nx % r || B.ny % r || B.nz % r) return fail(h, FPCLBM_ERR_ARG, "nx, ny, nz must be multiples of r");
    if (!X || !T) return fail(h, FPCLBM_ERR_ARG, "null output");
    if (!(tau_coarse > 0.5) || !std::isfinite(tau_coarse)) return fail(h, FPCLBM_ERR_ARG, "tau_coarse must be > 1/2");
    const int cx = B.nx / r, cy = B.ny / r, cz = B.nz / r;
    if (h->bc != FPCLBM_BC_PERIODIC && h->bc != FPCLBM_BC_WALLS_Y)
        return fail(h, FPCLBM_ERR_ARG, "closure sampling needs a periodic or channel box");
    const bool walls = h->bc == FPCLBM_BC_WALLS_Y;
    if (walls && cy < 2) return fail(h, FPCLBM_ERR_ARG, "walls need ny / r >= 2");
    const size_t nc = (size_t)cx * cy * cz;
    double* acc = nullptr;
    float *dX = X, *dT = T;
    cudaError_t e = rt_malloc(&acc, sizeof(double) * 10 * nc);
    if (e == cudaSuccess && !on_device) {
        e = rt_malloc(&dX, sizeof(float) * 9 * nc);
        if (e == cudaSuccess) e = rt_malloc(&dT, sizeof(float) * nc);
    }
    if (e != cudaSuccess) {
        rt_free(acc);
        if (!on_device) {
            rt_free(dX != X ? dX : nullptr);
        }
        return fail(h, FPCLBM_ERR_ALLOC, "closure_sample scratch");
    }
    BoxGeom g;
    g.buf = static_cast<char*>(h->d_pop) + B.off * elem_size(h->precision);
    g.stride = B.stride;
    g.ncells = B.ncells;
    g.nx = B.nx;
    g.ny = B.ny;
    g.nz = B.nz;
    g.walls = walls;
    g.div_nx = make_fastdiv((unsigned)B.nx);
    g.div_nxny = make_fastdiv((unsigned)(B.nx * B.ny));
    // threads of a filter block: few enough that every SM has two, but a column each where one cell has
    // more than a warp's
    int threads = kFilterThreads, group = std::max(1, threads / r);
    while (threads > 32 && threads / 2 >= r && (nc + group - 1) / group < 2 * (size_t)h->sm_count) {
        threads /= 2;
        group = threads / r;
    }
    threads = std::min(kFilterThreads, (group * r + 31) / 32 * 32);
    const size_t smem = 10 * sizeof(double) * threads;
    const int force = h->F[0] != 0.0 || h->F[1] != 0.0 || h->F[2] != 0.0;
    FilterArgs fa{g, (int)(h->steps & 1), r, cx, cy, cz, group, force, h->F[0], h->F[1], h->F[2], acc};
    const unsigned blocks = (unsigned)((nc + 127) / 128);
    const unsigned fblocks = (unsigned)((nc + group - 1) / group);
    switch (h->precision) {
        case FPCLBM_FP64: k_cl_filter<double><<<fblocks, threads, smem, h->stream>>>(fa); break;
        case FPCLBM_FP32: k_cl_filter<float><<<fblocks, threads, smem, h->stream>>>(fa); break;
        case FPCLBM_FP32_STORE_FP16: k_cl_filter<__half><<<fblocks, threads, smem, h->stream>>>(fa); break;
        default: k_cl_filter<__nv_bfloat16><<<fblocks, threads, smem, h->stream>>>(fa); break;
    }
    k_cl_label<<<blocks, 128, 0, h->stream>>>(acc, cx, cy, cz, walls, tau_coarse, dX, dT);
    e = cudaGetLastError();
    if (e == cudaSuccess && !on_device) {
        e = cudaMemcpyAsync(X, dX, sizeof(float) * 9 * nc, cudaMemcpyDeviceToHost, h->stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(T, dT, sizeof(float) * nc, cudaMemcpyDeviceToHost, h->stream);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    rt_free(acc);
    if (!on_device) {
        rt_free(dX);
        rt_free(dT);
    }
    if (e != cudaSuccess) return fail(h, FPCLBM_ERR_CUDA, std::string("closure_sample: ") + cudaGetErrorString(e));
    return FPCLBM_OK;
}

namespace {

// Run the forward/backward kernel over `count` samples starting at epoch position `first`: one
// block per kMB samples, each writing its gradient and loss to a.part / a.part_loss.
int batch_blocks(unsigned long long count) { return (int)((count + kMB - 1) / kMB); }

cudaError_t run_batch(const NetArgs& a, cudaStream_t st)
{
    const size_t smem = sizeof(TrainSmem);
    static bool attr = false;
    if (!attr) {
        const cudaError_t e = cudaFuncSetAttribute(k_cl_mma, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    k_cl_mma<<<batch_blocks(a.count), kTrainThreads, smem, st>>>(a);
    return cudaGetLastError();
}

int epoch_chunk(int blocks) { return (CL_N + blocks - 1) / blocks; }

// query: whether batches of `blocks` tiles can run as one cluster per epoch on the current device (a
// cluster of more than eight blocks may not fit a partition of the chip), and the kernel's attributes;
// otherwise the launch of an epoch.
cudaError_t epoch_launch(const EpochArgs& a, int blocks, cudaStream_t st, bool query, bool* fits)
{
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)blocks;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kTrainThreads);
    cfg.dynamicSmemBytes = epoch_smem(blocks, epoch_chunk(blocks));
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    if (!query) return cudaLaunchKernelEx(&cfg, k_cl_epoch, a);
    *fits = false;
    if (blocks > kMaxCluster) return cudaSuccess;
    int dev = 0, optin = 0, clusters = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    if (cfg.dynamicSmemBytes > (size_t)optin) return cudaSuccess;
    e = cudaFuncSetAttribute(k_cl_epoch, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
    if (e == cudaSuccess && blocks > 8) e = cudaFuncSetAttribute(k_cl_epoch, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&clusters, k_cl_epoch, &cfg);
    if (e != cudaSuccess) {
        cudaGetLastError();  // not an error of the training: the two-kernel path runs
        return cudaSuccess;
    }
    *fits = clusters > 0;
    return cudaSuccess;
}

}  // namespace

extern "C" int fpclbm_closure_grad(const float* X, const float* T, int n, const unsigned short* w, float* grad,
                                   double* loss, void* cuda_stream)
{
    g_create_error.clear();
    if (!X || !T || !w || !grad || !loss || n < 1) return err(FPCLBM_ERR_ARG, "closure_grad: bad arguments");
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    const int blocks = batch_blocks((unsigned long long)n);
    __nv_bfloat16* dW = nullptr;
    float *dG = nullptr, *dP = nullptr;
    double *dL = nullptr, *dPL = nullptr;
    cudaError_t e = rt_malloc(&dW, sizeof(__nv_bfloat16) * CL_N);
    if (e == cudaSuccess) e = rt_malloc(&dG, sizeof(float) * CL_N);
    if (e == cudaSuccess) e = rt_malloc(&dL, sizeof(double));
    if (e == cudaSuccess) e = rt_malloc(&dP, sizeof(float) * CL_N * (size_t)blocks);
    if (e == cudaSuccess) e = rt_malloc(&dPL, sizeof(double) * (size_t)blocks);
    auto cleanup = [&]() {
        rt_free(dW);
        rt_free(dG);
        rt_free(dL);
        rt_free(dP);
        rt_free(dPL);
    };
    if (e != cudaSuccess) {
        cleanup();
        return err(FPCLBM_ERR_ALLOC, "closure_grad buffers");
    }
    NetArgs a;
    std::memset(&a, 0, sizeof a);
    a.X = X;
    a.T = T;
    a.n = (unsigned long long)n;
    a.first = 0;
    a.count = (unsigned long long)n;
    a.perm_a = 1;
    a.perm_c = 0;
    for (int k = 0; k < 10; ++k) {
        a.mu[k] = 0.f;
        a.inv_sd[k] = 1.f;
    }
    a.scale = 2.0f / (float)n;
    a.W = dW;
    a.part = dP;
    a.part_loss = dPL;
    e = cudaMemcpyAsync(dW, w, sizeof(unsigned short) * CL_N, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(dL, 0, sizeof(double), st);
    if (e == cudaSuccess) e = run_batch(a, st);
    if (e == cudaSuccess) {
        k_cl_reduce_grad<<<(CL_N + 255) / 256, 256, 0, st>>>(dP, dPL, blocks, dG, dL);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(grad, dG, sizeof(float) * CL_N, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(loss, dL, sizeof(double), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cleanup();
    if (e != cudaSuccess) return err(FPCLBM_ERR_CUDA, std::string("closure_grad: ") + cudaGetErrorString(e));
    *loss /= n;
    return FPCLBM_OK;
}

extern "C" int fpclbm_closure_train(const float* X, const float* T, long long n, int epochs, int batch, double lr,
                                    unsigned long long seed, unsigned short* out_w, double* loss_per_epoch,
                                    void* cuda_stream)
{
    g_create_error.clear();
    if (!X || !T || !out_w || n < 2 || epochs < 1 || batch < 1 || !(lr > 0) || !std::isfinite(lr))
        return err(FPCLBM_ERR_ARG, "closure_train: bad arguments");
    cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
    // standardisation of inputs and target
    double* dS = nullptr;
    FPC_CL_CK(rt_malloc(&dS, sizeof(double) * 20 * kStatBlocks), "closure_train stats");
    k_cl_stats<<<kStatBlocks, kStatThreads, 0, st>>>(X, T, (unsigned long long)n, dS);
    std::vector<double> parts(20 * kStatBlocks);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(parts.data(), dS, sizeof(double) * parts.size(), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    rt_free(dS);
    double sums[20] = {0};
    for (int b = 0; b < kStatBlocks; ++b)
        for (int k = 0; k < 20; ++k) sums[k] += parts[20 * b + k];
    if (e != cudaSuccess) return err(FPCLBM_ERR_CUDA, std::string("closure_train stats: ") + cudaGetErrorString(e));
    double mu[10], sd[10];
    for (int k = 0; k < 10; ++k) {
        mu[k] = sums[k] / n;
        const double var = sums[10 + k] / n - mu[k] * mu[k];
        sd[k] = var > 0 ? std::sqrt(var) : 1.0;
        if (!(sd[k] > 1e-30)) sd[k] = 1.0;
    }
    // initial weights (standardised space): uniform(+-1/sqrt(fan_in)), zero biases
    std::vector<float> w0(CL_N, 0.f);
    uint64_t rs = seed;
    auto unif = [&](double lim) { return (float)(lim * (2.0 * ((splitmix(rs) >> 11) * 0x1.0p-53) - 1.0)); };
    for (int i = 0; i < 576; ++i) w0[CL_W1 + i] = unif(1.0 / 3.0);
    for (int i = 0; i < 4096; ++i) w0[CL_W2 + i] = unif(1.0 / 8.0);
    for (int i = 0; i < 64; ++i) w0[CL_W3 + i] = unif(1.0 / 8.0);
    std::vector<unsigned short> wb0(CL_N);
    for (int i = 0; i < CL_N; ++i) wb0[i] = bf16_bits(w0[i]);
    const int max_blocks = batch_blocks((unsigned long long)std::min<long long>(batch, n));
    float *dw = nullptr, *dm = nullptr, *dv = nullptr, *dP = nullptr;
    __nv_bfloat16* dwb = nullptr;
    double *dL = nullptr, *dPL = nullptr;
    const long long batches = (n + batch - 1) / batch;
    EpochArgs ea;
    std::memset(&ea, 0, sizeof ea);
    bool cluster = false;  // batches of few tiles: one cluster runs many of them in a launch
    e = epoch_launch(ea, max_blocks, st, true, &cluster);
    if (e == cudaSuccess) e = rt_malloc(&dw, sizeof(float) * CL_N);
    if (e == cudaSuccess) e = rt_malloc(&dm, sizeof(float) * CL_N);
    if (e == cudaSuccess) e = rt_malloc(&dv, sizeof(float) * CL_N);
    if (e == cudaSuccess && !cluster) e = rt_malloc(&dP, sizeof(float) * CL_N * (size_t)max_blocks);
    if (e == cudaSuccess && !cluster) e = rt_malloc(&dPL, sizeof(double) * (size_t)max_blocks);
    if (e == cudaSuccess) e = rt_malloc(&dwb, sizeof(__nv_bfloat16) * CL_N);
    if (e == cudaSuccess) e = rt_malloc(&dL, sizeof(double));
    auto cleanup = [&]() {
        rt_free(dw);
        rt_free(dm);
        rt_free(dv);
        rt_free(dP);
        rt_free(dPL);
        rt_free(dwb);
        rt_free(dL);
    };
    if (e != cudaSuccess) {
        cleanup();
        return err(FPCLBM_ERR_ALLOC, "closure_train buffers");
    }
    e = cudaMemcpyAsync(dw, w0.data(), sizeof(float) * CL_N, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dwb, wb0.data(), sizeof(unsigned short) * CL_N, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(dm, 0, sizeof(float) * CL_N, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(dv, 0, sizeof(float) * CL_N, st);
    NetArgs a;
    std::memset(&a, 0, sizeof a);
    a.X = X;
    a.T = T;
    a.n = (unsigned long long)n;
    for (int k = 0; k < 10; ++k) {
        a.mu[k] = (float)mu[k];
        a.inv_sd[k] = (float)(1.0 / sd[k]);
    }
    a.W = dwb;
    a.part = dP;
    a.part_loss = dPL;
    const float b1 = 0.9f, b2 = 0.999f;
    long long step = 0;
    // Adam's bias corrections of step k
    auto correction = [&](long long k) {
        return make_float2((float)(1.0 / (1.0 - std::pow((double)b1, (double)k))),
                           (float)(1.0 / (1.0 - std::pow((double)b2, (double)k))));
    };
    if (cluster) {
        ea.batch = std::min<long long>(batch, n);
        ea.lr = (float)lr;
        ea.b1 = b1;
        ea.b2 = b2;
        ea.eps = 1e-8f;
        ea.w = dw;
        ea.m = dm;
        ea.v = dv;
        ea.wb = dwb;
        ea.loss = dL;
        ea.chunk = make_fastdiv((unsigned)epoch_chunk(max_blocks));
    }
    for (int ep = 0; ep < epochs && e == cudaSuccess; ++ep) {
        // epoch order: i -> (perm_a i + perm_c) mod n with gcd(perm_a, n) = 1
        uint64_t pa = splitmix(rs) % (uint64_t)n;
        while (pa == 0 || gcd64(pa, (uint64_t)n) != 1) pa = (pa + 1) % (uint64_t)n;
        a.perm_a = pa;
        a.perm_c = splitmix(rs) % (uint64_t)n;
        e = cudaMemsetAsync(dL, 0, sizeof(double), st);
        ea.net = a;
        for (long long b = 0; cluster && b < batches && e == cudaSuccess; b += ea.batches) {
            ea.first = b;
            ea.batches = (int)std::min<long long>(batches - b, kEpochBatches);
            for (int k = 0; k < ea.batches; ++k) ea.corr[k] = correction(++step);
            e = epoch_launch(ea, max_blocks, st, false, nullptr);
        }
        for (long long first = 0; !cluster && first < n && e == cudaSuccess; first += batch) {
            const long long cnt = (n - first < batch) ? n - first : batch;
            a.first = (unsigned long long)first;
            a.count = (unsigned long long)cnt;
            a.scale = 2.0f / (float)cnt;
            e = run_batch(a, st);
            ++step;
            const float2 c = correction(step);
            if (e == cudaSuccess) {
                k_cl_reduce_adam<<<(CL_N + 255) / 256, 256, 0, st>>>(dw, dm, dv, dP, dPL, batch_blocks(a.count), dL, dwb,
                                                                     (float)lr, b1, b2, c.x, c.y, 1e-8f);
                e = cudaGetLastError();
            }
        }
        if (loss_per_epoch && e == cudaSuccess) {
            double l = 0;
            e = cudaMemcpyAsync(&l, dL, sizeof(double), cudaMemcpyDeviceToHost, st);
            if (e == cudaSuccess) e = cudaStreamSynchronize(st);
            loss_per_epoch[ep] = l / n;
        }
    }
    std::vector<float> w(CL_N);
    if (e == cudaSuccess) e = cudaMemcpyAsync(w.data(), dw, sizeof(float) * CL_N, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cleanup();
    if (e != cudaSuccess) return err(FPCLBM_ERR_CUDA, std::string("closure_train: ") + cudaGetErrorString(e));
    // fold the standardisation into the first and last layers (raw inputs, raw output)
    std::vector<double> out(CL_N);
    for (int j = 0; j < 64; ++j) {
        double b = w[CL_B1 + j];
        for (int i = 0; i < 9; ++i) {
            const double wij = (double)w[CL_W1 + 9 * j + i] / sd[i];
            out[CL_W1 + 9 * j + i] = wij;
            b -= wij * mu[i];
        }
        out[CL_B1 + j] = b;
    }
    for (int i = 0; i < 4096; ++i) out[CL_W2 + i] = w[CL_W2 + i];
    for (int j = 0; j < 64; ++j) out[CL_B2 + j] = w[CL_B2 + j];
    for (int j = 0; j < 64; ++j) out[CL_W3 + j] = (double)w[CL_W3 + j] * sd[9];
    out[CL_B3] = (double)w[CL_B3] * sd[9] + mu[9];
    for (int i = 0; i < CL_N; ++i) out_w[i] = bf16_bits((float)out[i]);
    return FPCLBM_OK;
}
