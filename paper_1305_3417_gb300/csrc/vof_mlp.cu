// The initial-guess network: 33 features of an interface cell -> 64 -> 64 ->
// 4 (a unit normal and the plane offset s = (d - d_min) / (d_max - d_min)),
// ReLU hidden layers, BF16 weights and activations, FP32 accumulation on the
// tensor cores (mma.sync m16n8k16; the layers are 48-64 wide, far below the
// tile sizes where tcgen05 and TMEM would pay), trained by Adam on the mean
// squared error with the forward and backward kernels here.  The paper has no
// learned part: the network only moves the start of the plane positioning,
// whose root and stop are unchanged.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <new>
#include <vector>

#include "vof_device.cuh"
#include "vof_internal.h"

namespace {

constexpr int IN = VOF_MLP_IN, K0 = 48, HID = VOF_MLP_HID, OUT = VOF_MLP_OUT, OUTP = 16;
// flat FP32 parameter layout: W1 [IN x HID], b1, W2 [HID x HID], b2, W3 [HID x OUT], b3
constexpr int OW1 = 0, OB1 = OW1 + IN * HID, OW2 = OB1 + HID, OB2 = OW2 + HID * HID, OW3 = OB2 + HID,
              OB3 = OW3 + HID * OUT, NPARAM = OB3 + OUT;
static_assert(NPARAM == VOF_MLP_NPARAM, "parameter count");

using bf = unsigned short;

__device__ __forceinline__ bf to_bf(float x) { return __bfloat16_as_ushort(__float2bfloat16_rn(x)); }
__device__ __forceinline__ uint32_t pk(bf lo, bf hi) { return (uint32_t)lo | ((uint32_t)hi << 16); }

__device__ __forceinline__ void mma16816(float c[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// ---------------------------------------------------------------- features
// Per interface cell: the volume fractions of its 3x3x3 lattice neighbourhood
// (the cells sharing a point with it, placed by the sign of their centre
// offset beyond half the cell size; missing slots take the cell's own value)
// and six scale-free shape numbers: box extents / V^(1/3) (3), V / box volume,
// faces / 24, points / 8.
__device__ void mlp_features_one(const DevMesh &m, const double *__restrict__ alpha, int c, float *f)
{
    const double ac = alpha[c];
    for (int k = 0; k < 27; ++k) f[k] = (float)ac;
    const double V = m.vc[c], h = cbrt(V);
    const vofd::V3 cc = vofd::ld3(m.cc, m.nc, c);
    for (int j = m.cpptr[c]; j < m.cpptr[c + 1]; ++j) {
        const int p = m.cpts[j];
        for (int q = m.pptr[p]; q < m.pptr[p + 1]; ++q) {
            const int nb = m.pcell[q];
            vofd::V3 d = vofd::ld3(m.cc, m.nc, nb) - cc;
            if (m.pcode) d = d + vofd::tshift(m, m.pcode[q]);  // periodic: the cell next to c
            const int sx = (d.x > 0.5 * h) - (d.x < -0.5 * h), sy = (d.y > 0.5 * h) - (d.y < -0.5 * h),
                      sz = (d.z > 0.5 * h) - (d.z < -0.5 * h);
            f[(sx + 1) + 3 * (sy + 1) + 9 * (sz + 1)] = (float)alpha[nb];
        }
    }
    const double *bx = m.cbox + 6 * (size_t)c;
    const double ex = bx[3] - bx[0], ey = bx[4] - bx[1], ez = bx[5] - bx[2];
    f[27] = (float)(ex / h);
    f[28] = (float)(ey / h);
    f[29] = (float)(ez / h);
    f[30] = (float)(V / (ex * ey * ez));
    f[31] = (float)((m.cptr[c + 1] - m.cptr[c]) / 24.0);
    f[32] = (float)((m.cpptr[c + 1] - m.cpptr[c]) / 8.0);
}

__global__ void k_mlp_features(DevMesh m, const double *__restrict__ alpha, const int *cells, int ncells,
                               const int *ndev, float *feat)
{
    const int nn = ndev ? min(*ndev, ncells) : ncells;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nn; i += gridDim.x * blockDim.x)
        mlp_features_one(m, alpha, cells ? cells[i] : i, feat + (size_t)i * IN);
}

// ---------------------------------------------------------------- weights
// BF16 copies of the FP32 master weights, zero padded: W1 [K0 x HID] transposed,
// W2 [HID x HID] and transpose, W3 [HID x OUTP] and transpose
__global__ void k_mlp_pack(const float *p, bf *W1t, bf *W2, bf *W2t, bf *W3, bf *W3t)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < K0 * HID) {
        const int k = i / HID, j = i % HID;
        W1t[j * K0 + k] = k < IN ? to_bf(p[OW1 + k * HID + j]) : (bf)0;
    }
    if (i < HID * HID) {
        const int k = i / HID, j = i % HID;
        const bf v = to_bf(p[OW2 + k * HID + j]);
        W2[k * HID + j] = v;
        W2t[j * HID + k] = v;
    }
    if (i < HID * OUTP) {
        const int k = i / OUTP, j = i % OUTP;
        const bf v = j < OUT ? to_bf(p[OW3 + k * OUT + j]) : (bf)0;
        W3[k * OUTP + j] = v;
        W3t[j * HID + k] = v;
    }
}

// ---------------------------------------------------- forward and backward
// One kernel for the network's whole pass over a tile of 64 samples (four
// warps, 16 samples each), the layers chained through registers: the
// accumulators of two 8-column tiles are the next layer's 16-column operand,
// forward and backward.  GRAD: the operands of the weight gradients
// (activations and BF16 upstream gradients) go to shared memory transposed,
// [column][sample], so that a pair of samples is one 32-bit operand load, and
// the block's 60 weight-gradient tiles (16 x 8) stay in registers over all the
// tiles that the block takes; a block writes one partial gradient in the flat
// parameter layout.  Rows of 72 (56, 24) 16-bit values: conflict-free operand
// loads.  Bound by latency (a few hundred small mma per tile on one SM): a tile
// of 64 samples spreads a batch of 4096 over 64 SMs.  Against one kernel per
// layer and per gradient with everything through global memory (13 launches,
// the weight gradients read with 16-bit loads): 4096 samples 251 -> 56 us a
// gradient call with its loss.
constexpr int TILE = 64, GT = 128, LT = TILE + 8, L1 = K0 + 8, L2 = HID + 8, L3 = OUTP + 8;
struct MlpShared {
    bf W1t[HID * L1], W2t[HID * L2], W2[HID * L2], W3t[8 * L2], W3[HID * L3];
    bf X[TILE * L1];
    bf XT[K0 * LT], H1T[HID * LT], H2T[HID * LT], D1T[HID * LT], D2T[HID * LT], DYT[8 * LT];
    float b1[HID], b2[HID], b3[8];
    float red[4][2 * HID + 8];
    double loss[4];
};
struct MlpWeights {
    const float *p;
    const bf *W1t, *W2, *W2t, *W3, *W3t;
};

__device__ __forceinline__ uint32_t ld2(const bf *q) { return *reinterpret_cast<const uint32_t *>(q); }

template <bool GRAD>
__global__ void __launch_bounds__(GT) k_mlp_pass(MlpWeights w, const float *__restrict__ feat,
                                                 const float *__restrict__ target, int n, float *out, float *part,
                                                 double *lpart)
{
    vofd::next_kernel();
    extern __shared__ __align__(16) unsigned char mlp_smem[];
    MlpShared &sh = *reinterpret_cast<MlpShared *>(mlp_smem);
    const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5, g = lane >> 2, t = lane & 3;
    // weights: rows of the packed copies, two values a load
    auto rows = [&](bf *dst, const bf *src, int nr, int len, int ld) {
        for (int i = tid; i < nr * (len / 2); i += GT) {
            const int r = i / (len / 2), c = 2 * (i % (len / 2));
            *reinterpret_cast<uint32_t *>(dst + r * ld + c) = ld2(src + r * len + c);
        }
    };
    rows(sh.W1t, w.W1t, HID, K0, L1);
    rows(sh.W2t, w.W2t, HID, HID, L2);
    rows(sh.W3t, w.W3t, 8, HID, L2);
    if (GRAD) {
        rows(sh.W2, w.W2, HID, HID, L2);
        rows(sh.W3, w.W3, HID, OUTP, L3);
    }
    for (int i = tid; i < HID; i += GT) { sh.b1[i] = w.p[OB1 + i]; sh.b2[i] = w.p[OB2 + i]; }
    if (tid < 8) sh.b3[tid] = tid < OUT ? w.p[OB3 + tid] : 0.0f;

    float wacc[15][4];           // weight-gradient tiles wp, wp + 4, ...: 24 of W1, 32 of W2, 4 of W3
    float s1[8][2], s2[8][2], s3[2] = {0.0f, 0.0f};  // bias gradients: column sums over this thread's rows
    double loss = 0.0;
    if (GRAD) {
#pragma unroll
        for (int i = 0; i < 15; ++i) wacc[i][0] = wacc[i][1] = wacc[i][2] = wacc[i][3] = 0.0f;
#pragma unroll
        for (int j = 0; j < 8; ++j) s1[j][0] = s1[j][1] = s2[j][0] = s2[j][1] = 0.0f;
    }
    const int ntile = (n + TILE - 1) / TILE;
    for (int tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
        const int r00 = tile * TILE;
        // features to BF16, zero beyond the batch and beyond the 33 columns
        for (int i = tid; i < TILE * K0; i += GT) {
            const int r = i / K0, k = i % K0;
            const bf v = (k < IN && r00 + r < n) ? to_bf(feat[(size_t)(r00 + r) * IN + k]) : (bf)0;
            sh.X[r * L1 + k] = v;
            if (GRAD) sh.XT[k * LT + r] = v;
        }
        __syncthreads();
        const int ra = 16 * wp + g, rb = ra + 8;  // this thread's rows of the tile
        float h[8][4];
        // bias and ReLU of a layer's accumulators: the next layer's operand
        // pairs (first row, second row) per 8-column tile, and the ReLU's mask
        auto relu = [&](const float *bias, uint32_t (&pa)[8], uint32_t (&pb)[8], uint32_t &mask, bf *HT) {
            mask = 0u;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int c = 8 * j + 2 * t;
                const float z0 = h[j][0] + bias[c], z1 = h[j][1] + bias[c + 1], z2 = h[j][2] + bias[c],
                            z3 = h[j][3] + bias[c + 1];
                mask |= (z0 > 0.0f ? 1u : 0u) << (4 * j) | (z1 > 0.0f ? 2u : 0u) << (4 * j) |
                        (z2 > 0.0f ? 4u : 0u) << (4 * j) | (z3 > 0.0f ? 8u : 0u) << (4 * j);
                const bf v0 = to_bf(fmaxf(z0, 0.0f)), v1 = to_bf(fmaxf(z1, 0.0f)), v2 = to_bf(fmaxf(z2, 0.0f)),
                         v3 = to_bf(fmaxf(z3, 0.0f));
                pa[j] = pk(v0, v1);
                pb[j] = pk(v2, v3);
                if (GRAD) {
                    HT[c * LT + ra] = v0; HT[(c + 1) * LT + ra] = v1;
                    HT[c * LT + rb] = v2; HT[(c + 1) * LT + rb] = v3;
                }
            }
        };
        auto zero = [&]() {
#pragma unroll
            for (int j = 0; j < 8; ++j) h[j][0] = h[j][1] = h[j][2] = h[j][3] = 0.0f;
        };
        uint32_t pa[8], pb[8], m1, m2;
        // layer 1
        zero();
#pragma unroll
        for (int k0 = 0; k0 < K0; k0 += 16) {
            const bf *xa = sh.X + ra * L1 + k0 + 2 * t, *xb = sh.X + rb * L1 + k0 + 2 * t;
            const uint32_t a0 = ld2(xa), a1 = ld2(xb), a2 = ld2(xa + 8), a3 = ld2(xb + 8);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const bf *bt = sh.W1t + (8 * j + g) * L1 + k0 + 2 * t;
                mma16816(h[j], a0, a1, a2, a3, ld2(bt), ld2(bt + 8));
            }
        }
        relu(sh.b1, pa, pb, m1, sh.H1T);
        // layer 2
        zero();
#pragma unroll
        for (int kk = 0; kk < HID / 16; ++kk)
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const bf *bt = sh.W2t + (8 * j + g) * L2 + 16 * kk + 2 * t;
                mma16816(h[j], pa[2 * kk], pb[2 * kk], pa[2 * kk + 1], pb[2 * kk + 1], ld2(bt), ld2(bt + 8));
            }
        relu(sh.b2, pa, pb, m2, sh.H2T);
        // output layer (columns 0..7, of which 0..3 exist)
        float y[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int kk = 0; kk < HID / 16; ++kk) {
            const bf *bt = sh.W3t + g * L2 + 16 * kk + 2 * t;
            mma16816(y, pa[2 * kk], pb[2 * kk], pa[2 * kk + 1], pb[2 * kk + 1], ld2(bt), ld2(bt + 8));
        }
        if constexpr (!GRAD) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int r = r00 + (e < 2 ? ra : rb), c = 2 * t + (e & 1);
                if (r < n && c < OUT) out[(size_t)r * OUT + c] = y[e] + sh.b3[c];
            }
        } else {
        // gradient of the mean squared error: 2 (Y - T) / n
        bf db[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int r = r00 + (e < 2 ? ra : rb), c = 2 * t + (e & 1);
            float d = 0.0f;
            if (r < n && c < OUT) {
                const float er = y[e] + sh.b3[c] - target[(size_t)r * OUT + c];
                const float l = er * er;
                loss += (double)l;
                d = 2.0f * er / (float)n;
            }
            db[e] = to_bf(d);
            s3[e & 1] += d;
            sh.DYT[c * LT + (e < 2 ? ra : rb)] = db[e];
        }
        // back through a layer: accumulators masked by the ReLU, their column
        // sums, and the next operand pairs
        auto back = [&](uint32_t mask, float (&s)[8][2], bf *DT) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int c = 8 * j + 2 * t;
                const float d0 = mask >> (4 * j) & 1u ? h[j][0] : 0.0f, d1 = mask >> (4 * j) & 2u ? h[j][1] : 0.0f,
                            d2 = mask >> (4 * j) & 4u ? h[j][2] : 0.0f, d3 = mask >> (4 * j) & 8u ? h[j][3] : 0.0f;
                s[j][0] += d0 + d2;
                s[j][1] += d1 + d3;
                const bf v0 = to_bf(d0), v1 = to_bf(d1), v2 = to_bf(d2), v3 = to_bf(d3);
                pa[j] = pk(v0, v1);
                pb[j] = pk(v2, v3);
                DT[c * LT + ra] = v0; DT[(c + 1) * LT + ra] = v1;
                DT[c * LT + rb] = v2; DT[(c + 1) * LT + rb] = v3;
            }
        };
        zero();
        {
            const uint32_t a0 = pk(db[0], db[1]), a1 = pk(db[2], db[3]);
#pragma unroll
            for (int j = 0; j < 8; ++j) mma16816(h[j], a0, a1, 0u, 0u, ld2(sh.W3 + (8 * j + g) * L3 + 2 * t), 0u);
        }
        back(m2, s2, sh.D2T);
        zero();
#pragma unroll
        for (int kk = 0; kk < HID / 16; ++kk)
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const bf *bt = sh.W2 + (8 * j + g) * L2 + 16 * kk + 2 * t;
                mma16816(h[j], pa[2 * kk], pb[2 * kk], pa[2 * kk + 1], pb[2 * kk + 1], ld2(bt), ld2(bt + 8));
            }
        back(m1, s1, sh.D1T);
        __syncthreads();
        // weight gradients of the tile: A^T . D over its 64 samples
        auto wtile = [&](float (&acc)[4], const bf *AT, const bf *DT, int k0, int c0) {
#pragma unroll
            for (int sb = 0; sb < TILE; sb += 16) {
                const bf *a = AT + (k0 + g) * LT + sb + 2 * t, *d = DT + (c0 + g) * LT + sb + 2 * t;
                mma16816(acc, ld2(a), ld2(a + 8 * LT), ld2(a + 8), ld2(a + 8 * LT + 8), ld2(d), ld2(d + 8));
            }
        };
#pragma unroll
        for (int i = 0; i < 6; ++i) wtile(wacc[i], sh.XT, sh.D1T, 16 * ((wp + 4 * i) / 8), 8 * ((wp + 4 * i) % 8));
#pragma unroll
        for (int i = 0; i < 8; ++i) wtile(wacc[6 + i], sh.H1T, sh.D2T, 16 * ((wp + 4 * i) / 8), 8 * ((wp + 4 * i) % 8));
        wtile(wacc[14], sh.H2T, sh.DYT, 16 * wp, 0);
        }
        __syncthreads();  // every operand read before the next tile
    }
    if (!GRAD) return;
    float *o = part + (size_t)blockIdx.x * NPARAM;
    auto put = [&](int base, int ld, int k, int c, int kmax, int cmax, const float (&acc)[4]) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int kk = k + g + (e >= 2 ? 8 : 0), cc = c + 2 * t + (e & 1);
            if (kk < kmax && cc < cmax) o[base + kk * ld + cc] = acc[e];
        }
    };
#pragma unroll
    for (int i = 0; i < 6; ++i) put(OW1, HID, 16 * ((wp + 4 * i) / 8), 8 * ((wp + 4 * i) % 8), IN, HID, wacc[i]);
#pragma unroll
    for (int i = 0; i < 8; ++i) put(OW2, HID, 16 * ((wp + 4 * i) / 8), 8 * ((wp + 4 * i) % 8), HID, HID, wacc[6 + i]);
    put(OW3, OUT, 16 * wp, 0, HID, OUT, wacc[14]);
    // bias gradients: over the rows of a warp (lanes of one t), then the warps
    auto rsum = [&](float v) {
#pragma unroll
        for (int x = 4; x < 32; x <<= 1) v += __shfl_xor_sync(0xffffffffu, v, x);
        return v;
    };
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const float v1 = rsum(s1[j][e]), v2 = rsum(s2[j][e]);
            if (g == 0) { sh.red[wp][8 * j + 2 * t + e] = v1; sh.red[wp][HID + 8 * j + 2 * t + e] = v2; }
        }
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const float v = rsum(s3[e]);
        if (g == 0) sh.red[wp][2 * HID + 2 * t + e] = v;
    }
    loss = vofd::warp_sum(loss);
    if (lane == 0) sh.loss[wp] = loss;
    __syncthreads();
    for (int i = tid; i < 2 * HID + OUT; i += GT) {
        const float v = (sh.red[0][i] + sh.red[1][i]) + (sh.red[2][i] + sh.red[3][i]);
        o[i < HID ? OB1 + i : i < 2 * HID ? OB2 + (i - HID) : OB3 + (i - 2 * HID)] = v;
    }
    if (tid == 0) lpart[blockIdx.x] = (sh.loss[0] + sh.loss[1]) + (sh.loss[2] + sh.loss[3]);
}

// sums the blocks' partials in block order into the flat gradient (and the
// caller's copy of it), and the squared errors into *loss (host memory)
constexpr int RED_T = 64;
__global__ void __launch_bounds__(RED_T) k_mlp_reduce(const float *part, const double *lpart, int nb, float *grad,
                                                      float *copy, float *loss)
{
    vofd::previous_kernel();
    const int i = blockIdx.x * RED_T + threadIdx.x;
    if (i < NPARAM) {
        float s = 0.0f;
#pragma unroll 8
        for (int b = 0; b < nb; ++b) s += part[(size_t)b * NPARAM + i];
        grad[i] = s;
        if (copy) copy[i] = s;
    }
    if (i == 0 && loss) {
        double s = 0.0;
        for (int b = 0; b < nb; ++b) s += lpart[b];
        *loss = (float)s;  // sum of squared errors; the host divides by n
    }
}

__global__ void k_mlp_adam(float *p, const float *g, float *m1, float *m2, float lr, float c1, float c2)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= NPARAM) return;
    const float b1 = 0.9f, b2 = 0.999f;
    const float m = b1 * m1[i] + (1.0f - b1) * g[i], v = b2 * m2[i] + (1.0f - b2) * g[i] * g[i];
    m1[i] = m;
    m2[i] = v;
    p[i] -= lr * (m / c1) / (sqrtf(v / c2) + 1e-8f);
}



// Per cell, once (vof_set_guess): the 27 lattice slots as cell indices (-1:
// the cell itself) and the 6 shape numbers, as vof_mlp_features places them
__global__ void k_mlp_tables(DevMesh m, int *nbr, float *geo)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= m.nc) return;
    int *t = nbr + 27 * (size_t)c;
    for (int k = 0; k < 27; ++k) t[k] = -1;
    const double V = m.vc[c], h = cbrt(V);
    const vofd::V3 cc = vofd::ld3(m.cc, m.nc, c);
    for (int j = m.cpptr[c]; j < m.cpptr[c + 1]; ++j) {
        const int p = m.cpts[j];
        for (int q = m.pptr[p]; q < m.pptr[p + 1]; ++q) {
            const int nb = m.pcell[q];
            vofd::V3 d = vofd::ld3(m.cc, m.nc, nb) - cc;
            if (m.pcode) d = d + vofd::tshift(m, m.pcode[q]);  // periodic: the cell next to c
            const int sx = (d.x > 0.5 * h) - (d.x < -0.5 * h), sy = (d.y > 0.5 * h) - (d.y < -0.5 * h),
                      sz = (d.z > 0.5 * h) - (d.z < -0.5 * h);
            t[(sx + 1) + 3 * (sy + 1) + 9 * (sz + 1)] = nb;
        }
    }
    const double *bx = m.cbox + 6 * (size_t)c;
    const double ex = bx[3] - bx[0], ey = bx[4] - bx[1], ez = bx[5] - bx[2];
    float *g = geo + 6 * (size_t)c;
    g[0] = (float)(ex / h);
    g[1] = (float)(ey / h);
    g[2] = (float)(ez / h);
    g[3] = (float)(V / (ex * ey * ez));
    g[4] = (float)((m.cptr[c + 1] - m.cptr[c]) / 24.0);
    g[5] = (float)((m.cpptr[c + 1] - m.cpptr[c]) / 8.0);
}

// The guess of a step in one kernel: one warp per 16 listed cells gathers
// their features straight into the tensor-core operand layout (from the
// tables), runs the three layers chaining each layer's accumulators into the
// next layer's operands in registers, and writes the clamped offsets.
__global__ void __launch_bounds__(128) k_mlp_guess_fused(const int *nbr, const float *geo,
                                                          const double *__restrict__ alpha, const int *list,
                                                          const int *count, int cap, const bf *W1t, const bf *W2t,
                                                          const bf *W3t, const float *p, float *s0)
{
    const int n = min(*count, cap);
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int wstride = (gridDim.x * blockDim.x) >> 5;
    for (int r0 = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 16; r0 < n; r0 += wstride * 16) {
        // feature (row r, column k) of the tile
        const int ra = r0 + g, rb = r0 + g + 8;
        const int ca = ra < n ? list[ra] : -1, cb = rb < n ? list[rb] : -1;
        auto feat = [&](int c, int k) -> bf {
            if (c < 0 || k >= IN) return (bf)0;
            if (k < 27) {
                const int q = nbr[27 * (size_t)c + k];
                return to_bf((float)alpha[q < 0 ? c : q]);
            }
            return to_bf(geo[6 * (size_t)c + (k - 27)]);
        };
        // layer 1: [16 x 48] . [48 x 64]
        float h1[8][4];
#pragma unroll
        for (int j = 0; j < 8; ++j) h1[j][0] = h1[j][1] = h1[j][2] = h1[j][3] = 0.0f;
#pragma unroll
        for (int k0 = 0; k0 < K0; k0 += 16) {
            const uint32_t a0 = pk(feat(ca, k0 + 2 * t), feat(ca, k0 + 2 * t + 1));
            const uint32_t a1 = pk(feat(cb, k0 + 2 * t), feat(cb, k0 + 2 * t + 1));
            const uint32_t a2 = pk(feat(ca, k0 + 2 * t + 8), feat(ca, k0 + 2 * t + 9));
            const uint32_t a3 = pk(feat(cb, k0 + 2 * t + 8), feat(cb, k0 + 2 * t + 9));
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const bf *bt = W1t + (size_t)(8 * j + g) * K0 + k0 + 2 * t;
                mma16816(h1[j], a0, a1, a2, a3, pk(bt[0], bt[1]), pk(bt[8], bt[9]));
            }
        }
        // bias, ReLU, BF16: the accumulators of two n-tiles form one k-step of
        // the next layer's operand
        auto act = [&](float (*h)[4], const float *bias, int kk, uint32_t &a0, uint32_t &a1, uint32_t &a2,
                       uint32_t &a3) {
            const int c0 = 16 * kk + 2 * t, c1 = c0 + 8;
            a0 = pk(to_bf(fmaxf(h[2 * kk][0] + bias[c0], 0.f)), to_bf(fmaxf(h[2 * kk][1] + bias[c0 + 1], 0.f)));
            a1 = pk(to_bf(fmaxf(h[2 * kk][2] + bias[c0], 0.f)), to_bf(fmaxf(h[2 * kk][3] + bias[c0 + 1], 0.f)));
            a2 = pk(to_bf(fmaxf(h[2 * kk + 1][0] + bias[c1], 0.f)),
                    to_bf(fmaxf(h[2 * kk + 1][1] + bias[c1 + 1], 0.f)));
            a3 = pk(to_bf(fmaxf(h[2 * kk + 1][2] + bias[c1], 0.f)),
                    to_bf(fmaxf(h[2 * kk + 1][3] + bias[c1 + 1], 0.f)));
        };
        float h2[8][4];
#pragma unroll
        for (int j = 0; j < 8; ++j) h2[j][0] = h2[j][1] = h2[j][2] = h2[j][3] = 0.0f;
#pragma unroll
        for (int kk = 0; kk < HID / 16; ++kk) {
            uint32_t a0, a1, a2, a3;
            act(h1, p + OB1, kk, a0, a1, a2, a3);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const bf *bt = W2t + (size_t)(8 * j + g) * HID + 16 * kk + 2 * t;
                mma16816(h2[j], a0, a1, a2, a3, pk(bt[0], bt[1]), pk(bt[8], bt[9]));
            }
        }
        float y[4] = {0.f, 0.f, 0.f, 0.f};  // output columns 0..7 (the offset is column 3)
#pragma unroll
        for (int kk = 0; kk < HID / 16; ++kk) {
            uint32_t a0, a1, a2, a3;
            act(h2, p + OB2, kk, a0, a1, a2, a3);
            const bf *bt = W3t + (size_t)g * HID + 16 * kk + 2 * t;
            mma16816(y, a0, a1, a2, a3, pk(bt[0], bt[1]), pk(bt[8], bt[9]));
        }
        if (t == 1) {  // column 2t + 1 = 3
            const float b3 = p[OB3 + 3];
            if (ra < n) s0[ra] = fminf(fmaxf(y[1] + b3, 0.02f), 0.98f);
            if (rb < n) s0[rb] = fminf(fmaxf(y[3] + b3, 0.02f), 0.98f);
        }
    }
}

inline int cdiv(long a, long b) { return (int)((a + b - 1) / b); }

}  // namespace

struct vof_mlp {
    int device, max_batch, nblk, adam_t;   // nblk: blocks (partial gradients) of a pass at most
    float *p, *grad, *m1, *m2;
    bf *W1t, *W2, *W2t, *W3, *W3t;
    float *part;
    double *lpart;
    float *y;                              // outputs of a forward pass over its own features
    float *h_loss;                         // pinned host memory that the device writes
    std::vector<void *> bufs;
};

namespace {

template <class T>
T *mlp_alloc(vof_mlp *q, size_t n, bool *ok)
{
    void *p = nullptr;
    if (*ok && cudaMalloc(&p, std::max<size_t>(n, 1) * sizeof(T)) == cudaSuccess) {
        q->bufs.push_back(p);
        return (T *)p;
    }
    *ok = false;
    return nullptr;
}

MlpWeights mlp_weights(const vof_mlp *q) { return MlpWeights{q->p, q->W1t, q->W2, q->W2t, q->W3, q->W3t}; }

int mlp_forward(vof_mlp *q, const float *feat, int n, float *out, cudaStream_t s)
{
    k_mlp_pass<false><<<std::min(cdiv(n, TILE), q->nblk), GT, sizeof(MlpShared), s>>>(mlp_weights(q), feat, nullptr, n,
                                                                                      out, nullptr, nullptr);
    return cudaGetLastError() == cudaSuccess ? VOF_OK : VOF_ERR_CUDA;
}

// forward and backward: the flat gradient into q->grad (and copy, if given),
// the sum of squared errors into q->h_loss if wanted
int mlp_gradient(vof_mlp *q, const float *feat, const float *target, int n, float *copy, bool want_loss, cudaStream_t s)
{
    const int nb = std::min(cdiv(n, TILE), q->nblk);
    k_mlp_pass<true><<<nb, GT, sizeof(MlpShared), s>>>(mlp_weights(q), feat, target, n, nullptr, q->part, q->lpart);
    if (cudaGetLastError() != cudaSuccess) return VOF_ERR_CUDA;
    return launch_after(k_mlp_reduce, cdiv(NPARAM, RED_T), RED_T, 0, s, q->part, q->lpart, nb, q->grad, copy,
                        want_loss ? q->h_loss : nullptr);
}

int mlp_pack(vof_mlp *q, cudaStream_t s)
{
    k_mlp_pack<<<cdiv(HID * HID, 256), 256, 0, s>>>(q->p, q->W1t, q->W2, q->W2t, q->W3, q->W3t);
    return cudaGetLastError() == cudaSuccess ? VOF_OK : VOF_ERR_CUDA;
}

}  // namespace

// the reconstruction guess of a step: for the first max_batch listed
// interface cells (device count), the clamped offsets by list position in
// c->mlp_s0 (one fused kernel)
int launch_mlp_guess(vof_ctx *c, const double *alpha, const int *cells, const int *count, int nmax, cudaStream_t s)
{
    vof_mlp *q = c->mlp;
    if (!q) return VOF_OK;
    const int cap = std::min(q->max_batch, nmax);
    if (!cells || !count) return VOF_ERR_INVALID_ARG;
    k_mlp_guess_fused<<<std::min(cdiv(cap, 64), 1024), 128, 0, s>>>(c->mlp_nbr, c->mlp_geo, alpha, cells, count,
                                                                     cap, q->W1t, q->W2t, q->W3t, q->p, c->mlp_s0);
    return cudaGetLastError() == cudaSuccess ? VOF_OK : VOF_ERR_CUDA;
}

int mlp_cap(const vof_ctx *c) { return c->mlp ? c->mlp->max_batch : 0; }

extern "C" {

int vof_mlp_create(int max_batch, const float *params, int device, vof_mlp **out)
{
    if (max_batch < 16 || !params || !out) return VOF_ERR_INVALID_ARG;
    *out = nullptr;
    if (cudaSetDevice(device) != cudaSuccess) return VOF_ERR_CUDA;
    vof_mlp *q = new (std::nothrow) vof_mlp();
    if (!q) return VOF_ERR_CUDA;
    q->device = device;
    q->max_batch = max_batch;
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    q->nblk = std::min(cdiv(max_batch, TILE), std::max(sms, 1));  // a block per SM at most: its shared memory
    bool ok = true;
    q->p = mlp_alloc<float>(q, NPARAM, &ok);
    q->grad = mlp_alloc<float>(q, NPARAM, &ok);
    q->m1 = mlp_alloc<float>(q, NPARAM, &ok);
    q->m2 = mlp_alloc<float>(q, NPARAM, &ok);
    q->W1t = mlp_alloc<bf>(q, K0 * HID, &ok);
    q->W2 = mlp_alloc<bf>(q, HID * HID, &ok);
    q->W2t = mlp_alloc<bf>(q, HID * HID, &ok);
    q->W3 = mlp_alloc<bf>(q, HID * OUTP, &ok);
    q->W3t = mlp_alloc<bf>(q, HID * OUTP, &ok);
    q->part = mlp_alloc<float>(q, (size_t)q->nblk * NPARAM, &ok);
    q->lpart = mlp_alloc<double>(q, q->nblk, &ok);
    q->y = mlp_alloc<float>(q, (size_t)max_batch * OUT, &ok);
    ok = ok && cudaMallocHost(&q->h_loss, sizeof(float)) == cudaSuccess &&
         cudaFuncSetAttribute(k_mlp_pass<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, sizeof(MlpShared)) ==
             cudaSuccess &&
         cudaFuncSetAttribute(k_mlp_pass<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sizeof(MlpShared)) ==
             cudaSuccess;
    ok = ok && cudaMemcpy(q->p, params, sizeof(float) * NPARAM, cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemset(q->m1, 0, sizeof(float) * NPARAM) == cudaSuccess &&
         cudaMemset(q->m2, 0, sizeof(float) * NPARAM) == cudaSuccess && mlp_pack(q, 0) == VOF_OK &&
         cudaDeviceSynchronize() == cudaSuccess;
    if (!ok) { vof_mlp_destroy(q); return VOF_ERR_CUDA; }
    *out = q;
    return VOF_OK;
}

void vof_mlp_destroy(vof_mlp *q)
{
    if (!q) return;
    cudaSetDevice(q->device);
    for (void *p : q->bufs) cudaFree(p);
    if (q->h_loss) cudaFreeHost(q->h_loss);
    delete q;
}

int vof_mlp_params(vof_mlp *q, float *params)
{
    if (!q || !params) return VOF_ERR_INVALID_ARG;
    if (cudaSetDevice(q->device) != cudaSuccess) return VOF_ERR_CUDA;
    return cudaMemcpy(params, q->p, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost) == cudaSuccess ? VOF_OK
                                                                                                   : VOF_ERR_CUDA;
}

int vof_mlp_features(vof_ctx *c, const double *alpha, const int32_t *cells, int ncells, float *feat, void *stream)
{
    if (!c || !alpha || !feat || ncells < 0) return VOF_ERR_INVALID_ARG;
    if (cudaSetDevice(c->device) != cudaSuccess) return VOF_ERR_CUDA;
    if (ncells == 0) return VOF_OK;
    k_mlp_features<<<std::min(cdiv(ncells, 128), 4096), 128, 0, (cudaStream_t)stream>>>(c->m, alpha, cells, ncells,
                                                                                         nullptr, feat);
    return cudaGetLastError() == cudaSuccess ? VOF_OK : VOF_ERR_CUDA;
}

int vof_mlp_forward(vof_mlp *q, const float *feat, int n, float *out, void *stream)
{
    if (!q || !feat || !out || n < 1 || n > q->max_batch) return VOF_ERR_INVALID_ARG;
    if (cudaSetDevice(q->device) != cudaSuccess) return VOF_ERR_CUDA;
    cudaStream_t s = (cudaStream_t)stream;
    // out may lie over feat: a block would write rows that another has yet to read
    const std::uintptr_t f = reinterpret_cast<std::uintptr_t>(feat), o = reinterpret_cast<std::uintptr_t>(out);
    const size_t fb = sizeof(float) * IN * (size_t)n, ob = sizeof(float) * OUT * (size_t)n;
    if (o >= f + fb || f >= o + ob) return mlp_forward(q, feat, n, out, s);
    const int r = mlp_forward(q, feat, n, q->y, s);
    if (r) return r;
    return cudaMemcpyAsync(out, q->y, ob, cudaMemcpyDeviceToDevice, s) == cudaSuccess ? VOF_OK : VOF_ERR_CUDA;
}

int vof_mlp_gradient(vof_mlp *q, const float *feat, const float *target, int n, float *grad, float *loss,
                     void *stream)
{
    if (!q || !feat || !target || n < 1 || n > q->max_batch) return VOF_ERR_INVALID_ARG;
    if (cudaSetDevice(q->device) != cudaSuccess) return VOF_ERR_CUDA;
    cudaStream_t s = (cudaStream_t)stream;
    const int r = mlp_gradient(q, feat, target, n, grad, loss != nullptr, s);
    if (r) return r;
    if (loss) {
        if (cudaStreamSynchronize(s) != cudaSuccess) return VOF_ERR_CUDA;
        *loss = *static_cast<volatile float *>(q->h_loss) / (float)n;
    }
    return VOF_OK;
}

int vof_mlp_train_step(vof_mlp *q, const float *feat, const float *target, int n, float lr, float *loss,
                       void *stream)
{
    int r = vof_mlp_gradient(q, feat, target, n, nullptr, loss, stream);
    if (r) return r;
    cudaStream_t s = (cudaStream_t)stream;
    ++q->adam_t;
    const float c1 = 1.0f - powf(0.9f, (float)q->adam_t), c2 = 1.0f - powf(0.999f, (float)q->adam_t);
    k_mlp_adam<<<cdiv(NPARAM, 256), 256, 0, s>>>(q->p, q->grad, q->m1, q->m2, lr, c1, c2);
    return mlp_pack(q, s);
}

int vof_set_guess(vof_ctx *c, vof_mlp *q)
{
    if (!c) return VOF_ERR_INVALID_ARG;
    if (cudaSetDevice(c->device) != cudaSuccess) return VOF_ERR_CUDA;
    if (q && q->device != c->device) return VOF_ERR_INVALID_ARG;
    // (a buffer that cannot be had leaves the context as it was: the network
    // attached before keeps its own)
    auto get = [](void **p, size_t bytes) {
        if (cudaMalloc(p, bytes) == cudaSuccess) return true;
        cudaGetLastError();
        return false;
    };
    if (q && !c->mlp_nbr) {
        void *nbr = nullptr, *geo = nullptr;
        if (!get(&nbr, sizeof(int) * 27 * (size_t)c->nc) || !get(&geo, sizeof(float) * 6 * (size_t)c->nc)) {
            cudaFree(nbr);
            return VOF_ERR_CUDA;
        }
        c->mlp_nbr = static_cast<int *>(nbr);
        c->mlp_geo = static_cast<float *>(geo);
        k_mlp_tables<<<cdiv(c->nc, 128), 128>>>(c->m, c->mlp_nbr, c->mlp_geo);
        if (cudaDeviceSynchronize() != cudaSuccess) return VOF_ERR_CUDA;
    }
    if (q && c->mlp_s0_cap < q->max_batch) {
        // offsets for the network's batch (kept until vof_destroy)
        void *s0 = nullptr;
        if (!get(&s0, sizeof(float) * (size_t)q->max_batch)) return VOF_ERR_CUDA;
        cudaFree(c->mlp_s0);
        c->mlp_s0 = static_cast<float *>(s0);
        c->mlp_s0_cap = q->max_batch;
    }
    ++c->cfg_gen;  // (also for the same network again: its weights or buffers may be new ones)
    c->mlp = q;
    return VOF_OK;
}

}  // extern "C"
