// dg_mlp_fused.cuh -- the network of the learned correction (60-128-128-12 and
// the like: up to 64 inputs, 128 hidden units, up to 16 outputs) with a whole
// sample tile's forward and backward pass in one block.  Included by dg_mlp.cu.
//
// What bounds it and why this shape.  The layers are small (25 868 parameters,
// 0.31 GFMA for a training step of 4096 samples: 8 us of the FP32 pipe), so
// layer-by-layer GEMMs spend their time on launches of a few blocks and on
// uncoalesced operand reads.  Here a block of 256 threads keeps the
// activations of 32 samples in shared memory from the first layer to the
// weight gradients; the weights come from a 16-bit copy stored in the order of
// use (k-major, refreshed with the parameters), so that every load of it is
// contiguous.  A thread owns 4 samples x 4 units of a layer, and 8 x 8 of a
// weight gradient, whose sum over the block's samples runs on paired FP32
// instructions (even and odd samples).  The blocks' partial gradients are
// summed in block order by one kernel, which also takes the Adam step.
// Training step of 4096 samples, host call included: 2010 -> 70 us.
#pragma once

namespace {

constexpr int FH = 128;      // hidden units
constexpr int FIN = 64;      // most inputs
constexpr int FOUT = 16;     // most outputs
constexpr int FS = 32;       // samples of a block
constexpr int FLD = FS + 4;  // stride of one unit's samples: 9 16-byte blocks, an odd number
constexpr int FMAXB = MAXB / FS;

// shared memory of the training block, in floats
constexpr int F_W2 = 0;                       // W2^T [k][u], then W2 [u][k]
constexpr int F_W1 = F_W2 + FH * FH;          // W1^T [k][u]
constexpr int F_W3T = F_W1 + FIN * FH;        // W3^T [k][16]
constexpr int F_W3 = F_W3T + FH * FOUT;       // W3 [o][k]
constexpr int F_X = F_W3 + FOUT * FH;         // inputs [k][samples]
constexpr int F_A1 = F_X + FIN * FLD;
constexpr int F_G1 = F_A1 + FH * FLD;         // gelu' of layer 1, then dZ1
constexpr int F_A2 = F_G1 + FH * FLD;
constexpr int F_G2 = F_A2 + FH * FLD;         // gelu' of layer 2, then dZ2
constexpr int F_DY = F_G2 + FH * FLD;
constexpr int F_LEN = F_DY + FOUT * FLD;
constexpr size_t F_BYTES = sizeof(float) * F_LEN;
static_assert(F_BYTES <= 227 * 1024, "shared memory of one block");

// 16-bit weights in the order of use: W1^T [k][128], W2^T [k][128], W3^T [k][16]
// (zero padded), W2 [u][128], W3 [o][128]
constexpr size_t T_W1 = 0, T_W2T = T_W1 + (size_t)FIN * FH, T_W3T = T_W2T + (size_t)FH * FH,
                 T_W2 = T_W3T + (size_t)FH * FOUT, T_W3 = T_W2 + (size_t)FH * FH, T_LEN = T_W3 + (size_t)FOUT * FH;

// positions of parameter t in the transposed copy (second = -1: only one)
__device__ __forceinline__ void fused_places(size_t t, int nin, int nout, long long &a, long long &b)
{
    const size_t ob1 = (size_t)FH * nin, oW2 = ob1 + FH, ob2 = oW2 + (size_t)FH * FH, oW3 = ob2 + FH, ob3 = oW3 + (size_t)nout * FH;
    a = b = -1;
    if (t < ob1) {
        a = T_W1 + (t % nin) * FH + t / nin;
    } else if (t >= oW2 && t < ob2) {
        const size_t r = t - oW2;
        a = T_W2T + (r % FH) * FH + r / FH;
        b = T_W2 + r;
    } else if (t >= oW3 && t < ob3) {
        const size_t r = t - oW3;
        a = T_W3T + (r % FH) * FOUT + r / FH;
        b = T_W3 + r;
    }
}

__global__ void fused_weights_kernel(const float *__restrict__ w, __nv_bfloat16 *__restrict__ wt, int nin, int nout, size_t np)
{
    for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < np; t += (size_t)gridDim.x * blockDim.x) {
        long long a, b;
        fused_places(t, nin, nout, a, b);
        const __nv_bfloat16 v = __float2bfloat16_rn(w[t]);
        if (a >= 0) wt[a] = v;
        if (b >= 0) wt[b] = v;
    }
}

// n (a multiple of 8) 16-bit weights to FP32 in shared memory, by a block of NT
// threads
template <int NT>
__device__ __forceinline__ void fused_load(float *dst, const __nv_bfloat16 *__restrict__ src, int n)
{
    constexpr int BATCH = 8;   // loads of a thread in flight together
#pragma unroll 1
    for (int v0 = threadIdx.x; v0 < n / 8; v0 += BATCH * NT) {
        uint4 r[BATCH];
#pragma unroll
        for (int i = 0; i < BATCH; ++i)
            if (v0 + i * NT < n / 8) r[i] = __ldg(reinterpret_cast<const uint4 *>(src) + v0 + i * NT);
#pragma unroll
        for (int i = 0; i < BATCH; ++i) {
            if (v0 + i * NT >= n / 8) break;
            const uint4 u = r[i];
            float4 *d = reinterpret_cast<float4 *>(dst) + 2 * (v0 + i * NT);
            d[0] = make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16),
                               __uint_as_float(u.y & 0xffff0000u));
            d[1] = make_float4(__uint_as_float(u.z << 16), __uint_as_float(u.z & 0xffff0000u), __uint_as_float(u.w << 16),
                               __uint_as_float(u.w & 0xffff0000u));
        }
    }
}

// acc[i][j] = sum_k A[k][s + i] W[k][u + j], k ascending (s, u: the thread's
// first sample and unit; A has LD samples a row, W 128 units)
template <int LD>
__device__ __forceinline__ void fused_gemm(const float *A, const float *W, int K, int s, int u, float (*acc)[4])
{
    float2 c[4][2];
#pragma unroll
    for (int i = 0; i < 4; ++i) c[i][0] = c[i][1] = make_float2(0.f, 0.f);
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
        const float4 a = *reinterpret_cast<const float4 *>(A + k * LD + s);
        const float4 w = *reinterpret_cast<const float4 *>(W + k * FH + u);
        const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            c[i][0] = __ffma2_rn(make_float2(av[i], av[i]), make_float2(w.x, w.y), c[i][0]);
            c[i][1] = __ffma2_rn(make_float2(av[i], av[i]), make_float2(w.z, w.w), c[i][1]);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i][0] = c[i][0].x, acc[i][1] = c[i][0].y, acc[i][2] = c[i][1].x, acc[i][3] = c[i][1].y;
}

// activation and its derivative of one layer's 4 x 4 values, to [unit][sample]
template <int LD, bool GRAD>
__device__ __forceinline__ void fused_gelu(const float (*z)[4], const float *__restrict__ bias, int s, int u, float *A, float *G)
{
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const float b = __ldg(bias + u + j);
        float a[4], g[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float x = z[i][j] + b;
            const float c = 0.5f * (1.0f + erff(x * 0.70710678118654752f));
            a[i] = x * c;
            if (GRAD) g[i] = c + x * 0.39894228040143268f * expf(-0.5f * x * x);
        }
        *reinterpret_cast<float4 *>(A + (u + j) * LD + s) = make_float4(a[0], a[1], a[2], a[3]);
        if (GRAD) *reinterpret_cast<float4 *>(G + (u + j) * LD + s) = make_float4(g[0], g[1], g[2], g[3]);
    }
}

// G[u][s] *= acc (dZ from dA and the activation's derivative)
__device__ __forceinline__ void fused_dz(const float (*acc)[4], int s, int u, float *G)
{
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float4 *p = reinterpret_cast<float4 *>(G + (u + j) * FLD + s);
        float4 g = *p;
        g.x *= acc[0][j], g.y *= acc[1][j], g.z *= acc[2][j], g.w *= acc[3][j];
        *p = g;
    }
}

// out[u][i] = sum_s dZ[u][s] X[i][s] for rows u < FH and i < ni (i in steps of
// 16 from the thread's), out row-major with ld columns
template <int NI>
__device__ __forceinline__ void fused_wgrad(const float *dZ, const float *X, int ni, float *__restrict__ out, int ld)
{
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    float2 c[8][NI];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < NI; ++j) c[i][j] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int s = 0; s < FS; s += 4) {
        float4 a[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) a[i] = *reinterpret_cast<const float4 *>(dZ + (ty + 16 * i) * FLD + s);
#pragma unroll
        for (int j = 0; j < NI; ++j) {
            const float4 x = *reinterpret_cast<const float4 *>(X + (tx + 16 * j) * FLD + s);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                c[i][j] = __ffma2_rn(make_float2(a[i].x, a[i].y), make_float2(x.x, x.y), c[i][j]);
                c[i][j] = __ffma2_rn(make_float2(a[i].z, a[i].w), make_float2(x.z, x.w), c[i][j]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < NI; ++j)
            if (tx + 16 * j < ni) out[(size_t)(ty + 16 * i) * ld + tx + 16 * j] = c[i][j].x + c[i][j].y;
}

// Forward (and with GRAD backward) of samples [32 b, 32 b + 32) of a batch in
// block b: normalised outputs to y, or the block's partial gradients (layout
// of the parameters) and its squared error.
template <bool GRAD>
__global__ void __launch_bounds__(256, 1) fused_mlp_kernel(const float *__restrict__ x, const float *__restrict__ t, int batch,
                                                           int nin, int nout, const __nv_bfloat16 *__restrict__ wt,
                                                           const float *__restrict__ w, const float *__restrict__ norm,
                                                           float *__restrict__ y, float *__restrict__ part, size_t np,
                                                           double *__restrict__ lpart)
{
    extern __shared__ __align__(16) float fsm[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int s = 4 * (lane & 7), u = 4 * (4 * warp + (lane >> 3));
    const int b0 = blockIdx.x * FS, nb = min(FS, batch - b0);
    const size_t ob1 = (size_t)FH * nin, oW2 = ob1 + FH, ob2 = oW2 + (size_t)FH * FH, oW3 = ob2 + FH, ob3 = oW3 + (size_t)nout * FH;
    const float *const out_mean = norm + 2 * nin, *const out_std = out_mean + nout;
    fused_load<256>(fsm + F_W1, wt + T_W1, nin * FH);
    fused_load<256>(fsm + F_W2, wt + T_W2T, FH * FH);
    fused_load<256>(fsm + F_W3T, wt + T_W3T, FH * FOUT);
    if (GRAD) fused_load<256>(fsm + F_W3, wt + T_W3, FOUT * FH);
    {   // normalised inputs, the loads of a thread in flight together
        constexpr int IT = FS * FIN / 256;
        float xv[IT];
#pragma unroll
        for (int i = 0; i < IT; ++i) {
            const int v = tid + 256 * i;
            xv[i] = v < nb * nin ? __ldg(x + (size_t)b0 * nin + v) : 0.0f;
        }
#pragma unroll
        for (int i = 0; i < IT; ++i) {
            const int v = tid + 256 * i, r = v / nin, c = v - r * nin;
            if (v < FS * nin) fsm[F_X + c * FLD + r] = r < nb ? (xv[i] - __ldg(norm + c)) / __ldg(norm + nin + c) : 0.0f;
        }
    }
    __syncthreads();
    float acc[4][4];
    fused_gemm<FLD>(fsm + F_X, fsm + F_W1, nin, s, u, acc);
    fused_gelu<FLD, GRAD>(acc, w + ob1, s, u, fsm + F_A1, fsm + F_G1);
    __syncthreads();
    fused_gemm<FLD>(fsm + F_A1, fsm + F_W2, FH, s, u, acc);
    fused_gelu<FLD, GRAD>(acc, w + ob2, s, u, fsm + F_A2, fsm + F_G2);
    __syncthreads();
    if (GRAD) fused_load<256>(fsm + F_W2, wt + T_W2, FH * FH);
    // outputs: sample = lane, outputs warp and warp + 8
    {
        float o0 = 0.f, o1 = 0.f;
#pragma unroll 8
        for (int k = 0; k < FH; ++k) {
            const float a = fsm[F_A2 + k * FLD + lane];
            o0 = fmaf(a, fsm[F_W3T + k * FOUT + warp], o0);
            o1 = fmaf(a, fsm[F_W3T + k * FOUT + warp + 8], o1);
        }
        double err = 0.0;
        const float scale = 2.0f / (float)((size_t)batch * nout);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int o = warp + 8 * h;
            float dy = 0.0f;
            if (o < nout && lane < nb) {
                const float v = (h ? o1 : o0) + __ldg(w + ob3 + o);
                const size_t at = (size_t)(b0 + lane) * nout + o;
                if (GRAD) {
                    const float d = v - (t[at] - out_mean[o]) / out_std[o];
                    dy = scale * d;
                    err += (double)d * d;
                } else {
                    y[at] = v;
                }
            }
            if (GRAD) fsm[F_DY + o * FLD + lane] = dy;
        }
        if (!GRAD) return;
        __shared__ double red[8];
        for (int m = 16; m > 0; m >>= 1) err += __shfl_xor_sync(0xffffffffu, err, m);
        if (lane == 0) red[warp] = err;
        __syncthreads();
        if (tid == 0) {
            double e = 0.0;
            for (int i = 0; i < 8; ++i) e += red[i];
            lpart[blockIdx.x] = e;
        }
    }
    float *const g = part + (size_t)blockIdx.x * np;
    // layer 3: dA2 = dY W3, dZ2; its weight and bias gradients
    fused_gemm<FLD>(fsm + F_DY, fsm + F_W3, nout, s, u, acc);
    fused_dz(acc, s, u, fsm + F_G2);
    {
        const int c = tid & 127, o0 = (tid >> 7) * 8;
        float a3[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) a3[i] = 0.f;
#pragma unroll 2
        for (int q = 0; q < FS; q += 4) {
            const float4 a = *reinterpret_cast<const float4 *>(fsm + F_A2 + c * FLD + q);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float4 d = *reinterpret_cast<const float4 *>(fsm + F_DY + (o0 + i) * FLD + q);
                a3[i] = fmaf(d.w, a.w, fmaf(d.z, a.z, fmaf(d.y, a.y, fmaf(d.x, a.x, a3[i]))));
            }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (o0 + i < nout) g[oW3 + (size_t)(o0 + i) * FH + c] = a3[i];
    }
    __syncthreads();
    // layer 2: dA1 = dZ2 W2, dZ1; layer 2's weight gradient
    fused_gemm<FLD>(fsm + F_G2, fsm + F_W2, FH, s, u, acc);
    fused_dz(acc, s, u, fsm + F_G1);
    fused_wgrad<8>(fsm + F_G2, fsm + F_A1, FH, g + oW2, FH);
    __syncthreads();
    // layer 1's weight gradient, and the bias gradients
    fused_wgrad<4>(fsm + F_G1, fsm + F_X, nin, g, nin);
    for (int v = tid; v < 2 * FH + nout; v += 256) {
        const float *r = fsm + (v < FH ? F_G1 + v * FLD : v < 2 * FH ? F_G2 + (v - FH) * FLD : F_DY + (v - 2 * FH) * FLD);
        float sum = 0.f;
#pragma unroll
        for (int q = 0; q < FS; q += 4) {
            const float4 d = *reinterpret_cast<const float4 *>(r + q);
            sum += d.x;
            sum += d.y;
            sum += d.z;
            sum += d.w;
        }
        g[v < FH ? ob1 + v : v < 2 * FH ? ob2 + v - FH : ob3 + v - 2 * FH] = sum;
    }
}

// Gradient = the blocks' partials summed in block order (in four consecutive
// quarters); with ADAM also the optimiser step and the refreshed 16-bit copies.
// Block 0 sums the squared errors.
template <bool ADAM>
__global__ void __launch_bounds__(256) fused_reduce_kernel(const float *__restrict__ part, const double *__restrict__ lpart, int nblocks,
                                                           size_t np, int nin, int nout, float *__restrict__ g, double *__restrict__ lsum,
                                                           float *__restrict__ w, float *__restrict__ m, float *__restrict__ v,
                                                           __nv_bfloat16 *__restrict__ wb, __nv_bfloat16 *__restrict__ wt, float lr,
                                                           float b1, float b2, float eps, float c1, float c2)
{
    __shared__ float q[4][64];
    const int tx = threadIdx.x & 63, seg = threadIdx.x >> 6;
    const size_t i = blockIdx.x * (size_t)64 + tx;
    const int per = (nblocks + 3) / 4, lo = seg * per, hi = min(nblocks, lo + per);
    float s = 0.f;
    if (i < np) {
#pragma unroll 16
        for (int b = lo; b < hi; ++b) s += __ldg(part + (size_t)b * np + i);
    }
    q[seg][tx] = s;
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x == 64) {
        double l = 0.0;
        for (int b = 0; b < nblocks; ++b) l += lpart[b];
        *lsum = l;
    }
    if (seg || i >= np) return;
    const float gi = ((q[0][tx] + q[1][tx]) + q[2][tx]) + q[3][tx];
    g[i] = gi;
    if (!ADAM) return;
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    w[i] = wi;
    const __nv_bfloat16 h = __float2bfloat16_rn(wi);
    wb[i] = h;
    long long a, b;
    fused_places(i, nin, nout, a, b);
    if (a >= 0) wt[a] = h;
    if (b >= 0) wt[b] = h;
}

}  // namespace
