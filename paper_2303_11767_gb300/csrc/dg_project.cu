// dg_project.cu -- cos(theta)-weighted L2 projection of point values onto the
// modal basis of a sphere mesh: the nm x nm values of an element and field are
// contracted over the lambda points, then over the theta points weighted by
// cos(theta), then multiplied by the row's inverse mass matrix, in FP64 and in
// that order of sums.
//
// The values arrive from host memory, 8 nm^2 bytes for 8 n^2 of result, so the
// copy bounds it (180x90 degree 3: 56 MB, 0.33 ms at 170 GB/s); one host thread
// took 14.4 ms for the sums.
#include <cuda_runtime.h>

#include "dg_internal.h"

namespace {

constexpr int PT = 128;   // threads of a block
constexpr int PE = 8;     // (element, field) pairs of a block

// pl: [n][nm] w_q L_a(x_q); cosm: [rows][nm] cos(theta) at the points of the
// mesh rows from the first; v: the values of npairs pairs from pair p0 of the
// mesh on, of 3 per element and 3 nlon per row
template <int N>
__global__ void __launch_bounds__(PT) project_kernel(const double *__restrict__ v, size_t p0, int npairs, int nlon, int nm,
                                                     const double *__restrict__ pl, const double *__restrict__ cosm,
                                                     const RowTab<double> *__restrict__ rows, double *__restrict__ out)
{
    constexpr int QM = DG_MAXN + 8, NP = N * N;   // most points per direction
    __shared__ double sv[PE * QM * QM], ss[PE * QM * N], sr[PE * NP], spl[N * QM];
    const int tid = threadIdx.x, nq = nm * nm;
    const int b0 = blockIdx.x * PE, np = min(PE, npairs - b0);
    for (int t = tid; t < N * nm; t += PT) spl[t] = pl[t];
#pragma unroll 4
    for (int t = tid; t < np * nq; t += PT) sv[t] = __ldg(v + (size_t)b0 * nq + t);
    __syncthreads();
    for (int t = tid; t < np * nm; t += PT) {   // (pair, theta point): its N sums over the lambda points
        const double *row = sv + (size_t)t * nm;
        double acc[N];
#pragma unroll
        for (int a = 0; a < N; ++a) acc[a] = 0.0;
        for (int q = 0; q < nm; ++q) {
            const double x = row[q];
#pragma unroll
            for (int a = 0; a < N; ++a) acc[a] = fma(spl[a * nm + q], x, acc[a]);
        }
#pragma unroll
        for (int a = 0; a < N; ++a) ss[t * N + a] = acc[a];
    }
    __syncthreads();
    for (int t = tid; t < np * NP; t += PT) {   // (pair, b, a): the sum over the theta points
        const int pr = t / NP, m = t - pr * NP, b = m / N, a = m - b * N;
        const size_t j = (p0 + b0 + pr) / ((size_t)3 * nlon);
        double acc = 0.0;
        for (int q = 0; q < nm; ++q) acc = fma(spl[b * nm + q] * __ldg(cosm + j * nm + q), ss[(pr * nm + q) * N + a], acc);
        sr[t] = acc;
    }
    __syncthreads();
    for (int t = tid; t < np * NP; t += PT) {
        const int pr = t / NP, m = t - pr * NP, b = m / N, a = m - b * N;
        const size_t j = (p0 + b0 + pr) / ((size_t)3 * nlon);
        double acc = 0.0;
#pragma unroll
        for (int c = 0; c < N; ++c) acc = fma(__ldg(&rows[j].Ci[b][c]), sr[pr * NP + c * N + a], acc);
        out[(p0 + b0) * NP + t] = acc;
    }
}

}  // namespace

int dg_launch_project(int n, const double *v, size_t pair0, int npairs, int nlon, int nm, const double *pl, const double *cosm,
                      const RowTab<double> *rows, double *out, void *stream)
{
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int blocks = (npairs + PE - 1) / PE;
    switch (n) {
    case 1: project_kernel<1><<<blocks, PT, 0, s>>>(v, pair0, npairs, nlon, nm, pl, cosm, rows, out); break;
    case 2: project_kernel<2><<<blocks, PT, 0, s>>>(v, pair0, npairs, nlon, nm, pl, cosm, rows, out); break;
    case 3: project_kernel<3><<<blocks, PT, 0, s>>>(v, pair0, npairs, nlon, nm, pl, cosm, rows, out); break;
    case 4: project_kernel<4><<<blocks, PT, 0, s>>>(v, pair0, npairs, nlon, nm, pl, cosm, rows, out); break;
    case 5: project_kernel<5><<<blocks, PT, 0, s>>>(v, pair0, npairs, nlon, nm, pl, cosm, rows, out); break;
    default: return 1;
    }
    return cudaPeekAtLastError() == cudaSuccess ? 0 : 1;
}
