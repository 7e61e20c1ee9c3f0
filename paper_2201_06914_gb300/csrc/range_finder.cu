// Range-finder probes on the device (Sec. 2.1): [Q, ~] = qr(A Z) with A = (D D^T)^p, the
// power-iteration form of the randomized range finder, for a batch of shots.
//
// D is an nt x ncols matrix per shot (or one shared by all shots): the shot's data
// (ncols = receivers) or the causal convolution matrix of the source wavelet (ncols = nt),
// the two readings of A this library offers.  The two products of each power step,
// T = D^T Y and Y = D T, run on the tensor-core probe contraction (probe_pipe.cu); this
// file holds what is left: a tiled transpose and a thin QR by classical Gram-Schmidt with
// one full reorthogonalisation (CGS2) in FP64, one cluster of CTAs per shot.  CGS2 gives Q orthonormal
// to working precision for any numerically full-rank Y and the positive diagonal of R
// (the sign convention of the oracle's qr).  Y is re-orthonormalised after every power
// step; in exact arithmetic that leaves the final Q unchanged (the intermediate R factors
// only multiply the sketch from the right by triangular matrices with positive diagonals).
#include <cooperative_groups.h>

#include "qr_plan.cuh"
#include "wp_internal.cuh"

namespace wp {

// out[s][c][r] = in[s][r][c] for an R x C matrix per shot (32 x 32 tiles through shared
// memory, both sides coalesced).
__global__ void transpose_kernel(const float *__restrict__ in, long long in_ss, int R, int C,
                                 float *__restrict__ out, long long out_ss)
{
    __shared__ float tile[32][33];
    const long long s = blockIdx.z;
    const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
    const float *src = in + s * in_ss;
    float *dst = out + s * out_ss;
    for (int k = threadIdx.y; k < 32; k += blockDim.y) {
        const int r = r0 + k, c = c0 + threadIdx.x;
        if (r < R && c < C) tile[k][threadIdx.x] = src[(long long)r * C + c];
    }
    __syncthreads();
    for (int k = threadIdx.y; k < 32; k += blockDim.y) {
        const int c = c0 + k, r = r0 + threadIdx.x;
        if (r < R && c < C) dst[(long long)c * R + r] = tile[threadIdx.x][k];
    }
}

cudaError_t launch_transpose(const float *in, long long in_ss, int R, int C, int nmat, float *out,
                             long long out_ss, cudaStream_t s)
{
    dim3 grid((C + 31) / 32, (R + 31) / 32, nmat);
    transpose_kernel<<<grid, dim3(32, 8), 0, s>>>(in, in_ss, R, C, out, out_ss);
    count_launch();
    return cudaGetLastError();
}

// Thin QR of Y (nt x r per shot, given column-major as Yt[s][i][t]) by CGS2 in FP64.  Writes
// Q[s][t][i] (row-major, the probe layout) and raises *err (value 3) when a column has no
// component left outside the span of the previous ones (a rank-deficient sketch); that column is
// written as zero.
//
// What bounds it: FP64 arithmetic, 2 r^2 nt multiply-adds per shot at the two an SM starts per
// clock, and a chain of 2 r reductions.  A cluster of CTAs therefore shares a shot: each keeps
// `rows` of the nt rows in shared memory (or, where they do not fit, in its part of W), computes
// their share of every dot product and reads the others' shares through distributed shared
// memory, in rank order; one cluster barrier per pass.  Columns stay unnormalised until the end:
// a column's squared norm is one more dot product of the next column's first pass, so it costs
// no reduction of its own.  16 shots of 2000 x 64: 1.14 ms in clusters of six (5.0 ms with one
// CTA per shot, 2.7 ms in clusters of eight that ran in two rounds and reduced through shuffles);
// one shot 0.9 ms.
__global__ void __launch_bounds__(QR_THREADS) cgs2_qr_kernel(const float *__restrict__ Yt, int nt, int r, int rows,
                                                             bool in_smem, double *__restrict__ W,
                                                             float *__restrict__ Q, int *err)
{
    namespace cg = cooperative_groups;
    extern __shared__ double qr_smem[];
    double *part = qr_smem;                          // [2][QR_MAXR + 1] this CTA's dot products
    double *coef = part + 2 * (QR_MAXR + 1);         // [QR_MAXR] projections onto the previous columns
    double *inv2 = coef + QR_MAXR;                   // [QR_MAXR] 1 / squared norm (0 for a zero column)
    double *psum = inv2 + QR_MAXR;                   // [QR_THREADS]
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const long long s = blockIdx.x / C;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = QR_THREADS / 32;
    const int t0 = min(rank * rows, nt), n = min(rows, nt - t0);   // rows t0 .. t0 + n - 1
    const float *Ys = Yt + s * (long long)nt * r + t0;
    double *w = in_smem ? psum + QR_THREADS : W + s * (long long)nt * r + t0;
    const long long ld = in_smem ? rows | 1 : nt;   // odd: 32 columns of a row in different banks
    for (int i = warp; i < r; i += nw)
        for (int t = lane; t < n; t += 32) w[i * ld + t] = (double)Ys[(long long)i * nt + t];
    __syncthreads();
    int buf = 0;
    // dot product i of part[buf] summed over the cluster in rank order
    auto total = [&](int i) {
        double x[8], v = 0.0;
#pragma unroll
        for (int k = 0; k < 8; k++) x[k] = k < C ? cl.map_shared_rank(part, k)[buf * (QR_MAXR + 1) + i] : 0.0;
#pragma unroll
        for (int k = 0; k < 8; k++) v += x[k];
        return v;
    };
    // Dot products of column j with the previous ones and, if `norm`, of column j - 1 with itself,
    // summed over the cluster: coef and inv2.  A thread owns one product and one of `sl` slices
    // of the rows (no shuffles: a 32-lane tree would add 160 FP64 additions to the 250 or so
    // multiply-adds of a product).  The barrier also orders the two buffers: a CTA reaches the
    // next one only after it has read this one's, and writes it two steps later.
    auto project = [&](int j, bool norm) {
        const double *wj = w + j * ld, *wl = w + (j - 1) * ld;
        const int m = j + (norm ? 1 : 0), P = (m + 31) & ~31, sl = max(1, QR_THREADS / P);
        for (int i0 = 0; i0 < m; i0 += QR_THREADS) {   // one round up to 512 products
            const int i = i0 + tid % P, k = tid / P;
            double acc = 0.0;
            if (k < sl && i < m) {
                const double *a = i < j ? w + i * ld : wl, *b = i < j ? wj : wl;
                for (int t = k; t < n; t += sl) acc = fma(a[t], b[t], acc);
            }
            psum[tid] = acc;
            __syncthreads();
            if (tid < P && i < m) {
                for (int q = 1; q < sl; q++) acc += psum[q * P + tid];
                part[buf * (QR_MAXR + 1) + i] = acc;
            }
        }
        cl.sync();
        for (int i = tid; i < j; i += QR_THREADS) {
            if (norm && i == j - 1) {
                const double n2 = total(j);
                inv2[i] = n2 > 0.0 ? 1.0 / n2 : 0.0;
            }
            coef[i] = total(i) * inv2[i];
        }
        __syncthreads();
        buf ^= 1;
    };
    // threads per row: the block covers min(n, 512) rows, `split` threads to a row
    const int R = min(QR_THREADS, max(32, (n + 31) & ~31)), split = QR_THREADS / R, sp = tid / R, tr = tid - sp * R;
    for (int j = 1; j < r; j++) {
        double *wj = w + j * ld;
        for (int pass = 0; pass < 2; pass++) {
            project(j, pass == 0);
            for (int tb = 0; tb < n; tb += R) {
                const int t = tb + tr;
                double v = 0.0;
                if (sp < split && t < n)
                    for (int i = sp; i < j; i += split) v = fma(coef[i], w[i * ld + t], v);
                if (split > 1) {
                    psum[tid] = v;
                    __syncthreads();
                    if (sp == 0)
                        for (int k = 1; k < split; k++) v += psum[k * R + tr];
                }
                if (sp == 0 && t < n) wj[t] -= v;
                __syncthreads();
            }
        }
    }
    // the last column's norm: its product with itself as "column r" (only the norm is used)
    if (warp == 0) {
        const double *wl = w + (r - 1) * ld;
        double acc = 0.0;
        for (int t = lane; t < n; t += 32) acc = fma(wl[t], wl[t], acc);
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lane == 0) part[buf * (QR_MAXR + 1)] = acc;
    }
    cl.sync();
    if (tid == 0) {
        const double n2 = total(0);
        inv2[r - 1] = n2 > 0.0 ? 1.0 / n2 : 0.0;
    }
    __syncthreads();
    for (int i = tid; i < r; i += QR_THREADS) {
        coef[i] = sqrt(inv2[i]);
        if (rank == 0 && !(inv2[i] > 0.0)) atomicExch(err, 3);
    }
    __syncthreads();
    float *Qs = Q + s * (long long)nt * r + (long long)t0 * r;
    for (int k = tid; k < n * r; k += QR_THREADS) {
        const int t = k / r, i = k - t * r;
        Qs[k] = (float)(w[i * ld + t] * coef[i]);
    }
    cl.sync();   // no CTA leaves while another may still read its partial sums
}

cudaError_t launch_cgs2_qr(const float *Yt, int nt, int r, int nshots, double *W, float *Q, int *err,
                           cudaStream_t s)
{
    if (r > QR_MAXR) return cudaErrorInvalidValue;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(QR_THREADS);
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaError_t e = cudaFuncSetAttribute(cgs2_qr_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)QR_SMEM);
    if (e != cudaSuccess) return e;
    auto shape = [&](int c, size_t smem) {
        cfg.dynamicSmemBytes = smem;
        cfg.gridDim = dim3((unsigned)(nshots * c));
        at.val.clusterDim.x = c;
    };
    const int C = qr_cluster(nt, r, nshots, [&](int c, bool in_smem) {
        shape(c, in_smem ? QR_SMEM : QR_HEAD);   // all of an SM's shared memory: one CTA an SM
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, cgs2_qr_kernel, &cfg) != cudaSuccess) {
            (void)cudaGetLastError();
            return 0;
        }
        return n;
    });
    const int rows = (nt + C - 1) / C;
    const size_t smem = qr_rows_smem(nt, r, C);
    shape(C, smem ? smem : QR_HEAD);
    e = cudaLaunchKernelEx(&cfg, cgs2_qr_kernel, Yt, nt, r, rows, smem > 0, W, Q, err);
    if (e != cudaSuccess) return e;
    count_launch();
    return cudaGetLastError();
}

}  // namespace wp
