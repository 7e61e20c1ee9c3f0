// Probe accumulation on the tensor cores (Eq. 3) for operands of any alignment: for a block of
// time steps given as rows of N points,
//   P[i][x] += scale * sum_t A[t][x] * Q[t0 + t][i]
// an [N x cnt] . [cnt x r] contraction per shot (wp_probe_accumulate on row lengths that no
// tensor map covers, wp_probe_accumulate_static, the two products of the range finder).  A is
// split into bfloat16 hi + lo in registers and stored in the K-major 128-byte-swizzled layout
// that tcgen05.mma reads; the probes arrive as swizzled hi/lo images (launch_probe_images).
// Four bf16 products (hi*hi, lo*hi, hi*lo, lo*lo) accumulate in FP32 in tensor memory, which
// keeps the contraction faithful to FP32 (relative error ~2^-17) for any probe matrix; the two
// with the probes' lo part are skipped when it is all zero (Rademacher).  One CTA owns 128 grid
// points (M = 128) and all r probes (N = r rounded up to 16); K runs over the block in chunks of
// 64 time steps.
//
// What bounds it: the latency of its 4-byte loads (rows may start at any 4-byte boundary).  A
// thread has all 64 loads of its column's next chunk in flight while the current one is
// multiplied, bulk copies bring the probe images, and three or four CTAs per SM are in different
// phases.  16 shots of 281 x 281 points, 256 steps, r = 64: 494 us = 3.9 TB/s of its bytes
// (939 us with index multiplies and predicates on every load, the image copied by the threads
// after it, P read one value at a time).
#include <algorithm>

#include "wp_internal.cuh"

namespace wp {

constexpr int KCH = 64;  // time steps per K chunk: one 128-byte swizzle row of bf16

__host__ __device__ inline uint32_t tmem_cols_for(int r_pad)
{
    uint32_t c = 32;
    while (c < (uint32_t)r_pad) c <<= 1;
    return c;
}

__global__ void __launch_bounds__(128, 4) probe_gemm_kernel(const GemmArgs A)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);   // stays a shared pointer
    uint8_t *a_hi = smem;
    uint8_t *a_lo = smem + 16384;
    uint8_t *b_hi = smem + 32768;
    __shared__ uint64_t mma_bar, img_bar[2];
    __shared__ uint32_t tmem_holder;

    const int tile = blockIdx.x, shot = blockIdx.y, m = threadIdx.x, warp = m >> 5;
    const long long p = (long long)tile * 128 + m, N = A.N;
    const bool valid = p < N;
    const uint32_t ncols = tmem_cols_for(A.r_pad);
    const uint32_t img_bytes = (uint32_t)A.r_pad * 128u;
    uint8_t *b_lo = b_hi + img_bytes;
    const bool qlo = *(volatile const int *)A.lo_nz != 0;   // written before this launch

    if (warp == 0) tmem_alloc(&tmem_holder, ncols);
    if (m == 0) {
        mbar_init(&mma_bar, 1);
        mbar_init(&img_bar[0], 1);
        mbar_init(&img_bar[1], 1);
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_holder;

    const float *col = A.a + (long long)shot * A.a_ss + (valid ? p : 0);
    const uint32_t idesc = idesc_bf16_f32(128, A.r_pad);
    const int nchunks = (A.cnt + KCH - 1) / KCH;
    bool failed = false;   // a wait of this thread gave up; the block votes and stops together
    bool stop = false;
    // Image of chunk c into its buffer: without the lo part the two buffers alternate and a copy
    // runs one chunk ahead; with it they hold one chunk's hi and lo.
    int issued = 0;        // images whose copy thread 0 has started
    auto issue_img = [&](int c) {
        if (m != 0 || c >= nchunks) return;
        const long long im = ((long long)shot * nchunks + c) * A.img_ld;
        uint64_t *bar = &img_bar[c & 1];
        mbar_arrive_expect_tx(bar, qlo ? 2u * img_bytes : img_bytes);
        bulk_g2s(!qlo && (c & 1) ? b_lo : b_hi, A.img_hi + im, img_bytes, bar);
        if (qlo) bulk_g2s(b_lo, A.img_lo + im, img_bytes, bar);
        issued = c + 1;
    };
    float v[KCH];
    auto load = [&](int c) {
        const int tb = c * KCH;
        const float *q = col + (long long)tb * N;
        if (valid && tb + KCH <= A.cnt) {
#pragma unroll
            for (int t = 0; t < KCH; t++) {
                v[t] = __ldg(q);
                q += N;
            }
        } else {
#pragma unroll
            for (int t = 0; t < KCH; t++) v[t] = (valid && tb + t < A.cnt) ? __ldg(q + (long long)t * N) : 0.f;
        }
    };
    issue_img(0);
    load(0);
    for (int c = 0; c < nchunks; c++) {
        // the MMAs of the previous chunk have read both operands
        if (c > 0 && !mbar_wait_bounded(&mma_bar, (uint32_t)((c - 1) & 1))) failed = true;
        if (!failed) {
            if (qlo && c > 0) issue_img(c);
            if (!qlo) issue_img(c + 1);
        }
#pragma unroll
        for (int cc = 0; cc < 8; cc++) {
            uint4 h, l;
            split_bf16x2(v[cc * 8], v[cc * 8 + 1], h.x, l.x);
            split_bf16x2(v[cc * 8 + 2], v[cc * 8 + 3], h.y, l.y);
            split_bf16x2(v[cc * 8 + 4], v[cc * 8 + 5], h.z, l.z);
            split_bf16x2(v[cc * 8 + 6], v[cc * 8 + 7], h.w, l.w);
            const uint32_t off = (uint32_t)m * 128u + ((uint32_t)(cc ^ (m & 7)) << 4);
            *(uint4 *)(a_hi + off) = h;
            *(uint4 *)(a_lo + off) = l;
        }
        if (c + 1 < nchunks) load(c + 1);   // in flight during this chunk's MMAs
        fence_proxy_async_smem();
        stop = __syncthreads_or(failed);
        if (stop) break;
        if (m == 0) {
            if (!mbar_wait_bounded(&img_bar[c & 1], (uint32_t)((c >> 1) & 1))) {
                failed = true;   // the others' wait for these MMAs gives up too
            } else {
                tc_fence_after();
                const uint32_t ah = smem_u32(a_hi), al = smem_u32(a_lo);
                const uint32_t bh = smem_u32(!qlo && (c & 1) ? b_lo : b_hi), bl = smem_u32(b_lo);
#pragma unroll
                for (int k = 0; k < KCH / 16; k++) {
                    const uint32_t ko = (uint32_t)k * 32u;
                    const uint64_t dah = sdesc_k_sw128(ah + ko), dal = sdesc_k_sw128(al + ko);
                    const uint64_t dbh = sdesc_k_sw128(bh + ko), dbl = sdesc_k_sw128(bl + ko);
                    umma_bf16(tmem, dah, dbh, idesc, (c > 0 || k > 0) ? 1u : 0u);
                    umma_bf16(tmem, dal, dbh, idesc, 1u);
                    if (qlo) {
                        umma_bf16(tmem, dah, dbl, idesc, 1u);
                        umma_bf16(tmem, dal, dbl, idesc, 1u);
                    }
                }
                umma_commit(&mma_bar);
            }
        }
    }

    float *P = A.P + (long long)shot * A.P_ss + (valid ? p : 0);
    float old[16];   // P of the slice of 16 probes that is written next, read one slice ahead
    auto read_p = [&](int c0) {
#pragma unroll
        for (int j = 0; j < 16; j++) old[j] = (valid && c0 + j < A.r) ? P[(long long)(c0 + j) * N] : 0.f;
    };
    if (!stop) {
        read_p(0);
        if (!mbar_wait_bounded(&mma_bar, (uint32_t)((nchunks - 1) & 1))) failed = true;
        stop = __syncthreads_or(failed);
    }
    if (!stop) {
        tc_fence_after();
        for (int c0 = 0; c0 < A.r_pad; c0 += 16) {
            uint32_t r16[16];
            tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, r16);
            float nv[16];
#pragma unroll
            for (int j = 0; j < 16; j++) nv[j] = fmaf(A.scale, __uint_as_float(r16[j]), old[j]);
            if (c0 + 16 < A.r_pad) read_p(c0 + 16);
#pragma unroll
            for (int j = 0; j < 16; j++)
                if (valid && c0 + j < A.r) P[(long long)(c0 + j) * N] = nv[j];
        }
    } else {
        if (m == 0) {
            atomicExch(A.err, 1);
            // copies in flight land
            for (int c = std::max(0, issued - 2); c < issued; c++) mbar_wait_bounded(&img_bar[c & 1], (uint32_t)((c >> 1) & 1));
        }
        // Give in-flight MMAs one more bounded chance to retire, then free the TMEM whether
        // or not they did: a block that exits still holding its columns leaves them
        // allocated for the rest of the context, so every later launch that allocates on
        // this SM would wait forever.  The cost of freeing is that an MMA still in flight
        // could write columns a block of a later launch has just allocated; the error flag
        // this call reports tells the caller that results computed on the stream since then
        // are suspect.
        mbar_wait_bounded(&mma_bar, (uint32_t)((nchunks - 1) & 1));
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, ncols);
}

size_t probe_gemm_smem(int r_pad)
{
    const size_t need = 1024 + 32768 + (size_t)2 * r_pad * 128;
    // Keep (co-resident CTAs) x (TMEM columns) within the 512 columns of an SM.
    const int max_ctas = 512 / (int)tmem_cols_for(r_pad);
    const size_t cap = (size_t)233472 / (size_t)(max_ctas + 1) + 1024;
    return need > cap ? need : cap;
}

cudaError_t launch_probe_gemm(const GemmArgs &A, int nshots, cudaStream_t s)
{
    const size_t smem = probe_gemm_smem(A.r_pad);
    cudaError_t e = cudaFuncSetAttribute(probe_gemm_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)((A.N + 127) / 128), nshots);
    cudaEvent_t ev = prof_begin(PROF_GEMM, s);
    probe_gemm_kernel<<<grid, 128, smem, s>>>(A);
    prof_end(PROF_GEMM, ev, s);
    count_launch();
    return cudaGetLastError();
}

}  // namespace wp
