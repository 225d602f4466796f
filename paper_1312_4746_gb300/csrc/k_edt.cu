// Exact squared distance from every pixel to the nearest scribble sample of
// each label (Sec. 3.1: rho_i(x) = alpha |x - x_v|, x_v the closest scribble
// location of label i).
//
// Separable exact transform in integers:
//   1. seed bitmaps: one bit per pixel and label;
//   2. row pass (one warp per label and row): horizontal distance h to the
//      nearest seed in the same row, from bit scans of the bitmap words;
//   3. column pass (2 to 8 builder threads per label and column, one per
//      row segment, and 8 or 32 readers): lower envelopes of the parabolas
//      (y - q)^2 + h(q)^2 over each segment's rows q with finite h, each
//      built in one sweep and read back by row ranges; intersection
//      abscissae are compared as exact rationals with 64-bit cross products,
//      so the result equals the brute-force minimum bit for bit. For images
//      up to labels x width x height^2 = 2e7 an outward scan per pixel with early
//      exit gives the same minimum with far more parallelism.
// majority_kernel: for the factorised form, the majority co-support of each label
// (Eq. tex-rep: bit set iff 2 * count >= m).
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "internal.h"

namespace {

constexpr int32_t INF = 0x7FFFFFFF;

__device__ __forceinline__ int label_of(const int32_t* __restrict__ off, int n_labels, int s) {
    int lo = 0, hi = n_labels - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= s)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// Seed bitmap: bit (x & 31) of word [i][y][x >> 5] is set when (y, x) is a
// sample of label i.
__global__ void seed_kernel(const int32_t* __restrict__ off, int n_labels,
                            const int32_t* __restrict__ sample_pix, int n_samples, int H, int W,
                            uint32_t* __restrict__ bm, int* __restrict__ d_err) {
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n_samples) return;
    const int pix = sample_pix[s];
    if (pix < 0 || pix >= H * W) {  // reject out-of-image sample indices, never write them
        if (atomicCAS(d_err, 0, CS_DEVERR_BAD_SAMPLE) == 0) d_err[1] = s;
        return;
    }
    const int i = label_of(off, n_labels, s);
    const int y = pix / W, x = pix % W, Wb = (W + 31) >> 5;
    atomicOr(bm + ((size_t)i * H + y) * Wb + (x >> 5), 1u << (x & 31));
}

// Pass 1 (one warp per label and row): horizontal distance to the nearest
// seed of the same row (INF if the row has none), from the seed bitmap with
// ballot-free bit scans; a forward sweep finds the last seed at or left of
// each pixel, a backward sweep the next seed at or right of it.
__global__ void rows_binary_kernel(int H, int W, int n_labels, const uint32_t* __restrict__ bm,
                                   int32_t* __restrict__ h) {
    const long long row = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (row >= (long long)n_labels * H) return;
    const int Wb = (W + 31) >> 5;
    const uint32_t* b = bm + (size_t)row * Wb;
    int32_t* out = h + (size_t)row * W;
    int carry = -1;  // last seed column seen so far
    for (int c = 0; c < Wb; ++c) {
        const uint32_t word = b[c];
        const uint32_t le = word & (lane == 31 ? 0xFFFFFFFFu : ((2u << lane) - 1u));
        const int last = le ? 32 * c + 31 - __clz(le) : carry;
        const int x = 32 * c + lane;
        if (x < W) out[x] = last < 0 ? INF : x - last;
        if (word) carry = 32 * c + 31 - __clz(word);
    }
    carry = -1;  // next seed column seen so far (from the right)
    for (int c = Wb - 1; c >= 0; --c) {
        const uint32_t word = b[c];
        const uint32_t ge = word & (0xFFFFFFFFu << lane);
        const int next = ge ? 32 * c + __ffs(ge) - 1 : carry;
        const int x = 32 * c + lane;
        if (x < W && next >= 0 && next - x < out[x]) out[x] = next - x;
        if (word) carry = 32 * c + __ffs(word) - 1;
    }
}

// Column pass, split: a block of 256 threads takes CB columns. S threads per
// column build the lower envelopes of its S row segments (one sweep over the
// segment's rows with finite h: a row's parabola (y - q)^2 + h(q)^2 replaces the
// stack top while it lies below it from the top's breakpoint on, compared exactly
// with 64-bit cross products); then NRD threads per column read them back, each
// for a range of rows: it finds the segment of its first row in each of the S
// envelopes by binary search over the breakpoints (the same exact comparison,
// monotone in the segment index), walks on, and keeps the smallest of the S
// values, the minimum over all rows.
//
// Bound with few columns (labels x width): the sweeps' and the reads' latency,
// about 0.2 us a row swept and 0.13 us a row and envelope read. Few columns per
// block give many readers (H / 32 rows each) and blocks for every SM, and with them
// more segments pay. With many columns: the loads and the reads of each envelope, so
// that 32 columns per block (whole lines of h and of the result) and few segments do.

__device__ __forceinline__ int env_build(const int32_t* __restrict__ col, int W, int q_lo, int q_hi,
                                         int32_t* v, int32_t* F, long long stride) {
    int kk = -1;
    constexpr int PF = 16;  // rows of h fetched ahead (independent loads)
    for (int q0 = q_lo; q0 < q_hi; q0 += PF) {
        int32_t hv[PF];
#pragma unroll
        for (int u = 0; u < PF; ++u) hv[u] = q0 + u < q_hi ? col[(size_t)(q0 + u) * W] : INF;
#pragma unroll
        for (int u = 0; u < PF; ++u) {
            const int q = q0 + u;
            const int32_t hq = hv[u];
            if (hq == INF) continue;
            const int32_t Fq = hq * hq + q * q;
            while (kk > 0) {
                const int vk = v[kk * stride], vp = v[(kk - 1) * stride];
                const int32_t Fv = F[kk * stride], Fp = F[(kk - 1) * stride];
                if ((long long)(Fq - Fv) * (vk - vp) <= (long long)(Fv - Fp) * (q - vk))
                    --kk;
                else
                    break;
            }
            ++kk;
            v[kk * stride] = q;
            F[kk * stride] = Fq;
        }
    }
    return kk;
}

// Reader state on one envelope: current segment j (vertex vj, value Fj).
struct EnvCursor {
    int j, kk, vj;
    int32_t Fj;
};
__device__ __forceinline__ EnvCursor env_seek(const int32_t* v, const int32_t* F,
                                              long long stride, int kk, int y0) {
    int lo = 0, hi = kk;
    while (lo < hi) {  // first segment whose right breakpoint is not left of y0
        const int mid = (lo + hi) >> 1;
        const int vm = v[mid * stride], vn = v[(mid + 1) * stride];
        const int32_t Fm = F[mid * stride], Fn = F[(mid + 1) * stride];
        if ((long long)(Fn - Fm) < 2ll * y0 * (vn - vm)) lo = mid + 1;  // z(v_mid, v_mid+1) < y0
        else hi = mid;
    }
    return {lo, kk, v[lo * stride], F[lo * stride]};
}
__device__ __forceinline__ int32_t env_value(EnvCursor& c, const int32_t* v, const int32_t* F,
                                             long long stride, int y) {
    while (c.j < c.kk) {
        const int vn = v[(c.j + 1) * stride];
        const int32_t Fn = F[(c.j + 1) * stride];
        if ((long long)(Fn - c.Fj) < 2ll * y * (vn - c.vj)) {  // z(vj, vn) < y
            ++c.j;
            c.vj = vn;
            c.Fj = Fn;
        } else {
            break;
        }
    }
    return (y - c.vj) * (y - c.vj) + (c.Fj - c.vj * c.vj);
}

template <bool SHARED, int S, int CB>  // CB columns per block
__global__ void __launch_bounds__(256) cols_envelope_split_kernel(
    int H, int W, int n_labels, const int32_t* __restrict__ h, int32_t* __restrict__ gv,
    int32_t* __restrict__ gF, int32_t* __restrict__ dist2) {
    constexpr int NRD = 256 / CB;  // reader threads per column
    static_assert(S >= 1 && S <= NRD, "segments");
    extern __shared__ int32_t smem[];
    __shared__ int s_kk[S][CB];
    const long long ncol = (long long)n_labels * W;
    const int c = threadIdx.x % CB, seg = threadIdx.x / CB;
    const long long col_id = blockIdx.x * (long long)CB + c;
    const bool valid = col_id < ncol;
    const int i = valid ? (int)(col_id / W) : 0, x = valid ? (int)(col_id % W) : 0;
    const int HS = (H + S - 1) / S;  // rows (and stack entries) per segment
    int32_t *v, *F;
    long long stride;
    if (SHARED) {
        v = smem + c;
        F = smem + (size_t)S * HS * CB + c;
        stride = CB;
    } else {
        v = gv + col_id;
        F = gF + col_id;
        stride = ncol;
    }
    const int32_t* col = h + (size_t)i * H * W + x;
    if (seg < S && valid) {
        const int q_lo = seg * HS, q_hi = min(H, q_lo + HS);
        s_kk[seg][c] = q_lo < q_hi ? env_build(col, W, q_lo, q_hi, v + (size_t)seg * HS * stride,
                                               F + (size_t)seg * HS * stride, stride)
                                   : -1;
    }
    __syncthreads();  // envelopes complete (shared or global) for the whole block
    if (!valid) return;
    int32_t* out = dist2 + (size_t)i * H * W + x;
    const int y0 = (int)((long long)H * seg / NRD), y1 = (int)((long long)H * (seg + 1) / NRD);
    EnvCursor cur[S];
    int kk[S];
#pragma unroll
    for (int b = 0; b < S; ++b) {
        kk[b] = s_kk[b][c];
        if (kk[b] >= 0 && y0 < y1)
            cur[b] = env_seek(v + (size_t)b * HS * stride, F + (size_t)b * HS * stride, stride,
                              kk[b], y0);
    }
    for (int y = y0; y < y1; ++y) {
        int32_t d = INF;  // INF when the label has no valid seed (a bad sample index)
#pragma unroll
        for (int b = 0; b < S; ++b)
            if (kk[b] >= 0)
                d = min(d, env_value(cur[b], v + (size_t)b * HS * stride,
                                     F + (size_t)b * HS * stride, stride, y));
        out[(size_t)y * W] = d;
    }
}

// Column pass for small images: D(y) = min over rows q of h(q)^2 + (y - q)^2,
// scanning q outwards from y and stopping once (y - q)^2 alone reaches the best
// value found, which no farther row can beat. Exact (integer arithmetic). A
// block holds 32 columns' h^2 in shared memory and scans `rows` rows of them,
// one row per warp at a time, SCAN_D rows each way per step. (Past the image's
// edge the edge row's h^2 is taken again with the larger distance: a value that
// the edge row itself has beaten.) O(min(H, sqrt(D))) per pixel with full
// parallelism, where the envelopes' sequential sweeps leave most of the chip
// idle (at 481 x 321, 5 labels the scan takes about 110 us: the distances are
// long). Measured at 96 x 64, 3 labels: 5.2 us against 17 us of a scan in global
// memory, one row per step.
constexpr int SCAN_D = 4;
constexpr int32_t SCAN_INF = 0x40000000;  // + any (y - q)^2 stays below 2^31
__global__ void __launch_bounds__(256) cols_scan_kernel(int H, int W, int n_labels, int rows,
                                                        const int32_t* __restrict__ h,
                                                        int32_t* __restrict__ dist2) {
    extern __shared__ int32_t hh[];  // H x 32
    const long long ncol = (long long)n_labels * W;
    const int c = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long col_id = blockIdx.x * 32ll + c;
    const bool valid = col_id < ncol;
    const int i = valid ? (int)(col_id / W) : 0, x = valid ? (int)(col_id % W) : 0;
    const size_t base = (size_t)i * H * W + x;
    for (int q = warp; q < H; q += 8) {
        const int32_t v = valid ? h[base + (size_t)q * W] : INF;
        hh[q * 32 + c] = v == INF ? SCAN_INF : v * v;
    }
    __syncthreads();
    const int y1 = min(H, ((int)blockIdx.y + 1) * rows);
    for (int y = blockIdx.y * rows + warp; y < y1; y += 8) {
        int32_t D = hh[y * 32 + c];
        const int reach = max(y, H - 1 - y);
        for (int d = 1; d <= reach && d * d < D; d += SCAN_D) {
            int32_t m = SCAN_INF;
#pragma unroll
            for (int r = 0; r < SCAN_D; ++r) {
                const int e = d + r;
                const int32_t up = hh[max(y - e, 0) * 32 + c], dn = hh[min(y + e, H - 1) * 32 + c];
                m = min(m, min(up, dn) + e * e);
            }
            D = min(D, m);
        }
        if (valid) dist2[base + (size_t)y * W] = D >= SCAN_INF ? INF : D;
    }
}

// Majority co-support of a label, one block per (word, label): each warp
// transposes the words of 32 samples by five shuffles, so that lane b holds
// bit b of all of them, and adds its population count. Bound: latency.
// Measured at 4 labels of up to 3100 samples, k = 98: 7 us, against 100 us
// with one thread per (label, bit) walking the samples.
constexpr int MJ = 1024;
__global__ void __launch_bounds__(MJ) majority_kernel(const int32_t* __restrict__ off, int k,
                                                      int Wk, long long P,
                                                      const int32_t* __restrict__ sample_pix,
                                                      const uint32_t* __restrict__ bitmask,
                                                      uint32_t* __restrict__ rep) {
    __shared__ int s_cnt[MJ / 32][32];
    const int w = blockIdx.x, i = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int s0 = off[i], s1 = off[i + 1];
    int cnt = 0;
    for (int s = s0 + 32 * warp; s < s1; s += MJ) {
        uint32_t v = 0u;
        if (s + lane < s1) {
            int pix = sample_pix[s + lane];
            if (pix < 0 || pix >= P) pix = 0;  // reported by seed_kernel
            v = bitmask[(size_t)pix * Wk + w];
        }
        uint32_t m = 0x0000FFFFu;
#pragma unroll
        for (int j = 16; j > 0; j >>= 1, m ^= m << j) {
            const uint32_t o = __shfl_xor_sync(0xffffffffu, v, j);
            v = (lane & j) ? (v & ~m) | ((o & ~m) >> j) : (v & m) | ((o & m) << j);
        }
        cnt += __popc(v);
    }
    s_cnt[warp][lane] = cnt;
    __syncthreads();
    if (warp) return;
    for (int q = 1; q < MJ / 32; ++q) cnt += s_cnt[q][lane];
    const unsigned word = __ballot_sync(0xffffffffu, 32 * w + lane < k && 2 * cnt >= s1 - s0);
    if (lane == 0) rep[(size_t)i * Wk + w] = word;
}

__global__ void set_offsets_kernel(OffsetsParam p, int n, int32_t* __restrict__ dst) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = p.v[i];
}

}  // namespace

cudaError_t launch_set_offsets(const OffsetsParam& p, int n, int32_t* dst, cudaStream_t st) {
    set_offsets_kernel<<<1, 128, 0, st>>>(p, n, dst);
    return cudaGetLastError();
}

cudaError_t launch_edt(const EdtArgs& a, cudaStream_t st) {
    const int Wb = (a.W + 31) / 32;
    const long long nrow = (long long)a.n_labels * a.H;
    cudaError_t e = cudaMemsetAsync(a.seedbits, 0, sizeof(uint32_t) * nrow * Wb, st);
    if (e != cudaSuccess) return e;
    seed_kernel<<<(a.n_samples + 255) / 256, 256, 0, st>>>(a.d_label_off, a.n_labels,
                                                           a.sample_pix, a.n_samples, a.H, a.W,
                                                           a.seedbits, a.d_err);
    rows_binary_kernel<<<(unsigned)((nrow * 32 + 127) / 128), 128, 0, st>>>(
        a.H, a.W, a.n_labels, a.seedbits, a.colbuf);
    const long long ncol = (long long)a.n_labels * a.W;
    // the scan's work is at most about ncol H^2 / 1.5 row visits (all of them when
    // the distances exceed the height): up to SCAN_MOST it stays below the
    // envelopes' time (at 240 x 160, 8 labels, 4.9e7, the two are equal); a column
    // block's h^2 must fit shared memory (H <= 880)
    constexpr long long SCAN_MOST = 20000000ll;
    if (ncol * a.H * a.H <= SCAN_MOST && a.H <= 880) {
        const unsigned cb = (unsigned)((ncol + 31) / 32);
        // rows per block: about two blocks per SM, a multiple of the 8 warps
        int rows = (int)std::min<long long>(64, std::max<long long>(8, (long long)cb * a.H / 304));
        rows = (rows + 7) / 8 * 8;
        cudaError_t e2 = cs_smem_limit((const void*)cols_scan_kernel, 880 * 128);
        if (e2 != cudaSuccess) return e2;
        cols_scan_kernel<<<dim3(cb, (a.H + rows - 1) / rows), 256, (size_t)a.H * 128, st>>>(
            a.H, a.W, a.n_labels, rows, a.colbuf, a.dist2);
        return cudaGetLastError();
    }
    // envelopes of CB columns per block (S segments) in shared memory when they fit
    auto run = [&](auto seg_c, auto cb_c) -> cudaError_t {
        constexpr int S = decltype(seg_c)::value, CB = decltype(cb_c)::value;
        const unsigned nblk = (unsigned)((ncol + CB - 1) / CB);
        const size_t smem = (size_t)((a.H + S - 1) / S) * S * 2 * sizeof(int32_t) * CB;
        if (smem <= 110u * 1024u) {
            // (the limit of every size: captured launches of several sizes share it)
            cudaError_t e2 =
                cs_smem_limit((const void*)cols_envelope_split_kernel<true, S, CB>, 110 * 1024);
            if (e2 != cudaSuccess) return e2;
            cols_envelope_split_kernel<true, S, CB><<<nblk, 256, smem, st>>>(
                a.H, a.W, a.n_labels, a.colbuf, nullptr, nullptr, a.dist2);
        } else {
            cols_envelope_split_kernel<false, S, CB><<<nblk, 256, 0, st>>>(
                a.H, a.W, a.n_labels, a.colbuf, a.vbuf, a.fbuf, a.dist2);
        }
        return cudaSuccess;
    };
    using std::integral_constant;
    // Measured, the transform's launches alone, us, columns per block / segments, on
    // brush strokes of 60 and of 2000 samples per label (a label's rows are then few,
    // and segments without seeds idle):
    //                    columns   8/6       8/8       32/2      32/4
    //   60 x 2000 x 5        300   82, 148   84, 134   177, 316  180, 300
    //   481 x 321 x 5       2405   36, 42    37, 44    46, 72    48, 62
    //   2000 x 200 x 5     10000   52, 63    58, 68    44, 60    47, 56
    //   640 x 480 x 16     10240   63, 81    68, 84    74, 102   70, 102
    //   1024 x 768 x 10    10240   102, 153  112, 156  102, 181  100, 151
    //   1024 x 1024 x 16   16384   190, 285  212, 290  145, 211  142, 199
    //   5000 x 100 x 5     25000   77, 85    81, 91    52, 61    56, 62
    //   3000 x 400 x 16    48000   213, 292  241, 315  210, 325  204, 273
    e = ncol >= 6000 && a.H <= 256   ? run(integral_constant<int, 2>{}, integral_constant<int, 32>{})
        : ncol >= 16000              ? run(integral_constant<int, 4>{}, integral_constant<int, 32>{})
        : ncol < 4000 && a.H > 1536  ? run(integral_constant<int, 8>{}, integral_constant<int, 8>{})
                                     : run(integral_constant<int, 6>{}, integral_constant<int, 8>{});
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

cudaError_t launch_majority(int H, int W, const uint32_t* bitmask, int k, int n_labels,
                            const int32_t* d_label_off, const int32_t* sample_pix, uint32_t* rep,
                            cudaStream_t st) {
    const int Wk = (k + 31) / 32;
    majority_kernel<<<dim3(Wk, n_labels), MJ, 0, st>>>(d_label_off, k, Wk, (long long)H * W,
                                                       sample_pix, bitmask, rep);
    return cudaGetLastError();
}
