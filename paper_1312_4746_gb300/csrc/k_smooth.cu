// Smooth co-sparse texture (mode CS_MODE_SMOOTH): Sec. 2 Eq. (map_tsm)
// iota_sigma(a)_j = exp(-a_j^2 / sigma), Eq. (approx_cosupp) and Sec. 3.1
// c_i = elementwise median of the iota of label i's scribble samples, and
// Eq. (post_text) P(s_x, x | i) = softmax_i(-||c_i - iota(O s_x)||_1 / beta_i(x)),
// added to the Parzen colour-location log-likelihood of Eq. (joined).
//
// Codes here are FP32 dot products of the FP32-normalised patch (the
// arithmetic of the FP32 codes kernel: Kahan mean, reciprocal norm); a patch
// whose centred norm is within the FP32 bound of zero is taken as flat
// (s = 0, every code 0, iota = 1). Three launches after the sum:
//   smooth_iota_samples_kernel  iota of every scribble sample (code-major)
//   smooth_median_kernel        c_i by exact radix selection (one block per
//                               label and code; the mean of the two middle
//                               values for an even count)
//   smooth_texture_kernel       per pixel: iota, l1 to each c_i, the texture
//                               log-posterior added to -L, label posteriors
#include <cstdint>

#include "internal.h"

namespace {

constexpr int TX = 32, TY = 4, TPX = 2;  // threads of the texture kernel, pixel rows TY apart per thread
constexpr int SL = 128;                // samples per block of the sample kernel
constexpr float SU32 = 5.9604645e-08f;  // 2^-24

__device__ __forceinline__ float gray_of(const float* px) {
    return __fadd_rn(__fadd_rn(__fmul_rn(0.299f, px[0]), __fmul_rn(0.587f, px[1])),
                     __fmul_rn(0.114f, px[2]));
}
__device__ __forceinline__ float gabs_of(const float* px) {
    return (0.299f * fabsf(px[0]) + 0.587f * fabsf(px[1]) + 0.114f * fabsf(px[2])) *
           (1.f + 4 * SU32);
}

// Normalised masked patch s (N values, padded to NP with zeros) from gray
// values g(t) and bounds ga(t) of window position t = dy P + dx.
template <int P, class GF, class AF>
__device__ __forceinline__ void norm_patch(const float* w, GF g, AF ga, float (&s)[(P * P + 3) & ~3]) {
    constexpr int N = P * P, NP = (N + 3) & ~3;
#pragma unroll
    for (int t = N; t < NP; ++t) s[t] = 0.f;
    float sum = 0.f, kc = 0.f, vabs = 0.f, e2 = 0.f;
#pragma unroll
    for (int t = 0; t < N; ++t) {
        const float v = __fmul_rn(w[t], g(t));
        s[t] = v;
        const float yk = __fsub_rn(v, kc);
        const float tk = __fadd_rn(sum, yk);
        kc = __fsub_rn(__fsub_rn(tk, sum), yk);
        sum = tk;
        vabs += fabsf(v);
        const float ew = fabsf(w[t]) * ga(t);
        e2 = fmaf(ew, ew, e2);
    }
    const float mu = __fdiv_rn(sum, (float)N);
    float ss = 0.f;
#pragma unroll
    for (int t = 0; t < N; ++t) {
        s[t] = __fsub_rn(s[t], mu);
        ss = fmaf(s[t], s[t], ss);
    }
    const float cn = sqrtf(ss);
    const float dc = (2.f * 5.1f * SU32) * sqrtf(e2) * 1.0001f +
                     3.1f * SU32 * vabs * rsqrtf((float)N) * 1.0001f + SU32 * cn;
    const float inv = cn > 4.f * dc ? __frcp_rn(cn) : 0.f;  // flat: s = 0
#pragma unroll
    for (int t = 0; t < N; ++t) s[t] = __fmul_rn(s[t], inv);
}

// Loads rows j0 .. j0 + 31 of O into shared memory (NP floats per row).
template <int P>
__device__ __forceinline__ void load_rows(float* s_om, const float* omega, int k, int j0,
                                          int tid, int nthr) {
    constexpr int N = P * P, NP = (N + 3) & ~3;
    const int rows = min(32, k - j0);
    for (int i = tid; i < 32 * NP; i += nthr) {
        const int jj = i / NP, t = i % NP;
        s_om[i] = (jj < rows && t < N) ? omega[(size_t)(j0 + jj) * N + t] : 0.f;
    }
}

// The dot products of an operator row in shared memory with PX patches held as
// packed pairs: two interleaved sums per patch (even and odd elements), one
// packed FMA for both. Each row element is read once for all PX patches (a
// broadcast read still fills a register in every lane, so reads and packed
// multiply-adds balance at four patches).
template <int NP, int PX>
__device__ __forceinline__ void dot_rows(const float* row, const uint64_t (&s2)[PX][NP / 2],
                                         float (&out)[PX]) {
    const ulonglong2* o2 = reinterpret_cast<const ulonglong2*>(row);
    uint64_t a[PX];
#pragma unroll
    for (int u = 0; u < PX; ++u) a[u] = 0;  // (0.f, 0.f)
#pragma unroll
    for (int t4 = 0; t4 < NP / 4; ++t4) {
        const ulonglong2 o = o2[t4];
#pragma unroll
        for (int u = 0; u < PX; ++u)
            asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(a[u]) : "l"((uint64_t)o.x), "l"(s2[u][2 * t4]));
#pragma unroll
        for (int u = 0; u < PX; ++u)
            asm("fma.rn.f32x2 %0, %1, %2, %0;"
                : "+l"(a[u])
                : "l"((uint64_t)o.y), "l"(s2[u][2 * t4 + 1]));
    }
#pragma unroll
    for (int u = 0; u < PX; ++u)
        out[u] = __uint_as_float((uint32_t)a[u]) + __uint_as_float((uint32_t)(a[u] >> 32));
}
template <int NP>
__device__ __forceinline__ void pack_patch(const float (&s)[NP], uint64_t (&s2)[NP / 2]) {
#pragma unroll
    for (int t = 0; t < NP / 2; ++t)
        asm("mov.b64 %0, {%1, %2};" : "=l"(s2[t]) : "f"(s[2 * t]), "f"(s[2 * t + 1]));
}

// iota of every scribble sample (every pixel when sample_pix is null),
// code-major: iota_smp[j * S + s]. PX samples per thread share each operator
// row's shared-memory reads; blockIdx.y takes `jgroup` codes (a multiple of
// 32), which splits a short sample list over the whole GPU.
//
// Bound: instruction issue (26 packed multiply-adds and an exponential per code
// and sample, at 8 to 12 warps per SM: the patches fill the registers); the
// multiply-adds alone (7.6e8 at 154,401 pixels x 98 x 49) would take 20 us.
// Measured there: 71 us, against 76 us with one sample per thread and
// unpacked multiply-adds (13 shared-memory reads per 49 multiply-adds); 10,000
// samples: 24 us against 27 us in 79 blocks.
template <int P, int PX>
__global__ void __launch_bounds__(SL) smooth_iota_samples_kernel(
    const float* __restrict__ img, int H, int W, const float* __restrict__ omega, int k,
    const float* __restrict__ mask, const int32_t* __restrict__ sample_pix, int S, float sigma,
    int jgroup, float* __restrict__ iota_smp) {
    constexpr int N = P * P, NP = (N + 3) & ~3, R = (P - 1) / 2;
    __shared__ __align__(16) float s_om[32 * NP];
    __shared__ float s_w[N];
    for (int i = threadIdx.x; i < N; i += SL) s_w[i] = mask[i];
    __syncthreads();
    int s_idx[PX];
    uint64_t s2[PX][NP / 2];
#pragma unroll
    for (int u = 0; u < PX; ++u) {
        s_idx[u] = (blockIdx.x * PX + u) * SL + threadIdx.x;
        const bool live = s_idx[u] < S;
        int pix = live ? (sample_pix ? sample_pix[s_idx[u]] : s_idx[u]) : 0;
        if (pix < 0 || pix >= H * W) pix = 0;  // reported by the distance transform's seed pass
        const int y = pix / W, x = pix % W;
        auto px_at = [&](int t) {
            const int yy = min(max(y + t / P - R, 0), H - 1), xx = min(max(x + t % P - R, 0), W - 1);
            return img + ((size_t)yy * W + xx) * 3;
        };
        float s[NP];
        norm_patch<P>(s_w, [&](int t) { return gray_of(px_at(t)); },
                      [&](int t) { return gabs_of(px_at(t)); }, s);
        pack_patch<NP>(s, s2[u]);
        asm volatile("" ::: "memory");  // one sample's loads at a time in registers
    }
    const float nsig = -1.f / sigma;
    const int jb = blockIdx.y * jgroup, je = min(k, jb + jgroup);
    for (int j0 = jb; j0 < je; j0 += 32) {
        __syncthreads();
        load_rows<P>(s_om, omega, k, j0, threadIdx.x, SL);
        __syncthreads();
        const int rows = min(32, je - j0);
        for (int jj = 0; jj < rows; ++jj) {
            float a[PX];
            dot_rows<NP, PX>(s_om + jj * NP, s2, a);
#pragma unroll
            for (int u = 0; u < PX; ++u)
                if (s_idx[u] < S)
                    iota_smp[(size_t)(j0 + jj) * S + s_idx[u]] = expf(a[u] * a[u] * nsig);
        }
    }
}

// Order-preserving map of a float's bits to an unsigned key, and back.
__device__ __forceinline__ unsigned f2key(float f) {
    const unsigned u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key2f(unsigned k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// c[i * k + j] = median over label i's samples of iota_smp[j][s], one block
// per (code, label): radix selection over the order-preserving keys with
// digits of 11, 11 and 10 bits, each digit's histogram scanned by the whole
// block. For an even count the upper middle value is the lower one, the next
// occupied bin of the last histogram, or the least key of the next occupied
// bin noted in an earlier pass.
//
// Bound: latency (three passes over a label's few thousand values). Measured
// at 5 labels x 2000 samples x 98 codes: 13 us, against 48 us for two
// selections of four 8-bit digits with one thread scanning each histogram.
constexpr int DB = 256;   // threads per block of the median kernel
constexpr int HB = 2048;  // histogram bins: 8 per thread
__global__ void __launch_bounds__(DB) smooth_median_kernel(
    const float* __restrict__ iota_smp, int S, int k, const int32_t* __restrict__ label_off,
    float* __restrict__ reps) {
    __shared__ __align__(16) unsigned hist[HB];
    __shared__ unsigned s_warp[DB / 32];
    __shared__ unsigned s_found[4];  // digit, rank within its bin, bin count, next occupied bin
    __shared__ unsigned s_min;
    const int i = blockIdx.y, j = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int off = label_off[i], m = label_off[i + 1] - off;
    const float* v = iota_smp + (size_t)j * S + off;
    const bool even = m % 2 == 0;
    unsigned pre = 0, r = (unsigned)(m - 1) / 2, succ = 0, sshift = 32;
    if (tid == 0) s_min = 0xffffffffu;
    for (int pass = 0; pass < 3; ++pass) {
        const int shift = pass == 0 ? 21 : pass == 1 ? 10 : 0;
        const unsigned dmask = pass == 2 ? 1023u : 2047u;
        for (int t = tid; t < HB / 4; t += DB)
            reinterpret_cast<uint4*>(hist)[t] = make_uint4(0u, 0u, 0u, 0u);
        if (tid == 0) s_found[3] = 0xffffffffu;
        __syncthreads();
        for (int e = tid; e < m; e += DB) {
            const unsigned key = f2key(v[e]);
            if (pass == 0 || key >> (pass == 1 ? 21 : 10) == pre)
                atomicAdd(hist + ((key >> shift) & dmask), 1u);
            else if (pass == 2 && sshift < 32 && key >> sshift == succ)
                atomicMin(&s_min, key);
        }
        __syncthreads();
        unsigned h[8], own = 0;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const uint4 x = reinterpret_cast<const uint4*>(hist)[2 * tid + q];
            h[4 * q] = x.x;
            h[4 * q + 1] = x.y;
            h[4 * q + 2] = x.z;
            h[4 * q + 3] = x.w;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) own += h[q];
        unsigned inc = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned up = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += up;
        }
        if (lane == 31) s_warp[warp] = inc;
        __syncthreads();
        unsigned acc = inc - own;
#pragma unroll
        for (int w = 0; w < DB / 32; ++w) acc += w < warp ? s_warp[w] : 0u;
        if (r >= acc && r < acc + own) {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                if (r >= acc && r < acc + h[q]) {
                    s_found[0] = 8u * tid + q;
                    s_found[1] = r - acc;
                    s_found[2] = h[q];
                }
                acc += h[q];
            }
        }
        __syncthreads();
        const unsigned dig = s_found[0];
        unsigned nx = 0xffffffffu;
#pragma unroll
        for (int q = 7; q >= 0; --q)
            if (h[q] && 8u * tid + q > dig) nx = 8u * tid + q;
        nx = __reduce_min_sync(0xffffffffu, nx);
        if (lane == 0 && nx != 0xffffffffu) atomicMin(s_found + 3, nx);
        __syncthreads();
        nx = s_found[3];
        r = s_found[1];
        if (pass < 2) {
            if (even && nx != 0xffffffffu) {
                succ = (pre << 11) | nx;
                sshift = (unsigned)shift;
            }
            pre = (pre << 11) | dig;
        } else if (tid == 0) {
            const float lo = key2f((pre << 10) | dig);
            float out = lo;
            if (even) {
                float hi = lo;
                if (s_found[2] - r < 2u) hi = key2f(nx != 0xffffffffu ? (pre << 10) | nx : s_min);
                out = __fmul_rn(0.5f, __fadd_rn(lo, hi));
            }
            reps[(size_t)i * k + j] = out;
        }
        __syncthreads();  // the digit is taken: s_found and hist are free again
    }
}

// Per pixel: iota of its codes, l1 to each representative, the texture
// log-posterior added to L (neglog holds -L of the Parzen sum), then the
// label posteriors. The l1 sums of NB labels at a time stay in registers; more
// than NB labels take further sweeps over the codes (cheaper than sums in
// shared memory, whose read-modify-write per label and code cost more than the
// dot product itself).
//
// Bound: instruction issue (the dot products, an exponential and two operations
// per label and code, 12 warps per SM). Measured there with 5 labels: 87 us, against
// 130 us with the sums in shared memory and unpacked multiply-adds.
template <int P, int NB>
__global__ void __launch_bounds__(TX* TY) smooth_texture_kernel(
    const float* __restrict__ img, int H, int W, const float* __restrict__ omega, int k,
    const float* __restrict__ mask, float sigma, const float* __restrict__ reps, int n_labels,
    const int32_t* __restrict__ dist2, float alpha, float d_min, float kappa_beta,
    float* __restrict__ neglog, float* __restrict__ post) {
    constexpr int N = P * P, NP = (N + 3) & ~3, R = (P - 1) / 2, TW = TX + P - 1;
    constexpr int TH = TPX * TY + P - 1, NT = TX * TY;
    extern __shared__ __align__(16) float sm[];
    float* s_om = sm;                          // 32 x NP
    float* s_rep = s_om + 32 * NP;             // k x NB (this sweep's labels)
    float* s_gray = s_rep + (size_t)k * NB;    // TH x TW
    float* s_gabs = s_gray + TW * TH;          // TH x TW
    float* s_w = s_gabs + TW * TH;             // N
    float* s_acc = s_w + ((N + 3) & ~3);       // n_labels x TPX x NT
    const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
    const int y0 = blockIdx.y * TPX * TY, x0 = blockIdx.x * TX;
    for (int i = tid; i < TW * TH; i += NT) {
        const int ly = i / TW, lx = i % TW;
        const int yy = min(max(y0 + ly - R, 0), H - 1), xx = min(max(x0 + lx - R, 0), W - 1);
        const float* px = img + ((size_t)yy * W + xx) * 3;
        s_gray[i] = gray_of(px);
        s_gabs[i] = gabs_of(px);
    }
    for (int i = tid; i < N; i += NT) s_w[i] = mask[i];
    __syncthreads();
    uint64_t s2[TPX][NP / 2];
#pragma unroll
    for (int u = 0; u < TPX; ++u) {
        float s[NP];
        const int r0 = ty + u * TY;
        norm_patch<P>(s_w, [&](int t) { return s_gray[(r0 + t / P) * TW + tx + t % P]; },
                      [&](int t) { return s_gabs[(r0 + t / P) * TW + tx + t % P]; }, s);
        pack_patch<NP>(s, s2[u]);
        asm volatile("" ::: "memory");  // one patch at a time in registers
    }
    const float nsig = -1.f / sigma;
    for (int i0 = 0; i0 < n_labels; i0 += NB) {
        __syncthreads();
        for (int t = tid; t < k * NB; t += NT) {
            const int jj = t / NB, i = i0 + t % NB;
            s_rep[t] = i < n_labels ? reps[(size_t)i * k + jj] : 0.f;
        }
        float acc[TPX][NB];
#pragma unroll
        for (int u = 0; u < TPX; ++u)
#pragma unroll
            for (int b = 0; b < NB; ++b) acc[u][b] = 0.f;
        for (int j0 = 0; j0 < k; j0 += 32) {
            __syncthreads();
            load_rows<P>(s_om, omega, k, j0, tid, NT);
            __syncthreads();
            const int rows = min(32, k - j0);
            for (int jj = 0; jj < rows; ++jj) {
                float a[TPX];
                dot_rows<NP, TPX>(s_om + jj * NP, s2, a);
                const float4* rp = reinterpret_cast<const float4*>(s_rep + (j0 + jj) * NB);
                float4 c[NB / 4];
#pragma unroll
                for (int b = 0; b < NB / 4; ++b) c[b] = rp[b];
#pragma unroll
                for (int u = 0; u < TPX; ++u) {
                    const float io = expf(a[u] * a[u] * nsig);
#pragma unroll
                    for (int b = 0; b < NB / 4; ++b) {
                        acc[u][4 * b] += fabsf(c[b].x - io);
                        acc[u][4 * b + 1] += fabsf(c[b].y - io);
                        acc[u][4 * b + 2] += fabsf(c[b].z - io);
                        acc[u][4 * b + 3] += fabsf(c[b].w - io);
                    }
                }
            }
        }
#pragma unroll
        for (int u = 0; u < TPX; ++u)
#pragma unroll
            for (int b = 0; b < NB; ++b)
                if (i0 + b < n_labels) s_acc[((i0 + b) * TPX + u) * NT + tid] = acc[u][b];
    }
    const long long P_ = (long long)H * W;
    const int x = x0 + tx;
    for (int u = 0; u < TPX; ++u) {
        const int y = y0 + ty + u * TY;
        if (y >= H || x >= W) continue;
        const int pix = y * W + x;
        float* sa = s_acc + u * NT + tid;
        constexpr int SS = TPX * NT;
        // texture log-posterior, Eq. (post_text), beta_i = kappa_beta rho_i
        float tmax = -INFINITY;
        for (int i = 0; i < n_labels; ++i) {
            const float rho = alpha * fmaxf(sqrtf((float)dist2[(size_t)i * P_ + pix]), d_min);
            const float t = -sa[i * SS] / (kappa_beta * rho);
            sa[i * SS] = t;
            tmax = fmaxf(tmax, t);
        }
        float ts = 0.f;
        for (int i = 0; i < n_labels; ++i) ts += expf(sa[i * SS] - tmax);
        const float tl = tmax + logf(ts);
        float lmax = -INFINITY;
        for (int i = 0; i < n_labels; ++i) {
            const float L = -neglog[(size_t)i * P_ + pix] + sa[i * SS] - tl;
            sa[i * SS] = L;
            lmax = fmaxf(lmax, L);
        }
        float ls = 0.f;
        for (int i = 0; i < n_labels; ++i) ls += expf(sa[i * SS] - lmax);
        const float lse = lmax + logf(ls);
        for (int i = 0; i < n_labels; ++i) {
            const float L = sa[i * SS];
            neglog[(size_t)i * P_ + pix] = -L;
            if (post) post[(size_t)i * P_ + pix] = expf(L - lse);
        }
    }
}

template <int P, int NB>
constexpr size_t texture_smem(int k, int n_labels) {
    constexpr int N = P * P, NP = (N + 3) & ~3, TW = TX + P - 1, TH = TPX * TY + P - 1;
    return sizeof(float) * ((size_t)32 * NP + (size_t)k * NB + 2 * TW * TH + NP +
                            (size_t)n_labels * TPX * TX * TY);
}

template <int P, int NB>
cudaError_t texture_p(const SmoothArgs& a, cudaStream_t st) {
    const size_t smem = texture_smem<P, NB>(a.k, a.n_labels);
    // (likelihoods take at most 256 codes)
    cudaError_t e = cs_smem_limit((const void*)smooth_texture_kernel<P, NB>,
                                  texture_smem<P, NB>(256, CS_MAX_LABELS));
    if (e != cudaSuccess) return e;
    dim3 grd((a.W + TX - 1) / TX, (a.H + TPX * TY - 1) / (TPX * TY));
    smooth_texture_kernel<P, NB><<<grd, TX * TY, smem, st>>>(
        a.img, a.H, a.W, a.omega, a.k, a.mask, a.sigma, a.reps, a.n_labels, a.dist2, a.alpha,
        a.d_min, a.kappa_beta, a.neglog, a.post);
    return cudaGetLastError();
}

template <int P>
cudaError_t smooth_p(const SmoothArgs& a, cudaStream_t st) {
    // the samples are few: one group of 32 codes per block
    smooth_iota_samples_kernel<P, 2>
        <<<dim3((a.S + 2 * SL - 1) / (2 * SL), (a.k + 31) / 32), SL, 0, st>>>(
            a.img, a.H, a.W, a.omega, a.k, a.mask, a.sample_pix, a.S, a.sigma, 32, a.iota_smp);
    smooth_median_kernel<<<dim3(a.k, a.n_labels), DB, 0, st>>>(a.iota_smp, a.S, a.k,
                                                                a.d_label_off, a.reps);
    if (a.n_labels <= 4) return texture_p<P, 4>(a, st);
    if (a.n_labels <= 8) return texture_p<P, 8>(a, st);
    return texture_p<P, 16>(a, st);
}

template <int P>
cudaError_t iota_pixels_p(const float* img, int H, int W, const float* omega, int k,
                          const float* mask, float sigma, float* iota, cudaStream_t st) {
    const int S = H * W;
    constexpr int PX = P <= 7 ? 4 : 2;
    smooth_iota_samples_kernel<P, PX><<<(S + PX * SL - 1) / (PX * SL), SL, 0, st>>>(
        img, H, W, omega, k, mask, nullptr, S, sigma, (k + 31) / 32 * 32, iota);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_iota_pixels(const float* img, int H, int W, const float* omega, int k, int p,
                               const float* mask, float sigma, float* iota, cudaStream_t st) {
    switch (p) {
        case 3: return iota_pixels_p<3>(img, H, W, omega, k, mask, sigma, iota, st);
        case 5: return iota_pixels_p<5>(img, H, W, omega, k, mask, sigma, iota, st);
        case 7: return iota_pixels_p<7>(img, H, W, omega, k, mask, sigma, iota, st);
        case 9: return iota_pixels_p<9>(img, H, W, omega, k, mask, sigma, iota, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_smooth(const SmoothArgs& a, cudaStream_t st) {
    switch (a.p) {
        case 3: return smooth_p<3>(a, st);
        case 5: return smooth_p<5>(a, st);
        case 7: return smooth_p<7>(a, st);
        case 9: return smooth_p<9>(a, st);
        default: return cudaErrorInvalidValue;
    }
}
