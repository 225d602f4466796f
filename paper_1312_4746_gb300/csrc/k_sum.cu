// Pixel x sample likelihood sum, plain FP32 form (Sec. 3.1, Eq. color,
// Eq. post_text, Eq. joined, Eq. energy1).
//
// For pixel x and label i, with rho = alpha * max(sqrt(D_i(x)), d_min) and
// beta = kappa_beta * rho, every sample j of the label contributes
//   e_j = -|x - x_j|^2 / (2 rho^2) - |I(x) - I_j|^2 / (2 sigma_c2)
//         - w_t TSM(b_x, b_j) / beta            (w_t = 1 per-sample, 0 factorised)
// and L_i(x) = logsumexp_j e_j - log m_i - log(2 pi rho^2) - 1.5 log(2 pi sigma_c2).
// The factorised form adds the texture log-posterior of Eq. (post_text) with
// the label's majority co-support. Posteriors are the softmax of L over
// labels; the data term is f_i = -L_i.
//
// The differences, squares, exponents (log2 units) and sums are FP32 on the CUDA
// cores, in packed pairs (f32x2) of samples; location distances are exact
// integers carried in FP32 (coordinates < 2^24). The TSM is an exact integer too,
// from the tensor cores (tcgen05): with the pixel's codes as +-1 and the
// sample's as 1 / 0 in e4m3 the dot product of the two is 2 b_x.b_j - |b_j|, and
// two further columns, the two exact parts of -|b_x| against 1, make it -TSM
// (sums of at most 512 in FP32). XOR and population count of the bit words took
// four population counts (16 per clock and SM) and eleven integer operations a
// pair; mma.sync in e4m3 is no way around them either (its operands are
// converted in the general pipes: about ten instructions a pair, 1.8 ms).
//
// Layout: one CTA of 8 warps per (PT x 128 pixels, label). The pixels' operand
// rows (one tensor-memory lane each) are written once; the label's samples come
// in tiles of 64 (positions and colours as planes, codes as operand slabs), laid
// out once per call (plain_tiles_kernel) and copied through a ring in shared
// memory. One thread issues a tile's MMAs into one of two accumulators while the
// warps form the exponents of the tile before from the other: warp w reads the
// lanes 32 (w % 4) .. and half the tile's columns, so a thread has one pixel of
// each of the PT operand tiles, which share the samples' reads, and every other
// 32 samples. It keeps an online log-sum-exp per pixel: a running maximum per 16
// samples and a TwoSum-compensated running sum per 32; the two threads of a
// pixel merge at the label's end. A second kernel normalises over the labels.
//
// Few samples per label on enough pixels (plain_few) take sum_few_kernel instead: a
// thread per pixel over all labels, the TSM by population counts, the normalisation at
// its end. There the operand rows, the waits and the merge of every (pixels, label)
// unit and the tiles' padding cost more than the population counts.
#include <cstdint>
#include <type_traits>

#include "internal.h"
#include "mma_phase.h"
#include "tc_ptx.cuh"

namespace {

constexpr int THREADS = 256;
constexpr int TS = 64;     // samples per tile
constexpr int STAGES = 4;  // tiles in the ring: one copied, one ahead, one multiplied, one summed
constexpr float LOG2E = 1.4426950408889634f;
constexpr float LN2 = 0.6931471805599453f;
constexpr float FAR = 1.0e18f;
constexpr float LOWEST = -3.0e38f;
constexpr uint64_t PLAIN_WAIT_NS = 1000000000ull;  // default limit of a wait for an MMA

// 32-column steps of the texture operands: k codes and the two columns of -|b_x|
__host__ __device__ constexpr int steps_for(int k) { return (k + 2 + 31) / 32; }
// bytes of a tile: x, y, r, g, b planes, then KS operand slabs of 64 rows
__host__ __device__ constexpr int tile_bytes(int KS) { return 5 * TS * 4 + KS * TS * 32; }
// shared memory: pixel operand slabs, ring, column-half exchange, barriers
__host__ __device__ constexpr int off_ring(int KS, int PT) { return PT * KS * 4096; }
__host__ __device__ constexpr int off_xchg(int KS, int PT) { return off_ring(KS, PT) + STAGES * tile_bytes(KS); }
__host__ __device__ constexpr int off_bars(int KS, int PT) { return off_xchg(KS, PT) + PT * 128 * 12; }
// (a floor on it keeps a third CTA off the SM, so that tensor memory never runs out)
__host__ __device__ constexpr int smem_bytes(int KS, int PT) {
    return off_bars(KS, PT) + 32 < 80 * 1024 ? 80 * 1024 : off_bars(KS, PT) + 32;
}

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ uint64_t pk2(float lo, float hi) {
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ void unpk2(uint64_t v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}

// 2^x of both halves.
__device__ __forceinline__ uint64_t ex2x2(uint64_t v) {
    uint64_t d;
    asm("{\n\t.reg .f32 x, y;\n\tmov.b64 {x, y}, %1;\n\t"
        "ex2.approx.ftz.f32 x, x;\n\tex2.approx.ftz.f32 y, y;\n\t"
        "mov.b64 %0, {x, y};\n\t}"
        : "=l"(d)
        : "l"(v));
    return d;
}
__device__ __forceinline__ uint64_t neg2(uint64_t v) { return v ^ 0x8000000080000000ull; }

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src)
                 : "memory");
}

// rho, -log2(e)/(2 s2), -log2(e)/beta and the location variance s2
// (rho^2, or rho itself when rho is read as the variance)
__device__ __forceinline__ void label_consts(int D, float alpha, float d_min, float kappa_beta,
                                             bool rho_var, float& rho, float& nA, float& nB) {
    float d = sqrtf((float)D);
    rho = alpha * fmaxf(d, d_min);
    nA = -LOG2E / (2.f * (rho_var ? rho : rho * rho));
    nB = -LOG2E / (kappa_beta * rho);
}

// The four bytes of a nibble's codes: `one` where the bit is set, else 0.
__device__ __forceinline__ uint32_t spread(uint32_t nibble, uint32_t one) {
    return (nibble * 0x00204081u & 0x01010101u) * one;
}
constexpr uint32_t E4M3_ONE = 0x38u, E4M3_MINUS = 0xB8u;
// e4m3 of -v, v an integer below 16 times a power of two (four significant bits: exact)
__device__ __forceinline__ uint32_t e4m3_minus(int v) {
    if (v == 0) return 0u;
    const int ex = 31 - __clz(v);
    return 0x80u | (uint32_t)(ex + 7) << 3 | (uint32_t)(((v << 3) >> ex) & 7);
}

// Bytes of a tile of the few-samples form: the planes, then the codes' words as planes.
__host__ __device__ constexpr int few_tile_bytes(int Wk) { return (5 + Wk) * TS * 4; }

// Sample tiles: one thread per (tile, sample). Padded samples lie far away (their
// terms vanish) and have no codes. words > 0: the few-samples form's layout.
__global__ void __launch_bounds__(256) plain_tiles_kernel(
    const float* __restrict__ img, int W, long long P, const uint32_t* __restrict__ bitmask, int Wk,
    const int32_t* __restrict__ label_off, const int32_t* __restrict__ tile_off, int n_labels,
    const int32_t* __restrict__ sample_pix, int total_tiles, int k, int KS, int words,
    uint8_t* __restrict__ blob) {
    const long long gid = blockIdx.x * 256ll + threadIdx.x;
    if (gid >= (long long)total_tiles * TS) return;
    const int tile = (int)(gid / TS), r = (int)(gid % TS);
    int lo = 0, hi = n_labels - 1;  // label of this tile
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (tile_off[mid] <= tile) lo = mid; else hi = mid - 1;
    }
    const int s = label_off[lo] + (tile - tile_off[lo]) * TS + r;
    const bool ok = s < label_off[lo + 1];
    uint8_t* base = blob + (size_t)tile * (words ? few_tile_bytes(words) : tile_bytes(KS));
    float* f = reinterpret_cast<float*>(base);
    int pix = ok ? sample_pix[s] : 0;
    if (pix < 0 || pix >= P) pix = 0;  // reported by the distance transform's seed pass
    f[r] = ok ? (float)(pix % W) : FAR;
    f[TS + r] = ok ? (float)(pix / W) : 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) f[(2 + c) * TS + r] = ok ? img[(size_t)pix * 3 + c] : 0.f;
    for (int w = 0; w < words; ++w)
        reinterpret_cast<uint32_t*>(f)[(5 + w) * TS + r] =
            ok ? bitmask[(size_t)pix * Wk + w] & code_mask(w, k) : 0u;
    for (int w = 0; w < KS; ++w) {
        uint32_t bits = ok && w < Wk ? bitmask[(size_t)pix * Wk + w] & code_mask(w, k) : 0u;
        for (int c = k; c < k + 2; ++c)  // the columns of -|b_x|
            if (c >> 5 == w) bits |= 1u << (c & 31);
        uint8_t* slab = base + 5 * TS * 4 + w * TS * 32;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            uint32_t v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = spread((bits >> (16 * h + 4 * q)) & 15u, E4M3_ONE);
            *reinterpret_cast<uint4*>(slab + tc::slab_off(r, 16 * h)) =
                make_uint4(v[0], v[1], v[2], v[3]);
        }
    }
}

// Waits for the MMAs of one tile, for wait_ns (0: PLAIN_WAIT_NS) at most.
__device__ __forceinline__ bool plain_wait(uint64_t* bars, MmaPhase p, uint64_t wait_ns) {
    uint64_t deadline = 0;
    for (uint32_t n = 0;; ++n) {
        if (tc::mbar_try_wait(bars + p.bar, p.parity, 1000u)) return true;
        if ((n & 63u) == 63u) {
            const uint64_t now = tc::globaltimer();
            if (deadline == 0) deadline = now + (wait_ns ? wait_ns : PLAIN_WAIT_NS);
            else if (now > deadline) return false;
        }
    }
}

// KS: 32-column steps of the texture (0: no texture in the pairs, the factorised
// and smooth forms); PT: 128-pixel operand tiles per CTA (one where two would
// leave SMs without a CTA). Bound: the FP32 pipe (15 packed operations per two pairs
// with the texture, the running maximum beside them in the integer pipe: 0.63 ms at
// 481 x 321, 10,000 samples). Measured there: 0.97 ms, against 1.65 ms with population
// counts, nine shared-memory words read per pair and scalar arithmetic.
template <int KS, int PT>
__global__ void __launch_bounds__(THREADS, 2) sum_plain_kernel(SumArgs a) {
    constexpr bool TEX = KS > 0;
    constexpr int TB = tile_bytes(KS), BP = 128 * PT;
    constexpr uint32_t NCOL = 2 * PT * TS;  // tensor-memory columns: two accumulators
    extern __shared__ __align__(1024) uint8_t smem[];
    uint8_t* ring = smem + off_ring(KS, PT);
    float* xchg = reinterpret_cast<float*>(smem + off_xchg(KS, PT));  // [3][PT][128]
    // [2] MMA commits, then one that nothing completes (the timeout-path test)
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + off_bars(KS, PT));
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(bars + 3);
    const long long P = (long long)a.H * a.W;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int row = 32 * (warp & 3) + lane, hf = warp >> 2;  // operand row, column half
    const float nC = -LOG2E / (2.f * a.sigma_c2);
    const float log_col_norm = 1.5f * logf(6.283185307179586f * a.sigma_c2);
    const uint64_t nC2 = pk2(nC, nC);
    // work items: every pixel, or the pixels of a device list (count on the device)
    const long long n_items = a.pix_list ? (long long)min(*a.list_count, a.list_cap) : P;
    const long long n_units = (n_items + BP - 1) / BP * a.n_labels;
    const int32_t* tile_off = a.d_label_off + a.n_labels + 1;
    auto pixel_of = [&](long long it) {
        return it < n_items ? (a.pix_list ? (long long)a.pix_list[it] : it) : 0ll;
    };
    uint32_t tmem = 0;
    if (TEX) {
        if (tid == 0) {
            tc::mbar_init(bars, 1);
            tc::mbar_init(bars + 1, 1);
            tc::mbar_init(bars + 2, 1);
            tc::fence_mbar_init();
        }
        if (warp == 0) {
            tc::tmem_alloc(s_tmem, NCOL);
            tc::tmem_relinquish();
        }
        tc::fence_before_sync();
        __syncthreads();
        tc::fence_after_sync();
        tmem = *s_tmem;
    }
    uint32_t it0 = 0;  // tiles issued before this unit
    bool ok = true;
    // the timeout-path test: the last block gives up before it issues anything
    if (TEX && a.stall && blockIdx.x == gridDim.x - 1)
        ok = __syncthreads_and(tid != 0 || plain_wait(bars, MmaPhase{2u, 0u}, a.wait_ns));

    for (long long unit = blockIdx.x; ok && unit < n_units; unit += gridDim.x) {
        const int i = (int)(unit % a.n_labels);
        const long long item0 = unit / a.n_labels * BP;
        const int nt = tile_off[i + 1] - tile_off[i];
        const uint8_t* src = a.t.blob + (size_t)tile_off[i] * TB;
        __syncthreads();  // the ring, the operands and the exchange are free (the unit before)
        auto copy = [&](int T) {
            if (T < nt) {
                uint8_t* dst = ring + (T % STAGES) * TB;
                for (int c = 16 * tid; c < TB; c += 16 * THREADS)
                    cp_async16(dst + c, src + (size_t)T * TB + c);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        copy(0);
        copy(1);
        // operand row of pixel tid (PT = 1: the first 128 threads)
        if (TEX && tid < BP) {
            const uint32_t* bx = a.bitmask + pixel_of(item0 + tid) * a.Wk;
            int pop = -__popc(bx[a.Wk - 1] & ~code_mask(a.Wk - 1, a.k));  // (bits that are no codes)
            for (int w = 0; w < a.Wk; ++w) pop += __popc(bx[w]);
            const uint32_t hi = e4m3_minus(pop & ~15), lo = e4m3_minus(pop & 15);
#pragma unroll
            for (int w = 0; w < KS; ++w) {
                const int left = a.k - 32 * w;  // codes from this step on
                const uint32_t valid = code_mask(w, a.k);
                const uint32_t bits = left > 0 ? bx[w] : 0u;
                uint32_t v[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    v[q] = spread(((bits & valid) >> (4 * q)) & 15u, E4M3_ONE) |
                           spread(((~bits & valid) >> (4 * q)) & 15u, E4M3_MINUS);
                    const int c0 = left - 4 * q, c1 = c0 + 1;  // the columns of -|b_x|
                    if (c0 >= 0 && c0 < 4) v[q] |= hi << (8 * c0);
                    if (c1 >= 0 && c1 < 4) v[q] |= lo << (8 * c1);
                }
                uint8_t* slab = smem + ((tid >> 7) * KS + w) * 4096;
                *reinterpret_cast<uint4*>(slab + tc::slab_off(tid & 127, 0)) =
                    make_uint4(v[0], v[1], v[2], v[3]);
                *reinterpret_cast<uint4*>(slab + tc::slab_off(tid & 127, 16)) =
                    make_uint4(v[4], v[5], v[6], v[7]);
            }
        }
        // this thread's pixels: values negated (differences by additions) and doubled
        uint64_t px[PT], py[PT], pr[PT], pg[PT], pb[PT], nA2[PT], nB2[PT];
        float M[PT], S[PT], Cc[PT];
#pragma unroll
        for (int t = 0; t < PT; ++t) {
            const long long pq = pixel_of(item0 + 128 * t + row);
            const float x = -(float)(pq % a.W), y = -(float)(pq / a.W);
            const float r = -a.img[pq * 3], gr = -a.img[pq * 3 + 1], b = -a.img[pq * 3 + 2];
            float rho, nA, nB;
            label_consts(a.dist2[(size_t)i * P + pq], a.alpha, a.d_min, a.kappa_beta, a.rho_var, rho,
                         nA, nB);
            px[t] = pk2(x, x);
            py[t] = pk2(y, y);
            pr[t] = pk2(r, r);
            pg[t] = pk2(gr, gr);
            pb[t] = pk2(b, b);
            nA2[t] = pk2(nA, nA);
            nB2[t] = pk2(-nB, -nB);  // times -TSM
            M[t] = LOWEST;
            S[t] = Cc[t] = 0.f;
        }

        // the exponents and sums of tile T
        auto sum_tile = [&](int T) {
            const uint32_t it = it0 + (uint32_t)T, b = mma_phase(it).bar;
            if (TEX) {
                // (one decision per warp: the load below takes the whole warp)
                ok = __all_sync(0xffffffffu, plain_wait(bars, mma_phase(it), a.wait_ns));
                if (!ok) return;
                tc::fence_after_sync();
            }
            const ulonglong2* sp =
                reinterpret_cast<const ulonglong2*>(ring + (T % STAGES) * TB) + 8 * hf;
            float ts[PT];  // the tile's sums, relative to M
#pragma unroll
            for (int t = 0; t < PT; ++t) ts[t] = 0.f;
#pragma unroll
            for (int c = 0; c < 2; ++c) {  // 16 samples at a time
                uint64_t e[PT][8];         // -TSM, then the exponents
                if (TEX) {
#pragma unroll
                    for (int t = 0; t < PT; ++t)
                        tc::tmem_ld16_wait_pk(tmem + ((uint32_t)(32 * (warp & 3)) << 16) +
                                                  (b * PT + t) * TS + 32 * hf + 16 * c,
                                              e[t]);
                }
#pragma unroll
                for (int n = 0; n < 4; ++n) {
                    const ulonglong2 x = sp[4 * c + n], y = sp[TS / 4 + 4 * c + n],
                                     r = sp[TS / 2 + 4 * c + n], g = sp[3 * TS / 4 + 4 * c + n],
                                     bl = sp[TS + 4 * c + n];
                    auto expo = [&](int t, uint64_t sx, uint64_t sy, uint64_t sr, uint64_t sg,
                                    uint64_t sb, uint64_t h) {
                        const uint64_t dx = add2(sx, px[t]), dy = add2(sy, py[t]);
                        const uint64_t d2 = fma2(dx, dx, mul2(dy, dy));
                        const uint64_t dr = add2(sr, pr[t]), dg = add2(sg, pg[t]),
                                       db = add2(sb, pb[t]);
                        const uint64_t c2 = fma2(dr, dr, fma2(dg, dg, mul2(db, db)));
                        const uint64_t col = TEX ? fma2(nC2, c2, mul2(nB2[t], h)) : mul2(nC2, c2);
                        return fma2(nA2[t], d2, col);
                    };
#pragma unroll
                    for (int t = 0; t < PT; ++t) {
                        e[t][2 * n] = expo(t, x.x, y.x, r.x, g.x, bl.x, e[t][2 * n]);
                        e[t][2 * n + 1] = expo(t, x.y, y.y, r.y, g.y, bl.y, e[t][2 * n + 1]);
                    }
                }
#pragma unroll
                for (int t = 0; t < PT; ++t) {
                    float mx = LOWEST;
#pragma unroll
                    for (int n = 0; n < 8; ++n) {
                        float lo, hi;
                        unpk2(e[t][n], lo, hi);
                        mx = fmaxf(mx, fmaxf(lo, hi));
                    }
                    if (mx > M[t]) {
                        const float sc = ex2(M[t] - mx);
                        S[t] *= sc;
                        Cc[t] *= sc;
                        ts[t] *= sc;
                        M[t] = mx;
                    }
                    const uint64_t nM = pk2(-M[t], -M[t]);
                    uint64_t s0 = 0, s1 = 0;  // (0.f, 0.f)
#pragma unroll
                    for (int n = 0; n < 8; n += 2) {
                        s0 = add2(s0, ex2x2(add2(e[t][n], nM)));
                        s1 = add2(s1, ex2x2(add2(e[t][n + 1], nM)));
                    }
                    float lo, hi;
                    unpk2(add2(s0, s1), lo, hi);
                    ts[t] += lo + hi;
                }
            }
#pragma unroll
            for (int t = 0; t < PT; ++t) {
                // TwoSum: S + ts = s + err exactly
                const float s = S[t] + ts[t];
                const float bb = s - S[t];
                Cc[t] += (S[t] - (s - bb)) + (ts[t] - bb);
                S[t] = s;
            }
        };

        int T = 0;
        for (; T <= nt; ++T) {
            if (T < nt) asm volatile("cp.async.wait_group 1;" ::: "memory");
            if (TEX) {
                tc::fence_proxy_async_smem();  // this thread's copies and operand rows
                tc::fence_before_sync();       // and its tensor-memory reads (tile T - 2)
            }
            // tile T is here; tile T - 2 is summed: its accumulator and place are free
            if (!(ok = __syncthreads_and(ok))) break;
            if (T < nt) {
                if (TEX && tid == 0) {
                    tc::fence_after_sync();
                    const uint32_t b = mma_phase(it0 + (uint32_t)T).bar;
                    const uint32_t al = tc::desc_lo(smem);
                    const uint32_t bl = tc::desc_lo(ring + (T % STAGES) * TB + 5 * TS * 4);
                    constexpr uint32_t id = tc::idesc(128, TS, 0, 0);
#pragma unroll
                    for (int t = 0; t < PT; ++t)
#pragma unroll
                        for (int w = 0; w < KS; ++w)
                            tc::mma_fp8(tmem + (b * PT + t) * TS,
                                        tc::desc_of(al + (t * KS + w) * 256, tc::DESC_HI),
                                        tc::desc_of(bl + w * (TS * 32 / 16), tc::DESC_HI), id, w > 0);
                    tc::mma_commit(bars + b);
                }
                copy(T + 2);
            }
            if (T > 0) sum_tile(T - 1);
        }
        it0 += (uint32_t)min(T, nt);  // (a wait that gave up leaves the loop before tile T)

        // the pixel's two threads: common maximum, scaled sums
        if (hf == 1)
#pragma unroll
            for (int t = 0; t < PT; ++t) {
                xchg[t * 128 + row] = M[t];
                xchg[(PT + t) * 128 + row] = S[t];
                xchg[(2 * PT + t) * 128 + row] = Cc[t];
            }
        if (!(ok = __syncthreads_and(ok))) break;
        if (hf == 1) continue;
        const float logm = logf((float)(a.d_label_off[i + 1] - a.d_label_off[i]));
#pragma unroll
        for (int t = 0; t < PT; ++t) {
            const long long it = item0 + 128 * t + row;
            if (it >= n_items) continue;
            const float M1 = xchg[t * 128 + row], mx = fmaxf(M[t], M1);
            const float w0 = ex2(M[t] - mx), w1 = ex2(M1 - mx);
            const float s = S[t] * w0 + xchg[(PT + t) * 128 + row] * w1;
            const float c = Cc[t] * w0 + xchg[(2 * PT + t) * 128 + row] * w1;
            const float lse = (mx + log2f(s + c)) * LN2;
            if (a.T_out) {  // log kernel sum only (surrogate targets), compact layout
                a.T_out[(size_t)i * a.list_cap + it] = lse;
                continue;
            }
            const long long pq = pixel_of(it);
            float rho, nA, nB;
            label_consts(a.dist2[(size_t)i * P + pq], a.alpha, a.d_min, a.kappa_beta, a.rho_var, rho,
                         nA, nB);
            const float s2 = a.rho_var ? rho : rho * rho;
            const float L = lse - logm - logf(6.283185307179586f * s2) - log_col_norm;
            a.neglog[(size_t)i * P + pq] = -L;
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (TEX) {
        if (!ok && tid == 0) {
            if (atomicCAS(a.d_err, 0, CS_DEVERR_TIMEOUT) == 0) a.d_err[1] = 51;
            // MMAs still in flight: they must finish before the tensor memory is
            // freed and the operands' shared memory goes to another CTA
            MmaPhase last;
            if (mma_last(it0, last)) plain_wait(bars, last, a.wait_ns);
        }
        tc::fence_before_sync();
        __syncthreads();
        if (warp == 0) {
            tc::fence_after_sync();
            tc::tmem_dealloc(tmem, NCOL);
        }
    }
}

// Label normalisation (and the factorised texture posterior) of pixel q.
__device__ __forceinline__ void normalise_plain(const SumArgs& a, long long P, long long q) {
    if (a.mode == CS_MODE_FACTORISED) {
        const uint32_t* bx = a.bitmask + (size_t)q * a.Wk;
        const int pad = __popc(bx[a.Wk - 1] & ~code_mask(a.Wk - 1, a.k));  // bits that are no codes
        auto logit = [&](int i) {
            float rho, nA, nB;
            label_consts(a.dist2[(size_t)i * P + q], a.alpha, a.d_min, a.kappa_beta, a.rho_var,
                         rho, nA, nB);
            int h = -pad;
            for (int w = 0; w < a.Wk; ++w) h += __popc(bx[w] ^ a.t.rep[i * a.Wk + w]);
            return nB * (float)h;
        };
        float tmax = -INFINITY;
        for (int i = 0; i < a.n_labels; ++i) tmax = fmaxf(tmax, logit(i));
        float ts = 0.f;
        for (int i = 0; i < a.n_labels; ++i) ts += ex2(logit(i) - tmax);
        const float tlse2 = tmax + log2f(ts);
        for (int i = 0; i < a.n_labels; ++i)  // texture log-posterior, natural log
            a.neglog[(size_t)i * P + q] -= (logit(i) - tlse2) * LN2;
    }
    if (!a.post) return;
    float lmax = -INFINITY;
    for (int i = 0; i < a.n_labels; ++i) lmax = fmaxf(lmax, -a.neglog[(size_t)i * P + q]);
    float ls = 0.f;
    for (int i = 0; i < a.n_labels; ++i) ls += expf(-a.neglog[(size_t)i * P + q] - lmax);
    const float lse = lmax + logf(ls);
    for (int i = 0; i < a.n_labels; ++i)
        a.post[(size_t)i * P + q] = expf(-a.neglog[(size_t)i * P + q] - lse);
}
__global__ void __launch_bounds__(256) normalise_plain_kernel(SumArgs a) {
    const long long P = (long long)a.H * a.W;
    const long long n_items = a.pix_list ? (long long)min(*a.list_count, a.list_cap) : P;
    for (long long it = blockIdx.x * 256ll + threadIdx.x; it < n_items;
         it += (long long)gridDim.x * 256)
        normalise_plain(a, P, a.pix_list ? (long long)a.pix_list[it] : it);
}

// The few-samples form: a thread per pixel, all labels in turn; sums as in the general
// form's comment, with the running maximum and the TwoSum per 16 samples. Bound: with
// the texture, the population counts (WK a pair, 16 per clock and SM). WK: words of the
// texture (0: none in the pairs). Measured, sum and normalisation, us, against the
// general form: 2048 x 1024, 4 labels of 10 samples, k = 50: 190, 865; factorised: 232,
// 607; 481 x 321, 5 x 60, k = 98: 66, 99; 320 x 240, 64 x 40, k = 98: 318, 560.
constexpr int FEW_THREADS = 128;
template <int WK>
__global__ void __launch_bounds__(FEW_THREADS) sum_few_kernel(SumArgs a) {
    constexpr int TB = few_tile_bytes(WK), CH = 16;
    __shared__ __align__(16) float s_tile[TB / 4];  // x, y, r, g, b, words
    const uint32_t* s_bits = reinterpret_cast<const uint32_t*>(s_tile + 5 * TS);
    const long long P = (long long)a.H * a.W;
    const int tid = threadIdx.x;
    const float nC = -LOG2E / (2.f * a.sigma_c2);
    const float log_col_norm = 1.5f * logf(6.283185307179586f * a.sigma_c2);
    const int n_items = a.pix_list ? min(*a.list_count, a.list_cap) : (int)P;
    const int32_t* tile_off = a.d_label_off + a.n_labels + 1;
    // a tile is read ahead into registers while the one before is summed (the labels'
    // tiles follow one another)
    constexpr int NV = (TB / 16 + FEW_THREADS - 1) / FEW_THREADS;
    const int n_tiles = tile_off[a.n_labels];
    uint4 ahead[NV];
    auto read = [&](int T) {
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            const int c = tid + v * FEW_THREADS;
            if (c < TB / 16 && T < n_tiles)
                ahead[v] = reinterpret_cast<const uint4*>(a.t.blob + (size_t)T * TB)[c];
        }
    };
    for (long long base = (long long)blockIdx.x * FEW_THREADS; base < n_items;
         base += (long long)gridDim.x * FEW_THREADS) {
        read(0);
        const int it = (int)base + tid;
        const bool live = it < n_items;
        const int q = live ? (a.pix_list ? a.pix_list[it] : it) : 0;
        const float px = (float)(q % a.W), py = (float)(q / a.W);
        const float* I = a.img + (size_t)q * 3;
        const float pr = I[0], pg = I[1], pb = I[2];
        uint32_t bits[WK > 0 ? WK : 1];
#pragma unroll
        for (int w = 0; w < WK; ++w) bits[w] = a.bitmask[(size_t)q * WK + w] & code_mask(w, a.k);
        for (int i = 0; i < a.n_labels; ++i) {
            float rho, nA, nB, M = LOWEST, S = 0.f, Cc = 0.f;
            label_consts(a.dist2[(size_t)i * P + q], a.alpha, a.d_min, a.kappa_beta, a.rho_var, rho,
                         nA, nB);
            const int m = a.d_label_off[i + 1] - a.d_label_off[i];
            for (int T = tile_off[i]; T < tile_off[i + 1]; ++T) {
                __syncthreads();
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    const int c = tid + v * FEW_THREADS;
                    if (c < TB / 16) reinterpret_cast<uint4*>(s_tile)[c] = ahead[v];
                }
                __syncthreads();
                read(T + 1);
                const int nvalid = min(TS, m - (T - tile_off[i]) * TS);
                for (int c0 = 0; c0 < nvalid; c0 += CH) {
                    float e[CH], mx = LOWEST;
#pragma unroll
                    for (int c = 0; c < CH; ++c) {
                        const int j = c0 + c;
                        const float dx = px - s_tile[j], dy = py - s_tile[TS + j];
                        const float dr = pr - s_tile[2 * TS + j], dg = pg - s_tile[3 * TS + j],
                                    db = pb - s_tile[4 * TS + j];
                        const float d2 = fmaf(dx, dx, dy * dy);
                        const float c2 = fmaf(dr, dr, fmaf(dg, dg, db * db));
                        float col = nC * c2;
                        if (WK > 0) {
                            int h = 0;
#pragma unroll
                            for (int w = 0; w < WK; ++w) h += __popc(bits[w] ^ s_bits[w * TS + j]);
                            col = fmaf(nC, c2, nB * (float)h);
                        }
                        e[c] = fmaf(nA, d2, col);
                        mx = fmaxf(mx, e[c]);
                    }
                    if (mx > M) {
                        const float sc = ex2(M - mx);
                        S *= sc;
                        Cc *= sc;
                        M = mx;
                    }
                    float ts = 0.f;
#pragma unroll
                    for (int c = 0; c < CH; ++c) ts += ex2(e[c] - M);
                    // TwoSum: S + ts = s + err exactly
                    const float s = S + ts, bb = s - S;
                    Cc += (S - (s - bb)) + (ts - bb);
                    S = s;
                }
            }
            if (!live) continue;
            const float lse = (M + log2f(S + Cc)) * LN2;
            if (a.T_out) {  // log kernel sum only (surrogate targets), compact layout
                a.T_out[(size_t)i * a.list_cap + it] = lse;
                continue;
            }
            const float s2 = a.rho_var ? rho : rho * rho;
            a.neglog[(size_t)i * P + q] =
                -(lse - logf((float)m) - logf(6.283185307179586f * s2) - log_col_norm);
        }
        if (live && !a.T_out) normalise_plain(a, P, q);
    }
}

int steps_of(const SumArgs& a) { return a.mode == CS_MODE_PERSAMPLE ? steps_for(a.k) : 0; }

template <class F>
cudaError_t with_steps(int KS, F&& f) {
    switch (KS) {
        case 0: return f(std::integral_constant<int, 0>{});
        case 1: return f(std::integral_constant<int, 1>{});
        case 2: return f(std::integral_constant<int, 2>{});
        case 3: return f(std::integral_constant<int, 3>{});
        case 4: return f(std::integral_constant<int, 4>{});
        case 5: return f(std::integral_constant<int, 5>{});
        case 6: return f(std::integral_constant<int, 6>{});
        case 7: return f(std::integral_constant<int, 7>{});
        case 8: return f(std::integral_constant<int, 8>{});
        case 9: return f(std::integral_constant<int, 9>{});
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

int plain_tiles_per_label(int m) { return (m + TS - 1) / TS; }

// The few-samples form? Its cost goes with the samples, padded to 16 per label, and
// their words; the general form's with 64-sample tiles and units. With the texture the
// two meet near 200 samples a label at four words, 128 at six; and the few-samples form
// needs pixels, which is all it works on in parallel. Measured, tiles, sum and
// normalisation, us, few and general (k = 98; samples per label x labels):
//   481 x 321: 16 x 5 36, 105; 64 x 5 71, 105; 130 x 5 138, 161; 200 x 5 191, 191
//   320 x 240: 130 x 16 .90 of the general form's; 240 x 180: 64 x 16 .91, 100 x 16
//   1.17; 200 x 100: 16 x 16 .69, 40 x 16 1.06; 96 x 64: 64 x 2 .88, 100 x 2 1.07
//   (factorised, 481 x 321: 16 x 5 .51, 64 x 5 .77, 200 x 5 .85)
bool plain_few(int H, int W, int k, int n_labels, const int32_t* label_off, bool persample) {
    const long long P = (long long)H * W;
    long long padded = 0;
    for (int i = 0; i < n_labels; ++i) padded += (label_off[i + 1] - label_off[i] + 15) / 16 * 16;
    const int most = persample && (k + 31) / 32 > 4 ? 768 / ((k + 31) / 32) : 192;
    return padded <= (long long)most * n_labels && (P >= 60000 || 40 * padded <= P);
}

size_t plain_tile_bytes(int k, bool persample, bool few) {
    return few ? (size_t)few_tile_bytes(persample ? (k + 31) / 32 : 0)
               : (size_t)tile_bytes(persample ? steps_for(k) : 0);
}

cudaError_t launch_plain_tiles(const float* img, int H, int W, const uint32_t* bitmask, int k,
                               int n_labels, const int32_t* d_label_off,
                               const int32_t* sample_pix, int total_tiles, bool persample,
                               bool few, uint8_t* blob, cudaStream_t st) {
    const long long n = (long long)total_tiles * TS;
    plain_tiles_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(
        img, W, (long long)H * W, bitmask, (k + 31) / 32, d_label_off, d_label_off + n_labels + 1,
        n_labels, sample_pix, total_tiles, k, persample && !few ? steps_for(k) : 0,
        persample && few ? (k + 31) / 32 : 0, blob);
    return cudaGetLastError();
}

cudaError_t launch_sum_plain(const SumArgs& a, cudaStream_t st) {
    const long long n = a.pix_list ? (long long)a.list_cap : (long long)a.H * a.W;
    const long long most = 16ll * a.n_sm;
    if (a.few)
        return with_steps(a.mode == CS_MODE_PERSAMPLE ? a.Wk : 0, [&](auto wk) {
            constexpr int WK = decltype(wk)::value;
            long long blocks = (n + FEW_THREADS - 1) / FEW_THREADS;
            if (a.pix_list && blocks > most) blocks = most;  // grid-stride over the list
            sum_few_kernel<WK><<<(unsigned)(blocks < 1 ? 1 : blocks), FEW_THREADS, 0, st>>>(a);
            return cudaGetLastError();
        });
    const cudaError_t e = with_steps(steps_of(a), [&](auto ks) {
        constexpr int KS = decltype(ks)::value;
        auto run = [&](auto pt) {
            constexpr int PT = decltype(pt)::value;
            constexpr int smem = smem_bytes(KS, PT);
            static_assert(smem <= 227 * 1024, "shared memory budget");
            cudaError_t e2 = cudaFuncSetAttribute(
                sum_plain_kernel<KS, PT>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
            if (e2 != cudaSuccess) return e2;
            long long blocks = (n + 128 * PT - 1) / (128 * PT) * a.n_labels;
            if (a.pix_list && blocks > most) blocks = most;  // grid-stride over the list
            if (blocks > 0x7fffffffll) blocks = 0x7fffffffll;
            sum_plain_kernel<KS, PT><<<(unsigned)(blocks < 1 ? 1 : blocks), THREADS, smem, st>>>(a);
            return cudaGetLastError();
        };
        // two operand tiles share the samples' reads; one where the units of two
        // would not fill the SMs twice
        return (n + 255) / 256 * a.n_labels >= 2 * a.n_sm ? run(std::integral_constant<int, 2>{})
                                                          : run(std::integral_constant<int, 1>{});
    });
    if (e != cudaSuccess || a.T_out || (!a.post && a.mode != CS_MODE_FACTORISED)) return e;
    const long long blocks = (n + 255) / 256;
    normalise_plain_kernel<<<(unsigned)(blocks < most ? (blocks < 1 ? 1 : blocks) : most), 256, 0,
                             st>>>(a);
    return cudaGetLastError();
}
