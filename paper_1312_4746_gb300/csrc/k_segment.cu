// Convex multilabel segmentation on the data term (Sec. 4): the relaxed
// energy of Eq. (energy1) / Eq. (sets) minimised by the primal-dual
// iteration of Eq. (algo), then binarised by argmax.
//
// Discretisation (the paper gives none): forward differences with a zero
// difference across the last row / column for grad, its negative adjoint for
// div; edge weight g(x) = exp(-|grad I(x)| / gamma) / (2 gamma) with |grad I|
// the Euclidean norm of the forward differences of the three channels of
// 255 I; step sizes by diagonal preconditioning: 1/2 for xi and mu, 1/5 for
// u, 1/|Omega| for m; start u = 1/n, m = 1, xi = mu = 0.
//
// One persistent cooperative launch runs every iteration, in one of two forms:
//
// seg_tile_kernel  (images whose state fits the SMs' registers and shared
//   memory) One block per SM owns a 2D tile of the image: u and mu (and f where
//   the registers allow) live in registers, xi and ub in shared memory, with a
//   halo of one pixel. Each block also advances xi of the pixels left of and
//   above its tile (their state is part of its own), so that an iteration needs
//   one exchange only: the tile borders' ub, through global memory, and with a
//   label cost (nu > 0) the blocks' sums of mu. Every value travels with its
//   iteration's number in one 64-bit word, so the reader polls the values
//   themselves: no flag, no fence, no grid barrier. The buffers alternate; a
//   block writes one again only after it has read what its neighbours published
//   after reading it. Without a label cost m stays 1 exactly (m - (0 + sum mu) /
//   |Omega| >= 1 is clamped to 1), so the sums are not formed.
// seg_solve_kernel  (larger images, more than 16 labels) Each block owns a
//   contiguous range of pixels (all labels) and keeps its own copy of m in
//   shared memory; per iteration: the dual step (xi, mu and the block's sums of
//   mu per label), a grid barrier, the m step (every block sums the per-block
//   parts in the same fixed order, so all copies agree), the primal step, a
//   grid barrier. The state lies in global memory (in L2 while it fits).
//
// All waits are bounded: on timeout the kernel records the site in the error
// word, raises an abort flag that every other block sees, and returns.
#include <algorithm>
#include <atomic>
#include <cstdint>
#include <mutex>

#include "internal.h"

namespace {

constexpr int SB = 512;                         // threads per block
constexpr int NW = SB / 32;
constexpr unsigned long long SEG_WAIT_NS = 1000000000ull;  // 1 s per barrier

__device__ __forceinline__ uint64_t seg_clock() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Grid barrier on a monotonic arrival counter: barrier number `k` (from 1)
// completes when the counter reaches k * gridDim.x. bar[0] = counter,
// bar[1] = abort flag. Returns false (for the whole block) when this block
// gave up or another block raised the abort flag. `arrive` false (the
// timeout-path test) skips this block's arrival, so that no block's wait
// completes: every block gives up after `wait_ns` or on the abort flag.
__device__ bool grid_barrier(unsigned* bar, unsigned k, int* d_err, int site, int* s_ok,
                             uint64_t wait_ns, bool arrive = true) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (arrive) atomicAdd(bar, 1u);
        const unsigned target = k * gridDim.x;
        const uint64_t deadline = seg_clock() + wait_ns;
        int ok = 1;
        for (unsigned n = 0;; ++n) {
            if ((int)(ld_acquire(bar) - target) >= 0) break;
            if ((n & 63u) == 63u) {
                if (ld_acquire(bar + 1)) {
                    ok = 0;
                    break;
                }
                if (seg_clock() > deadline) {
                    if (atomicCAS(d_err, 0, CS_DEVERR_TIMEOUT) == 0) d_err[1] = site;
                    atomicExch(bar + 1, 1u);
                    ok = 0;
                    break;
                }
            }
        }
        __threadfence();
        *s_ok = ok;
    }
    __syncthreads();
    return *s_ok != 0;
}

// Ascent and projection of one xi: (vx, vy) + 1/2 (dx, dy), scaled back to
// length bd where it is longer. (The minimum also takes the 1 where the length
// is 0 or its square denormal: the reciprocal root is then infinite.)
__device__ __forceinline__ void dual_step(float dx, float dy, float bd, float& vx, float& vy) {
    vx += 0.5f * dx;
    vy += 0.5f * dy;
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(vx * vx + vy * vy));
    const float sc = fminf(1.f, bd * r);
    vx *= sc;
    vy *= sc;
}

// Michelot's projection of v[0 .. n-1] onto the simplex: returns the shift t,
// the projection being max(v - t, 0). Each round takes the mean excess of the
// entries that the last shift left non-negative; the shifts only grow, so an
// entry dropped once stays dropped, and the rounds end when none is. The first
// shift comes from the entries with start[i] > 0, the support that the last
// iteration ended with: the shift of any set is at most the final one, so every
// entry of the final support passes it, and two rounds usually do where the
// full set takes five or six. (Comparisons are negated so that a NaN keeps
// every entry, as the definition does, and spreads.)
template <int N>
__device__ __forceinline__ float michelot(const float (&v)[N], const float (&start)[N], int n) {
    float s = 0.f, cnt = 0.f;
#pragma unroll
    for (int i = 0; i < N; ++i)
        if (i < n && start[i] > 0.f) {
            s += v[i];
            cnt += 1.f;
        }
    float t = __fdividef(s - 1.f, cnt);
    cnt = 0.f;
    for (int round = 0; round <= n; ++round) {
        float s2 = 0.f, c2 = 0.f;
#pragma unroll
        for (int i = 0; i < N; ++i)
            if (i < n && !(v[i] < t)) {
                s2 += v[i];
                c2 += 1.f;
            }
        if (c2 == cnt) break;
        cnt = c2;
        t = __fdividef(s2 - 1.f, cnt);
    }
    return t;
}

// State that other blocks write during the launch (u, ub, px, py, mu, parts)
// is read through plain pointers (no read-only cache path).
struct SegState {
    const float* f;
    const float* img;
    float* u;
    float* ub;
    float* px;
    float* py;
    float* mu;
    float* bound;
    float* parts;  // n x gridDim.x sums of mu
    unsigned* bar;
    int32_t* labels;
    int* d_err;
    int H, W, n, iterations;
    float lambda, nu, gamma;
    uint64_t wait_ns;  // limit of each grid-barrier wait
    bool stall;        // the last block skips its arrival at the first barrier of the iterations
};

// N: the label count when it is at most 8 (every label loop unrolled
// exactly), else an upper bound (16 or CS_MAX_LABELS, loops guarded by
// i < n). I: the element index type, int when n |Omega| fits. The dual step
// takes the labels in groups of 4 so that each group's loads are in flight
// together; the primal step holds the pixel's labels in registers.
template <int N, typename I>
__global__ void __launch_bounds__(SB, 2) seg_solve_kernel(SegState S) {
    constexpr bool EXACT = N <= 8;
    __shared__ float red[CS_MAX_LABELS][NW];
    __shared__ float s_m[CS_MAX_LABELS], s_mb[CS_MAX_LABELS];
    __shared__ int s_ok;
    const int P = S.H * S.W;  // H W < 2^31 (checked by the caller)
    const int n = EXACT ? N : S.n;
    const int W = S.W, H = S.H;
    const int G = gridDim.x, b = blockIdx.x;
    const int chunk = (int)(((long long)P + G - 1) / G);
    const int q0 = (int)((long long)b * chunk < P ? (long long)b * chunk : P);
    const int q1 = (int)((long long)q0 + chunk < P ? (long long)q0 + chunk : P);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

    // edge weight bound lambda g / 2 and the start point, own pixels
    for (int q = q0 + threadIdx.x; q < q1; q += SB) {
        const int y = q / W, x = q - y * W;
        float s = 0.f;
        for (int c = 0; c < 3; ++c) {
            const float v = 255.f * S.img[(size_t)q * 3 + c];
            const float dx = x + 1 < W ? 255.f * S.img[(size_t)(q + 1) * 3 + c] - v : 0.f;
            const float dy = y + 1 < H ? 255.f * S.img[(size_t)(q + W) * 3 + c] - v : 0.f;
            s = fmaf(dx, dx, fmaf(dy, dy, s));
        }
        S.bound[q] = 0.5f * S.lambda * (expf(-sqrtf(s) / S.gamma) / (2.f * S.gamma));
        for (int i = 0; i < n; ++i) {
            const I e = (I)i * P + q;
            S.u[e] = 1.f / (float)n;
            S.ub[e] = 1.f / (float)n;
            S.px[e] = 0.f;
            S.py[e] = 0.f;
            S.mu[e] = 0.f;
        }
    }
    for (int i = threadIdx.x; i < n; i += SB) s_m[i] = s_mb[i] = 1.f;
    unsigned nbar = 0;
    if (!grid_barrier(S.bar, ++nbar, S.d_err, 40, &s_ok, S.wait_ns)) return;

    const float inv_area = 1.f / (float)P;
    for (int it = 0; it < S.iterations; ++it) {
        // dual step: xi <- Pi_Kg(xi + 1/2 grad ub), mu <- min(0, mu + 1/2 (mb - ub))
#pragma unroll 1
        for (int i0 = 0; i0 < n; i0 += 4) {
            float acc[4] = {0.f, 0.f, 0.f, 0.f};
            for (int q = q0 + threadIdx.x; q < q1; q += SB) {
                const int y = q / W, x = q - y * W;
                const bool hr = x + 1 < W, hd = y + 1 < H;
                const float bd = S.bound[q];
                float c[4], gx[4], gy[4], ax[4], ay[4], m0[4];
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (i0 + j < n) {
                        const I e = (I)(i0 + j) * P + q;
                        c[j] = S.ub[e];
                        gx[j] = hr ? S.ub[e + 1] : 0.f;
                        gy[j] = hd ? S.ub[e + W] : 0.f;
                        ax[j] = S.px[e];
                        ay[j] = S.py[e];
                        m0[j] = S.mu[e];
                    }
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (i0 + j < n) {
                        const I e = (I)(i0 + j) * P + q;
                        dual_step(hr ? gx[j] - c[j] : 0.f, hd ? gy[j] - c[j] : 0.f, bd, ax[j],
                                  ay[j]);
                        S.px[e] = ax[j];
                        S.py[e] = ay[j];
                        const float m = fminf(0.f, m0[j] + 0.5f * (s_mb[i0 + j] - c[j]));
                        S.mu[e] = m;
                        acc[j] += m;
                    }
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float a = acc[j];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
                if (lane == 0 && i0 + j < n) red[i0 + j][warp] = a;
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += SB) {
            float s = 0.f;
            for (int w = 0; w < NW; ++w) s += red[i][w];
            S.parts[(size_t)i * G + b] = s;
        }
        if (!grid_barrier(S.bar, ++nbar, S.d_err, 41, &s_ok, S.wait_ns,
                          !(S.stall && it == 0 && b == G - 1)))
            return;

        // m step: m <- clamp(m - (nu + sum mu) / |Omega|, 0, 1), mb = 2 m_new - m;
        // one warp per label, the same summation order in every block
        for (int i = warp; i < n; i += NW) {
            float s = 0.f;
            for (int k = lane; k < G; k += 32) s += S.parts[(size_t)i * G + k];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) {
                const float mo = s_m[i];
                const float mn = fminf(1.f, fmaxf(0.f, mo - inv_area * (S.nu + s)));
                s_mb[i] = 2.f * mn - mo;
                s_m[i] = mn;
            }
        }

        // primal step per pixel: u <- Pi_simplex(u - 1/5 (-div xi + f - mu)) by
        // Michelot's algorithm over the labels, ub = 2 u_new - u
        for (int q = q0 + threadIdx.x; q < q1; q += SB) {
            const int y = q / W, x = q - y * W;
            float v[N], uo[N];
#pragma unroll
            for (int i = 0; i < N; ++i)
                if (EXACT || i < n) {
                    const I e = (I)i * P + q;
                    const float pxr = x + 1 < W ? S.px[e] : 0.f;
                    const float pxl = x > 0 ? S.px[e - 1] : 0.f;
                    const float pyd = y + 1 < H ? S.py[e] : 0.f;
                    const float pyu = y > 0 ? S.py[e - W] : 0.f;
                    const float d = (pxr - pxl) + (pyd - pyu);  // div xi
                    uo[i] = S.u[e];
                    v[i] = uo[i] - 0.2f * (-d + S.f[e] - S.mu[e]);
                }
            const float t = michelot<N>(v, uo, n);
#pragma unroll
            for (int i = 0; i < N; ++i)
                if (EXACT || i < n) {
                    const I e = (I)i * P + q;
                    const float un = v[i] < t ? 0.f : v[i] - t;
                    S.ub[e] = 2.f * un - uo[i];
                    S.u[e] = un;
                }
        }
        if (!grid_barrier(S.bar, ++nbar, S.d_err, 42, &s_ok, S.wait_ns)) return;
    }

    if (S.labels)
        for (int q = q0 + threadIdx.x; q < q1; q += SB) {
            int best = 0;
            float bv = S.u[q];
            for (int i = 1; i < n; ++i) {
                const float v = S.u[(I)i * P + q];
                if (v > bv) {
                    bv = v;
                    best = i;
                }
            }
            S.labels[q] = best;
        }
}

// the element index n P + P (the last label's plane plus a row) fits an int?
bool seg_narrow(long long P, int n) { return (long long)(n + 1) * P < (1ll << 31); }

// ---------------------------------------------------------------- tiles on chip

constexpr int TNT = 640;         // threads per block at most (5 warps per scheduler: 96 registers)
constexpr size_t SEG_SMEM = 227 * 1024;

// Shared-memory planes per label: xi's two (PS floats: tile plus the column
// left of it and the row above) and ub's (US: tile plus a ring). The strides
// are constants so that a label's offset is part of the instruction.
__host__ __device__ constexpr int seg_ps(int N, int PPT) {
    const int words = (int)(SEG_SMEM - 4096) / 4;
    const int room = (words - 96 * N) / (3 * N + 1), want = TNT * PPT + 48 + 32 * PPT;
    return room < want ? room : want;
}
__host__ __device__ constexpr int seg_us(int N, int PPT) { return seg_ps(N, PPT) + 96; }
__host__ __device__ constexpr size_t seg_tile_smem(int N, int PPT) {
    return sizeof(float) * ((size_t)N * (2 * seg_ps(N, PPT) + seg_us(N, PPT)) + seg_ps(N, PPT));
}

// border pixels of a tw x th tile
__host__ __device__ constexpr int seg_border(int tw, int th) {
    return tw < 3 || th < 3 ? tw * th : 2 * (tw + th) - 4;
}

// Place of border pixel (lx, ly) in the tile's order of border pixels.
__host__ __device__ constexpr int seg_border_place(int tw, int th, int lx, int ly) {
    return ly == 0        ? lx
           : ly == th - 1 ? tw + lx
           : lx == 0      ? 2 * tw + ly - 1
                          : 2 * tw + (th - 2) + ly - 1;
}

struct SegTile {
    const float* f;
    const float* img;
    float* u;
    // by iteration parity: ub of every tile's border pixels [tile][label][place]
    // and the blocks' sums of mu [label][tile], as (iteration << 32 | bits)
    unsigned long long* xch[2];
    unsigned long long* parts[2];
    unsigned* abort_flag;  // then a word that nothing sets (the timeout-path test)
    int32_t* labels;
    int* d_err;
    int H, W, iterations;
    int tw, th, gx, gy;  // tile size and tiles per row and column
    float lambda, nu, gamma;
    uint64_t wait_ns;
    bool stall;
};

// The same value, which with many labels the compiler does not know to be the
// same: what is formed from it is formed again in every iteration instead of
// taking the registers that the pixels' state needs.
template <int N>
__device__ __forceinline__ int opaque(int v) {
    if (N > 8) asm volatile("" : "+r"(v));
    return v;
}

__device__ __forceinline__ void put_tagged(unsigned long long* p, unsigned tag, float v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p),
                 "l"((unsigned long long)tag << 32 | __float_as_uint(v))
                 : "memory");
}
__device__ __forceinline__ unsigned long long get_tagged(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// The value at p once its tag is `tag`. Gives up (ok = 0) after the time limit,
// which it records and tells every block, or when another block has.
__device__ float wait_tagged(const SegTile& S, const unsigned long long* p, unsigned tag, int site,
                             int& ok) {
    unsigned long long v = get_tagged(p);
    uint64_t deadline = 0;
    for (unsigned t = 0; (unsigned)(v >> 32) != tag; ++t) {
        if ((t & 63u) == 63u) {
            const uint64_t now = seg_clock();
            if (deadline == 0) deadline = now + S.wait_ns;
            const bool late = now > deadline;
            if (late) {
                if (atomicCAS(S.d_err, 0, CS_DEVERR_TIMEOUT) == 0) S.d_err[1] = site;
                atomicExch(S.abort_flag, 1u);
            }
            if (late || ld_acquire(S.abort_flag)) {
                ok = 0;
                break;
            }
        }
        v = get_tagged(p);
    }
    return __uint_as_float((unsigned)v);
}

// lambda g / 2 at pixel (x, y)
__device__ __forceinline__ float seg_bound(const SegTile& S, int x, int y) {
    const size_t q = (size_t)y * S.W + x;
    float s = 0.f;
    for (int c = 0; c < 3; ++c) {
        const float v = 255.f * S.img[q * 3 + c];
        const float dx = x + 1 < S.W ? 255.f * S.img[(q + 1) * 3 + c] - v : 0.f;
        const float dy = y + 1 < S.H ? 255.f * S.img[(q + S.W) * 3 + c] - v : 0.f;
        s = fmaf(dx, dx, fmaf(dy, dy, s));
    }
    return 0.5f * S.lambda * (expf(-sqrtf(s) / S.gamma) / (2.f * S.gamma));
}

// N labels, PPT pixels per thread. The tile's border pixels come first in the
// threads' order. An iteration: the neighbours' border ub (and m), xi of the
// border and halo pixels; the border's primal step, published at once; then the
// interior's primal step and the interior's xi for the next iteration, under
// which the exchange runs. SUMS: nu > 0 (m varies, and mu waits for it).
//
// Bound: instruction issue (the two steps and the projection's rounds) and,
// for few labels, the exchange's latency that the interior does not cover.
// Measured at 481 x 321, 300 iterations: 1.06 ms (5 labels), 3.99 ms (16
// labels, nu = 1100), against 3.36 and 11.9 ms with the state in L2 and two grid
// barriers an iteration.
template <int N, int PPT, bool SUMS>
__global__ void __launch_bounds__(TNT, 1) seg_tile_kernel(SegTile S) {
    constexpr int PS = seg_ps(N, PPT), US = seg_us(N, PPT);
    constexpr bool FREG = 3 * N * PPT + N + 40 <= 96;  // f in registers too
    constexpr int NR = N <= 8 ? 8 : 16;                // labels of the sum reduction
    extern __shared__ __align__(16) float sm[];
    float* s_px = sm;                 // N x PS
    float* s_py = s_px + N * PS;      // N x PS
    float* s_ub = s_py + N * PS;      // N x US
    float* s_bd = s_ub + N * US;      // PS
    __shared__ float s_red[NR][TNT / 32 + 1];
    __shared__ float s_m[16], s_mb[16];
    const int tid = threadIdx.x, NT = blockDim.x, lane = tid & 31, warp = tid >> 5;
    const int W = S.W, H = S.H, tw = S.tw, th = S.th, G = gridDim.x;
    const int P = H * W;  // (N + 1) P < 2^31: the image fits the chip
    const int x0 = (int)(blockIdx.x % S.gx) * tw, y0 = (int)(blockIdx.x / S.gx) * th;
    const int pw = tw + 1, uw = tw + 2;  // row strides of the xi and ub windows

    // windows: xi = 0, ub = 1/n, bounds of the tile, its left column, its top row
    const float u0 = 1.f / (float)N;
    for (int t = tid; t < N * PS; t += NT) s_px[t] = s_py[t] = 0.f;
    for (int t = tid; t < N * US; t += NT) s_ub[t] = u0;
    for (int t = tid; t < pw * (th + 1); t += NT) {
        const int x = x0 - 1 + t % pw, y = y0 - 1 + t / pw;
        s_bd[t] = x >= 0 && y >= 0 && x < W && y < H ? seg_bound(S, x, y) : 0.f;
    }
    if (tid < 16) s_m[tid] = s_mb[tid] = 1.f;
    // this thread's pixels: the tile's nbord border pixels, then its interior
    const int nbord = seg_border(tw, th), iw = tw - 2;
    float u[PPT][N], mu[PPT][N], f[FREG ? PPT : 1][FREG ? N : 1];
    int pq[PPT];  // place in the image (-1: none)
    // places in the xi and ub windows and the steps to the right and lower neighbour
    // in the latter (0 at the image's edge), packed where registers are short
    constexpr bool PACK = N > 8;
    int at[PPT], ui[PACK ? 1 : PPT], rs[PACK ? 1 : PPT], ds[PACK ? 1 : PPT];
#pragma unroll
    for (int k = 0; k < PPT; ++k) {
        const int t = tid + k * NT;
        int lx, ly;
        if (t < nbord) {
            if (t < tw) {
                lx = t, ly = 0;
            } else if (t < 2 * tw && th > 1) {
                lx = t - tw, ly = th - 1;
            } else {
                const int c = t - 2 * tw, r = c < th - 2 ? c : c - (th - 2);
                lx = c < th - 2 ? 0 : tw - 1;
                ly = r + 1;
            }
        } else {
            const int c = t - nbord;
            ly = iw > 0 ? c / iw : th;
            lx = c - ly * iw + 1;
            ly = iw > 0 && ly < th - 2 ? ly + 1 : th;  // th: no such pixel
        }
        const int x = x0 + lx, y = y0 + ly;
        const bool live = ly < th && x < W && y < H;
        pq[k] = live ? y * W + x : -1;
        const int p = live ? (ly + 1) * pw + lx + 1 : 0, q = live ? (ly + 1) * uw + lx + 1 : 0;
        at[k] = PACK ? p | q << 14 | (x + 1 < W ? 1 << 28 : 0) | (y + 1 < H ? 1 << 29 : 0) : p;
        if (!PACK) {
            ui[PACK ? 0 : k] = q;
            rs[PACK ? 0 : k] = x + 1 < W ? 1 : 0;
            ds[PACK ? 0 : k] = y + 1 < H ? uw : 0;
        }
#pragma unroll
        for (int i = 0; i < N; ++i) {
            u[k][i] = u0;
            mu[k][i] = 0.f;
            if (FREG) f[FREG ? k : 0][FREG ? i : 0] = live ? S.f[i * P + pq[k]] : 0.f;
        }
    }
    const bool bord = tid < nbord;               // slot 0 holds a border pixel
    // Pixels around the tile: each thread takes one (more when the tile is thin)
    // for every ng-th label, and likewise the halo pixels whose xi the block
    // advances, those counted from the other end of the threads.
    const int ring = 2 * (tw + 2) + 2 * th, hp = th + tw;
    const int ng = max(1, NT / ring), hg = max(1, NT / hp);
    const int g_own = tid / ring, h_own = (NT - 1 - tid) / hp;
    auto fetch = [&](int r, int g, int step, unsigned tag, int& ok) {
        int lx, ly;
        if (r < 2 * uw) {
            ly = r < uw ? -1 : th;
            lx = (r < uw ? r : r - uw) - 1;
        } else {
            const int c = r - 2 * uw;
            lx = c < th ? -1 : tw;
            ly = c < th ? c : c - th;
        }
        const int x = x0 + lx, y = y0 + ly;
        if (x < 0 || y < 0 || x >= W || y >= H) return;
        const int dx = lx < 0 ? -1 : lx == tw ? 1 : 0, dy = ly < 0 ? -1 : ly == th ? 1 : 0;
        const unsigned long long* src =
            S.xch[tag & 1] + (size_t)(blockIdx.x + dy * S.gx + dx) * N * nbord +
            seg_border_place(tw, th, lx - dx * tw, ly - dy * th);
        float* dst = s_ub + (ly + 1) * uw + lx + 1;
        for (int i = g; i < N; i += step) dst[i * US] = wait_tagged(S, src + i * nbord, tag, 41, ok);
    };
    __syncthreads();

    auto ub_of = [&](int k) { return s_ub + (PACK ? at[k] >> 14 & 0x3fff : ui[PACK ? 0 : k]); };
    // xi <- Pi_Kg(xi + 1/2 grad ub) of one pixel
    // (a difference across the image's last column or row is that of a value
    // with itself), and without a label cost mu, whose m is 1
    auto ascend = [&](int k) {
        const int p = PACK ? at[k] & 0x3fff : at[k];
        const float bd = s_bd[p];
        const float* ubc = ub_of(k);
        const float* ubr = ubc + (PACK ? at[k] >> 28 & 1 : rs[PACK ? 0 : k]);
        const float* ubd = ubc + (PACK ? (at[k] >> 29 & 1 ? uw : 0) : ds[PACK ? 0 : k]);
        float *qx = s_px + p, *qy = s_py + p;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const float c = ubc[i * US];
            float vx = qx[i * PS], vy = qy[i * PS];
            dual_step(ubr[i * US] - c, ubd[i * US] - c, bd, vx, vy);
            qx[i * PS] = vx;
            qy[i * PS] = vy;
            if (!SUMS) mu[k][i] = fminf(0.f, mu[k][i] + 0.5f * (1.f - c));
        }
    };
    // u <- Pi_simplex(u - 1/5 (-div xi + f - mu)), ub = 2 u_new - u of one pixel
    auto descend = [&](int k, float (&v)[N]) {
        const int p = PACK ? at[k] & 0x3fff : at[k];
        const float *qx = s_px + p, *qy = s_py + p, *qu = qy - pw;
        const int Pv = opaque<N>(P);  // (multiples of P formed here, not kept over the iterations)
#pragma unroll
        for (int i = 0; i < N; ++i)  // every load of f in flight together
            v[i] = FREG ? f[FREG ? k : 0][FREG ? i : 0] : __ldg(S.f + (i * Pv + pq[k]));
#pragma unroll
        for (int i = 0; i < N; ++i) {
            // xi is 0 across the last column and row, and outside the image
            const float d = (qx[i * PS] - qx[i * PS - 1]) + (qy[i * PS] - qu[i * PS]);
            v[i] = u[k][i] - 0.2f * (-d + v[i] - mu[k][i]);
        }
        const float t = michelot<N>(v, u[k], N);
        float* ub = ub_of(k);
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const float un = v[i] < t ? 0.f : v[i] - t;
            v[i] = 2.f * un - u[k][i];
            ub[i * US] = v[i];
            u[k][i] = un;
        }
    };

    const float inv_area = 1.f / (float)P;
    for (int it = 0; it < S.iterations; ++it) {
        if (it > 0) {
            int ok = 1;
            if (ring <= NT) {
                const int g0 = N > 8 ? opaque<N>(tid) / ring : g_own;
                if (g0 < ng) fetch(tid - g0 * ring, g0, ng, (unsigned)it, ok);
            } else {
                for (int r = tid; r < ring; r += NT) fetch(r, 0, 1, (unsigned)it, ok);
            }
            if (SUMS) {
                // m <- clamp(m - (nu + sum mu) / |Omega|, 0, 1), mb = 2 m_new - m; one
                // warp per label, the same summation order in every block
                const unsigned long long* pt = S.parts[it & 1];
                for (int i = warp; i < N; i += NT / 32) {
                    float s = 0.f;
                    for (int k = lane; k < G; k += 32) s += wait_tagged(S, pt + i * G + k, (unsigned)it, 41, ok);
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                    if (lane == 0) {
                        const float mo = s_m[i];
                        const float mn = fminf(1.f, fmaxf(0.f, mo - inv_area * (S.nu + s)));
                        s_mb[i] = 2.f * mn - mo;
                        s_m[i] = mn;
                    }
                }
            }
            if (!__syncthreads_and(ok)) return;
        }
        // xi of the border, and of the pixels left of and above the tile (by the
        // threads at the other end)
        if (bord && pq[0] >= 0) ascend(0);
        auto ascend_halo = [&](int h, int g, int step) {
            const int lx = h < th ? -1 : h - th, ly = h < th ? h : -1;
            const int x = x0 + lx, y = y0 + ly;
            if (x < 0 || y < 0 || x >= W || y >= H) return;
            const int p = (ly + 1) * pw + lx + 1;
            const float* ubc = s_ub + (ly + 1) * uw + lx + 1;
            const float *ubr = ubc + (x + 1 < W ? 1 : 0), *ubd = ubc + (y + 1 < H ? uw : 0);
            const float bd = s_bd[p];
            for (int i = g; i < N; i += step) {
                const float c = ubc[i * US];
                float vx = s_px[i * PS + p], vy = s_py[i * PS + p];
                dual_step(ubr[i * US] - c, ubd[i * US] - c, bd, vx, vy);
                s_px[i * PS + p] = vx;
                s_py[i * PS + p] = vy;
            }
        };
        const int rt = NT - 1 - tid;
        if (hp <= NT) {
            const int g0 = N > 8 ? opaque<N>(rt) / hp : h_own;
            if (g0 < hg) ascend_halo(rt - g0 * hp, g0, hg);
        } else {
            for (int h = rt; h < hp; h += NT) ascend_halo(h, 0, 1);
        }
        if (it == 0) {  // the interior's xi, later advanced at the end of the iteration before
#pragma unroll
            for (int k = 0; k < PPT; ++k)
                if (pq[k] >= 0 && (k > 0 || !bord)) ascend(k);
        }
#pragma unroll
        for (int k = 0; SUMS && k < PPT; ++k) {  // mu <- min(0, mu + 1/2 (mb - ub))
            if (pq[k] < 0) continue;
            const float* ub = ub_of(k);
#pragma unroll
            for (int i = 0; i < N; ++i)
                mu[k][i] = fminf(0.f, mu[k][i] + 0.5f * (s_mb[i] - ub[i * US]));
        }
        if (SUMS) {
            // the block's sums of mu: halving exchanges leave lane l with label
            // l * NR / 32's sum over the warp
            float a[NR];
#pragma unroll
            for (int i = 0; i < NR; ++i) {
                a[i] = 0.f;
                if (i < N)
#pragma unroll
                    for (int k = 0; k < PPT; ++k) a[i] += mu[k][i < N ? i : 0];
            }
            int w = NR;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                if (w > 1) {
                    w >>= 1;
                    const bool up = lane & o;
#pragma unroll
                    for (int i = 0; i < NR / 2; ++i)
                        if (i < w) {
                            const float send = up ? a[i] : a[i + w], keep = up ? a[i + w] : a[i];
                            a[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                        }
                } else {
                    a[0] += __shfl_xor_sync(0xffffffffu, a[0], o);
                }
            }
            if (lane % (32 / NR) == 0) s_red[lane / (32 / NR)][warp] = a[0];
        }
        __syncthreads();
        float v[N];
        const unsigned tag = (unsigned)it + 1u;
        const bool publish = !(S.stall && it == 0 && blockIdx.x == G - 1);
        if (SUMS && tid < N && publish) {
            float s = 0.f;
            for (int w = 0; w < NT / 32; ++w) s += s_red[tid][w];
            put_tagged(S.parts[tag & 1] + tid * G + blockIdx.x, tag, s);
        }
        if (pq[0] >= 0) {
            descend(0, v);
            if (bord && publish) {
                const int nb = opaque<N>(nbord);
                unsigned long long* o = S.xch[tag & 1] + (size_t)blockIdx.x * N * nb + tid;
#pragma unroll
                for (int i = 0; i < N; ++i) put_tagged(o + i * nb, tag, v[i]);
            }
        }
#pragma unroll
        for (int k = 1; k < PPT; ++k)
            if (pq[k] >= 0) descend(k, v);
        __syncthreads();
        if (it + 1 < S.iterations) {
#pragma unroll
            for (int k = 0; k < PPT; ++k)
                if (pq[k] >= 0 && (k > 0 || !bord)) ascend(k);
        }
    }
    if (S.stall) {  // the timeout-path test: wait for what nobody publishes
        int ok = 1;
        if (tid == 0)
            wait_tagged(S, reinterpret_cast<unsigned long long*>(S.abort_flag + 2), 1u, 41, ok);
        if (!__syncthreads_and(ok)) return;
    }

#pragma unroll
    for (int k = 0; k < PPT; ++k) {
        if (pq[k] < 0) continue;
        int best = 0;
        float bv = u[k][0];
#pragma unroll
        for (int i = 0; i < N; ++i) {
            S.u[i * P + pq[k]] = u[k][i];
            if (u[k][i] > bv) {
                bv = u[k][i];
                best = i;
            }
        }
        if (S.labels) S.labels[pq[k]] = best;
    }
}

using SegTileKernel = void (*)(SegTile);

template <int PPT, bool SUMS>
SegTileKernel seg_tile_kernel_n(int n, size_t& smem, int& ps, int& us) {
#define CS_SEG_CASE(NN)                  \
    case NN:                             \
        smem = seg_tile_smem(NN, PPT);   \
        ps = seg_ps(NN, PPT);            \
        us = seg_us(NN, PPT);            \
        return seg_tile_kernel<NN, PPT, SUMS>;
    switch (n) {
        CS_SEG_CASE(1)
        CS_SEG_CASE(2)
        CS_SEG_CASE(3)
        CS_SEG_CASE(4)
        CS_SEG_CASE(5)
        CS_SEG_CASE(6)
        CS_SEG_CASE(7)
        CS_SEG_CASE(8)
        default: break;
    }
    if constexpr (PPT <= 2) {
        switch (n) {
            CS_SEG_CASE(9)
            CS_SEG_CASE(10)
            CS_SEG_CASE(11)
            CS_SEG_CASE(12)
            CS_SEG_CASE(13)
            CS_SEG_CASE(14)
            CS_SEG_CASE(15)
            CS_SEG_CASE(16)
            default: break;
        }
    }
#undef CS_SEG_CASE
    return nullptr;
}

// Tiling of an H x W image for the on-chip form: the fewest pixels per thread
// whose windows fit, then the split of the SMs into gx x gy tiles with the
// least area and perimeter per tile. Tiles below 128 pixels would add blocks
// to wait for and no work to share. kernel == nullptr: the state does not fit.
struct SegPlan {
    SegTileKernel kernel = nullptr;
    size_t smem = 0;
    int tw = 0, th = 0, gx = 0, gy = 0, threads = 0;
};
template <bool SUMS>
SegPlan seg_plan_t(int H, int W, int n, int n_sm) {
    SegPlan best;
    const long long P = (long long)H * W;
    if (n > 16 || !seg_narrow(P, n)) return best;
    const int blocks = (int)std::min<long long>(n_sm, std::max<long long>(1, (P + 127) / 128));
    for (int ppt = 1; ppt <= 4 && !best.kernel; ppt *= 2) {
        size_t smem = 0;
        int ps = 0, us = 0;
        SegTileKernel k = ppt == 1   ? seg_tile_kernel_n<1, SUMS>(n, smem, ps, us)
                          : ppt == 2 ? seg_tile_kernel_n<2, SUMS>(n, smem, ps, us)
                                     : seg_tile_kernel_n<4, SUMS>(n, smem, ps, us);
        if (!k) continue;
        double cost = 0;
        for (int gx = 1; gx <= blocks && gx <= W; ++gx) {
            const int tw = (W + gx - 1) / gx, rows = blocks / gx;
            const int th = (H + rows - 1) / rows;
            if ((long long)tw * th > (long long)TNT * ppt ||
                (long long)(tw + 1) * (th + 1) > ps || (long long)(tw + 2) * (th + 2) > us)
                continue;
            const int threads = std::max(64, ((tw * th + ppt - 1) / ppt + 31) / 32 * 32);
            if (seg_border(tw, th) > threads) continue;  // border pixels fill slot 0 at most
            const double c = (double)tw * th + 2.0 * (tw + th);
            if (best.kernel && c >= cost) continue;
            cost = c;
            best.kernel = k;
            best.smem = smem;
            best.tw = tw;
            best.th = th;
            best.gx = (W + tw - 1) / tw;
            best.gy = (H + th - 1) / th;
            best.threads = threads;
        }
    }
    return best;
}

using SegKernel = void (*)(SegState);

template <typename I>
SegKernel seg_kernel_t(int n) {
    switch (n) {
        case 1: return seg_solve_kernel<1, I>;
        case 2: return seg_solve_kernel<2, I>;
        case 3: return seg_solve_kernel<3, I>;
        case 4: return seg_solve_kernel<4, I>;
        case 5: return seg_solve_kernel<5, I>;
        case 6: return seg_solve_kernel<6, I>;
        case 7: return seg_solve_kernel<7, I>;
        case 8: return seg_solve_kernel<8, I>;
        default: return n <= 16 ? seg_solve_kernel<16, I> : seg_solve_kernel<CS_MAX_LABELS, I>;
    }
}

SegKernel seg_kernel(long long P, int n) {
    return seg_narrow(P, n) ? seg_kernel_t<int>(n) : seg_kernel_t<long long>(n);
}

int seg_grid(long long P, int n, int n_sm) {
    // co-resident blocks per SM, per variant (labels 1..8, 16, 64; narrow /
    // wide index); -1 until queried (calls from several threads store the
    // same value)
    static std::atomic<int> per_sm[2][10];
    static std::once_flag init;
    std::call_once(init, [] {
        for (auto& row : per_sm)
            for (auto& v : row) v.store(-1);
    });
    const int v = n <= 8 ? n - 1 : n <= 16 ? 8 : 9;
    std::atomic<int>& slot = per_sm[seg_narrow(P, n) ? 0 : 1][v];
    int nb = slot.load();
    if (nb < 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, seg_kernel(P, n), SB, 0) !=
            cudaSuccess)
            nb = 0;
        slot.store(nb);
    }
    const int k = nb < 2 ? nb : 2;
    return k * n_sm;
}

SegPlan seg_plan(int H, int W, int n, int n_sm, bool sums) {
    return sums ? seg_plan_t<true>(H, W, n, n_sm) : seg_plan_t<false>(H, W, n, n_sm);
}

// Words of the exchange buffers (both parities): border ub, sums of mu, then the
// abort flag and a word that nothing sets.
size_t seg_exchange_words(const SegPlan& p, int n) {
    return 2 * (size_t)p.gx * p.gy * n * ((size_t)seg_border(p.tw, p.th) + 1) + 2;
}

}  // namespace

size_t seg_scratch_bytes(int H, int W, int n, int nblk, int n_sm, bool sums) {
    const long long P = (long long)H * W;
    const SegPlan pl = seg_plan(H, W, n, n_sm, sums);
    if (pl.kernel) return 8 * seg_exchange_words(pl, n);

    return sizeof(float) * ((size_t)4 * n * P + (size_t)P + (size_t)n * nblk) + 1024;
}

int seg_blocks(long long P, int n, int n_sm) {
    const long long need = (P + SB - 1) / SB;
    const int g = seg_grid(P, n, n_sm);
    return (int)(need < g ? need : g);
}

cudaError_t launch_segment(const SegArgs& a, cudaStream_t st) {
    const long long P = (long long)a.H * a.W;
    const int n = a.n_labels;
    if (a.nblk < 1) return cudaErrorInvalidConfiguration;
    const SegPlan pl = seg_plan(a.H, a.W, n, a.n_sm, a.nu != 0.f);
    if (pl.kernel) {
        const int G = pl.gx * pl.gy;
        const size_t per = (size_t)G * n * seg_border(pl.tw, pl.th);
        SegTile S;
        S.f = a.f;
        S.img = a.img;
        S.u = a.u;
        S.xch[0] = reinterpret_cast<unsigned long long*>(a.scratch);
        S.xch[1] = S.xch[0] + per;
        S.parts[0] = S.xch[1] + per;
        S.parts[1] = S.parts[0] + (size_t)n * G;
        S.abort_flag = reinterpret_cast<unsigned*>(S.parts[1] + (size_t)n * G);
        S.labels = a.labels;
        S.d_err = a.d_err;
        S.H = a.H;
        S.W = a.W;
        S.iterations = a.iterations;
        S.tw = pl.tw;
        S.th = pl.th;
        S.gx = pl.gx;
        S.gy = pl.gy;
        S.lambda = a.lambda;
        S.nu = a.nu;
        S.gamma = a.gamma;
        S.wait_ns = a.wait_ns ? a.wait_ns : SEG_WAIT_NS;
        S.stall = a.stall && a.iterations > 0;
        cudaError_t e = cudaFuncSetAttribute((const void*)pl.kernel,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)pl.smem);
        if (e == cudaSuccess)
            e = cudaMemsetAsync(S.xch[0], 0, 8 * seg_exchange_words(pl, n), st);  // no tag is 0
        if (e != cudaSuccess) return e;
        void* args[] = {&S};
        return cudaLaunchCooperativeKernel((const void*)pl.kernel, dim3(G), dim3(pl.threads), args,
                                           pl.smem, st);
    }
    SegState S;
    S.f = a.f;
    S.img = a.img;
    S.u = a.u;
    S.ub = a.scratch;
    S.px = S.ub + (size_t)n * P;
    S.py = S.px + (size_t)n * P;
    S.mu = S.py + (size_t)n * P;
    S.bound = S.mu + (size_t)n * P;
    S.parts = S.bound + P;
    // the barrier words sit 256-byte aligned after the parts
    const uintptr_t end = reinterpret_cast<uintptr_t>(S.parts + (size_t)n * a.nblk);
    S.bar = reinterpret_cast<unsigned*>((end + 255) & ~(uintptr_t)255);
    S.labels = a.labels;
    S.d_err = a.d_err;
    S.H = a.H;
    S.W = a.W;
    S.n = n;
    S.iterations = a.iterations;
    S.lambda = a.lambda;
    S.nu = a.nu;
    S.gamma = a.gamma;
    S.wait_ns = a.wait_ns ? a.wait_ns : SEG_WAIT_NS;
    S.stall = a.stall && a.iterations > 0;
    cudaError_t e = cudaMemsetAsync(S.bar, 0, 2 * sizeof(unsigned), st);
    if (e != cudaSuccess) return e;
    void* args[] = {&S};
    return cudaLaunchCooperativeKernel((const void*)seg_kernel(P, n), dim3(a.nblk), dim3(SB), args,
                                       0, st);
}
