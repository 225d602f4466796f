// The solver's on-chip form (k_segment.cu has the method and both forms): the
// tile kernel and its tiling, shared by the translation units that instantiate
// it with and without a label cost.
#pragma once

#include <algorithm>
#include <cstdint>

#include "internal.h"

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

// the tilings (kernel == nullptr: the state does not fit the chip)
SegPlan seg_plan_plain(int H, int W, int n, int n_sm);  // nu = 0
SegPlan seg_plan_mdl(int H, int W, int n, int n_sm);    // nu > 0

namespace {

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

}  // namespace
