// Unsupervised mode (Sec. 3.2, "Unsupervised Segmentation"): k-means on the
// colour pixels, k-medians on the smooth co-supports iota(O s_x) of Eq.
// (map_tsm), segments = (colour class, texture class) pairs, each pixel's
// colour and texture likelihood as in Eq. (post_text).
//
// Both clusterings start from caller-given pixels and run a fixed number of
// rounds (assignment, then update), then a last assignment to the final
// centres. Assignments are decided in FP32 with the distances accumulated in
// a fixed order (colour ((d0^2 + d1^2) + d2^2), texture over codes
// j = 0 .. k-1), ties to the lower class, so they are reproducible bit for
// bit. A k-means centroid is the exact mean of the members' values rounded
// to multiples of 2^-24: integer sums (order-free atomics), one double
// division, one rounding to FP32. A k-medians centre is the elementwise
// median by radix selection, all classes of a code at once on a cluster of
// blocks that split the points. A class without members keeps its centre.
#include <cooperative_groups.h>

#include <cstdint>
#include <type_traits>

#include "internal.h"

namespace {

constexpr int UB = 256;             // threads per block
constexpr int MB = 512;             // threads per block of the median kernel
constexpr float QSCALE = 16777216.f;  // 2^24

__global__ void kmeans_init_kernel(const float* __restrict__ X, UnsupInit init, int n,
                                   float* __restrict__ C) {
    const int t = threadIdx.x;
    if (t < 3 * n) C[t] = X[(size_t)init.v[t / 3] * 3 + t % 3];
}

__device__ __forceinline__ int nearest_colour(const float* x, const float* C, int n) {
    int best = 0;
    float bd = 0.f;
    for (int a = 0; a < n; ++a) {
        const float t0 = __fsub_rn(x[0], C[3 * a]);
        const float t1 = __fsub_rn(x[1], C[3 * a + 1]);
        const float t2 = __fsub_rn(x[2], C[3 * a + 2]);
        const float d =
            __fadd_rn(__fadd_rn(__fmul_rn(t0, t0), __fmul_rn(t1, t1)), __fmul_rn(t2, t2));
        if (a == 0 || d < bd) {
            bd = d;
            best = a;
        }
    }
    return best;
}

// Assignment to the nearest centre; with sums != null also the members'
// fixed-point sums and counts (per block in shared memory, then atomics).
//
// Bound: the sums. 64-bit shared-memory atomics are compare-and-swap loops, whose
// cost is a class's members in the warp; adding those up first costs a few warp
// reductions per class present. A warp of many classes has few members of each: up
// to KM_GROUPS classes the reductions, above that the atomics. Measured, five rounds,
// 1e6 points, us (reductions always, atomics always, by this rule): random points,
// 4 classes 144, 329, 144; 16 classes 332, 163, 167; an image's points, 4 classes 124,
// 417, 123; 16 classes 236, 288, 226.
constexpr int KM_GROUPS = 6;
__global__ void __launch_bounds__(UB) kmeans_assign_kernel(
    const float* __restrict__ X, int N, const float* __restrict__ Cg, int n,
    int32_t* __restrict__ assign, unsigned long long* __restrict__ sums,
    unsigned* __restrict__ counts) {
    __shared__ float C[3 * CS_MAX_CLASSES];
    __shared__ unsigned long long s_sum[3 * CS_MAX_CLASSES];
    __shared__ unsigned s_cnt[CS_MAX_CLASSES];
    for (int t = threadIdx.x; t < 3 * n; t += UB) {
        C[t] = Cg[t];
        s_sum[t] = 0ull;
    }
    for (int t = threadIdx.x; t < n; t += UB) s_cnt[t] = 0u;
    __syncthreads();
    for (int q = blockIdx.x * UB + threadIdx.x; q < N; q += gridDim.x * UB) {
        const float x[3] = {X[(size_t)q * 3], X[(size_t)q * 3 + 1], X[(size_t)q * 3 + 2]};
        const int a = nearest_colour(x, C, n);
        if (assign) assign[q] = a;
        if (sums) {
            const unsigned act = __activemask(), grp = __match_any_sync(act, (unsigned)a);
            const bool lead = (int)(threadIdx.x & 31u) == __ffs(grp) - 1;
            if (__popc(__ballot_sync(act, lead)) > KM_GROUPS) {
                for (int c = 0; c < 3; ++c)
                    atomicAdd(s_sum + 3 * a + c,
                              (unsigned long long)__float2ll_rn(__fmul_rn(x[c], QSCALE)));
                atomicAdd(s_cnt + a, 1u);
                continue;
            }
            // the warp's members of each class are added up first: 24 low bits
            // and the signed rest, whose 32-lane sum fits 32 bits while
            // |value| < 2^25; larger values go one by one
            for (int c = 0; c < 3; ++c) {
                const long long v = __float2ll_rn(__fmul_rn(x[c], QSCALE));
                const long long hi = v >> 24;
                if (__any_sync(grp, hi >= (1ll << 25) || hi < -(1ll << 25))) {
                    atomicAdd(s_sum + 3 * a + c, (unsigned long long)v);
                } else {
                    const unsigned lo = __reduce_add_sync(grp, (unsigned)(v & 0xffffffll));
                    const int hs = __reduce_add_sync(grp, (int)hi);
                    if (lead)
                        atomicAdd(s_sum + 3 * a + c,
                                  (unsigned long long)((long long)hs * (1ll << 24) + lo));
                }
            }
            if (lead) atomicAdd(s_cnt + a, (unsigned)__popc(grp));
        }
    }
    if (!sums) return;
    __syncthreads();
    for (int t = threadIdx.x; t < 3 * n; t += UB)
        if (s_sum[t]) atomicAdd(sums + t, s_sum[t]);
    for (int t = threadIdx.x; t < n; t += UB)
        if (s_cnt[t]) atomicAdd(counts + t, s_cnt[t]);
}

// C = float(S / (cnt 2^24)) for classes with members; clears the sums.
__global__ void kmeans_update_kernel(float* __restrict__ C, unsigned long long* __restrict__ sums,
                                     unsigned* __restrict__ counts, int n) {
    const int t = threadIdx.x;
    if (t < 3 * n) {
        const unsigned cnt = counts[t / 3];
        if (cnt) C[t] = (float)((double)(long long)sums[t] / ((double)cnt * 16777216.0));
    }
    __syncthreads();
    if (t < 3 * n) sums[t] = 0ull;
    if (t < n) counts[t] = 0u;
}

__global__ void kmedians_init_kernel(const float* __restrict__ V, int N, int k, UnsupInit init,
                                     int n, float* __restrict__ C) {
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n * k; t += gridDim.x * blockDim.x)
        C[t] = V[(size_t)(t % k) * N + init.v[t / k]];
}

// l1 distances of pixel q's column of V to the n centres in shared memory
// (code-major rows of cpad(NC) floats), summed over codes j = 0 .. k-1 in turn
// (FP32, no contraction). NC: the class count when it is at most 8 (every
// class loop unrolled exactly), else CS_MAX_CLASSES with the classes from n on
// ignored. The loads of L1_J codes are in flight together: one pixel per
// thread leaves too few warps to hide one load at a time.
constexpr int L1_J = 14;
__host__ __device__ constexpr int cpad(int nc) { return nc <= 2 ? nc : (nc + 3) & ~3; }

template <int NC>
__device__ __forceinline__ void l1_all(const float* __restrict__ V, int N, int k, int q,
                                       const float* C, float (&d)[NC]) {
    constexpr int CP = cpad(NC);
#pragma unroll
    for (int b = 0; b < NC; ++b) d[b] = 0.f;
    auto add = [&](int j, float v) {
        float c[CP];
#pragma unroll
        for (int b = 0; b < CP; ++b) c[b] = C[j * CP + b];
#pragma unroll
        for (int b = 0; b < NC; ++b) d[b] = __fadd_rn(d[b], fabsf(__fsub_rn(c[b], v)));
    };
    const float* col = V + q;
    int j = 0;
    for (; j + L1_J <= k; j += L1_J) {
        float v[L1_J];
#pragma unroll
        for (int u = 0; u < L1_J; ++u) v[u] = col[(size_t)(j + u) * N];
#pragma unroll
        for (int u = 0; u < L1_J; ++u) add(j + u, v[u]);
    }
    for (; j < k; ++j) add(j, col[(size_t)j * N]);
}

// centres n x k (class-major) into the layout l1_all reads, padding zeroed
template <int NC>
__device__ __forceinline__ void load_centres(float* C, const float* __restrict__ Cg, int n, int k) {
    constexpr int CP = cpad(NC);
    for (int t = threadIdx.x; t < k * CP; t += UB) {
        const int j = t / CP, b = t % CP;
        C[t] = b < n ? Cg[(size_t)b * k + j] : 0.f;
    }
}

template <int NC>
__device__ __forceinline__ int nearest_l1(const float (&d)[NC], int n, float& bd) {
    int best = 0;
    bd = d[0];
#pragma unroll
    for (int b = 1; b < NC; ++b)
        if ((NC <= 8 || b < n) && d[b] < bd) {
            bd = d[b];
            best = b;
        }
    return best;
}

// Assignment to the nearest centre, as bytes for the median rounds (assign8)
// or as the call's result (assign).
//
// Bound: one read of V from L2 (60 MB at 154,401 points x 98 codes) and two
// FP32 adds per point, code and class. Measured there with 4 classes:
// 17 us a launch (cold L2), against 37 us with 16 guarded classes, 4 loads in flight
// and class-major centres (a shared-memory load per class and code).
template <int NC>
__global__ void __launch_bounds__(UB) kmedians_assign_kernel(
    const float* __restrict__ V, int N, int k, const float* __restrict__ Cg, int n,
    int32_t* __restrict__ assign, uint8_t* __restrict__ assign8) {
    extern __shared__ __align__(16) float C[];  // k x cpad(NC)
    load_centres<NC>(C, Cg, n, k);
    __syncthreads();
    for (int q = blockIdx.x * UB + threadIdx.x; q < N; q += gridDim.x * UB) {
        float d[NC];
        l1_all<NC>(V, N, k, q, C, d);
        float bd;
        const int best = nearest_l1<NC>(d, n, bd);
        if (assign)
            assign[q] = best;
        else
            assign8[q] = (uint8_t)best;
    }
}

// Order-preserving map of a float's bits to an unsigned key, and back.
__device__ __forceinline__ unsigned key_of(float f) {
    const unsigned u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float float_of(unsigned k) {
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// One cluster of MC blocks per code j: the elementwise median of every class
// over the points assigned to it, all classes at once, by narrowing a range of
// keys per class that holds the lower middle value. Each pass histograms the
// range's keys of the block's slice of the points (row j of V and the
// byte-wide assignment, coalesced) into HB bins with plain shared-memory
// increments; the classes are then shared out among the cluster's blocks, each
// of which adds up its classes' histograms through distributed shared memory,
// scans them in parallel and writes the chosen bin to every block as the next
// range. The first pass bins by value (fine steps over iota's range,
// [0, 1]), the later ones by key. The second pass first
// copies the keys of the ranges into a list, which it and the later passes read
// in place of the slice (unless they do not fit). A class with an even count needs
// the least key above its lower middle value too: a scan notes the next
// occupied bin, and the next pass takes the least key in it. Classes without
// points keep their centre. The cluster barriers are the hardware's.
//
// Bound: instruction issue, about 12 per point, code and pass over the slice
// (V stays in L2 between rounds). The value steps spread a warp's increments
// (iota crowds the top of [0, 1], where the leading key bits that a radix digit
// takes are nearly all equal) and leave few keys in any one bin, so that they
// fit the list: equal steps over [0, 1] alone crowd the lowest one. The list pays because nearly every warp has some
// key in range, so that the second pass would run the histogram's code for all
// of them (78 us so, and with digits of 11, 11 and 10 key bits). Three blocks
// per SM hold 98 codes' clusters in one wave. Measured on 154,401 points x 98 codes, 4 classes:
// 50 us a launch (cold L2), against 233 us for four 8-bit digits with match_any and
// one thread scanning each histogram.
constexpr int MC = 4;        // blocks per code
constexpr int HB = 2048;     // histogram bins per class
constexpr int MU = 8;        // points per thread in flight
constexpr int list_cap(bool h16) { return h16 ? 2048 : 4096; }  // keys a block's list holds
constexpr int MED_PASSES = 8;  // more than any narrowing takes (2^32 keys, 2^11 a pass)

struct MedState {
    uint2 rng[CS_MAX_CLASSES];      // first key of the range; distance to the last key of interest
    unsigned khi[CS_MAX_CLASSES];   // last key of the range (above it: the next occupied bin)
    unsigned shift[CS_MAX_CLASSES];  // bin of a key: (key - rng.x) >> shift
    unsigned slo[CS_MAX_CLASSES];   // the next occupied bin's keys (slo > shi: none)
    unsigned shi[CS_MAX_CLASSES];
    unsigned rank[CS_MAX_CLASSES];  // rank of the lower middle value within the range
    unsigned cnt[CS_MAX_CLASSES];
    unsigned smin[CS_MAX_CLASSES];  // least key of the block's slice in the next occupied bin
    unsigned done[CS_MAX_CLASSES];
};

// First-pass bins, monotone in the key (which puts a NaN beyond the infinity
// of its sign): 1024 steps of 1/32 octave from 2^-35 to 1/8 (below: bin 0), then
// steps of 1/1024 up to 1, then one bin for 1 and above.
constexpr int VB_LOW = 92 * 32;  // 2^-35's bits >> 18
constexpr unsigned VB_TOP = 1920u;
__device__ __forceinline__ unsigned value_bin(float v) {
    const int b = __float_as_int(v);
    const unsigned low = (unsigned)max((b >> 18) - VB_LOW, 0);
    // 2^23 + 896 + floor(1024 v), exactly
    const float c = __int_as_float(min(b, 0x3F800000));
    const unsigned high = __float_as_uint(__fmaf_rz(c, 1024.f, 8388608.f + 896.f)) - 0x4B000000u;
    return b >= 0x3E000000 ? high : low;
}
__device__ __forceinline__ unsigned value_bin_first(unsigned d) {  // a bin's first key
    return d == 0u     ? 0u
           : d < 1024u ? ((d + VB_LOW) << 18) | 0x80000000u
                       : key_of((float)(d - 896u) * (1.f / 1024.f));
}
__device__ __forceinline__ void value_bin_keys(unsigned d, unsigned& lo, unsigned& hi) {
    lo = value_bin_first(d);
    hi = d >= VB_TOP ? 0xffffffffu : value_bin_first(d + 1u) - 1u;
}

//
// H16: 16-bit counters, two bins a word, and a shorter list. From 12 classes on, 32-bit
// counters would leave one block per SM (98 clusters in three waves); so there are
// three. Slices of at most 65535 points, so that no counter runs over (beyond that the
// sweeps, not the blocks in flight, take the time). Measured with 16 classes x 98 codes,
// five rounds, us (32-bit, 16-bit): 300 points 487, 256; 5000 points 498, 261; 154,401
// points 738, 470.
template <bool H16>
__global__ void __cluster_dims__(MC, 1, 1) __launch_bounds__(MB, 3)
    class_median_kernel(const float* __restrict__ V, int N, int k,
                        const uint8_t* __restrict__ assign, int n, float* __restrict__ C) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    constexpr int HW = H16 ? HB / 2 : HB;             // words of a class's histogram
    constexpr int cap = list_cap(H16);
    extern __shared__ __align__(16) unsigned hist[];  // n x HW, then the list's keys and classes
    unsigned* lkey = hist + (size_t)n * HW;
    uint8_t* lcls = reinterpret_cast<uint8_t*>(lkey + cap);
    __shared__ unsigned s_warp[MB / 32];
    __shared__ unsigned s_found[4];  // bin, rank within it, its count, next occupied bin
    __shared__ unsigned s_len;       // keys listed (more than cap: the list is incomplete)
    __shared__ MedState st;
    const int rank = (int)cluster.block_rank();
    const int j = blockIdx.x / MC;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float* v = V + (size_t)j * N;
    const int chunk = (N + MC - 1) / MC;
    const int q0 = min(rank * chunk, N), q1 = min(q0 + chunk, N);
    if (tid < CS_MAX_CLASSES) {
        st.done[tid] = 0u;
        st.smin[tid] = 0xffffffffu;
        st.slo[tid] = 1u;
        st.shi[tid] = 0u;
    }
    if (tid == 0) s_len = 0u;
    auto tally = [&](unsigned b, unsigned bin) {
        unsigned* w = hist + b * HW + (H16 ? bin >> 1 : bin);
        // (an increment by 1 is a unit of its own that takes a warp's increments of one
        // bin at once: the even bins keep it, among them that of iota = 1, flat patches)
        if (H16 && (bin & 1u))
            atomicAdd(w, 0x10000u);
        else
            atomicAdd(w, 1u);
    };
    for (int pass = 0; pass < MED_PASSES; ++pass) {
        for (int t = tid; t < n * (HW / 4); t += MB)
            reinterpret_cast<uint4*>(hist)[t] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        auto count = [&](unsigned b, unsigned key) {
            const unsigned d = key - st.rng[b].x;
            if (d > st.rng[b].y) return;
            if (key <= st.khi[b])
                tally(b, d >> st.shift[b]);
            else if (key >= st.slo[b])
                atomicMin(&st.smin[b], key);
        };
        // the slice's points, MU at a time
        auto sweep = [&](auto&& f) {
            for (int qb = q0 + tid; qb < q1; qb += MB * MU) {
                float val[MU];
                unsigned cls[MU];
                if (qb - tid + MB * MU <= q1) {
#pragma unroll
                    for (int u = 0; u < MU; ++u) {
                        cls[u] = assign[qb + u * MB];
                        val[u] = v[qb + u * MB];
                    }
#pragma unroll
                    for (int u = 0; u < MU; ++u) f(cls[u], val[u], true);
                } else {
                    for (int u = 0; u < MU; ++u) {
                        const int q = qb + u * MB;
                        f(q < q1 ? (unsigned)assign[q] : 0u, q < q1 ? v[q] : 0.f, q < q1);
                    }
                }
            }
        };
        if (pass == 0) {
            sweep([&](unsigned b, float x, bool live) {
                if (live) tally(b, value_bin(x));
            });
        } else {
            if (pass == 1) {  // list the keys in range
                sweep([&](unsigned b, float x, bool live) {
                    const unsigned key = key_of(x);
                    const uint2 r = st.rng[b];
                    if (live && key - r.x <= r.y) {
                        const unsigned e = atomicAdd(&s_len, 1u);
                        if (e < (unsigned)cap) {
                            lkey[e] = key;
                            lcls[e] = (uint8_t)b;
                        }
                    }
                });
                __syncthreads();
            }
            const unsigned len = s_len;
            if (len <= (unsigned)cap)
                for (unsigned e = tid; e < len; e += MB) count(lcls[e], lkey[e]);
            else
                sweep([&](unsigned b, float x, bool live) {
                    if (live) count(b, key_of(x));
                });
        }
        cluster.sync();  // every slice's histogram (and least keys) are complete
        for (int b = rank; b < n; b += MC) {  // this block's classes
            if (st.done[b]) continue;         // uniform over the block
            // bins 4 tid .. 4 tid + 3, summed over the slices, and their scan
            unsigned h[4] = {0u, 0u, 0u, 0u};
#pragma unroll
            for (int r = 0; r < MC; ++r) {
                const unsigned* hr = cluster.map_shared_rank(hist, r) + b * HW;
                if (H16) {
                    const uint2 x = reinterpret_cast<const uint2*>(hr)[tid];
                    h[0] += x.x & 0xffffu;
                    h[1] += x.x >> 16;
                    h[2] += x.y & 0xffffu;
                    h[3] += x.y >> 16;
                } else {
                    const uint4 x = reinterpret_cast<const uint4*>(hr)[tid];
                    h[0] += x.x;
                    h[1] += x.y;
                    h[2] += x.z;
                    h[3] += x.w;
                }
            }
            const unsigned own = h[0] + h[1] + h[2] + h[3];
            unsigned inc = own;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned up = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += up;
            }
            if (lane == 31) s_warp[warp] = inc;
            if (tid == 0) s_found[3] = 0xffffffffu;
            __syncthreads();
            unsigned base = 0, total = 0;
#pragma unroll
            for (int w = 0; w < MB / 32; ++w) {
                const unsigned x = s_warp[w];
                base += w < warp ? x : 0u;
                total += x;
            }
            const unsigned cnt = pass == 0 ? total : st.cnt[b];
            const unsigned r = pass == 0 ? (cnt ? (cnt - 1) / 2 : 0u) : st.rank[b];
            const unsigned excl = base + inc - own;
            if (r >= excl && r < excl + own) {
                unsigned acc = excl;
                int d = 0;
                while (d < 3 && r >= acc + h[d]) acc += h[d++];
                s_found[0] = 4u * tid + d;
                s_found[1] = r - acc;
                s_found[2] = h[d];
            }
            __syncthreads();
            const unsigned dig = s_found[0], rin = s_found[1], eq = s_found[2];
            if (cnt) {  // the next occupied bin above the chosen one
                unsigned nx = 0xffffffffu;
#pragma unroll
                for (int d = 3; d >= 0; --d)
                    if (h[d] && 4u * tid + d > dig) nx = 4u * tid + d;
                nx = __reduce_min_sync(0xffffffffu, nx);
                if (lane == 0 && nx != 0xffffffffu) atomicMin(s_found + 3, nx);
            }
            // the range this pass worked on, read by every thread before any writes it
            const unsigned lo0 = st.rng[b].x, hi0 = st.khi[b], sh = st.shift[b];
            const unsigned slo0 = st.slo[b], shi0 = st.shi[b];
            __syncthreads();
            if (tid < MC) {  // one thread per block of the cluster
                MedState* d = cluster.map_shared_rank(&st, tid);
                const unsigned nx = s_found[3];
                unsigned lo = 0, hi = 0, slo = slo0, shi = shi0;
                const bool even = !(cnt & 1u), next = even && nx != 0xffffffffu;
                if (!cnt) {  // no points: the centre stays
                    d->done[b] = 1u;
                } else {
                    if (pass == 0) {
                        value_bin_keys(dig, lo, hi);
                        if (next) value_bin_keys(nx, slo, shi);
                    } else {
                        lo = lo0 + (dig << sh);
                        hi = min(hi0 - lo, (1u << sh) - 1u) + lo;
                        if (next) {
                            slo = lo0 + (nx << sh);
                            shi = min(hi0 - slo, (1u << sh) - 1u) + slo;
                        }
                    }
                    if (lo == hi && tid == 0) {  // one key left (and then sh is 0 if nx exists)
                        const float x = float_of(lo);
                        float out = x;
                        if (even) {
                            float y = x;
                            if (eq - rin < 2u) {
                                unsigned m = 0xffffffffu;
                                if (next)
                                    m = slo;
                                else
                                    for (int q = 0; q < MC; ++q)
                                        m = min(m, cluster.map_shared_rank(&st, q)->smin[b]);
                                y = float_of(m);
                            }
                            out = __fmul_rn(0.5f, __fadd_rn(x, y));
                        }
                        C[(size_t)b * k + j] = out;
                    }
                    d->done[b] = lo == hi;
                    d->rng[b] = make_uint2(lo, (slo <= shi ? shi : hi) - lo);
                    d->khi[b] = hi;
                    const int bits = 32 - __clz((int)(hi - lo));
                    d->shift[b] = bits > 11 ? bits - 11 : 0;
                    d->slo[b] = slo;
                    d->shi[b] = shi;
                    d->rank[b] = rin;
                    d->cnt[b] = cnt;
                }
            }
            __syncthreads();  // s_warp and s_found are free; smin is read
            if (tid < MC && cnt && !(cnt & 1u) && s_found[3] != 0xffffffffu)
                cluster.map_shared_rank(&st, tid)->smin[b] = 0xffffffffu;  // a nearer bin
            __syncthreads();
        }
        cluster.sync();  // the choices are in every block, the histograms are read
        bool all = true;
        for (int b = 0; b < n; ++b) all = all && st.done[b] != 0u;
        if (all) break;  // uniform over the cluster: the states are equal
    }
    cluster.sync();  // no block exits while another may still read its shared memory
}

// Last step: colour and texture assignments to the final centres and the
// data term f_{a n_t + b} = -log P_colour(a) - log P_texture(b), each a
// softmax over its classes: logits -|I - mu_a|^2 / (2 sigma_c2) and
// -||c_b - iota||_1 / beta.
template <int NC>
__global__ void __launch_bounds__(UB) unsup_final_kernel(
    const float* __restrict__ img, int P, const float* __restrict__ V, int k,
    const float* __restrict__ Ccol, int nc, const float* __restrict__ Ctex, int nt,
    float inv2s2, float inv_beta, float* __restrict__ neglog, int32_t* __restrict__ cassign,
    int32_t* __restrict__ tassign) {
    extern __shared__ __align__(16) float C[];  // k x cpad(NC) texture centres
    __shared__ float Cc[3 * CS_MAX_CLASSES];
    load_centres<NC>(C, Ctex, nt, k);
    for (int t = threadIdx.x; t < 3 * nc; t += UB) Cc[t] = Ccol[t];
    __syncthreads();
    for (int q = blockIdx.x * UB + threadIdx.x; q < P; q += gridDim.x * UB) {
        const float x[3] = {img[(size_t)q * 3], img[(size_t)q * 3 + 1], img[(size_t)q * 3 + 2]};
        if (cassign) cassign[q] = nearest_colour(x, Cc, nc);
        float d[NC];
        l1_all<NC>(V, P, k, q, C, d);
        float bd;
        const int best = nearest_l1<NC>(d, nt, bd);
        if (tassign) tassign[q] = best;
        // texture log-softmax
        const float tmax = -bd * inv_beta;
        float ts = 0.f;
#pragma unroll
        for (int b = 0; b < NC; ++b)
            if (NC <= 8 || b < nt) ts += __expf(-d[b] * inv_beta - tmax);
        const float tlse = tmax + __logf(ts);
        // colour log-softmax; the logits are formed again below, not kept
        auto logit = [&](int a) {
            const float t0 = x[0] - Cc[3 * a], t1 = x[1] - Cc[3 * a + 1], t2 = x[2] - Cc[3 * a + 2];
            return -(t0 * t0 + t1 * t1 + t2 * t2) * inv2s2;
        };
        float cmax = -3.0e38f;
        for (int a = 0; a < nc; ++a) cmax = fmaxf(cmax, logit(a));
        float cs = 0.f;
        for (int a = 0; a < nc; ++a) cs += __expf(logit(a) - cmax);
        const float clse = cmax + __logf(cs);
        float* out = neglog + q;
        for (int a = 0; a < nc; ++a) {
            const float fc = clse - logit(a);
#pragma unroll
            for (int b = 0; b < NC; ++b)
                if (NC <= 8 || b < nt) out[(size_t)(a * nt + b) * P] = fc + (tlse + d[b] * inv_beta);
        }
    }
}

// Calls f with the class-count template argument for n classes.
template <class F>
cudaError_t with_classes(int n, F&& f) {
    switch (n) {
        case 1: return f(std::integral_constant<int, 1>{});
        case 2: return f(std::integral_constant<int, 2>{});
        case 3: return f(std::integral_constant<int, 3>{});
        case 4: return f(std::integral_constant<int, 4>{});
        case 5: return f(std::integral_constant<int, 5>{});
        case 6: return f(std::integral_constant<int, 6>{});
        case 7: return f(std::integral_constant<int, 7>{});
        case 8: return f(std::integral_constant<int, 8>{});
        default: return f(std::integral_constant<int, CS_MAX_CLASSES>{});
    }
}

int grid_for(long long N, int n_sm) {
    const long long need = (N + UB - 1) / UB, cap = 8ll * n_sm;
    return (int)(need < 1 ? 1 : need < cap ? need : cap);
}

// dynamic shared memory of the median kernel and of the kernels that hold k x cpad(NC) centres
constexpr size_t median_smem(int n, bool h16) {
    const size_t cap = list_cap(h16);
    return sizeof(unsigned) * ((size_t)n * (h16 ? HB / 2 : HB) + cap) + cap;
}
constexpr size_t centres_smem(int k, int nc) { return sizeof(float) * (size_t)k * cpad(nc); }

}  // namespace

size_t kmeans_scratch_bytes(int n) {
    return sizeof(unsigned long long) * 3 * (size_t)n + sizeof(unsigned) * (size_t)n + 256;
}

cudaError_t launch_kmeans(const KmeansArgs& a, cudaStream_t st) {
    unsigned long long* sums = reinterpret_cast<unsigned long long*>(a.scratch);
    unsigned* counts = reinterpret_cast<unsigned*>(sums + 3 * a.n);
    cudaError_t e = cudaMemsetAsync(a.scratch, 0, kmeans_scratch_bytes(a.n), st);
    if (e != cudaSuccess) return e;
    kmeans_init_kernel<<<1, 3 * CS_MAX_CLASSES, 0, st>>>(a.X, a.init, a.n, a.C);
    const int g = grid_for(a.N, a.n_sm);
    for (int it = 0; it < a.iterations; ++it) {
        kmeans_assign_kernel<<<g, UB, 0, st>>>(a.X, a.N, a.C, a.n, nullptr, sums, counts);
        kmeans_update_kernel<<<1, 3 * CS_MAX_CLASSES, 0, st>>>(a.C, sums, counts, a.n);
    }
    if (a.assign)
        kmeans_assign_kernel<<<g, UB, 0, st>>>(a.X, a.N, a.C, a.n, a.assign, nullptr, nullptr);
    return cudaGetLastError();
}

cudaError_t launch_kmedians(const KmediansArgs& a, cudaStream_t st) {
    // (from 12 classes on full counters would leave one block per SM)
    const bool h16 = a.n >= 12 && (a.N + MC - 1) / MC <= 65535;
    const auto median = h16 ? class_median_kernel<true> : class_median_kernel<false>;
    const size_t hbytes = median_smem(a.n, h16);
    cudaError_t e = cs_smem_limit((const void*)median, median_smem(CS_MAX_CLASSES, h16));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute((const void*)median,
                                 cudaFuncAttributePreferredSharedMemoryCarveout,
                                 cudaSharedmemCarveoutMaxShared);
    if (e != cudaSuccess) return e;
    kmedians_init_kernel<<<(a.n * a.k + UB - 1) / UB, UB, 0, st>>>(a.V, a.N, a.k, a.init, a.n,
                                                                   a.C);
    return with_classes(a.n, [&](auto nc) {
        constexpr int NC = decltype(nc)::value;
        const size_t smem = centres_smem(a.k, NC);
        cudaError_t e2 =
            cs_smem_limit((const void*)kmedians_assign_kernel<NC>, centres_smem(CS_MAX_K, NC));
        if (e2 != cudaSuccess) return e2;
        const int g = grid_for(a.N, a.n_sm);
        for (int it = 0; it < a.iterations; ++it) {
            kmedians_assign_kernel<NC>
                <<<g, UB, smem, st>>>(a.V, a.N, a.k, a.C, a.n, nullptr, a.work_assign);
            median<<<a.k * MC, MB, hbytes, st>>>(a.V, a.N, a.k, a.work_assign, a.n, a.C);
        }
        if (a.assign)
            kmedians_assign_kernel<NC>
                <<<g, UB, smem, st>>>(a.V, a.N, a.k, a.C, a.n, a.assign, nullptr);
        return cudaGetLastError();
    });
}

cudaError_t launch_unsup_final(const UnsupFinalArgs& a, cudaStream_t st) {
    return with_classes(a.nt, [&](auto nc) {
        constexpr int NC = decltype(nc)::value;
        const size_t smem = centres_smem(a.k, NC);
        cudaError_t e = cs_smem_limit((const void*)unsup_final_kernel<NC>, centres_smem(CS_MAX_K, NC));
        if (e != cudaSuccess) return e;
        unsup_final_kernel<NC><<<grid_for(a.P, a.n_sm), UB, smem, st>>>(
            a.img, a.P, a.V, a.k, a.Ccol, a.nc, a.Ctex, a.nt, a.inv2s2, a.inv_beta, a.neglog,
            a.cassign, a.tassign);
        return cudaGetLastError();
    });
}
