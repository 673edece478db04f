// graph.cu -- Algorithm 2's adjust step (Sec. 3.2) on the GPU.
//
// Steps (1)-(3) of graph_host.h run here, one warp per vertex: the NSG
// pruning of every vertex's own candidates (kernel 1), the reverse-edge
// lists, then the re-pruning with them and the adaptive angle rule (kernel
// 2), which writes the finished rows; the flood of the reachability repair
// runs here too.  The random fill of a short row and the repair itself stay
// on the host.  Every decision is the host's bit for bit: the exact distance
// in its canonical fp32 order (32 lane partial sums of fmaf over float4
// chunks, then the xor butterfly), the same (distance, id) order, the same
// cosine arithmetic.  A vertex whose lists do not fit a warp's shared-memory
// lists (a hub with many reverse candidates) is marked and refined on the
// host with the same code.  A degree-unaligned graph ("w/o GR", Sec. 5)
// skips the angle rule.
//
// What bounds it: the angle rule's pairwise distances (about 6,500 per
// vertex at R = 32).  One pair at a time, each ended by a 5-step shuffle
// butterfly and a square root and division in every lane, they took 60
// warp-instructions and a full latency per pair.  Here the distances of up to
// 64 pairs are accumulated side by side (4 candidates x 16 nearer ones,
// reading each row once for the 4), their 32-lane sums are formed by a
// reduce-scatter that leaves one pair per lane (31 shuffles for 32 pairs
// instead of 160), and each lane then takes its own pair's cosine.
// Measured at 20,000 vertices of d 128, R = 32, 96 candidates: refinement
// 18.4 -> 3.1 ms, pruning 1.80 -> 1.23 ms; the whole call 28-30 -> 4.9-5.4 ms
// with the reverse lists (host loops over all edges before), the rows and the
// flood on the device as well.
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>
#include <vector>

#include "../../include/sqg.h"
#include "graph_host.h"

namespace {

constexpr int kWarps = 4;      // warps (vertices in flight) per block
constexpr int kCap = 512;      // entries of a warp's two long lists
constexpr int kMaxR = 64;      // longest edge list the kernels keep
constexpr int kAll = 256;      // kept + angle-rule candidates: R' + 3R' <= 4 * 64
constexpr uint32_t kNone = 0xFFFFFFFFu;
constexpr uint32_t kFlagHost = 1u, kFlagFill = 2u;  // rows that the host finishes
// counters of a build: kept edges, rows the angle rule supplemented, rows left
// to the host's refinement and to the random fill, values that are not finite
enum { kSumKept, kSupplemented, kHostRows, kFillRows, kBadValues, kCounters };

typedef unsigned long long u64;

// A candidate (distance, id) as one key whose unsigned order is the
// (distance, id) order: distances are sums of squares from +0, never
// negative, so their bits order like their values.
__device__ __forceinline__ u64 key_di(float d, uint32_t id) { return ((u64)__float_as_uint(d) << 32) | id; }
__device__ __forceinline__ float key_d(u64 k) { return __uint_as_float((uint32_t)(k >> 32)); }
__device__ __forceinline__ uint32_t key_id(u64 k) { return (uint32_t)k; }
// the same candidate keyed by id first (for removing repeated ids)
__device__ __forceinline__ u64 swap_halves(u64 k) { return (k << 32) | (k >> 32); }

__device__ __forceinline__ uint32_t lanes_below(int lane) { return (1u << lane) - 1u; }

// Ascending bitonic sort of a[0, cnt) by one warp; a has room for the
// next power of 2 >= max(cnt, 32), padded with the largest key.
__device__ void warp_sort(u64 *a, int cnt, int lane) {
    int N = 32;
    while (N < cnt) N <<= 1;
    for (int i = cnt + lane; i < N; i += 32) a[i] = ~0ull;
    __syncwarp();
    for (int k = 2; k <= N; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = lane; i < N; i += 32) {
                const int ixj = i ^ j;
                if (ixj > i) {
                    const u64 x = a[i], y = a[ixj];
                    if ((x > y) == ((i & k) == 0)) {
                        a[i] = y;
                        a[ixj] = x;
                    }
                }
            }
            __syncwarp();
        }
}

// a[0, cnt) sorted by id-first keys: copy one entry per id to b, back in
// (distance, id) keys; returns the count.
__device__ int unique_by_id(const u64 *a, int cnt, u64 *b, int lane) {
    int m = 0;
    for (int base = 0; base < cnt; base += 32) {
        const int i = base + lane;
        const bool keep = i < cnt && (i == 0 || (a[i] >> 32) != (a[i - 1] >> 32));
        const uint32_t bal = __ballot_sync(0xffffffffu, keep);
        if (keep) b[m + __popc(bal & lanes_below(lane))] = swap_halves(a[i]);
        m += __popc(bal);
    }
    __syncwarp();
    return m;
}

// The canonical sums of P pairs whose lane partials are v[0, P): at butterfly
// step O a lane hands the half of its pairs that the partner keeps to the
// partner and adds the partner's partials to its own half -- the same two
// partials per addition as the plain xor butterfly, so the same sums.  Lane l
// ends with pair l >> (5 - log2 P).
template <int P, int O>
__device__ __forceinline__ float reduce_scatter(const float (&v)[P], int lane) {
    if constexpr (O == 0) {
        return v[0];
    } else if constexpr (P == 1) {
        const float w[1] = {__fadd_rn(v[0], __shfl_xor_sync(0xffffffffu, v[0], O))};
        return reduce_scatter<1, O / 2>(w, lane);
    } else {
        const bool up = (lane & O) != 0;
        float w[P / 2];
#pragma unroll
        for (int i = 0; i < P / 2; ++i) {
            const float keep = up ? v[i + P / 2] : v[i], give = up ? v[i] : v[i + P / 2];
            w[i] = __fadd_rn(keep, __shfl_xor_sync(0xffffffffu, give, O));
        }
        return reduce_scatter<P / 2, O / 2>(w, lane);
    }
}

__device__ __forceinline__ float add_sq(const float4 &p, const float4 &q, float acc) {
    const float dx = __fsub_rn(p.x, q.x), dy = __fsub_rn(p.y, q.y);
    const float dz = __fsub_rn(p.z, q.z), dw = __fsub_rn(p.w, q.w);
    acc = __fmaf_rn(dx, dx, acc);
    acc = __fmaf_rn(dy, dy, acc);
    acc = __fmaf_rn(dz, dz, acc);
    return __fmaf_rn(dw, dw, acc);
}

// Exact squared distances, in the canonical order, of row x to the rows of
// the candidates list[0, cnt), 1 <= cnt <= P (absent ones repeat the last):
// lane l returns that of candidate l >> (5 - log2 P).
template <int P>
__device__ __forceinline__ float row_dists(const float *data, uint32_t d, const float *x, const u64 *list, int cnt,
                                           int lane) {
    const uint32_t nch = d / 4;
    const float4 *x4 = reinterpret_cast<const float4 *>(x);
    float v[P];
#pragma unroll
    for (int p = 0; p < P; ++p) v[p] = 0.0f;
    for (uint32_t c = lane; c < nch; c += 32) {
        const float4 xc = __ldg(x4 + c);
#pragma unroll
        for (int p = 0; p < P; ++p) {
            const uint32_t id = key_id(list[min(p, cnt - 1)]);
            v[p] = add_sq(__ldg(reinterpret_cast<const float4 *>(data + (size_t)id * d) + c), xc, v[p]);
        }
    }
    return reduce_scatter<P, 16>(v, lane);
}

// NSG's rule over c[0, m) (sorted): keep c unless a kept w has
// d(w, c) < d(u, c); at most R kept, written to kept[].  Warp-uniform.  A
// candidate's distances to up to 16 kept ones are taken at once.
__device__ int nsg_prune_warp(const u64 *c, int m, u64 *kept, int R, const float *data, uint32_t d, int lane) {
    int nk = 0;
    for (int i = 0; i < m && nk < R; ++i) {
        const u64 ci = c[i];
        const float *xc = data + (size_t)key_id(ci) * d;
        bool occluded = false;
        for (int j = 0; j < nk && !occluded;) {
            const int cnt = nk - j;
            bool hit;
            if (cnt <= 4) {
                hit = row_dists<4>(data, d, xc, kept + j, cnt, lane) < key_d(ci);
                j += 4;
            } else if (cnt <= 8) {
                hit = row_dists<8>(data, d, xc, kept + j, cnt, lane) < key_d(ci);
                j += 8;
            } else {
                hit = row_dists<16>(data, d, xc, kept + j, min(cnt, 16), lane) < key_d(ci);
                j += 16;
            }
            occluded = __any_sync(0xffffffffu, hit);
        }
        if (!occluded) {
            if (lane == 0) kept[nk] = ci;
            ++nk;
            __syncwarp();
        }
    }
    return nk;
}

// The angle rule's score of extra candidates ext[0, ne) (sorted): the largest
// cosine to a nearer one of all[0, nall) (sorted), -2 if none is nearer.
__device__ __forceinline__ void angle_scores(const u64 *ext, int ne, const u64 *all, int nall, float *score,
                                             const float *data, uint32_t d, int lane) {
    const uint32_t nch = d / 4;
    for (int e0 = 0; e0 < ne; e0 += 4) {
        const u64 last = ext[min(e0 + 3, ne - 1)];  // its nearer ones include the others'
        u64 ce[2];
        float de[2], se[2], best[2];
#pragma unroll
        for (int g = 0; g < 2; ++g) {  // this lane's candidates: e0 + 2 g + (lane / 16)
            const int e = e0 + 2 * g + (lane >> 4);
            ce[g] = e < ne ? ext[e] : 0ull;  // (key 0: nothing is nearer)
            de[g] = key_d(ce[g]);
            se[g] = __fsqrt_rn(de[g]);
            best[g] = -2.0f;
        }
        for (int p0 = 0; p0 < nall && all[p0] < last; p0 += 16) {
            float v[2][32];  // pairs (e0 + 2 g + q / 16, p0 + q % 16)
#pragma unroll
            for (int g = 0; g < 2; ++g)
#pragma unroll
                for (int q = 0; q < 32; ++q) v[g][q] = 0.0f;
            for (uint32_t c = lane; c < nch; c += 32) {
                float4 x[4];
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    x[i] = __ldg(reinterpret_cast<const float4 *>(
                                     data + (size_t)key_id(ext[min(e0 + i, ne - 1)]) * d) + c);
                // eight rows on their way together: 168 registers and 12 warps per SM
                // instead of 127 and 16, and 5 % (d 128) to 18 % (d 256) faster
#pragma unroll
                for (int h = 0; h < 16; h += 8) {
                    float4 y[8];
#pragma unroll
                    for (int p = 0; p < 8; ++p)
                        y[p] = __ldg(reinterpret_cast<const float4 *>(
                                         data + (size_t)key_id(all[min(p0 + h + p, nall - 1)]) * d) + c);
#pragma unroll
                    for (int p = 0; p < 8; ++p)
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            v[i >> 1][(i & 1) * 16 + h + p] = add_sq(y[p], x[i], v[i >> 1][(i & 1) * 16 + h + p]);
                }
            }
            const int j = p0 + (lane & 15);
            const u64 kw = j < nall ? all[j] : ~0ull;
            const float dw = key_d(kw), sw = __fmul_rn(2.0f, __fsqrt_rn(dw));
#pragma unroll
            for (int g = 0; g < 2; ++g) {
                const float dwc = reduce_scatter<32, 16>(v[g], lane);
                if (kw < ce[g]) {
                    const float den = __fmul_rn(sw, se[g]);
                    const float cs = den > 0.0f ? __fdiv_rn(__fsub_rn(__fadd_rn(dw, de[g]), dwc), den) : 1.0f;
                    if (best[g] < cs) best[g] = cs;
                }
            }
        }
#pragma unroll
        for (int g = 0; g < 2; ++g) {
#pragma unroll
            for (int o = 8; o >= 1; o >>= 1) {
                const float b = __shfl_xor_sync(0xffffffffu, best[g], o);
                if (best[g] < b) best[g] = b;
            }
            const int e = e0 + 2 * g + (lane >> 4);
            if ((lane & 15) == 0 && e < ne) score[e] = best[g];
        }
    }
    __syncwarp();
}

struct WarpLists {
    u64 a[kCap], b[kCap];
    u64 k[kMaxR];
    float s[kAll];
};

// (1) own candidates of each vertex, kept by NSG's rule.
__global__ void __launch_bounds__(kWarps * 32) adjust_prune_kernel(const float *__restrict__ data, uint64_t n,
                                                                   uint32_t d, const uint32_t *__restrict__ cand,
                                                                   uint32_t L, uint32_t Rr, u64 *c_own,
                                                                   uint32_t *c_cnt, u64 *k1, uint32_t *n1,
                                                                   uint32_t *rcnt, u64 *counters) {
    __shared__ WarpLists lists[kWarps];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    WarpLists &S = lists[w];
    for (uint64_t u = (uint64_t)blockIdx.x * kWarps + w; u < n; u += (uint64_t)gridDim.x * kWarps) {
        int m = 0;  // valid ids (L <= kCap), keyed by id
        for (uint32_t base = 0; base < L; base += 32) {
            const uint32_t t = base + lane;
            const uint32_t v = t < L ? cand[u * L + t] : kNone;
            const bool ok = v != kNone && v < n && v != u;
            const uint32_t bal = __ballot_sync(0xffffffffu, ok);
            if (ok) S.a[m + __popc(bal & lanes_below(lane))] = (u64)v << 32;
            m += __popc(bal);
        }
        __syncwarp();
        warp_sort(S.a, m, lane);
        m = unique_by_id(S.a, m, S.b, lane);
        const float *xu = data + (size_t)u * d;
        for (int i = 0; i < m; i += 32) {
            const float dd = row_dists<32>(data, d, xu, S.b + i, min(m - i, 32), lane);
            __syncwarp();
            if (i + lane < m) S.b[i + lane] = key_di(dd, key_id(S.b[i + lane]));
        }
        __syncwarp();
        warp_sort(S.b, m, lane);
        for (int i = lane; i < m; i += 32) c_own[u * L + i] = S.b[i];
        const int nk = nsg_prune_warp(S.b, m, S.k, (int)Rr, data, d, lane);
        for (int i = lane; i < nk; i += 32) {
            k1[u * Rr + i] = S.k[i];
            atomicAdd(&rcnt[key_id(S.k[i])], 1u);  // a reverse candidate of its target
        }
        if (lane == 0) {
            c_cnt[u] = (uint32_t)m;
            n1[u] = (uint32_t)nk;
            atomicAdd(&counters[kSumKept], (u64)nk);
        }
        __syncwarp();
    }
}

// Reverse lists, offsets: exclusive prefix sum of the n counts, with the total
// at off[n]; the counts are cleared for the fill.  One block.
constexpr int kScanThreads = 1024, kScanItems = 8;
__global__ void __launch_bounds__(kScanThreads) reverse_offsets_kernel(uint32_t *cnt, uint64_t n, uint64_t *off) {
    __shared__ u64 warp_sum[kScanThreads / 32];
    __shared__ u64 carry;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    if (tid == 0) carry = 0;
    __syncthreads();
    for (uint64_t base = 0; base < n; base += kScanThreads * kScanItems) {
        const uint64_t i0 = base + (uint64_t)tid * kScanItems;
        uint32_t c[kScanItems];
        u64 sum = 0;
#pragma unroll
        for (int j = 0; j < kScanItems; ++j) {
            c[j] = i0 + j < n ? cnt[i0 + j] : 0u;
            if (i0 + j < n) cnt[i0 + j] = 0u;
            sum += c[j];
        }
        u64 x = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const u64 y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) warp_sum[w] = x;
        __syncthreads();
        if (w == 0) {
            u64 t = warp_sum[lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const u64 y = __shfl_up_sync(0xffffffffu, t, o);
                if (lane >= o) t += y;
            }
            warp_sum[lane] = t;
        }
        __syncthreads();
        u64 run = carry + (w > 0 ? warp_sum[w - 1] : 0) + x - sum;
#pragma unroll
        for (int j = 0; j < kScanItems; ++j) {
            if (i0 + j < n) off[i0 + j] = run;
            run += c[j];
        }
        __syncthreads();
        if (tid == kScanThreads - 1) carry = run;
        __syncthreads();
    }
    if (tid == 0) off[n] = carry;
}

// Reverse lists, entries: the edge u -> v as (distance, u) at v.  The order
// within a list is whatever the atomics give: its readers sort.
__global__ void reverse_fill_kernel(const u64 *__restrict__ k1, const uint32_t *__restrict__ n1, uint64_t n, uint32_t Rr,
                                    const uint64_t *__restrict__ off, uint32_t *cnt, u64 *rev) {
    const int lane = threadIdx.x & 31;
    const uint64_t u = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (u >= n) return;
    for (uint32_t j = lane; j < n1[u]; j += 32) {
        const u64 k = k1[u * Rr + j];
        const uint32_t v = key_id(k);
        rev[off[v] + atomicAdd(&cnt[v], 1u)] = key_di(key_d(k), (uint32_t)u);
    }
}

// Values that are not finite (the packed keys order finite distances only).
__global__ void finite_kernel(const float *__restrict__ x, uint64_t count, u64 *counters) {
    bool bad = false;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (uint64_t)gridDim.x * blockDim.x)
        bad |= !isfinite(x[i]);
    if (bad) atomicAdd(&counters[kBadValues], 1ull);
}

// One level of the flood from the entry point: the out-neighbours of every
// vertex of level `at` that have no level yet get the next one.  A warp looks
// at 32 vertices and walks the rows of those on the level together.
__global__ void flood_kernel(const uint32_t *__restrict__ adj, uint64_t n, uint32_t R, uint32_t *level, uint32_t at,
                             uint32_t *grew) {
    const int lane = threadIdx.x & 31;
    const uint64_t u0 = (((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32;
    if (u0 >= n) return;
    const bool on = u0 + lane < n && level[u0 + lane] == at;
    bool any = false;
    for (uint32_t m = __ballot_sync(0xffffffffu, on); m; m &= m - 1) {
        const uint64_t u = u0 + __ffs(m) - 1;
        for (uint32_t t = lane; t < R; t += 32) {
            const uint32_t v = adj[u * R + t];
            if (v != kNone && level[v] == kNone) {
                level[v] = at + 1;
                any = true;
            }
        }
    }
    if (any) *grew = 1u;
}

// (2)-(3) re-prune with the reverse candidates, then the angle rule; the
// finished rows go to adj (n x R).
__global__ void __launch_bounds__(kWarps * 32) adjust_refine_kernel(
    const float *__restrict__ data, uint64_t n, uint32_t d, uint32_t L, uint32_t Rr, const u64 *__restrict__ c_own,
    const uint32_t *__restrict__ c_cnt, u64 *k1, const uint32_t *__restrict__ n1, const u64 *__restrict__ rev,
    const uint64_t *__restrict__ roff, int regular, uint32_t R, uint32_t *n2, uint32_t *flag, uint32_t *adj,
    u64 *counters) {
    __shared__ WarpLists lists[kWarps];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    WarpLists &S = lists[w];
    const int cap = d >= 512 ? 2 * (int)Rr : 3 * (int)Rr;
    for (uint64_t u = (uint64_t)blockIdx.x * kWarps + w; u < n; u += (uint64_t)gridDim.x * kWarps) {
        const uint64_t r0 = roff[u], nrev = roff[u + 1] - r0;
        const int nk1 = (int)n1[u];
        if ((uint64_t)nk1 + nrev > (uint64_t)kCap || (uint64_t)c_cnt[u] + nrev > (uint64_t)kCap) {
            if (lane == 0) {
                flag[u] = kFlagHost;  // too long for the warp's lists
                atomicAdd(&counters[kHostRows], 1ull);
            }
            continue;
        }
        // pool = kept edges + reverse candidates, one per id, by (distance, id)
        int np = nk1 + (int)nrev;
        for (int i = lane; i < np; i += 32)
            S.a[i] = swap_halves(i < nk1 ? k1[u * Rr + i] : rev[r0 + (i - nk1)]);
        __syncwarp();
        warp_sort(S.a, np, lane);
        np = unique_by_id(S.a, np, S.b, lane);
        warp_sort(S.b, np, lane);
        int nk = nsg_prune_warp(S.b, np, S.k, (int)Rr, data, d, lane);
        if (regular && nk < (int)Rr) {
            if (lane == 0) atomicAdd(&counters[kSupplemented], 1ull);
            // own and reverse candidates not kept, the nearest `cap` of them
            const int nc = (int)c_cnt[u];
            int na = nc + (int)nrev;
            for (int i = lane; i < na; i += 32) S.a[i] = swap_halves(i < nc ? c_own[u * L + i] : rev[r0 + (i - nc)]);
            __syncwarp();
            warp_sort(S.a, na, lane);
            na = unique_by_id(S.a, na, S.b, lane);
            int ne = 0;
            for (int base = 0; base < na; base += 32) {
                const int i = base + lane;
                bool keep = i < na;
                if (keep)
                    for (int j = 0; j < nk; ++j) keep = keep && key_id(S.k[j]) != key_id(S.b[i]);
                const uint32_t bal = __ballot_sync(0xffffffffu, keep);
                if (keep) S.a[ne + __popc(bal & lanes_below(lane))] = S.b[i];
                ne += __popc(bal);
            }
            __syncwarp();
            warp_sort(S.a, ne, lane);
            if (ne > cap) ne = cap;
            const int need = (int)Rr - nk;
            if (ne > 0) {
                // all = kept + extra by (distance, id)
                const int nall = nk + ne;
                for (int i = lane; i < nall; i += 32) S.b[i] = i < nk ? S.k[i] : S.a[i - nk];
                __syncwarp();
                warp_sort(S.b, nall, lane);
                // each extra candidate's largest cosine to a nearer candidate
                angle_scores(S.a, ne, S.b, nall, S.s, data, d, lane);
                // the threshold: the take-th smallest score
                const int take = need < ne ? need : ne;
                for (int i = lane; i < ne; i += 32) {
                    const uint32_t bits = __float_as_uint(S.s[i]);
                    const uint32_t ord = (bits & 0x80000000u) ? ~bits : (bits | 0x80000000u);
                    S.b[i] = ((u64)ord << 32) | (uint32_t)i;
                }
                __syncwarp();
                warp_sort(S.b, ne, lane);
                const float thr = S.s[(uint32_t)S.b[take - 1]];
                // the nearest `take` candidates scoring at most the threshold
                int added = 0;
                for (int base = 0; base < ne && added < take; base += 32) {
                    const int i = base + lane;
                    const bool sel = i < ne && S.s[i] <= thr;
                    const uint32_t bal = __ballot_sync(0xffffffffu, sel);
                    const int pos = added + __popc(bal & lanes_below(lane));
                    if (sel && pos < take) S.k[nk + pos] = S.a[i];
                    added += __popc(bal);
                }
                __syncwarp();
                nk += added < take ? added : take;
                warp_sort(S.k, nk, lane);
            }
        }
        const bool fill = regular && nk < (int)Rr;  // the host adds random vertices
        for (uint32_t t = lane; t < R && !fill; t += 32)
            adj[u * R + t] = t < (uint32_t)nk ? key_id(S.k[t]) : regular ? key_id(S.k[t % nk]) : kNone;
        for (int i = lane; i < nk && fill; i += 32) k1[u * Rr + i] = S.k[i];  // (its kept edges are in the pool)
        if (lane == 0) {
            n2[u] = (uint32_t)nk;
            flag[u] = fill ? kFlagFill : 0u;
            if (fill) atomicAdd(&counters[kFillRows], 1ull);
        }
        __syncwarp();
    }
}

// One device allocation for the build's arrays (14 cudaMalloc and cudaFree
// pairs took 0.75 ms).
struct DevArena {
    char *base = nullptr;
    size_t size = 0;
    ~DevArena() {
        if (base) cudaFree(base);
    }
    size_t add(size_t bytes) {  // offset of an array; all before commit()
        const size_t at = size;
        size += (bytes + 255) / 256 * 256;
        return at;
    }
    bool commit() { return cudaMalloc(&base, size ? size : 256) == cudaSuccess; }
    template <class T>
    T *at(size_t off) const { return reinterpret_cast<T *>(base + off); }
};

inline sqg_graph::Cand unpack_host(uint64_t k) {
    sqg_graph::Cand c;
    const uint32_t bits = (uint32_t)(k >> 32);
    std::memcpy(&c.d, &bits, 4);
    c.id = (uint32_t)k;
    return c;
}

}  // namespace

extern "C" int sqg_build_graph_ex(const float *data, uint64_t n, uint32_t d, const uint32_t *cand, uint32_t L,
                                  uint32_t R, uint32_t entry, uint64_t seed, uint32_t flags, uint32_t *out_adj,
                                  uint64_t *out_stats, int threads, int device) {
    if ((flags & ~SQG_GRAPH_IRREGULAR) != 0) return SQG_ERR_INVALID_ARG;
    const bool regular = !(flags & SQG_GRAPH_IRREGULAR);
    if (device < 0) {
        if (out_stats) out_stats[4] = n;  // every vertex refined on the host
        return sqg_graph::build_graph_host(data, n, d, cand, L, R, entry, seed, regular, out_adj, out_stats, threads);
    }
    if (!data || !cand || !out_adj || n < 2 || d == 0 || d % 32 != 0 || R == 0 || R % 32 != 0 || L == 0 ||
        entry >= n || n > 0xFFFFFFF0ull)
        return SQG_ERR_INVALID_ARG;
    const uint32_t Rr = (uint32_t)std::min<uint64_t>(R, n - 1);
    if (L > (uint32_t)kCap || Rr > (uint32_t)kMaxR) return SQG_ERR_UNSUPPORTED;
    int prev = -1;
    cudaGetDevice(&prev);
    if (cudaSetDevice(device) != cudaSuccess) {
        cudaGetLastError();
        return SQG_ERR_INVALID_ARG;
    }
    int rc = SQG_OK;
    {
        // What is not needed at the same time shares memory: the rows take the
        // candidate ids' place once the pruning has read those, a row left to the
        // host its kept edges'; the reverse counts, the refined lists' counts and
        // the flood's levels follow one another.
        DevArena A;
        const size_t cand_bytes = sizeof(uint32_t) * n * L;
        const size_t rows_bytes = (sizeof(uint32_t) * n * R + 255) / 256 * 256;
        const size_t o_data = A.add(sizeof(float) * n * d), o_cand = A.add(std::max(cand_bytes, rows_bytes));
        const size_t o_own = A.add(sizeof(u64) * n * L), o_cnt = A.add(sizeof(uint32_t) * n);
        const size_t o_k1 = A.add(sizeof(u64) * n * Rr), o_n1 = A.add(sizeof(uint32_t) * n);
        const size_t o_roff = A.add(sizeof(uint64_t) * (n + 1)), o_rev = A.add(sizeof(u64) * n * Rr);
        const size_t o_n2 = A.add(sizeof(uint32_t) * n), o_flag = A.add(sizeof(uint32_t) * n);
        constexpr int kBatch = 8;  // flood levels between looks at the result
        const size_t o_ctr = A.add(sizeof(u64) * kCounters), o_grew = A.add(sizeof(uint32_t) * kBatch);
        if (!A.commit()) {
            cudaGetLastError();
            rc = SQG_ERR_OOM;
        }
        float *d_data = A.at<float>(o_data);
        uint32_t *c_cnt = A.at<uint32_t>(o_cnt), *n1 = A.at<uint32_t>(o_n1), *flag = A.at<uint32_t>(o_flag);
        uint32_t *d_cand = A.at<uint32_t>(o_cand), *d_adj = d_cand;
        uint32_t *n2 = A.at<uint32_t>(o_n2), *rcnt = n2, *level = n2;
        u64 *c_own = A.at<u64>(o_own), *k1 = A.at<u64>(o_k1), *d_rev = A.at<u64>(o_rev);
        uint64_t *d_roff = A.at<uint64_t>(o_roff);
        u64 *ctr = A.at<u64>(o_ctr), h_ctr[kCounters] = {};
        int sms = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
        sms = std::max(sms, 1);
        const long long want = ((long long)n + kWarps - 1) / kWarps;
        const int grid = (int)std::max(1LL, std::min<long long>(want, (long long)sms * 8));
        const unsigned warp_blocks = (unsigned)((n + 7) / 8), flood_blocks = (unsigned)((n + 255) / 256);
        auto ok = [&](cudaError_t e) {
            if (e != cudaSuccess && rc == SQG_OK) rc = SQG_ERR_CUDA;
            return rc == SQG_OK;
        };
        if (rc == SQG_OK && ok(cudaMemset(ctr, 0, sizeof(h_ctr))) && ok(cudaMemset(rcnt, 0, sizeof(uint32_t) * n)) &&
            ok(cudaMemcpy(d_data, data, sizeof(float) * n * d, cudaMemcpyHostToDevice))) {
            finite_kernel<<<sms * 4, 256>>>(d_data, n * d, ctr);
            ok(cudaGetLastError());
            ok(cudaMemcpy(d_cand, cand, cand_bytes, cudaMemcpyHostToDevice));
            ok(cudaMemcpy(h_ctr, ctr, sizeof(h_ctr), cudaMemcpyDeviceToHost));
            if (rc == SQG_OK && h_ctr[kBadValues]) rc = SQG_ERR_INVALID_ARG;
        }
        if (rc == SQG_OK) {  // (1)-(3)
            adjust_prune_kernel<<<grid, kWarps * 32>>>(d_data, n, d, d_cand, L, Rr, c_own, c_cnt, k1, n1, rcnt, ctr);
            reverse_offsets_kernel<<<1, kScanThreads>>>(rcnt, n, d_roff);
            reverse_fill_kernel<<<warp_blocks, 256>>>(k1, n1, n, Rr, d_roff, rcnt, d_rev);
            adjust_refine_kernel<<<grid, kWarps * 32>>>(d_data, n, d, L, Rr, c_own, c_cnt, k1, n1, d_rev, d_roff,
                                                        regular ? 1 : 0, R, n2, flag, d_adj, ctr);
            ok(cudaGetLastError());
            ok(cudaMemcpy(out_adj, d_adj, sizeof(uint32_t) * n * R, cudaMemcpyDeviceToHost));
            ok(cudaMemcpy(h_ctr, ctr, sizeof(h_ctr), cudaMemcpyDeviceToHost));
        }
        std::atomic<uint64_t> n_supp{0}, n_fill{0};
        const bool host_rows = h_ctr[kHostRows] != 0, fill_rows = h_ctr[kFillRows] != 0;
        if (rc == SQG_OK && (host_rows || fill_rows)) {  // the rows that the kernels left: refine, random fill
            std::vector<uint32_t> h_flag(n), h_n1(n), h_n2(n);
            std::vector<u64> h_k1((size_t)n * Rr), h_rev;  // kept edges of the rows to refine, refined lists of the others
            std::vector<uint64_t> roff;
            ok(cudaMemcpy(h_flag.data(), flag, sizeof(uint32_t) * n, cudaMemcpyDeviceToHost));
            ok(cudaMemcpy(h_k1.data(), k1, sizeof(u64) * h_k1.size(), cudaMemcpyDeviceToHost));
            if (host_rows) {
                h_rev.resize((size_t)h_ctr[kSumKept]);
                roff.resize(n + 1);
                ok(cudaMemcpy(h_n1.data(), n1, sizeof(uint32_t) * n, cudaMemcpyDeviceToHost));
                ok(cudaMemcpy(roff.data(), d_roff, sizeof(uint64_t) * (n + 1), cudaMemcpyDeviceToHost));
                ok(cudaMemcpy(h_rev.data(), d_rev, sizeof(u64) * h_rev.size(), cudaMemcpyDeviceToHost));
            }
            if (fill_rows) ok(cudaMemcpy(h_n2.data(), n2, sizeof(uint32_t) * n, cudaMemcpyDeviceToHost));
            std::vector<uint64_t> left;
            for (uint64_t u = 0; u < n; ++u)
                if (h_flag[u]) left.push_back(u);
            if (rc == SQG_OK)
                sqg_graph::parallel_for(left.size(), threads, [&](uint64_t i) {
                    const uint64_t u = left[i];
                    std::vector<sqg_graph::Cand> l2;
                    if (h_flag[u] & kFlagHost) {
                        std::vector<sqg_graph::Cand> own, rev;
                        for (uint32_t j = 0; j < h_n1[u]; ++j) own.push_back(unpack_host(h_k1[u * Rr + j]));
                        for (uint64_t j = roff[u]; j < roff[u + 1]; ++j) rev.push_back(unpack_host(h_rev[j]));
                        if (sqg_graph::refine_vertex(data, n, d, cand, L, Rr, u, own.data(), h_n1[u], rev.data(),
                                                     rev.size(), regular, l2))
                            n_supp++;
                    } else {
                        for (uint32_t j = 0; j < h_n2[u]; ++j) l2.push_back(unpack_host(h_k1[u * Rr + j]));
                    }
                    if (sqg_graph::fill_and_write(data, n, d, R, Rr, seed, u, regular, l2, out_adj)) n_fill++;
                }, 1);
        }
        if (rc == SQG_OK) {  // (5) reachability, flooded on the device from out_adj's current rows
            // A level is one launch that looks at every vertex, whatever it reaches:
            // 5.7 us with its share of the looks at the result (20,000 to 200,000
            // vertices; 6.6 at a million), while the host's flood looks at every
            // edge once, 40 to 180 ns per vertex of 32 edges.  A graph of very many
            // levels is the host's: n / 128 of them take 45 ns per vertex, so the
            // change costs at most about what the host takes.  A chain of 200,000
            // vertices: 15 ms for the call, 1,170 with a launch for each level.
            const uint64_t most = std::max<uint64_t>(64, n / 128);
            bool deep = false;
            bool current = !host_rows && !fill_rows;  // d_adj holds them
            const uint64_t repairs = sqg_graph::repair_reachability(
                n, cand, L, R, entry, out_adj, [&](std::vector<uint8_t> &seen) {
                    if (deep) {
                        seen = sqg_graph::reachable_host(n, R, entry, out_adj);
                        return true;
                    }
                    uint32_t *grew = A.at<uint32_t>(o_grew);
                    const uint32_t zero = 0;
                    if (!current) ok(cudaMemcpy(d_adj, out_adj, sizeof(uint32_t) * n * R, cudaMemcpyHostToDevice));
                    current = false;  // the repair may change rows before it asks again
                    ok(cudaMemset(level, 0xff, sizeof(uint32_t) * n));
                    ok(cudaMemcpy(level + entry, &zero, sizeof(zero), cudaMemcpyHostToDevice));
                    for (uint32_t at = 0; rc == SQG_OK; at += kBatch) {
                        uint32_t h_grew[kBatch];
                        ok(cudaMemset(grew, 0, sizeof(h_grew)));
                        for (int i = 0; i < kBatch; ++i)
                            flood_kernel<<<flood_blocks, 256>>>(d_adj, n, R, level, at + i, grew + i);
                        ok(cudaGetLastError());
                        ok(cudaMemcpy(h_grew, grew, sizeof(h_grew), cudaMemcpyDeviceToHost));
                        if (!h_grew[kBatch - 1]) break;
                        deep = at + kBatch >= most;
                        if (deep) {
                            seen = sqg_graph::reachable_host(n, R, entry, out_adj);
                            return rc == SQG_OK;
                        }
                    }
                    std::vector<uint32_t> h_level(n);
                    if (!ok(cudaMemcpy(h_level.data(), level, sizeof(uint32_t) * n, cudaMemcpyDeviceToHost))) return false;
                    seen.resize(n);
                    for (uint64_t v = 0; v < n; ++v) seen[v] = h_level[v] != kNone;
                    return true;
                });
            if (rc == SQG_OK && out_stats) {
                out_stats[0] = h_ctr[kSumKept] * 1000 / n;
                out_stats[1] = h_ctr[kSupplemented] + n_supp.load();
                out_stats[2] = n_fill.load();
                out_stats[3] = repairs;
                out_stats[4] = h_ctr[kHostRows];
            }
        }
    }
    if (prev >= 0) cudaSetDevice(prev);
    return rc;
}
