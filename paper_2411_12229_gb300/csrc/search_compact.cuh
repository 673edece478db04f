// search_compact.cuh -- the compact search kernel: one warp per query for
// d <= 1024, out-degree 32 or 64, k <= 32 and ef <= 128 (for d <= 256 also
// k <= 128 and ef <= 256), with multiple estimates (instantiated in
// search_compact.cu for d <= 256, search_compact_wide.cu for 256 < d <=
// 1024, search_compact_stop.cu with the learned stop and
// search_compact_big.cu for d <= 256 past k 32 or ef 128).
//
// It runs the same Algorithm 1 (Querying, Sec. 3.1.3) with multiple
// estimated distances and implicit re-ranking (Sec. 3.1.2) as
// search_kernel, takes every decision in the same precision and order, and
// returns the same ids, distances, hop counts and status bits; what differs
// is the bookkeeping, cut to a few warp instructions per step:
//
//   * a beam entry is one 64-bit word, (order-preserving key bits << 32) |
//     (id << 1) | visited, so the (key, id) order of reading R4 is one
//     unsigned compare and a duplicate (key, id) is one xor;
//   * the beam (at most 32 NB entries: NB = 2 for ef <= 64, 4 for ef <=
//     128, 8 for ef <= 256) sits in shared memory, sorted, and lane l also keeps entries
//     l + 32 s (s < NB) in registers for the select and the visited marks;
//     all 32 NB slots are always written, the empty entry (greater than
//     every entry, visited bit set) from the beam's length on, so the
//     binary search, the select and the marks need no bound on the length;
//   * the admitted candidates' beam positions come from a branch-free
//     binary search; the merged beam is gathered into the other of two
//     beam buffers, each output slot finding its source from a 32 NB-bit
//     mask of the candidates' final positions (no shifting loop);
//   * with out-degree 32 one or two admitted candidates are inserted into the
//     registers directly (position by ballots, later entries up by shuffles);
//   * the k <= 32 RK results live in registers, lane l holding results
//     l + 32 s (s < RK); without the stop, more than 32 results are logged
//     and sorted instead;
//   * with out-degree 64 (NR = 2) lane l estimates neighbours l and l + 32
//     and the step's candidates are staged 64 wide.
//
// The next vertex -- the smaller of the best admitted candidate and the
// first unvisited beam entry -- is known as soon as the estimates are, so
// its block copy (1-D bulk copy into shared memory, Sec. 3.1.4's
// prefetch) is issued before the merge, which then runs while the copy is
// in flight, together with the marks of the vertex's copies in the beam
// and its visited-set insert (one warp-wide probe of 32 slots).
#pragma once
#include "search.cuh"

namespace sqg {

namespace compact {

constexpr uint64_t kNone = ~0ull;  // an empty beam or result slot (greater than every entry)

// The learned stop's state carried from hop to hop (12 bytes of the warp's
// shared memory after its mbarrier).
struct StopCarry {
    int last_improve;
    float ema_improve, ema_insert;
};

// Order-preserving map of a float key (never NaN) to uint32: a < b as floats
// iff map(a) < map(b) as unsigned integers; -0 and +0 map to one value, as
// they compare equal as floats.
__device__ __forceinline__ uint32_t key_bits(float f) {
    const uint32_t b = __float_as_uint(__fadd_rn(f, 0.0f));  // -0 + 0 = +0
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ uint64_t pack_entry(uint32_t kb, uint32_t id) {
    return ((uint64_t)kb << 32) | ((uint64_t)id << 1);
}
__device__ __forceinline__ uint32_t entry_id(uint64_t e) { return (uint32_t)(e >> 1) & kIdMask; }
__device__ __forceinline__ uint64_t shfl64(uint64_t v, int src) {
    const uint32_t lo = __shfl_sync(kFull, (uint32_t)v, src), hi = __shfl_sync(kFull, (uint32_t)(v >> 32), src);
    return ((uint64_t)hi << 32) | lo;
}
__device__ __forceinline__ uint64_t shfl64_up(uint64_t v, int d) {
    const uint32_t lo = __shfl_up_sync(kFull, (uint32_t)v, d), hi = __shfl_up_sync(kFull, (uint32_t)(v >> 32), d);
    return ((uint64_t)hi << 32) | lo;
}

// Insert an id that is not in the table (an unvisited vertex) with the
// whole warp: lane l reads probe slot s + l, and the first empty slot of the
// window is the one a slot-by-slot linear probe would take.
__device__ __forceinline__ void hash_insert_warp(uint32_t *H, uint32_t bits, uint32_t id, int lane) {
    const uint32_t mask = (1u << bits) - 1u;
    uint32_t s = hslot(id, bits);
#pragma unroll 1
    for (;;) {
        const uint32_t slot = (s + lane) & mask;
        const uint32_t emp = __ballot_sync(kFull, H[slot] == kEmpty);
        if (emp) {
            if (lane == __ffs(emp) - 1) H[slot] = id;
            __syncwarp();
            return;
        }
        s += 32;
    }
}

// A full adder on bit slices: three words of one weight into a word of that
// weight (xor3) and the carries, a word of twice the weight (maj3), each as
// one three-input logic instruction (d 960: 4,600 cycles per expansion,
// against 5,560 with the plain expressions).
__device__ __forceinline__ uint32_t xor3(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0x96;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}
__device__ __forceinline__ uint32_t maj3(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0xE8;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}

// One expansion's exact-distance partial (exact_partial's arithmetic and
// order) and S = sum_i b_i qbar_i (Sec. 3.1.1) of neighbours lane + 32 n (n <
// NR), out-degree R = 32 NR: the sums over words w and planes b of 2^b
// popc(code word w of the neighbour, at w * R + j, AND word w of plane b),
// nw <= 4 CH words.
//
// A POPC holds its pipe for 8 cycles, an AND or ADD the ALU for 2: counted
// word by word, S of a long code is bound by the POPC pipe (8 cycles per word
// and plane; d 960 with out-degree 64: 5,850 of an expansion's 8,470 cycles
// with 12 warps per SM).  For d > 256 full adders in front halve the POPCs
// for 2 LOP3 each.  Exact partial, S and butterfly at d 960, out-degree 64,
// cycles per expansion, word by word / here: 4,160 / 2,780 for a lone warp,
// 6,250 / 4,600 with 12 warps per SM.  A second adder level gains nothing
// (4,800: the ALU is then the limit).  For d <= 256 other ALU work dominates a
// full SM, and adders cost more than they save (10k queries of d 128, ef 40:
// 262 us word by word, 273 with adders); where issue slots are free the chain
// they shorten counts (ADD: exact partial, S and butterfly of a lone warp 595
// -> 289 cycles).
template <int CH, int NR, bool ADD>
__device__ __forceinline__ void exact_and_S(const float4 (&qv)[CH], const unsigned char *blk, uint32_t off_codes,
                                            const uint32_t *planes, uint32_t nch, uint32_t nw, int lane, float (&acc)[1],
                                            int (&S)[NR]) {
    constexpr uint32_t R = 32 * NR;
    const uint32_t *codes = reinterpret_cast<const uint32_t *>(blk + off_codes) + lane;
    const uint4 *pl = reinterpret_cast<const uint4 *>(planes);
    if constexpr (CH <= 2) {
        exact_partial<CH, 32>(reinterpret_cast<const float4(&)[1][CH]>(qv), reinterpret_cast<const float *>(blk), nch,
                              Team<32>(lane), acc);
        if constexpr (NR == 1 && ADD) {
            // groups of four words, absent words zero; within a group the carries
            // of plane b join plane b + 1's words: 9 POPCs for 16
            S[0] = 0;
#pragma unroll
            for (uint32_t g = 0; g < 4 * CH; g += 4) {
                if (g > 0 && g >= nw) break;
                uint32_t c[4], p[4][4];  // [plane][word]
#pragma unroll
                for (uint32_t w = 0; w < 4; ++w) {
                    const bool in = g + w < nw;
                    const uint4 v = in ? pl[g + w] : make_uint4(0u, 0u, 0u, 0u);
                    p[0][w] = v.x;
                    p[1][w] = v.y;
                    p[2][w] = v.z;
                    p[3][w] = v.w;
                    c[w] = in ? codes[(g + w) * R] : 0u;
                }
                uint32_t s0[4], c0[4], a3[4], u[4], t[4];
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const uint32_t x = c[0] & p[b][0], y = c[1] & p[b][1], z = c[2] & p[b][2];
                    s0[b] = xor3(x, y, z);  // weight 2^b
                    c0[b] = maj3(x, y, z);  // weight 2^(b + 1)
                    a3[b] = c[3] & p[b][3];
                }
#pragma unroll
                for (int b = 1; b < 4; ++b) {
                    t[b] = xor3(c0[b - 1], s0[b], a3[b]);
                    u[b] = maj3(c0[b - 1], s0[b], a3[b]);
                }
                S[0] += __popc(s0[0]) + __popc(a3[0]) + 2 * __popc(t[1]) + 4 * (__popc(t[2]) + __popc(u[1])) +
                        8 * (__popc(t[3]) + __popc(u[2])) + 16 * (__popc(c0[3]) + __popc(u[3]));
            }
        } else {
            int s0[NR], s1[NR], s2[NR], s3[NR];
#pragma unroll
            for (int n = 0; n < NR; ++n) s0[n] = s1[n] = s2[n] = s3[n] = 0;
#pragma unroll
            for (uint32_t w = 0; w < 4 * CH; ++w)
                if (w < nw) {
                    const uint4 p = pl[w];
#pragma unroll
                    for (int n = 0; n < NR; ++n) {
                        const uint32_t c = codes[w * R + 32 * n];
                        s0[n] += __popc(c & p.x);
                        s1[n] += __popc(c & p.y);
                        s2[n] += __popc(c & p.z);
                        s3[n] += __popc(c & p.w);
                    }
                }
#pragma unroll
            for (int n = 0; n < NR; ++n) S[n] = s0[n] + 2 * s1[n] + 4 * s2[n] + 8 * s3[n];
        }
    } else {
        // chunk t: the lane's t-th float4 of the raw vector and words 4 t .. 4
        // t + 3; `one` carries each plane's sum of weight 1 from word to word
        const float4 *r4 = reinterpret_cast<const float4 *>(blk);
        uint32_t one[NR][4];
        int two[NR][4];  // counts of weight 2
#pragma unroll
        for (int n = 0; n < NR; ++n)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                one[n][b] = 0u;
                two[n][b] = 0;
            }
        float s = 0.0f;
#pragma unroll
        for (uint32_t t = 0; t < CH; ++t) {
            if (4 * t >= nw) break;
            const uint32_t c = lane + 32 * t;
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
            if (c < nch) x = r4[c];
            if (4 * t + 4 <= nw) {
                uint32_t p[4][4], cw[NR][4];
#pragma unroll
                for (uint32_t w = 0; w < 4; ++w) {
                    const uint4 v = pl[4 * t + w];
                    p[0][w] = v.x;
                    p[1][w] = v.y;
                    p[2][w] = v.z;
                    p[3][w] = v.w;
#pragma unroll
                    for (int n = 0; n < NR; ++n) cw[n][w] = codes[(4 * t + w) * R + 32 * n];
                }
#pragma unroll
                for (int n = 0; n < NR; ++n)
#pragma unroll
                    for (int b = 0; b < 4; ++b) {
                        const uint32_t a0 = cw[n][0] & p[b][0], a1 = cw[n][1] & p[b][1];
                        const uint32_t a2 = cw[n][2] & p[b][2], a3 = cw[n][3] & p[b][3];
                        const uint32_t o = one[n][b], o1 = xor3(o, a0, a1);
                        two[n][b] += __popc(maj3(o, a0, a1)) + __popc(maj3(o1, a2, a3));
                        one[n][b] = xor3(o1, a2, a3);
                    }
            } else {
                for (uint32_t w = 4 * t; w < nw; ++w) {
                    const uint4 v = pl[w];
#pragma unroll
                    for (int n = 0; n < NR; ++n) {
                        const uint32_t e = codes[w * R + 32 * n];
                        const uint32_t a[4] = {e & v.x, e & v.y, e & v.z, e & v.w};
#pragma unroll
                        for (int b = 0; b < 4; ++b) {
                            two[n][b] += __popc(one[n][b] & a[b]);
                            one[n][b] ^= a[b];
                        }
                    }
                }
            }
            if (c < nch) {
                const float dx = __fsub_rn(qv[t].x, x.x), dy = __fsub_rn(qv[t].y, x.y);
                const float dz = __fsub_rn(qv[t].z, x.z), dw = __fsub_rn(qv[t].w, x.w);
                s = __fmaf_rn(dx, dx, s);
                s = __fmaf_rn(dy, dy, s);
                s = __fmaf_rn(dz, dz, s);
                s = __fmaf_rn(dw, dw, s);
            }
        }
        acc[0] = s;
#pragma unroll
        for (int n = 0; n < NR; ++n) {
            S[n] = 0;
#pragma unroll
            for (int b = 0; b < 4; ++b) S[n] += (__popc(one[n][b]) + 2 * two[n][b]) << b;
        }
    }
}

// The key of neighbour j (the estimator of Sec. 3.1.1 and the bound-shifted
// key of reading R7), out-degree R, in two parts: what needs its S only, and
// the rest from the vertex's exact distance.  The same operations in the same
// order as estimate_from_S.
struct EstPart {
    float f_add, f_rescale, ip;
};
template <int R>
__device__ __forceinline__ EstPart est_part(const float *fac, const QuerySide &qs, uint32_t d, int j, int S) {
    EstPart e;
    e.f_add = fac[j];
    e.f_rescale = fac[R + j];
    const int pc = (int)reinterpret_cast<const uint32_t *>(fac)[3 * R + j];
    const float A = (float)(2 * S - qs.sq);
    const float B = __fmul_rn(qs.vl, (float)(2 * pc - (int)d));
    e.ip = __fmul_rn(__fmaf_rn(qs.delta, A, B), qs.inv_sqrt_d);
    return e;
}
template <int R>
__device__ __forceinline__ float est_key(const EstPart &e, const float *fac, int j, float dist_c, float eps0) {
    const float est = __fmaf_rn(e.f_rescale, e.ip, __fadd_rn(e.f_add, dist_c));
    if (eps0 == 0.0f) return est;
    const float bound = __fmul_rn(fac[2 * R + j], __fsqrt_rn(dist_c));
    return __fsub_rn(est, __fmul_rn(eps0, bound));
}

// hash_contains from the value `v` of the id's first slot on.
__device__ __forceinline__ bool hash_contains_from(uint32_t v, const uint32_t *H, uint32_t bits, uint32_t id) {
    if (v == id) return true;
    if (v == kEmpty) return false;
    const uint32_t mask = (1u << bits) - 1u;
    uint32_t s = hslot(id, bits);
#pragma unroll 1
    for (;;) {
        s = (s + 1) & mask;
        v = H[s];
        if (v == id) return true;
        if (v == kEmpty) return false;
    }
}

// With more than 32 results (RK 4) the expanded vertices are logged, as
// (distance bits << 32) | id, one per expansion that may enter the results,
// and the k smallest are selected when the log is full and at the end of the
// search: at k 100 nine expansions of ten enter the results, and keeping them
// in order as they come took 75 warp-instructions each, an eighth of the
// search (2,001 queries of d 128, k 100, ef 200: 430 -> 408 us; 10,000 at ef
// 100: 602 -> 527).  Up to k 32 one or two shuffles insert a result, and the
// log's selections cost more than that (10,000 queries at ef 40: 254 against
// 264 us, ef 96: 475 against 514).
constexpr int kLogSize = 256;  // k <= 128

// The min(n, k) smallest of log[0, n) to its front, in order (a bitonic sort
// of the next power of 2); returns their number.
__device__ __forceinline__ int log_select(uint64_t *log, int n, int k, int lane) {
    int N = 64;
    while (N < n) N <<= 1;
#pragma unroll 1
    for (int i = n + lane; i < N; i += 32) log[i] = kNone;
    __syncwarp();
#pragma unroll 1
    for (int run = 2; run <= N; run <<= 1)
#pragma unroll 1
        for (int j = run >> 1; j > 0; j >>= 1) {
#pragma unroll 2
            for (int i = lane; i < N / 2; i += 32) {
                const int x = ((i & ~(j - 1)) << 1) | (i & (j - 1)), y = x | j;
                const uint64_t ex = log[x], ey = log[y];
                if ((ex > ey) == ((x & run) == 0)) {
                    log[x] = ey;
                    log[y] = ex;
                }
            }
            __syncwarp();
        }
    return n < k ? n : k;
}

// The key a packed entry holds (the inverse of key_bits; -0 comes back as +0).
__device__ __forceinline__ float entry_key(uint64_t e) {
    const uint32_t kb = (uint32_t)(e >> 32);
    return __uint_as_float((kb & 0x80000000u) ? (kb & 0x7FFFFFFFu) : ~kb);
}

// Entry s of a lane's NB beam registers, s warp-uniform (an unrolled
// select: no local-memory array).
template <int NB>
__device__ __forceinline__ uint64_t pick(const uint64_t (&b)[NB], int s) {
    uint64_t v = b[0];
#pragma unroll
    for (int t = 1; t < NB; ++t)
        if (s == t) v = b[t];
    return v;
}

}  // namespace compact

// CH: float4 chunks of the raw vector per lane (d <= 128 CH).  NR:
// neighbours per lane (out-degree 32 NR).  NB: beam slots per lane (2: ef <=
// 64, 4: ef <= 128, 8: ef <= 256).  MINB: resident blocks of 4 warps per SM
// the build is made for (d <= 256 with NR 1: NB 2: 8 for up to 64 registers
// or 9 for 56; NB 4: 7 for up to 72 or 8 for 64).  STOP: the build with the
// learned early stop fused (the same features, network and decision points
// as search_kernel's, so the same hops, results and status bits).  RK:
// result slots per lane (1: k <= 32, 4: k <= 128), lane l holding results
// l + 32 s.  ADD: full adders in the estimates (exact_and_S).  What bounds
// it, measured: the chain of dependent steps of an expansion (without ADD 475
// warp-instructions; a lone warp takes 5.9 cycles for each) and with a full SM
// the issue slots (2.8 of 4 per cycle); no wait for a block finds it late at
// any load.
template <int CH, int NR, int NB, int MINB, bool STOP = false, int RK = 1, bool ADD = false>
__global__ void __launch_bounds__(128, MINB) search_compact_kernel(const SearchArgs a) {
    using namespace compact;
    constexpr bool kLog = RK > 1 && !STOP;  // (the stop's features need the results in order)
    // Up to this many admitted candidates are inserted one by one instead of
    // merged (out-degree 32; 26 % of the expansions admit none, 30 % one or
    // two): 45 warp-instructions each with two beam rows, against 140 for the
    // merge's search, ranks and gather.
    constexpr int kFew = NR == 1 ? (NB <= 4 ? 2 : 1) : 0;
    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t d = a.d, nch = d / 4;
    unsigned char *ws = smem + (size_t)warp * a.warp_bytes;
    unsigned char *const buf = ws + a.o_buf0;
    uint64_t *const bar = reinterpret_cast<uint64_t *>(ws + a.o_bar);
    uint64_t *beam_a = reinterpret_cast<uint64_t *>(ws + a.o_beam);  // two buffers of 32 NB entries
    uint64_t *beam_b = beam_a + 32 * NB;
    uint64_t *const stage = reinterpret_cast<uint64_t *>(ws + a.o_spos);  // this step's candidates by rank
    uint64_t *const rlog = reinterpret_cast<uint64_t *>(ws + a.o_log);
    uint32_t *const planes = reinterpret_cast<uint32_t *>(ws + a.o_planes);
    const uint32_t gwarp = blockIdx.x * (blockDim.x >> 5) + warp;
    uint32_t *const Hs = reinterpret_cast<uint32_t *>(ws + a.o_hash);
    uint32_t *const Hg = a.ghash ? a.ghash + ((size_t)gwarp << a.hash_bits) : nullptr;
    const Team<32> tm(lane);

    if (lane == 0) mbar_init(&bar[0], 1);
    fence_mbar_init();
    __syncwarp();
    uint32_t phase = 0;
    bool healthy = true;

    while (healthy) {
        int qi = 0;
        if (lane == 0) qi = (int)atomicAdd(a.queue_head, 1u);
        qi = __shfl_sync(kFull, qi, 0);
        if (qi >= a.nq) break;
        const int k = a.k ? a.k[qi] : a.uniform_k, ef = a.ef ? a.ef[qi] : a.one_ef;
        const long long off = a.uniform_k ? (long long)qi * a.uniform_k : a.offsets[qi];
        uint32_t status = 0;
        if (!(k >= 1 && k <= a.max_k && ef >= k && ef <= a.max_ef && (!a.uniform_k || k == a.uniform_k))) {
            const int kk = a.uniform_k ? a.uniform_k : (k < 0 ? 0 : (k > SQG_MAX_K ? SQG_MAX_K : k));
#pragma unroll 1
            for (int t = lane; t < kk; t += 32) {
                a.out_ids[off + t] = SQG_NO_ID;
                a.out_dists[off + t] = __int_as_float(0x7f800000);
            }
            if (lane == 0) {
                if (a.stats) a.stats[qi] = sqg_query_stats{0u, SQG_STATUS_BAD_PARAM};
                atomicOr(a.status_word, SQG_STATUS_BAD_PARAM);
            }
            continue;
        }
        const int hop_cap = a.hop_cap > 0 ? a.hop_cap : 4 * ef + 64;

        // ---- query setup: raw query in registers, quantized rotated query planes
        float4 qv[CH];
        const float4 *q4 = reinterpret_cast<const float4 *>(a.queries + (size_t)qi * d);
#pragma unroll
        for (int t = 0; t < CH; ++t) {
            const uint32_t c = lane + 32 * t;
            qv[t] = c < nch ? q4[c] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        QuerySide qs;
        if (a.qplanes) {
            const uint4 *src = reinterpret_cast<const uint4 *>(a.qplanes + (size_t)qi * 4 * (d / 32));
            if (lane < (int)(d / 32)) reinterpret_cast<uint4 *>(planes)[lane] = src[lane];
            const float4 sc = a.qscal[qi];
            qs.vl = sc.x;
            qs.delta = sc.y;
            qs.sq = (int)sc.z;
            qs.inv_sqrt_d = sc.w;
        } else {
            qs = quantize_team<32, CH <= 2>(a.qrot + (size_t)qi * d, d, planes, tm);
        }
        uint32_t *H = Hs;
        uint32_t hbits = a.shash_bits;
#pragma unroll 1
        for (uint32_t i = 4 * lane; i < (1u << hbits); i += 128)
            *reinterpret_cast<uint4 *>(H + i) = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);

        // ---- Algorithm 1, line 1: the beam holds the entry, which is expanded
        // first (its key, its exact distance, is set at that expansion)
        int m = 1;
        uint64_t b[NB];  // b[s] = beam[lane + 32 s]
#pragma unroll
        for (int s = 0; s < NB; ++s) {
            b[s] = s == 0 && lane == 0 ? pack_entry(0u, a.entry) | 1ull : kNone;
            beam_a[lane + 32 * s] = b[s];  // all 32 NB slots, kNone from m on: no bound on m below
        }
        // the results, in registers: res[s] = result[lane + 32 s], for lane + 32 s
        // < k; or nl entries of the log
        uint64_t res[RK];
#pragma unroll
        for (int s = 0; s < RK; ++s) res[s] = kNone;
        int nl = 0;
        uint64_t rworst = kNone;  // an entry that k results do not exceed: a new one must beat it
        uint64_t bworst = kNone;  // beam[ef - 1] once the beam holds ef entries (the early cut)
        uint32_t p = a.entry;
        __syncwarp();
        hash_insert_warp(H, hbits, p, lane);
        if (lane == 0) {
            fence_proxy_async();
            bulk_fetch(buf, a.blocks + (size_t)p * a.block_bytes, a.block_bytes, &bar[0]);
        }
        int hops = 1;
        // learned-stop state (STOP builds): the last hop whose vertex entered
        // the result and the moving averages of entering and of the inserted
        // share, kept by lane 0 in shared memory beside the barrier (no
        // registers held across the loop)
        StopCarry *const sst = reinterpret_cast<StopCarry *>(ws + a.o_bar + 8);
        if (STOP && lane == 0)
            *sst = StopCarry{0, 0.0f, 0.0f};

        for (;;) {
            if (__builtin_expect(!mbar_wait_bounded(&bar[0], phase & 1u), 0)) {
                status |= SQG_STATUS_TIMEOUT;
                healthy = false;
                break;
            }
            phase ^= 1u;
            const unsigned char *blk = buf;

            // ---- line 4: exact distance (implicit re-ranking); the neighbours'
            // integer sums S while the distance's butterfly is in flight
            float dacc[1];
            uint32_t cid[NR];
            int S[NR];
#pragma unroll
            for (int t = 0; t < NR; ++t) cid[t] = reinterpret_cast<const uint32_t *>(blk + a.off_ids)[lane + 32 * t];
            exact_and_S<CH, NR, ADD>(qv, blk, a.off_codes, planes, nch, d / 32, lane, dacc, S);
            EstPart part[NR];
            uint32_t hv[NR];  // each neighbour's first visited-set slot
#pragma unroll
            for (int t = 0; t < NR; ++t) {
                part[t] = est_part<32 * NR>(reinterpret_cast<const float *>(blk + a.off_factors), qs, d, lane + 32 * t,
                                            S[t]);
                hv[t] = H[hslot(cid[t], hbits)];
            }
            const float dist_c = exact_reduce<32>(dacc, tm);
            // ---- line 5: the estimate and key of every neighbour from the same block
            uint64_t cand[NR];
            bool adm[NR];
            uint32_t am[NR], anyam = 0;
#pragma unroll
            for (int t = 0; t < NR; ++t) {
                const float key = est_key<32 * NR>(part[t], reinterpret_cast<const float *>(blk + a.off_factors),
                                                   lane + 32 * t, dist_c, a.eps0);
                cand[t] = pack_entry(key_bits(key), cid[t]);
            }
            if (__builtin_expect(hops == 1, 0)) {  // reading R8: the entry's key is its exact distance
                if (lane == 0) {
                    b[0] = pack_entry(key_bits(dist_c), p) | 1ull;
                    beam_a[0] = b[0];
                }
                __syncwarp();
                if (ef == 1) bworst = shfl64(b[0], 0);
            }
#pragma unroll
            for (int t = 0; t < NR; ++t) {
                // ---- line 6: unvisited neighbours enter the beam; an entry the
                // cut to ef would drop at once is skipped early
                adm[t] = cid[t] != kEmpty && cand[t] < bworst;
                if (adm[t]) adm[t] = !hash_contains_from(hv[t], H, hbits, cid[t]);
                am[t] = __ballot_sync(kFull, adm[t]);
                anyam |= am[t];
            }

            // ---- lines 2-3 of the next step, taken now (Sec. 3.1.4: the next
            // block is fetched while this step's merge runs): the next vertex
            // is the smaller of the best admitted candidate and the first
            // unvisited beam entry.  A candidate equal in (key, id) to a beam
            // entry (dropped below as a duplicate) names that entry's vertex,
            // which is unvisited, so it may stand in for it here.
            uint64_t nxt;
            {  // the smallest of the lane's admitted candidates and unvisited
               // entries, then the warp's smallest (high word, then low word)
                uint64_t v = kNone;
#pragma unroll
                for (int t = 0; t < NR; ++t) v = adm[t] && cand[t] < v ? cand[t] : v;
#pragma unroll
                for (int s = 0; s < NB; ++s) v = !(b[s] & 1ull) && b[s] < v ? b[s] : v;  // kNone: visited
                const uint32_t chi = __reduce_min_sync(kFull, (uint32_t)(v >> 32));
                const uint32_t clo = __reduce_min_sync(kFull, (uint32_t)(v >> 32) == chi ? (uint32_t)v : 0xFFFFFFFFu);
                nxt = ((uint64_t)chi << 32) | clo;
            }
            const bool go = nxt != kNone && hops < hop_cap;  // a next expansion follows (the stop aside)
            const uint32_t pn = entry_id(nxt);
            __syncwarp();  // every lane's reads of the current block are done
            if (go && lane == 0) {
                fence_proxy_async();
                bulk_fetch(buf, a.blocks + (size_t)pn * a.block_bytes, a.block_bytes, &bar[0]);
            }
            bool improved = false;
            const uint64_t r = ((uint64_t)__float_as_uint(dist_c) << 32) | p;  // distances are >= 0
            if constexpr (kLog) {
                if (r < rworst) {
                    if (lane == 0) rlog[nl] = r;
                    if (__builtin_expect(++nl == kLogSize, 0)) {
                        nl = log_select(rlog, nl, k, lane);
                        rworst = rlog[k - 1];
                        __syncwarp();
                    }
                }
            } else {  // result top-k in registers
                if (r < rworst) {
                    improved = true;
                    int pos = 0;
#pragma unroll
                    for (int s = 0; s < RK; ++s) pos += __popc(__ballot_sync(kFull, lane + 32 * s < k && res[s] < r));
                    // entries pos .. k - 2 move up one slot: slot j takes old j - 1
                    // (lane 0 of row s from lane 31 of row s - 1)
                    uint64_t up[RK];
#pragma unroll
                    for (int s = 0; s < RK; ++s) {
                        const uint64_t u = shfl64_up(res[s], 1);
                        const uint64_t c = s > 0 ? shfl64(res[s > 0 ? s - 1 : 0], 31) : kNone;
                        up[s] = lane == 0 ? c : u;
                    }
#pragma unroll
                    for (int s = 0; s < RK; ++s) {
                        const int j = lane + 32 * s;
                        if (j == pos) res[s] = r;
                        else if (j > pos && j < k) res[s] = up[s];
                    }
                    rworst = shfl64(pick<RK>(res, (k - 1) >> 5), (k - 1) & 31);
                }
            }
            if constexpr (!STOP) {  // (with the stop these two ends follow its decision)
                if (nxt == kNone) break;  // no unvisited entry: the search ends (line 2)
                if (hops >= hop_cap) {    // reading R6
                    status |= SQG_STATUS_CAPACITY;
                    break;
                }
            }
            int inserted = 0;  // this step's candidates kept by the cut (the stop's features)

            // ---- line 6: merge the admitted candidates, cut the beam to ef
            const uint64_t *B = beam_a;
            int pos[NR];
            if (kFew > 0 && __popc(am[0]) <= kFew) {
                if (anyam) {
                    // a few candidates are inserted into the beam's registers one
                    // by one: position by ballots, later entries up by shuffles
                    int low = 32 * NB;
                    bool entered = false;  // this lane's candidate
#pragma unroll 1
                    for (uint32_t left = am[0]; left; left &= left - 1) {
                        const int src = __ffs(left) - 1;
                        const uint64_t c = shfl64(cand[0], src);
                        int at = 0;
                        bool same = false;
#pragma unroll
                        for (int s = 0; s < NB; ++s) {
                            at += __popc(__ballot_sync(kFull, b[s] < c));
                            same |= ((b[s] ^ c) >> 1) == 0;
                        }
                        if (__any_sync(kFull, same) || at >= ef) continue;  // there already, or cut
#pragma unroll
                        for (int s = NB - 1; s >= 0; --s) {
                            if (32 * s + 31 < at) continue;
                            const uint64_t u = shfl64_up(b[s], 1);
                            const uint64_t w = s > 0 ? shfl64(b[s > 0 ? s - 1 : 0], 31) : kNone;
                            const int o = lane + 32 * s;
                            if (o >= at) b[s] = o == at ? c : o >= ef ? kNone : lane == 0 ? w : u;
                        }
                        m = min(ef, m + 1);
                        low = min(low, at);
                        if (lane == src) entered = true;
                    }
#pragma unroll
                    for (int s = 0; s < NB; ++s)
                        if (32 * s + 31 >= low) beam_a[lane + 32 * s] = b[s];
                    bworst = m == ef ? shfl64(pick<NB>(b, (ef - 1) >> 5), (ef - 1) & 31) : kNone;
                    // (one that a smaller one pushed past the cut was not inserted)
                    if constexpr (STOP) inserted = __popc(__ballot_sync(kFull, entered && cand[0] <= bworst));
                }
                anyam = 0;
            } else if (anyam) {
                anyam = 0;
#pragma unroll
                for (int t = 0; t < NR; ++t) {
                    // beam position (lower bound) by a branch-free binary search;
                    // an identical (key, id) already in the beam is dropped
                    pos[t] = 0;
#pragma unroll
                    for (int step = 16 * NB; step >= 1; step >>= 1) {
                        const int u = pos[t] + step;
                        if (B[u - 1] < cand[t]) pos[t] = u;  // kNone from m on: pos <= m
                    }
                    if (adm[t] && ((B[pos[t]] ^ cand[t]) >> 1) == 0) adm[t] = false;
                    am[t] = __ballot_sync(kFull, adm[t]);
                    anyam |= am[t];
                }
            }
            if (anyam) {
                // rank among the admitted candidates (their ids are distinct):
                // the candidates are compacted into the stage, and every lane
                // counts the smaller ones with broadcast reads
                int nadm = 0;
#pragma unroll
                for (int t = 0; t < NR; ++t) {
                    if (adm[t]) stage[nadm + __popc(am[t] & ((1u << lane) - 1u))] = cand[t];
                    nadm += __popc(am[t]);
                }
                __syncwarp();
                int rank[NR];
#pragma unroll
                for (int t = 0; t < NR; ++t) rank[t] = 0;
                int j = 0;
#pragma unroll 1
                for (; j + 2 <= nadm; j += 2) {  // two staged candidates per 16-byte read
                    const ulonglong2 v = *reinterpret_cast<const ulonglong2 *>(stage + j);
#pragma unroll
                    for (int t = 0; t < NR; ++t) rank[t] += (v.x < cand[t] ? 1 : 0) + (v.y < cand[t] ? 1 : 0);
                }
                if (j < nadm) {
                    const uint64_t v = stage[j];
#pragma unroll
                    for (int t = 0; t < NR; ++t) rank[t] += v < cand[t] ? 1 : 0;
                }
                __syncwarp();
                int fp[NR];  // final positions in the merged beam
#pragma unroll
                for (int t = 0; t < NR; ++t) {
                    fp[t] = pos[t] + rank[t];
                    if (adm[t]) stage[rank[t]] = cand[t];
                    if constexpr (STOP) inserted += __popc(__ballot_sync(kFull, adm[t] && fp[t] < ef));
                }
                uint32_t mk[NB];  // bit l of mk[s]: a candidate lands in slot 32 s + l
#pragma unroll
                for (int s = 0; s < NB; ++s) {
                    uint32_t bits = 0;
#pragma unroll
                    for (int t = 0; t < NR; ++t) bits |= adm[t] && (fp[t] >> 5) == s ? 1u << (fp[t] & 31) : 0u;
                    mk[s] = __reduce_or_sync(kFull, bits);
                }
                const int m2 = min(ef, m + nadm);
                uint64_t *Bn = beam_b;
                __syncwarp();
                // output slot o: a candidate if bit o of the mask is set (the one
                // of rank = candidates placed before o), else old entry o - that count
                int cbase = 0;
#pragma unroll
                for (int s = 0; s < NB; ++s) {
                    const int o = lane + 32 * s;
                    const int c = cbase + __popc(mk[s] & ((1u << lane) - 1u));
                    const uint64_t v = o < m2 ? (((mk[s] >> lane) & 1u) ? stage[c] : B[o - c]) : kNone;
                    Bn[o] = v;
                    b[s] = v;
                    cbase += __popc(mk[s]);
                }
                beam_b = beam_a;
                beam_a = Bn;
                m = m2;
                // (a visited mark set below does not matter to the early cut: no
                // candidate shares an id with a visited entry)
                bworst = m == ef ? shfl64(pick<NB>(b, (ef - 1) >> 5), (ef - 1) & 31) : kNone;
            }

            // ---- learned early stop (not in the paper): after the merge, on
            // the merged beam, before the next vertex is marked -- the point
            // where search_kernel takes it
            if constexpr (STOP) {
                constexpr float inv_R = 1.0f / (32 * NR);  // a power of 2: exact, the division's value
                if (lane == 0) {
                    if (improved) sst->last_improve = hops;
                    sst->ema_improve =
                        __fadd_rn(__fmul_rn(0.75f, sst->ema_improve), __fmul_rn(0.25f, improved ? 1.0f : 0.0f));
                    sst->ema_insert =
                        __fadd_rn(__fmul_rn(0.75f, sst->ema_insert), __fmul_rn(0.25f, __fmul_rn((float)inserted, inv_R)));
                }
                // hops mod the period by a multiply-high with the host's
                // 2^64 / period + 1, exact for every hops < 2^32
                const uint64_t hq = __umul64hi((uint64_t)hops, a.stop_magic);
                const bool eval_now = a.stop_every == 1 || (uint64_t)hops == hq * (uint64_t)a.stop_every;
                if (a.stop_every > 0 && eval_now && rworst != kNone) {
                    // lane 0's stop state is visible to every lane after this, and
                    // the gather's reads of both beam buffers and the stage are done
                    __syncwarp();
                    const float rk = __uint_as_float((uint32_t)(rworst >> 32));
                    const float rk2 = __fmul_rn(1.25f, rk);
                    int u = 0, near1 = 0, near2 = 0;  // unvisited; of them with key <= rk, <= 1.25 rk
#pragma unroll
                    for (int s = 0; s < NB; ++s) {
                        const bool un = !(b[s] & 1ull);  // kNone reads as visited
                        const float kk = un ? entry_key(b[s]) : 0.0f;
                        u += __popc(__ballot_sync(kFull, un));
                        near1 += __popc(__ballot_sync(kFull, un && kk <= rk));
                        near2 += __popc(__ballot_sync(kFull, un && kk <= rk2));
                    }
                    const float den = rk > 1e-20f ? rk : 1e-20f;
                    const float since = (float)(hops - sst->last_improve);
                    const float inv_ef = __fdiv_rn(1.0f, (float)ef), inv_den = __fdiv_rn(1.0f, den);
                    const float inv_k = __fdiv_rn(1.0f, (float)k);
                    const float inv_h1 = __fdiv_rn(1.0f, __fadd_rn((float)hops, 1.0f));
                    const float r0 = __uint_as_float((uint32_t)(shfl64(res[0], 0) >> 32));
                    // d <= 256 (builds at their register limit): the features go to
                    // the beam buffer the next merge writes (idle until then), each
                    // as soon as it is known, so that few registers hold them;
                    // larger d: registers.  The stage holds the hidden layer.
                    constexpr bool kFeatSmem = CH <= 2;
                    float *const fs = reinterpret_cast<float *>(beam_b);
                    float f[SQG_MLP_IN];
                    auto put = [&](int i, float v) {
                        if constexpr (kFeatSmem) {
                            if (lane == 0) fs[i] = clamp8(v);
                        } else {
                            f[i] = clamp8(v);
                        }
                    };
                    put(0, __fmul_rn((float)hops, inv_ef));
                    put(1, __fmul_rn(since, inv_ef));
                    put(2, __fmul_rn((float)u, inv_ef));
                    put(3, __fmul_rn((float)m, inv_ef));
                    put(4, __fmul_rn(r0, inv_den));
                    put(5, u > 0 ? __fmul_rn(entry_key(nxt), inv_den) : 0.0f);  // nxt: the first unvisited entry
                    put(6, __fmul_rn(dist_c, inv_den));
                    put(7, __fmul_rn((float)inserted, inv_R));
                    put(8, __fmul_rn((float)k, inv_ef));
                    put(9, sst->ema_improve);
                    put(10, sst->ema_insert);
                    put(11, __fmul_rn((float)near1, inv_k));
                    put(12, __fmul_rn((float)near2, inv_k));
                    put(13, __fmul_rn(since, inv_h1));
                    put(14, dist_c <= rk ? 1.0f : 0.0f);
                    put(15, __fmul_rn((float)k, 0.01f));
                    __syncwarp();
                    float logit;
                    if constexpr (kFeatSmem)
                        logit = mlp_logit_warp(a.mlp, static_cast<const float *>(fs), lane, reinterpret_cast<float *>(stage));
                    else
                        logit = mlp_logit_warp(a.mlp, f, lane, reinterpret_cast<float *>(stage));
                    if (logit > a.stop_logit) {
                        status |= SQG_STATUS_LEARNED_STOP;
                        if (go) {  // the copy issued for the next vertex completes unused
                            if (mbar_wait_bounded(&bar[0], phase & 1u)) {
                                phase ^= 1u;
                            } else {
                                status |= SQG_STATUS_TIMEOUT;
                                healthy = false;
                            }
                        }
                        break;
                    }
                }
                if (nxt == kNone) break;  // no unvisited entry: the search ends (line 2)
                if (hops >= hop_cap) {    // reading R6
                    status |= SQG_STATUS_CAPACITY;
                    break;
                }
            }

            // ---- line 3: the next vertex is visited; every copy of it in the
            // beam is marked (reading R5: the copies keep their slots)
            p = pn;
#pragma unroll
            for (int s = 0; s < NB; ++s)
                if ((uint32_t)b[s] == p << 1) {  // id p, not yet visited (ids < 2^31)
                    b[s] |= 1ull;
                    beam_a[lane + 32 * s] = b[s];
                }
            hash_insert_warp(H, hbits, p, lane);  // its closing __syncwarp also orders the marks above
            ++hops;
            if (__builtin_expect(Hg && H == Hs && (uint32_t)hops >= (1u << hbits) / 2, 0)) {
                hash_migrate<32>(Hs, hbits, Hg, a.hash_bits, tm);
                H = Hg;
                hbits = a.hash_bits;
            }
        }
        // ---- line 8: the k nearest expanded vertices by exact distance
        const bool ok = !(status & SQG_STATUS_TIMEOUT);
        if constexpr (kLog) nl = log_select(rlog, nl, k, lane);
#pragma unroll
        for (int s = 0; s < RK; ++s) {
            const int j = lane + 32 * s;
            if (j < k) {
                if constexpr (kLog) res[s] = j < nl ? rlog[j] : kNone;
                const bool have = ok && res[s] != kNone;
                a.out_ids[off + j] = have ? (uint32_t)res[s] : SQG_NO_ID;
                a.out_dists[off + j] = have ? __uint_as_float((uint32_t)(res[s] >> 32)) : __int_as_float(0x7f800000);
            }
        }
        if (lane == 0) {
            if (a.stats) a.stats[qi] = sqg_query_stats{(uint32_t)hops, status};
            if (status) atomicOr(a.status_word, status);
        }
        __syncwarp();
    }
}

template <int CH, int NR, int NB, int MINB, bool STOP = false, int RK = 1, bool ADD = false>
static cudaError_t compact_launch_one(dim3 grid, dim3 block, size_t smem, cudaStream_t s, const SearchArgs &a) {
    auto fn = search_compact_kernel<CH, NR, NB, MINB, STOP, RK, ADD>;
    cudaError_t e = allow_dynamic_smem(fn);
    if (e != cudaSuccess) return e;
    fn<<<grid, block, smem, s>>>(a);
    return cudaGetLastError();
}

template <int CH, int NR, int NB, int MINB, bool STOP = false, int RK = 1, bool ADD = false>
static cudaError_t compact_occ_one(int block, size_t smem, int *nb) {
    auto fn = search_compact_kernel<CH, NR, NB, MINB, STOP, RK, ADD>;
    cudaError_t e = allow_dynamic_smem(fn);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(nb, fn, block, smem);
}

}  // namespace sqg
