// search_deep.cuh -- the deep-beam search kernel: one warp per query for
// beams past the compact kernel's range (search_compact.cuh) and for d >
// 1024: any ef up to SQG_MAX_EF, k <= 128, out-degree 32 or 64, d <= 2048,
// with multiple estimates; it can record the expansion order (the candidate
// search of index construction).  No learned stop and no feature trace.
//
// It runs the same Algorithm 1 with the same decisions as the other two
// kernels.  Merging an expansion's candidates into a sorted beam of several
// hundred entries costs passes over the whole beam at every expansion, which
// is where the general kernel spends its instructions (1,100 per expansion
// at ef 400, d = 128).  Here the beam is kept in two levels:
//
//   * the front: at most 32 NB entries (64 with out-degree 32, 128 with 64),
//     sorted, merged at every expansion exactly as the compact kernel's beam
//     (packed 64-bit entries, gathered merge, entries lane + 32 s in
//     registers);
//   * the main part: up to ef sorted entries in shared memory, into which
//     the front is merged only when it has no room for an expansion's
//     candidates.
//
// The beam of Algorithm 1 is the ef smallest entries of main part and front
// together.  What the search takes from it is its smallest unvisited entry,
// and whether there is one:
//
//   * 32 entries of the main part from its first unvisited entry on (the
//     window) sit in registers with their visited marks, so the smallest
//     unvisited entry is one warp minimum over candidates, front and window;
//     a copy of an expanded vertex outside the window is recognised by the
//     visited set when the window reaches it;
//   * an entry belongs to the beam if fewer than ef entries are smaller.
//     All entries smaller than the smallest unvisited one are visited; when
//     their number (an upper bound: an entry may be in both parts) reaches
//     ef, the parts are merged, duplicates dropped and the cut taken, and
//     the choice is made on the result.  An entry that Algorithm 1 cut
//     earlier has ef smaller entries for ever after, so cutting late drops
//     the same entries.
//
// A query with ef <= 32 NB needs no main part: its front is its beam, cut to
// ef at every merge.
//
// Measured (16,384 candidate searches of d 128 at ef 400, k 64, with the
// path): 5.29 ms with the general kernel, 2.60 ms here, 1,140 and 700
// warp-instructions per expansion; bound by issue (2.86 of 4 instructions per
// cycle, 26 warps per SM).  At d 1536 it is bound by the latency of one
// expansion (IPC 1.1, 9 warps per SM): the longest queries end the launch.
// Main parts in the workspace instead of shared memory raise the resident
// warps (9 to 12 at d 1536, ef 800) but lengthen every merge's binary search:
// 1-3 % slower up to ef 400, 7-14 % faster at ef 800 on batches of one ef, 6 %
// slower on the mixed batch, so they stay in shared memory.
#pragma once
#include "search_compact.cuh"

namespace sqg {

namespace deep {

using compact::kNone;

__device__ __forceinline__ uint64_t warp_min64(uint64_t v) {
    const uint32_t hi = __reduce_min_sync(kFull, (uint32_t)(v >> 32));
    const uint32_t lo = __reduce_min_sync(kFull, (uint32_t)(v >> 32) == hi ? (uint32_t)v : 0xFFFFFFFFu);
    return ((uint64_t)hi << 32) | lo;
}

}  // namespace deep

// CH: float4 chunks of the raw vector per lane (d <= 128 CH).  NR:
// neighbours per lane (out-degree 32 NR).  RK: result slots per lane (1: k <=
// 32, 4: k <= 128).  MINB: resident blocks of 4 warps per SM the build is
// made for.
template <int CH, int NR, int RK, int MINB>
__global__ void __launch_bounds__(128, MINB) search_deep_kernel(const SearchArgs a) {
    using namespace compact;
    using deep::warp_min64;
    constexpr int NB = 2 * NR, kFront = 32 * NB;
    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t below = (1u << lane) - 1u;
    const uint32_t d = a.d, nch = d / 4;
    unsigned char *ws = smem + (size_t)warp * a.warp_bytes;
    unsigned char *const buf = ws + a.o_buf0;
    uint64_t *const bar = reinterpret_cast<uint64_t *>(ws + a.o_bar);
    uint64_t *front_a = reinterpret_cast<uint64_t *>(ws + a.o_beam);  // two buffers of kFront entries
    uint64_t *front_b = front_a + kFront;
    uint64_t *const stage = reinterpret_cast<uint64_t *>(ws + a.o_spos);
    uint32_t *const planes = reinterpret_cast<uint32_t *>(ws + a.o_planes);
    const uint32_t gwarp = blockIdx.x * (blockDim.x >> 5) + warp;
    uint64_t *const M = reinterpret_cast<uint64_t *>(ws + a.o_res);  // the main part, max_ef entries
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
        const bool shallow = ef <= kFront;  // the front is the whole beam
        const int front_cap = shallow ? ef : kFront;

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
            for (uint32_t w = lane; w < d / 32; w += 32) reinterpret_cast<uint4 *>(planes)[w] = src[w];
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
        int mf = 1;  // entries in the front
        int m = 0;   // entries in the main part
        int wbase = 0;           // the window holds main entries wbase + lane
        uint64_t win = kNone;
        uint64_t b[NB];  // b[s] = front[lane + 32 s]
#pragma unroll
        for (int s = 0; s < NB; ++s) {
            b[s] = s == 0 && lane == 0 ? pack_entry(0u, a.entry) | 1ull : kNone;
            front_a[lane + 32 * s] = b[s];
        }
        uint64_t res[RK];  // res[s] = result[lane + 32 s], for lane + 32 s < k
#pragma unroll
        for (int s = 0; s < RK; ++s) res[s] = kNone;
        uint64_t rworst = kNone;  // result[k - 1]: the entry a new result must beat
        uint64_t bworst = kNone;  // an entry that ef entries are known not to exceed (the early cut)
        uint32_t p = a.entry;
        __syncwarp();
        hash_insert_warp(H, hbits, p, lane);
        if (lane == 0) {
            fence_proxy_async();
            bulk_fetch(buf, a.blocks + (size_t)p * a.block_bytes, a.block_bytes, &bar[0]);
            if (a.path) a.path[(size_t)qi * a.path_cap] = p;
        }
        int hops = 1;

        // the window from main entry wbase on, moved to the first 32 entries
        // with an unvisited one among them (or the last ones)
        auto load_window = [&]() {
            for (;;) {
                const int i = wbase + lane;
                uint64_t e = i < m ? M[i] : kNone;
                if (!(e & 1ull) && hash_contains(H, hbits, entry_id(e))) e |= 1ull;
                win = e;
                if (__ballot_sync(kFull, !(e & 1ull)) || wbase + 32 >= m) return;
                wbase += 32;
            }
        };

        for (;;) {
            if (!mbar_wait_bounded(&bar[0], phase & 1u)) {
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
            exact_and_S<CH, NR, false>(qv, blk, a.off_codes, planes, nch, d / 32, lane, dacc, S);
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
            uint32_t am[NR];
            int nadm = 0;
#pragma unroll
            for (int t = 0; t < NR; ++t) {
                const float key = est_key<32 * NR>(part[t], reinterpret_cast<const float *>(blk + a.off_factors),
                                                   lane + 32 * t, dist_c, a.eps0);
                cand[t] = pack_entry(key_bits(key), cid[t]);
            }
            if (hops == 1) {  // reading R8: the entry's key is its exact distance
                if (lane == 0) {
                    b[0] = pack_entry(key_bits(dist_c), p) | 1ull;
                    front_a[0] = b[0];
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
                nadm += __popc(am[t]);
            }

            // ---- lines 2-3 of the next step: the smallest unvisited entry of
            // candidates, front and window
            uint64_t v = win & 1ull ? kNone : win;
#pragma unroll
            for (int t = 0; t < NR; ++t) v = adm[t] && cand[t] < v ? cand[t] : v;
#pragma unroll
            for (int s = 0; s < NB; ++s) v = !(b[s] & 1ull) && b[s] < v ? b[s] : v;  // kNone: visited
            uint64_t nxt = warp_min64(v);
            bool late = false;  // nxt may be past the cut: choose after a full merge
            if (!shallow && nxt != kNone && wbase + 32 + mf >= ef) {
                int smaller = wbase + __popc(__ballot_sync(kFull, win < nxt));
#pragma unroll
                for (int s = 0; s < NB; ++s) smaller += __popc(__ballot_sync(kFull, b[s] < nxt));
                late = smaller >= ef;
            }
            __syncwarp();  // every lane's reads of the current block are done
            if (nxt != kNone && !late && hops < hop_cap && lane == 0) {
                fence_proxy_async();
                bulk_fetch(buf, a.blocks + (size_t)entry_id(nxt) * a.block_bytes, a.block_bytes, &bar[0]);
            }
            {  // result top-k in registers: (dist bits << 32) | id, dist >= 0
                const uint64_t r = ((uint64_t)__float_as_uint(dist_c) << 32) | p;
                if (r < rworst) {
                    int pos = 0;
#pragma unroll
                    for (int s = 0; s < RK; ++s) pos += __popc(__ballot_sync(kFull, lane + 32 * s < k && res[s] < r));
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
            if (nxt == kNone) break;  // no unvisited entry: the search ends (line 2)
            if (!late && hops >= hop_cap) {  // reading R6
                status |= SQG_STATUS_CAPACITY;
                break;
            }

            // ---- line 6: step 0 merges the candidates into the front (the
            // front into the main part before, if they do not fit); step 1, on
            // a late choice, merges the front into the main part
#pragma unroll 1
            for (int step = 0; step < 2; ++step) {
                if (step == 0 ? !shallow && mf + nadm > kFront : late) {
                    // positions in the main part; an identical (key, id) there
                    // already is dropped
                    int pos[NB], fp[NB];
                    bool keep[NB];
#pragma unroll
                    for (int s = 0; s < NB; ++s) pos[s] = 0;
                    for (int st = m > 0 ? 1 << (31 - __clz(m)) : 0; st >= 1; st >>= 1) {
#pragma unroll
                        for (int s = 0; s < NB; ++s) {
                            const int u = pos[s] + st;
                            if (u <= m && M[u - 1] < (b[s] & ~1ull)) pos[s] = u;
                        }
                    }
                    int nkeep = 0, nin = 0, first = 0x7fffffff, first_un = 0x7fffffff;
#pragma unroll
                    for (int s = 0; s < NB; ++s) {
                        keep[s] = b[s] != kNone && !(pos[s] < m && ((M[pos[s]] ^ b[s]) >> 1) == 0);
                        const uint32_t kb = __ballot_sync(kFull, keep[s]);
                        fp[s] = pos[s] + nkeep + __popc(kb & below);  // final position in the merged main part
                        nkeep += __popc(kb);
                        const bool in = keep[s] && fp[s] < ef;
                        if (in) front_b[fp[s] - pos[s]] = b[s];  // by rank
                        nin += __popc(__ballot_sync(kFull, in));
                        if (in && fp[s] < first) first = fp[s];
                        if (in && !(b[s] & 1ull) && fp[s] < first_un) first_un = fp[s];
                    }
                    first = __reduce_min_sync(kFull, first);
                    first_un = __reduce_min_sync(kFull, first_un);
                    const uint32_t wun = __ballot_sync(kFull, !(win & 1ull));
                    if (wun) {  // the window's first unvisited entry, moved up by the front's smaller ones
                        const int l0 = __ffs(wun) - 1;
                        const uint64_t wf = shfl64(win, l0);
                        int at = wbase + l0;
#pragma unroll
                        for (int s = 0; s < NB; ++s) at += __popc(__ballot_sync(kFull, keep[s] && b[s] < wf));
                        first_un = min(first_un, at);
                    }
                    // a bit per main slot that a front entry takes; slot o then
                    // holds front entry c or old entry o - c, c the set bits
                    // below o.  In place from the top: a row reads slots up to
                    // its own only.
                    uint32_t *const mw = reinterpret_cast<uint32_t *>(stage);
                    for (int i = lane; i < (ef + 31) / 32; i += 32) mw[i] = 0u;
                    __syncwarp();
#pragma unroll
                    for (int s = 0; s < NB; ++s)
                        if (keep[s] && fp[s] < ef) atomicOr(&mw[fp[s] >> 5], 1u << (fp[s] & 31));
                    const int m2 = min(ef, m + nkeep);
                    __syncwarp();
                    if (nin > 0) {
                        int cb = nin;
                        for (int r = (m2 - 1) >> 5; r >= first >> 5; --r) {
                            const uint32_t w = mw[r];
                            cb -= __popc(w);
                            const int o = 32 * r + lane, c = cb + __popc(w & below);
                            uint64_t e = 0;
                            if (o < m2) e = (w >> lane) & 1u ? front_b[c] : M[o - c];
                            __syncwarp();
                            if (o < m2) M[o] = e;
                        }
                        __syncwarp();
                    }
                    m = m2;
                    mf = 0;
#pragma unroll
                    for (int s = 0; s < NB; ++s) {
                        b[s] = kNone;
                        front_a[lane + 32 * s] = kNone;
                    }
                    if (m == ef) bworst = M[ef - 1];
                    wbase = min(first_un, m);
                    load_window();
                    __syncwarp();
                    if (step == 0) {  // the cut may have come down below some candidates
                        nadm = 0;
#pragma unroll
                        for (int t = 0; t < NR; ++t) {
                            adm[t] = adm[t] && cand[t] < bworst;
                            am[t] = __ballot_sync(kFull, adm[t]);
                            nadm += __popc(am[t]);
                        }
                    }
                }
                if (step == 0 && nadm > 0) {
                    // the compact kernel's merge: front position by a branch-free
                    // binary search (an identical (key, id) is dropped), rank
                    // among the admitted candidates, gather
                    const uint64_t *B = front_a;
                    int pos[NR];
                    nadm = 0;
#pragma unroll
                    for (int t = 0; t < NR; ++t) {
                        pos[t] = 0;
#pragma unroll
                        for (int st = 16 * NB; st >= 1; st >>= 1) {
                            const int u = pos[t] + st;
                            if (B[u - 1] < cand[t]) pos[t] = u;  // kNone from mf on: pos <= mf
                        }
                        if (adm[t] && ((B[pos[t]] ^ cand[t]) >> 1) == 0) adm[t] = false;
                        am[t] = __ballot_sync(kFull, adm[t]);
                        if (adm[t]) stage[nadm + __popc(am[t] & below)] = cand[t];
                        nadm += __popc(am[t]);
                    }
                    __syncwarp();
                    int rank[NR];
#pragma unroll
                    for (int t = 0; t < NR; ++t) rank[t] = 0;
                    int j = 0;
#pragma unroll 2
                    for (; j + 2 <= nadm; j += 2) {  // two staged candidates per 16-byte read
                        const ulonglong2 w = *reinterpret_cast<const ulonglong2 *>(stage + j);
#pragma unroll
                        for (int t = 0; t < NR; ++t) rank[t] += (w.x < cand[t] ? 1 : 0) + (w.y < cand[t] ? 1 : 0);
                    }
                    if (j < nadm) {
                        const uint64_t w = stage[j];
#pragma unroll
                        for (int t = 0; t < NR; ++t) rank[t] += w < cand[t] ? 1 : 0;
                    }
                    __syncwarp();
                    int fp[NR];
#pragma unroll
                    for (int t = 0; t < NR; ++t) {
                        fp[t] = pos[t] + rank[t];
                        if (adm[t]) stage[rank[t]] = cand[t];
                    }
                    uint32_t mk[NB];  // bit l of mk[s]: a candidate lands in slot 32 s + l
#pragma unroll
                    for (int s = 0; s < NB; ++s) {
                        uint32_t bits = 0;
#pragma unroll
                        for (int t = 0; t < NR; ++t) bits |= adm[t] && (fp[t] >> 5) == s ? 1u << (fp[t] & 31) : 0u;
                        mk[s] = __reduce_or_sync(kFull, bits);
                    }
                    const int mf2 = min(front_cap, mf + nadm);
                    uint64_t *Bn = front_b;
                    __syncwarp();
                    int cbase = 0;
#pragma unroll
                    for (int s = 0; s < NB; ++s) {
                        const int o = lane + 32 * s;
                        const int c = cbase + __popc(mk[s] & below);
                        const uint64_t e = o < mf2 ? (((mk[s] >> lane) & 1u) ? stage[c] : B[o - c]) : kNone;
                        Bn[o] = e;
                        b[s] = e;
                        cbase += __popc(mk[s]);
                    }
                    front_b = front_a;
                    front_a = Bn;
                    mf = mf2;
                    if (shallow) bworst = mf == ef ? shfl64(pick<NB>(b, (ef - 1) >> 5), (ef - 1) & 31) : kNone;
                    __syncwarp();
                }
                if (!late) break;
            }
            if (late) {  // the main part is the beam now: its first unvisited entry, if any
                const uint32_t wun = __ballot_sync(kFull, !(win & 1ull));
                if (!wun) break;  // line 2
                nxt = shfl64(win, __ffs(wun) - 1);
                if (hops >= hop_cap) {  // reading R6
                    status |= SQG_STATUS_CAPACITY;
                    break;
                }
                if (lane == 0) {
                    fence_proxy_async();
                    bulk_fetch(buf, a.blocks + (size_t)entry_id(nxt) * a.block_bytes, a.block_bytes, &bar[0]);
                }
            }

            // ---- line 3: the next vertex is visited; its copies in front and
            // window are marked (reading R5: the copies keep their slots), those
            // elsewhere in the main part when the window reaches them
            p = entry_id(nxt);
#pragma unroll
            for (int s = 0; s < NB; ++s)
                if ((uint32_t)b[s] == p << 1) {
                    b[s] |= 1ull;
                    front_a[lane + 32 * s] = b[s];
                }
            if ((uint32_t)win == p << 1) win |= 1ull;
            hash_insert_warp(H, hbits, p, lane);  // its closing __syncwarp also orders the marks above
            if (a.path && hops < a.path_cap && lane == 0) a.path[(size_t)qi * a.path_cap + hops] = p;
            ++hops;
            if (Hg && H == Hs && (uint32_t)hops >= (1u << hbits) / 2) {
                hash_migrate<32>(Hs, hbits, Hg, a.hash_bits, tm);
                H = Hg;
                hbits = a.hash_bits;
            }
            if (wbase + 32 < m && !__ballot_sync(kFull, !(win & 1ull))) {
                wbase += 32;
                load_window();
            }
        }
        // ---- line 8: the k nearest expanded vertices by exact distance
        const bool ok = !(status & SQG_STATUS_TIMEOUT);
#pragma unroll
        for (int s = 0; s < RK; ++s) {
            const int j = lane + 32 * s;
            if (j < k) {
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

template <int CH, int NR, int RK, int MINB>
static cudaError_t deep_launch_one(dim3 grid, dim3 block, size_t smem, cudaStream_t s, const SearchArgs &a) {
    auto fn = search_deep_kernel<CH, NR, RK, MINB>;
    cudaError_t e = allow_dynamic_smem(fn);
    if (e != cudaSuccess) return e;
    fn<<<grid, block, smem, s>>>(a);
    return cudaGetLastError();
}

template <int CH, int NR, int RK, int MINB>
static cudaError_t deep_occ_one(int block, size_t smem, int *nb) {
    auto fn = search_deep_kernel<CH, NR, RK, MINB>;
    cudaError_t e = allow_dynamic_smem(fn);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(nb, fn, block, smem);
}

}  // namespace sqg
