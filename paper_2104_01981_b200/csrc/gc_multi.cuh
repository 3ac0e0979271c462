// Exact top-k of MANY tensors (layer-wise plans) in one cooperative launch.
//
// The scheme of the one-tensor kernel, applied per tensor: sample -> bracket [tau, tau_hi) and a
// guess tau_z of the threshold -> fold + candidates + band histogram -> band bin of the k-th
// key -> short list ranked by every CTA that needs it -> index-ordered emission; four grid
// barriers.  What differs:
//   * CTA b owns a contiguous run of tiles, so it sees one to a few tensors ("segments") and
//     keeps one small record per segment in shared memory;
//   * all histograms and short lists exist once per tensor in global memory; a CTA only looks
//     at those of its own segments;
//   * the sample is a coarse histogram (top 11 key bits) per tensor plus the kept sampled keys;
//     after the first barrier ONE CTA per tensor computes the bracket (short samples, see
//     kRefineTiles: the kept keys give tau and tau_z a second radix level; long ones: tau is a
//     bin edge and tau_z interpolated inside its bin -- it is only a guess; tau_hi always is a
//     bin edge) and publishes it, so the fold pass of the many CTAs that share a tensor
//     only reads three words per segment;
//   * the slot of a segment's first entry = what the tensor's earlier tiles send: the sum of
//     their published counts + the sent short-list entries that lie before the segment;
//   * tensors that fit one tile ("small") are finished by one CTA each between the arrival at
//     and the wait on the barrier behind the fold, by the CTAs that arrive there first;
//   * a tensor whose bracket missed, or whose band bin holds more than kMultiMidCap candidates,
//     is flagged and redone by the exact multi-pass kernels at the end (the others are not);
//     if a CTA's candidate region overflows, everything is redone.
#pragma once
#include "gc_single.cuh"

namespace gc {

constexpr uint32_t kMultiMidCap = 4u * kMidFast; // short list per tensor (the first kMidFast entries stay in registers)
constexpr uint32_t kSegWords = 16;               // shared-memory words per segment record
constexpr uint32_t kRefineTiles = 32;            // samples of up to this many sample tiles are ranked a second time
// Short lists up to kWarpMid entries are settled by one warp (a CTA with many segments has eight at a time), up
// to kRankMid by the whole CTA, every entry against all others; longer ones by radix select.  A warp alone
// takes 4 us for 100 entries and radix select 3 us or more, and the CTAs of large tensors came that much
// later: 161 tensors of 25.6M elements at 0.1 % 100 -> 91 us, a dozen of 30M at 0.4 % 125 -> 113, 199 of 110M at 1 % 286 -> 279.
// (direct ranking up to 512 entries instead of 128: 110M in 199 tensors at 5 % 324.5 / 316.7, the dozen 111.8 / 109.3.)
constexpr uint32_t kWarpMid = 32;
constexpr uint32_t kRankMid = 128;

// Contiguous runs of tiles: CTAs below c1 take n1 tiles each, those from there below c2 take n2, the others share
// the rest evenly.  The CTAs launched last are the youngest on their SMs and advance the slowest
// (the oldest get the most issue slots).
struct RunMap {
    uint32_t c1, n1, c2, n2;
    __host__ __device__ __forceinline__ uint32_t begin(uint32_t b, uint32_t G, uint32_t ntiles) const {
        const uint32_t s1 = c1 * n1, s2 = s1 + (c2 - c1) * n2;
        const uint32_t at = b <= c1 ? b * n1 : b <= c2 ? s1 + (b - c1) * n2 : s2;
        if (b <= c2 || at >= ntiles) return at < ntiles ? at : ntiles;
        return s2 + (uint32_t)(((unsigned long long)(b - c2) * (ntiles - s2)) / (G - c2));
    }
};

struct MultiArgs {
    const TensorDesc* desc;
    uint32_t T, ntiles, nstiles;
    uint32_t per;                    // tiles per CTA (contiguous run), at most
    RunMap runs;                     // which tiles are CTA b's
    uint32_t pool_cap;               // candidate slots per CTA
    uint32_t pool_smem_words;        // words of shared memory reserved for one bit per candidate slot
    uint32_t ntab;                   // T if the tile tables fit in shared memory, else 0
    // threshold mode (see topk_multi_body): `desc` holds the bracket's sample and, as k, the rank in the definition's; the
    // table with the definition's sample stands in front of it (desc - T) and has so many sample tiles
    uint32_t nstiles_def;
    const uint32_t* small_ids;       // the tensors that fit one tile, the tiny ones (one warp each) first
    uint32_t n_small, n_tiny;
    const uint32_t* reg_ids;         // the tensors that are not small (and not empty)
    uint32_t n_reg;
    TensorSel* brk;                  // [T] bracket of every such tensor: .prefix = tau, .krem = tau_z, .T = shift
    const void* g;                   // fp32 or bf16, see the kernel's template argument
    float* r;
    uint32_t* out_idx;
    float* out_val;
    uint32_t* out_count;
    uint2* cand;                     // [gridDim.x * pool_cap]
    uint2* mid;                      // [T][kMultiMidCap] candidates inside the band bin of the threshold
    uint32_t* mid_n;                 // [T] their number (zeroed)
    uint32_t* shist;                 // [n_reg][kHistBins] coarse sample histogram (zeroed)
    uint32_t* bhist;                 // [n_reg][kHistBins] band histogram (zeroed)
    uint32_t* tile_cnt;              // [ntiles] candidates above the band bin, per tile
    uint4* skeys;                    // [nstiles * kBlock] the sampled keys, one group of four per entry
    WsView ws, gws;
    CleanArgs cl;                    // the control block is left clean for the next launch (early section: shist)
};

// segment record (one per tensor a CTA's tile run touches), kSegWords words in shared memory
enum : uint32_t {
    SG_T = 0, SG_TILE0, SG_NTILE, SG_BASE0, SG_BEGIN, SG_TAU, SG_TAUZ, SG_SHIFT,
    SG_A, SG_ABOVE, SG_M, SG_TKEY, SG_CUT, SG_OK, SG_OUT, SG_K,
    SG_END = SG_CUT                  // threshold mode: end of the tensor's slots (there is no tie cut)
};

// First half of a barrier; returns this CTA's place in the order of arrival (0 = first).
__device__ __forceinline__ uint32_t grid_arrive(WsHeader* hdr, uint32_t passed, uint32_t* s_place, uint32_t G) {
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        *s_place = atomicAdd(&hdr->barrier, 1u) - passed * G;
    }
    __syncthreads();
    return *s_place;
}
// second half of a barrier whose arrival was signalled with grid_arrive
__device__ __forceinline__ bool grid_wait(WsHeader* hdr, uint32_t& passed, int* s_ok, uint32_t G) {
    if (threadIdx.x == 0) {
        int ok = 1;
        const uint32_t target = (passed + 1u) * G;
        uint32_t spins = 0;
        while (ld_cg(&hdr->barrier) < target) {
            if (++spins > kSpinLimit || ((spins & 15u) == 0u && ld_cg(&hdr->abort) != 0u)) { ok = 0; break; }
            if (spins > 32) __nanosleep(spins > 4096 ? 400 : 60);
        }
        if (!ok) {
            record_status(hdr, -5 /*GC_E_TIMEOUT*/, 0xB0000000ull + passed);
            atomicExch(&hdr->abort, 1u);
        }
        __threadfence();
        *s_ok = ok;
    }
    __syncthreads();
    ++passed;
    return *s_ok != 0;
}
__device__ __forceinline__ bool grid_wait(WsHeader* hdr, uint32_t& passed, int* s_ok) {
    return grid_wait(hdr, passed, s_ok, gridDim.x);
}

// A segment, chunks [c0, c1), that does not fit the CTA's region gives its candidates back to the residual and its room to
// the next one (`used` = where it began), and its tensor is flagged.  The whole CTA calls.  (Out of line: rare, and its registers were
// spilled in the fold.)
static __device__ __noinline__ void give_back_segment(uint32_t* rec, uint32_t c0, uint32_t c1, const uint2* pool, float* r, uint32_t* s_used,
                                                      uint32_t used, uint32_t* flags, WsHeader* hdr) {
    for (uint32_t c = c0 + threadIdx.x; c < c1; c += kBlock) {
        const uint32_t rc = rec[c];
        for (uint32_t j = 0; j < (rc & 1023u); ++j) {
            const uint2 pr = pool[(rc >> 10) + j];
            r[pr.x] = __uint_as_float(pr.y);
        }
        rec[c] = 0u;
    }
    if (threadIdx.x == 0) {
        *s_used = used;
        if ((atomicOr(flags, kSelFailed) & kSelFailed) == 0u) atomicAdd(&hdr->n_failed, 1u);
    }
    __syncthreads();
}
// (gc_thr_multi.cuh)
static __device__ void tiny_threshold_warp(const TensorDesc& d, uint32_t t, uint32_t T, const float* __restrict__ g, float* __restrict__ r,
                                           uint32_t* __restrict__ out_idx, float* __restrict__ out_val, uint32_t* __restrict__ out_count,
                                           WsHeader* hdr, int lane);
static __device__ void small_threshold_body(BlockSmem& sm, const TensorDesc& d, uint32_t t, uint32_t T, const float* __restrict__ g,
                                            float* __restrict__ r, uint32_t* __restrict__ out_idx, float* __restrict__ out_val,
                                            uint32_t* __restrict__ out_count, WsHeader* hdr);

// Threshold mode, behind the counts: exact threshold, first slot and counts of every segment.  The wanted rank is one
// among the sampled entries of the short list, of which there are a handful: a warp per segment takes them
// from the top, one distinct key at a time; lists beyond kThrWarpMid entries take the block-wide radix select.  The CTA
// that holds a tensor's first tile totals its hits.
constexpr uint32_t kThrWarpMid = 256;
template <typename F>
__device__ __forceinline__ void thr_slots(const MultiArgs& a, uint32_t* seg, uint32_t nseg, uint32_t* rec2, uint32_t first, BlockSmem& sm,
                                          uint32_t& s_cnt, WsHeader* hdr, F chunk_of) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (uint32_t q = tid; q < nseg; q += kBlock) {
        uint32_t* s = seg + (size_t)q * kSegWords;
        s[SG_M] = ld_cg(a.mid_n + s[SG_T]);
        if (s[SG_M] > kMultiMidCap) s[SG_OK] = 0u;               // (flagged by the thread that came too late for the list)
    }
    __syncthreads();
    for (uint32_t sidx = (uint32_t)warp; sidx < nseg; sidx += kWarps) {
        uint32_t* s = seg + (size_t)sidx * kSegWords;
        const uint32_t m = s[SG_M];
        if (s[SG_OK] == 0u || m > kThrWarpMid) continue;
        const uint32_t t = s[SG_T];
        const TensorDesc d = a.desc[t];
        const InSample in{d.off, d.stride};
        const uint2* mid = a.mid + (size_t)t * kMultiMidCap;
        uint2 e[kThrWarpMid / 32];
        uint32_t sampled = 0;                                // one bit per own entry
#pragma unroll
        for (uint32_t u = 0; u < kThrWarpMid / 32; ++u) {
            e[u] = u * 32u + lane < m ? ld_cg(mid + u * 32u + lane) : make_uint2(0u, 0u);
            sampled |= u * 32u + lane < m && in(e[u].x) ? 1u << u : 0u;
        }
        const uint32_t nbefore = first + s[SG_TILE0] - d.tile0;
        uint32_t before = 0;
        for (uint32_t q = lane; q < nbefore; q += 32u) before += ld_cg(a.tile_cnt + d.tile0 + q);
        uint32_t left = s[SG_K] - s[SG_ABOVE], below = 0x80000000u, T = 0xFFFFFFFFu;
        while (true) {
            uint32_t best = 0, same = 0;                     // largest sampled key below the last one, plus 1
#pragma unroll
            for (uint32_t u = 0; u < kThrWarpMid / 32; ++u) {
                const uint32_t key = e[u].y & kKeyMask;
                if (((sampled >> u) & 1u) && key < below) best = max(best, key + 1u);
            }
            best = __reduce_max_sync(0xFFFFFFFFu, best);
            if (best == 0u) break;                           // (the list holds at least that many, unless it changed under us)
            below = best - 1u;
#pragma unroll
            for (uint32_t u = 0; u < kThrWarpMid / 32; ++u) same += ((sampled >> u) & 1u) && (e[u].y & kKeyMask) == below ? 1u : 0u;
            same = __reduce_add_sync(0xFFFFFFFFu, same);
            if (left <= same) { T = below; break; }
            left -= same;
        }
        const uint32_t seg_end = s[SG_BASE0] + s[SG_NTILE] * (uint32_t)kTile;
#pragma unroll
        for (uint32_t u = 0; u < kThrWarpMid / 32; ++u) {
            if (u * 32u + lane >= m || (e[u].y & kKeyMask) < T) continue;
            if (e[u].x < s[SG_BEGIN]) ++before;
            else if (e[u].x < seg_end) atomicAdd(&rec2[chunk_of(s, e[u].x)], 1u);
        }
        before = __reduce_add_sync(0xFFFFFFFFu, before);
        __syncwarp();
        if (lane == 0) {
            s[SG_TKEY] = T; s[SG_OUT] = d.out_off + before;
            if (T == 0xFFFFFFFFu) { s[SG_OK] = 0u; record_status(hdr, -1 /*GC_E_INVALID*/, 0xE0000000ull + t); }
        }
    }
    __syncthreads();
    for (uint32_t sidx = 0; sidx < nseg; ++sidx) {           // long lists: the whole CTA, one segment after the other
        uint32_t* s = seg + (size_t)sidx * kSegWords;
        const uint32_t m = s[SG_M];
        if (s[SG_OK] == 0u || m <= kThrWarpMid) continue;
        const uint32_t t = s[SG_T];
        const TensorDesc d = a.desc[t];
        const InSample in{d.off, d.stride};
        const uint2* mid = a.mid + (size_t)t * kMultiMidCap;
        uint2 e[kMidRegs];
#pragma unroll
        for (uint32_t u = 0; u < kMidRegs; ++u) e[u] = u * kBlock + tid < m ? ld_cg(mid + u * kBlock + tid) : make_uint2(0u, 0u);
        const uint32_t nbefore = first + s[SG_TILE0] - d.tile0;
        uint32_t before = 0;
        for (uint32_t q = tid; q < nbefore; q += kBlock) before += ld_cg(a.tile_cnt + d.tile0 + q);
        if (tid == 0) s_cnt = 0u;
        const uint32_t shift = s[SG_SHIFT], A = s[SG_A], binlo = s[SG_TAU] + (A << shift);
        uint32_t v, x0, x1;
        const bool good = short_list_select(sm, e, mid, m, A == 2047u ? 31 : max((int)shift, 1), s[SG_K] - s[SG_ABOVE],
                                            [&](const uint2& pr, uint32_t& w) { w = (pr.y & kKeyMask) - binlo; return in(pr.x); }, v, x0, x1);
        const uint32_t T = good ? binlo + v : 0xFFFFFFFFu, seg_end = s[SG_BASE0] + s[SG_NTILE] * (uint32_t)kTile;
        auto settle = [&](const uint2& pr) {
            if ((pr.y & kKeyMask) < T) return;
            if (pr.x < s[SG_BEGIN]) ++before;
            else if (pr.x < seg_end) atomicAdd(&rec2[chunk_of(s, pr.x)], 1u);
        };
#pragma unroll
        for (uint32_t u = 0; u < kMidRegs; ++u)
            if (u * kBlock + tid < m) settle(e[u]);
        for (uint32_t i = kMidFast + tid; i < m; i += kBlock) settle(ld_cg(mid + i));
        __syncthreads();
        before = __reduce_add_sync(0xFFFFFFFFu, before);
        if (lane == 0 && before) atomicAdd(&s_cnt, before);
        __syncthreads();
        if (tid == 0) {
            s[SG_TKEY] = T; s[SG_OUT] = d.out_off + s_cnt;
            if (!good) { s[SG_OK] = 0u; record_status(hdr, -1 /*GC_E_INVALID*/, 0xE0000000ull + t); }
        }
        __syncthreads();
    }
    for (uint32_t sidx = (uint32_t)warp; sidx < nseg; sidx += kWarps) {
        const uint32_t* s = seg + (size_t)sidx * kSegWords;
        const uint32_t t = s[SG_T], m = s[SG_M], T = s[SG_TKEY];
        if (first + s[SG_TILE0] != a.desc[t].tile0 || s[SG_OK] == 0u) continue;
        const TensorDesc d = a.desc[t];
        uint32_t hits = 0;
        for (uint32_t q0 = 0; q0 < d.ntiles; q0 += 256u) {
#pragma unroll
            for (uint32_t u = 0; u < 8; ++u) hits += q0 + u * 32u + lane < d.ntiles ? ld_cg(a.tile_cnt + d.tile0 + q0 + u * 32u + lane) : 0u;
        }
        for (uint32_t q = lane; q < m; q += 32u) hits += (ld_cg(a.mid + (size_t)t * kMultiMidCap + q).y & kKeyMask) >= T ? 1u : 0u;
        hits = __reduce_add_sync(0xFFFFFFFFu, hits);
        if (lane == 0) {
            if (a.out_count != nullptr) { a.out_count[t] = min(hits, d.cap); a.out_count[a.T + t] = hits; }
            if (hits > d.cap) record_status(hdr, 1 /*GC_W_TRUNCATED*/, t);
        }
    }
}

// The whole compress of one worker by the G CTAs of one group (this CTA is number b of them);
// the group's barriers count on the worker's own workspace header.
// (DENSE, VOTES: see k_topk_single)
// THR: threshold mode.  The threshold is the k_s-th largest key of the sample that the definition fixes, one group of
// four elements per `stride` groups, and reading those before the fold costs what as many scattered accesses cost.
// Here they are picked out of the stream instead: the bracket comes from a sample of 128-byte lines as in top-k mode, the
// band histogram counts the candidates that are in the definition's sample, the band bin of rank k_s and the short list
// (all candidates in it) give the exact threshold, and every candidate at or above it is a hit, up to the capacity.
// A tensor that fails (bracket missed, list full, no room in a region) is redone from the residual by radix levels over
// the definition's sample and the look-back emission (199 tensors of 110M elements rounded to bfloat16, a list of ties too
// long in the largest: 1036 us with all of them redone, 658 with that one; first calls on gradients with a log-normal scale of
// spread 0.4 per channel, where the sample of a layer or two sees so small entries that a region fills: eight 161-tensor workers at
// 0.1 % 696 -> 570 us, 0.5 % 994 -> 640, 199 tensors 926 -> 487).  Eight 161-tensor workers: sample and thresholds 95 -> 26 us, call
// with the decode 532 -> 494.
template <typename GL, bool DENSE, bool VOTES, bool THR = false>
__device__ __forceinline__ void topk_multi_body(const MultiArgs& a, const uint32_t G, const uint32_t b, BlockSmem& sm,
                                                uint32_t& s_used, uint32_t& s_cnt, unsigned char* s_dyn) {
    uint32_t* const rec = reinterpret_cast<uint32_t*>(s_dyn);                  // [per*kWarps] off<<10 | cnt
    uint32_t* const rec2 = rec + (size_t)a.per * kWarps;                       // [per*kWarps] counts, later slots
    uint32_t* const seg = rec2 + (size_t)a.per * kWarps;                       // [per][kSegWords]
    uint32_t* const sent_bits = seg + (size_t)a.per * kSegWords;               // [ceil(pool_cap / 32)]
    uint32_t* const tab_tile0 = sent_bits + (a.pool_smem_words);               // [ntab] first tile of every tensor
    uint32_t* const tab_stile0 = tab_tile0 + a.ntab;                           // [ntab] first sample tile
    uint2* const pool = a.cand + (size_t)b * a.pool_cap;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    WsHeader* hdr = a.ws.hdr;
    uint32_t passed = 0, n_stamp = 0;
    ClearWait cleared;
    if (!clean_begin(a.cl, hdr, G, b, tid, cleared)) return;
    const uint32_t first = a.runs.begin(b, G, a.ntiles), last = a.runs.begin(b + 1u, G, a.ntiles);
    const uint32_t ntl = last - first;                                         // own tiles
    for (int i = tid; i < 2048; i += kBlock) sm.hist[i] = 0u;
    for (uint32_t i = tid; i < ntl * kWarps; i += kBlock) { rec[i] = 0u; rec2[i] = 0u; }
    if (tid == 0) { s_used = 0u; s_cnt = 0u; }
    // first tile / first sample tile of every tensor, so that "which tensor owns this tile" is a
    // binary search in shared memory instead of a chain of dependent global loads
    for (uint32_t t = tid; t < a.ntab; t += kBlock) {
        tab_tile0[t] = a.desc[t].tile0;
        tab_stile0[t] = a.desc[t].stile0;
    }
    phase_stamp(hdr, n_stamp, b);
    __syncthreads();
    auto owner = [&](const uint32_t* tab, uint32_t tile) -> uint32_t {    // last t with tab[t] <= tile
        uint32_t lo = 0, hi = a.ntab;
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) >> 1;
            if (tab[mid] <= tile) lo = mid; else hi = mid;
        }
        return lo;
    };

    // ---------------------------------------------------------------- sample: coarse histogram per tensor
    if (a.nstiles) {
        const uint32_t sper = (a.nstiles + G - 1) / G;
        const uint32_t sfirst = min(a.nstiles, b * sper), slast = min(a.nstiles, sfirst + sper);
        uint32_t t = 0xFFFFFFFFu;
        TensorDesc d;
        for (uint32_t st = sfirst; st < slast;) {
            if (t == 0xFFFFFFFFu || st >= d.stile0 + d.nstiles) {
                if (t != 0xFFFFFFFFu) { cleared(); flush_hist(sm, a.shist + (size_t)d.reg * kHistBins, 1 << level_bits(0)); }
                __syncthreads();
                t = a.ntab ? owner(tab_stile0, st) : find_tensor<SampleSpace>(a.desc, a.T, st);
                d = a.desc[t];
            }
            // up to kSampleBatch sample tiles of this tensor at once: all their loads are in flight
            // together, so a CTA that owns several sample tiles (a group of CTAs that serves one of
            // several workers) pays one round trip for the batch instead of one per tile.  The counts are plain
            // shared-memory adds: aggregated over the warp first they were the phase's longest part (eight
            // 161-tensor workers 29 us against 14, one worker 10 against 7)
            constexpr uint32_t kSampleBatch = 4;
            const uint32_t nb = min(kSampleBatch, min(slast, d.stile0 + d.nstiles) - st);
            const uint32_t ngroups = (d.n + 3u) >> 2;
            const BracketSample def(d.n, d.stride, d.sstride);             // (threshold mode)
            const uint32_t nsg = THR ? def.count() : (ngroups + d.sstride - 1) / d.sstride;
            const bool vec_ok = (d.off & 3u) == 0u;           // the tensor's groups are 16-byte aligned in the flat buffers
            float gv[kSampleBatch][4], rv[kSampleBatch][4];
            uint32_t i0[kSampleBatch];
            bool live[kSampleBatch];
#pragma unroll
            for (uint32_t u = 0; u < kSampleBatch; ++u) {
                const uint64_t sg = (uint64_t)(st + u - d.stile0) * kBlock + tid;
                const uint64_t gi = THR ? def.group((uint32_t)sg, d.stride) : sample_group(sg, d.sstride);
                live[u] = u < nb && sg < nsg && gi < ngroups;
                i0[u] = live[u] ? (uint32_t)gi * 4u : 0u;
                if (vec_ok && live[u] && i0[u] + 3u < d.n) {
                    // the whole group in one 16-byte load each (a quarter of the load instructions and
                    // of the sectors the L1 has to look up: the groups lie `sstride` x 16 bytes apart)
                    const float4 g4 = GL::ld4(a.g, d.off + i0[u]);
                    const float4 r4 = ld_cg(reinterpret_cast<const float4*>(a.r + d.off + i0[u]));
                    gv[u][0] = g4.x; gv[u][1] = g4.y; gv[u][2] = g4.z; gv[u][3] = g4.w;
                    rv[u][0] = r4.x; rv[u][1] = r4.y; rv[u][2] = r4.z; rv[u][3] = r4.w;
                } else {
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const bool v = live[u] && i0[u] + e < d.n;
                        const uint32_t f = d.off + (v ? i0[u] + e : 0u);
                        gv[u][e] = v ? GL::ld1(a.g, f) : 0.f;
                        rv[u][e] = v ? ld_cg(a.r + f) : 0.f;
                    }
                }
            }
#pragma unroll
            for (uint32_t u = 0; u < kSampleBatch; ++u) {
                if (u < nb) {                             // (uniform over the CTA)
                    uint32_t key[4] = {0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu};     // = not a sample
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        if (live[u] && i0[u] + e < d.n) key[e] = key_of(__fadd_rn(gv[u][e], rv[u][e]));
                        if (key[e] != 0xFFFFFFFFu) atomicAdd(&sm.hist[key[e] >> level_shift(0)], 1u);
                    }
                    // the keys are kept: the fold pass ranks them a second time, and by then the residual
                    // they were computed from has been overwritten
                    if (d.nstiles <= kRefineTiles)
                        a.skeys[(size_t)(st + u) * kBlock + tid] = make_uint4(key[0], key[1], key[2], key[3]);
                }
            }
            st += nb;
        }
        cleared();
        if (t != 0xFFFFFFFFu) flush_hist(sm, a.shist + (size_t)d.reg * kHistBins, 1 << level_bits(0));
    }
    cleared();
    if (!grid_barrier(hdr, passed, &sm.ok, G)) return;
    phase_stamp(hdr, n_stamp, b);
    clean_in_use(hdr, b, tid);

    // ---------------------------------------------------------------- bracket per tensor, one CTA each
    // tau = the srank-th largest sampled key (21 bits when the kept keys allow the second radix
    // level, else the lower edge of its coarse bin), tau_hi = upper edge of the bin of the key
    // that stays below the expected rank by the same margin, tau_z = the key of the expected rank
    // itself (21 bits, or a place inside its bin); published as (tau, tau_z, shift of the band histogram).
    for (uint32_t q = b; q < a.n_reg; q += G) {
        const uint32_t cur = a.reg_ids[q];
        const TensorDesc d = a.desc[cur];
        uint32_t tau = 0, tau_z = 0;
        int shift = 0;
        {
            uint32_t tau_hi = 0x80000000u;
            if (d.sstride != 0u) {
                const uint32_t ngroups = (d.n + 3u) >> 2;
                float ks, sd;                              // expected rank of the threshold in the sample, its noise
                if constexpr (THR) {                       // (k is a rank in the definition's sample, this one a part of it: see thr_bracket)
                    const BracketSample def(d.n, d.stride, d.sstride);
                    const float part = fminf(1.0f, (float)def.count() / (float)def.of);
                    ks = (float)d.k * part; sd = sqrtf(ks * (1.0f - part));
                } else {
                    ks = (float)d.k * (4.0f * (float)((ngroups + d.sstride - 1) / d.sstride)) / (float)d.n; sd = sqrtf(ks);
                }
                const float hi = floorf(ks - 6.0f * sd - 8.0f);
                // (a sample too small for that margin: the largest sampled key bounds the band instead)
                const uint32_t want[3] = {d.srank, hi >= 1.0f ? (uint32_t)hi : 1u, max(1u, (uint32_t)ceilf(ks))};
                Picked pk[3];
                block_select_multi<(1 << level_bits(0)), 3>(sm, a.shist + (size_t)d.reg * kHistBins, want, pk);
                if (pk[0].ok) tau = pk[0].bin << level_shift(0);
                if (pk[0].ok && d.nstiles <= kRefineTiles) {
                    // second radix level of the lower bracket and of the guess over the kept sample keys:
                    // tau and tau_z get 21 significant bits
                    const uint4* sk = a.skeys + (size_t)d.stile0 * kBlock;
                    const uint32_t nk = d.nstiles * kBlock, bin0 = pk[0].bin, bin2 = pk[2].ok ? pk[2].bin : bin0;
                    for (uint32_t q0 = tid; q0 < nk; q0 += 4 * kBlock) {
                        uint4 kv[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            kv[u] = q0 + u * kBlock < nk ? ld_cg(sk + q0 + u * kBlock)
                                                         : make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu);
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            const uint32_t kk[4] = {kv[u].x, kv[u].y, kv[u].z, kv[u].w};
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const uint32_t c = kk[e] >> level_shift(0);
                                if (c == bin0 || c == bin2)
                                    atomicAdd(&sm.hist[((kk[e] >> (level_shift(0) - 10)) & 1023u) + (c == bin0 ? 0u : 1024u)], 1u);
                            }
                        }
                    }
                    __syncthreads();
                    uint32_t bin1, above1, bin3, above3;
                    const bool ok1 = block_select<1024, true>(sm, sm.hist, d.srank - pk[0].above, bin1, above1);
                    const bool ok3 = pk[2].ok && block_select<1024, true>(sm, sm.hist + (bin2 == bin0 ? 0 : 1024),
                                                                          want[2] - pk[2].above, bin3, above3);
                    for (int i2 = tid; i2 < 2048; i2 += kBlock) sm.hist[i2] = 0u;
                    __syncthreads();
                    if (ok1) tau |= bin1 << (level_shift(0) - 10);
                    if (ok3) tau_z = (bin2 << level_shift(0)) | (bin3 << (level_shift(0) - 10));
                }
                if (pk[1].ok) tau_hi = (pk[1].bin + 1u) << level_shift(0);
                if (pk[2].ok && tau_z == 0u) {
                    const float pos = ((float)(want[2] - pk[2].above) - 0.5f) / (float)pk[2].count;   // from the top of the bin
                    tau_z = (pk[2].bin << level_shift(0)) +
                            (uint32_t)((1.0f - pos) * (float)((1u << level_shift(0)) - 1u));
                }
            }
            if (tau_z < tau) tau_z = tau;
            if (tau_hi <= tau) tau_hi = 0x80000000u;
            shift = 0;
            while (((tau_hi - tau) >> shift) > 2046u) ++shift;
        }
        if (tid == 0) { a.brk[cur].prefix = tau; a.brk[cur].krem = tau_z; a.brk[cur].T = (uint32_t)shift; }
    }
    if (!grid_barrier(hdr, passed, &sm.ok, G)) return;
    phase_stamp(hdr, n_stamp, b);
    clean_early(a.cl, G, b, tid);      // the sample histograms have had their last reader (the brackets)

    // ---------------------------------------------------------------- fold + candidates, segment by segment
    uint32_t nseg = 0;
    {
        const uint32_t my_off = warp * kWarpChunk + lane * 4;
        bool block_overflow = false, open = false;
        uint32_t cur = 0xFFFFFFFFu, tau = 0, tau_z = 0;
        int shift = 0;
        TensorDesc d;
        for (uint32_t tile = first; tile < last; ++tile) {
            const uint32_t i = tile - first;
            if (cur == 0xFFFFFFFFu || tile >= d.tile0 + d.ntiles) {
                // Threshold mode: the definition's sample may have met entries so small that many times k are hits.  A tensor that
                // does not fit is redone alone.  (In top-k mode the number of candidates is a matter of the rank, and a full region
                // has everything redone.)
                if constexpr (THR) {
                    if (open && __syncthreads_or(block_overflow ? 1 : 0)) {
                        const uint32_t* q = seg + (size_t)(nseg - 1u) * kSegWords;
                        give_back_segment(rec, q[SG_TILE0] * kWarps, i * kWarps, pool, a.r, &s_used, q[SG_ABOVE], &a.ws.sel[cur].flags, hdr);
                        block_overflow = false;
                    }
                }
                if (open) flush_hist(sm, a.bhist + (size_t)d.reg * kHistBins, 2048);
                open = false;
                cur = a.ntab ? owner(tab_tile0, tile) : find_tensor(a.desc, a.T, tile);
                d = a.desc[cur];
                if (d.kind != kKindSmall) {
                    // bracket of this tensor, published by the CTA that computed it
                    tau = ld_cg(&a.brk[cur].prefix);
                    tau_z = ld_cg(&a.brk[cur].krem);
                    shift = (int)ld_cg(&a.brk[cur].T);
                    if (tid == 0) {
                        uint32_t* s = seg + (size_t)nseg * kSegWords;
                        const TileGeom tg0 = tile_geom(d, tile - d.tile0);
                        s[SG_T] = cur; s[SG_TILE0] = i; s[SG_NTILE] = min(last, d.tile0 + d.ntiles) - tile;
                        s[SG_BASE0] = (d.off & ~3u) + (tile - d.tile0) * (uint32_t)kTile; s[SG_BEGIN] = tg0.lo;
                        s[SG_TAU] = tau; s[SG_TAUZ] = tau_z; s[SG_SHIFT] = (uint32_t)shift;
                        s[SG_OK] = 1u; s[SG_OUT] = d.out_off; s[SG_K] = d.k;
                        s[SG_A] = d.reg;               // (until the band bin is known)
                        if (THR) { s[SG_END] = d.out_off + d.cap; s[SG_ABOVE] = s_used; }      // (where its candidates begin)
                    }
                    if (THR) __syncthreads();              // (before anyone adds to s_used again)
                    ++nseg;
                    open = true;
                }
            }
            if (d.kind == kKindSmall) continue;          // finished by its own CTA
            const TileGeom tg = tile_geom(d, tile - d.tile0);
            const bool interior = tg.lo == tg.base && tg.hi == tg.base + (uint32_t)kTile;
            float av[kVpt][4];
            uint32_t valid = 0xFFFFu;
            if (interior) {
                float4 gv[kVpt], rv[kVpt];
#pragma unroll
                for (int j = 0; j < kVpt; ++j) {
                    gv[j] = GL::ld4(a.g, tg.base + my_off + j * 128);
                    rv[j] = ld_cg(reinterpret_cast<const float4*>(a.r + tg.base + my_off + j * 128));
                }
#pragma unroll
                for (int j = 0; j < kVpt; ++j) {
                    av[j][0] = __fadd_rn(gv[j].x, rv[j].x); av[j][1] = __fadd_rn(gv[j].y, rv[j].y);
                    av[j][2] = __fadd_rn(gv[j].z, rv[j].z); av[j][3] = __fadd_rn(gv[j].w, rv[j].w);
                }
            } else {
                valid = 0u;
#pragma unroll
                for (int j = 0; j < kVpt; ++j) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const uint32_t f = tg.base + my_off + j * 128 + e;
                        float v = 0.0f;
                        if (f >= tg.lo && f < tg.hi) {
                            v = __fadd_rn(GL::ld1(a.g, f), ld_cg(a.r + f));
                            valid |= 1u << (4 * j + e);
                        }
                        av[j][e] = v;
                    }
                }
            }
            if constexpr (VOTES) {
                if constexpr (THR)
                    block_overflow |= !fold_tail_votes(sm, av, interior, valid, tau, tau_z, shift, tg.base + my_off, a.r, s_used, a.pool_cap, pool,
                                                       rec[i * kWarps + warp], lane, warp, InSample{d.off, d.stride});
                else
                    block_overflow |= !fold_tail_votes(sm, av, interior, valid, tau, tau_z, shift, tg.base + my_off, a.r, s_used, a.pool_cap, pool,
                                                       rec[i * kWarps + warp], lane, warp);
            } else {
                uint32_t cnt[kVpt], cm = 0, hm = 0;      // candidates; candidates that are zeroed right away
#pragma unroll
                for (int j = 0; j < kVpt; ++j) {
                    cnt[j] = 0;
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const uint32_t key = key_of(av[j][e]);
                        bool c = key >= tau;
                        if (!interior) c = c && ((valid >> (4 * j + e)) & 1u);
                        cnt[j] += c;
                        cm |= (uint32_t)c << (4 * j + e);
                        if (!interior) hm |= (uint32_t)(key >= tau_z) << (4 * j + e);
                    }
                }
                uint32_t rk[kVpt], wtot;
                warp_rank(cnt, lane, rk, wtot);
                uint32_t off = 0;
                if (lane == 0 && wtot) off = atomicAdd(&s_used, wtot);
                off = __shfl_sync(0xFFFFFFFFu, off, 0);
                const bool fits = off + wtot <= a.pool_cap;
                if (!fits) block_overflow = true;
                if (lane == 0) rec[i * kWarps + warp] = fits ? ((off << 10) | wtot) : 0u;
                const uint32_t em = fits ? cm : 0u;             // goes to the candidate list
                const uint32_t zm = fits ? (hm & cm) : 0u;      // ... and leaves +0 in the residual (probably sent)
                if (interior) {
                    // +0 where the key reaches tau_z (implies a candidate: tau_z >= tau), a elsewhere; a chunk
                    // that did not fit keeps all its values (no key reaches 2^31)
                    const uint32_t tz = fits ? tau_z : 0x80000000u;
#pragma unroll
                    for (int j = 0; j < kVpt; ++j) {
                        float4 o;
                        o.x = key_of(av[j][0]) >= tz ? 0.0f : av[j][0];
                        o.y = key_of(av[j][1]) >= tz ? 0.0f : av[j][1];
                        o.z = key_of(av[j][2]) >= tz ? 0.0f : av[j][2];
                        o.w = key_of(av[j][3]) >= tz ? 0.0f : av[j][3];
                        __stcs(reinterpret_cast<float4*>(a.r + tg.base + my_off + j * 128), o);    // streaming: evict first
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < kVpt; ++j) {
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            if ((valid >> (4 * j + e)) & 1u)
                                a.r[tg.base + my_off + j * 128 + e] = ((zm >> (4 * j + e)) & 1u) ? 0.0f : av[j][e];
                        }
                    }
                }
                const bool staged = wtot <= (uint32_t)kEmitStage;
                if (fits && wtot != 0u) {
                    // one round per candidate of the lane that has the most, instead of sixteen predicated
                    // blocks that every warp walks through (see the one-tensor kernel)
                    for (uint32_t m = em; m != 0u; m &= m - 1u) {
                        const uint32_t bq = (uint32_t)__ffs((int)m) - 1u, j = bq >> 2;      // element 4 j + e of this thread
                        float s8[8], s4[4];                                                 // its value by a select tree
#pragma unroll
                        for (int q = 0; q < 8; ++q) s8[q] = (bq & 8u) ? av[2 + q / 4][q % 4] : av[q / 4][q % 4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) s4[q] = (bq & 4u) ? s8[4 + q] : s8[q];
                        const float s20 = (bq & 2u) ? s4[2] : s4[0], s21 = (bq & 2u) ? s4[3] : s4[1];
                        const float v = (bq & 1u) ? s21 : s20;
                        const uint32_t rkj = (bq & 8u) ? ((bq & 4u) ? rk[3] : rk[2]) : ((bq & 4u) ? rk[1] : rk[0]);
                        const uint32_t pos = rkj + (uint32_t)__popc(em & ((1u << bq) - 1u) & (0xFu << (4u * j)));
                        const uint2 pr = make_uint2(tg.base + my_off + j * 128u + (bq & 3u), __float_as_uint(v));
                        if (staged) sm.emit[warp][pos] = pr; else pool[off + pos] = pr;
                        if (THR ? !staged && InSample{d.off, d.stride}(pr.x) : true) atomicAdd(&sm.hist[min((key_of(v) - tau) >> shift, 2047u)], 1u);
                    }
                    if (staged) {
                        __syncwarp();
                        for (uint32_t q = lane; q < wtot; q += 32) {
                            const uint2 pr = sm.emit[warp][q];
                            pool[off + q] = pr;
                            if (THR && InSample{d.off, d.stride}(pr.x)) atomicAdd(&sm.hist[min(((pr.y & kKeyMask) - tau) >> shift, 2047u)], 1u);
                        }
                        __syncwarp();
                    }
                }
            }
        }
        if constexpr (THR) {
            if (open && __syncthreads_or(block_overflow ? 1 : 0)) {
                const uint32_t* q = seg + (size_t)(nseg - 1u) * kSegWords;
                give_back_segment(rec, q[SG_TILE0] * kWarps, ntl * kWarps, pool, a.r, &s_used, q[SG_ABOVE], &a.ws.sel[cur].flags, hdr);
                block_overflow = false;
            }
        }
        if (open) flush_hist(sm, a.bhist + (size_t)d.reg * kHistBins, 2048);
        if (__syncthreads_or(block_overflow ? 1 : 0)) {
            if (tid == 0) atomicExch(&hdr->overflow, 1u);
        }
        if (tid == 0) atomicAdd(&hdr->cand_total, min(s_used, a.pool_cap));
    }
    const uint32_t used = s_used;      // read linearly only when no chunk anywhere overflowed
    // Small tensors need nothing from anyone, and nobody needs them: the CTAs that are through with their fold
    // first take them, in the order of their arrival, while the others are still folding (the first and the
    // last arrive 15 to 40 us apart).  In front of the brackets, where the last CTAs of the grid took them, all
    // others waited for their 10-15 us: brackets of 110M elements in 199 tensors 18.3 -> 12.9 us, of eight 161-tensor
    // workers 19.4 -> 10.8.
    if (a.n_small != 0u) {
        const uint32_t tiny = (a.n_tiny + kWarps - 1u) / kWarps, units = tiny + a.n_small - a.n_tiny;
        for (uint32_t u = grid_arrive(hdr, passed, &sm.tile, G); u < units; u += G) {
            if (u < tiny) {                                  // tiny ones: a warp each, eight at a time
                const uint32_t q = u * kWarps + (uint32_t)warp;
                if (q < a.n_tiny) {
                    const uint32_t t = a.small_ids[q];
                    const TensorDesc d = a.desc[t];
                    if constexpr (THR) tiny_threshold_warp(d, t, a.T, (const float*)a.g, a.r, a.out_idx, a.out_val, a.out_count, hdr, lane);
                    else tiny_tensor_warp<GL>(d.off, d.n, d.k, d.out_off, t, a.T, a.g, a.r, a.out_idx, a.out_val, a.out_count, lane);
                }
                continue;
            }
            const uint32_t t = a.small_ids[a.n_tiny + u - tiny];
            const TensorDesc d = a.desc[t];
            if constexpr (THR) small_threshold_body(sm, d, t, a.T, (const float*)a.g, a.r, a.out_idx, a.out_val, a.out_count, hdr);
            else if (d.k <= kFewK) small_tensor_fewk<GL>(sm, d, t, a.T, a.g, a.r, a.out_idx, a.out_val, a.out_count);
            else small_tensor_body<GL>(sm, d, t, a.T, a.g, a.r, a.out_idx, a.out_val, a.out_count);
            __syncthreads();
            for (int i = tid; i < 2048; i += kBlock) sm.hist[i] = 0u;
        }
        if (!grid_wait(hdr, passed, &sm.ok, G)) return;
    } else if (!grid_barrier(hdr, passed, &sm.ok, G)) {
        return;
    }
    phase_stamp(hdr, n_stamp, b);

    // segment of a candidate: the last one that begins at or before its index.  A thread's next candidate is
    // nearly always in the segment of its last one, whose indices are [cur_lo, cur_lo + cur_len): what the passes need
    // of it stays in registers (110M elements in 199 tensors at 5 % 336 -> 326 us; read anew for every candidate before).
    uint32_t cur_lo = 0u, cur_len = 0u;
    auto seg_of = [&](uint32_t idx) -> uint32_t* {
        uint32_t s = nseg - 1u, end = 0xFFFFFFFFu;
        while (s > 0u && seg[(size_t)s * kSegWords + SG_BEGIN] > idx) { end = seg[(size_t)s * kSegWords + SG_BEGIN]; --s; }
        uint32_t* const p = seg + (size_t)s * kSegWords;
        cur_lo = p[SG_BEGIN]; cur_len = end - cur_lo;
        return p;
    };
    auto chunk_of = [&](const uint32_t* s, uint32_t idx) -> uint32_t {
        const uint32_t rel = idx - s[SG_BASE0];
        return s[SG_TILE0] * kWarps + (rel >> 9);
    };
    static_assert(kWarpChunk == 512 && kWarps * kWarpChunk == kTile, "chunks side by side");

    const bool overflowed = ld_cg(&hdr->overflow) != 0u, by_chunk = DENSE && used >= kChunkWalk * ntl * kWarps;
    if (!overflowed && nseg != 0u) {
        // ------------------------------------------------------------ band bin per segment, counts above it
        for (uint32_t sidx = (uint32_t)warp; sidx < nseg; sidx += kWarps) {      // a warp per segment, all at once
            uint32_t* s = seg + (size_t)sidx * kSegWords;
            const uint32_t t = s[SG_T];
            const uint32_t flags = THR ? ld_cg(&a.ws.sel[t].flags) : 0u;
            const Picked pa = warp_select_2048(a.bhist + (size_t)s[SG_A] * kHistBins, s[SG_K], lane);
            // (threshold mode counts the sampled ones only; some CTA may have had no room for the tensor)
            const bool ok = pa.ok && (THR ? (flags & kSelFailed) == 0u : pa.count <= kMultiMidCap);
            if (lane == 0) {
                s[SG_A] = pa.bin; s[SG_ABOVE] = pa.above; s[SG_M] = pa.count; s[SG_OK] = ok ? 1u : 0u;
                if (!ok) {          // every CTA that sees this tensor decides the same; count it once
                    const uint32_t old = atomicOr(&a.ws.sel[t].flags, kSelFailed);
                    if ((old & kSelFailed) == 0u) atomicAdd(&hdr->n_failed, 1u);
                }
            }
        }
        __syncthreads();
        uint32_t c_t = 0, c_tau = 0, c_shift = 0, c_A = 0, c_base0 = 0;
        uint32_t* c_rec = rec2;
        auto classify = [&](const uint2& pr) {
            if (pr.x - cur_lo >= cur_len) {
                const uint32_t* s = seg_of(pr.x);
                c_t = s[SG_T]; c_tau = s[SG_TAU]; c_shift = s[SG_SHIFT]; c_base0 = s[SG_BASE0]; c_rec = rec2 + s[SG_TILE0] * kWarps;
                c_A = s[SG_OK] != 0u ? s[SG_A] : 2048u;          // (a tensor that is redone: no bin reaches it)
            }
            const uint32_t bin = min(((pr.y & kKeyMask) - c_tau) >> c_shift, 2047u);
            if (bin < c_A) return;
            if (bin > c_A) {
                atomicAdd(&c_rec[(pr.x - c_base0) >> 9], 1u);
            } else {
                const uint32_t slot = atomicAdd(a.mid_n + c_t, 1u);
                if (slot < kMultiMidCap) a.mid[(size_t)c_t * kMultiMidCap + slot] = pr;
                else if (THR && slot == kMultiMidCap) {      // (one thread per tensor gets here)
                    atomicOr(&a.ws.sel[c_t].flags, kSelFailed);
                    atomicAdd(&hdr->n_failed, 1u);
                }
            }
        };
        for (uint32_t i0 = tid; i0 < used; i0 += 4 * kBlock) {      // four loads in flight per thread
            uint2 pr[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t i = i0 + u * kBlock;
                pr[u] = i < used ? pool[i] : make_uint2(0u, 0u);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (i0 + u * kBlock < used) classify(pr[u]);
        }
        __syncthreads();
        for (uint32_t i = tid; i < ntl; i += kBlock) {
            uint32_t tot = 0;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) tot += rec2[i * kWarps + w];
            a.tile_cnt[first + i] = tot;
        }
    }
    if (!grid_barrier(hdr, passed, &sm.ok, G)) return;
    phase_stamp(hdr, n_stamp, b);

    if (!overflowed) {
        if (nseg != 0u) {
            if constexpr (THR) {
                thr_slots(a, seg, nseg, rec2, first, sm, s_cnt, hdr, chunk_of);
            } else {
            // -------------------------------------------------------- threshold, tie cut and slots per segment
            // Short lists of up to kWarpMid entries (nearly all: a band bin holds a handful of
            // candidates) are settled by a warp each, all segments of the CTA at once and without a
            // block-wide barrier: every entry's place in the order (key descending, index ascending)
            // is counted directly against all others, which settles threshold and tie cut in one go.
            for (uint32_t sidx = (uint32_t)warp; sidx < nseg; sidx += kWarps) {
                uint32_t* s = seg + (size_t)sidx * kSegWords;
                const uint32_t m = s[SG_M];
                if (s[SG_OK] == 0u || m > kWarpMid) continue;
                const uint32_t t = s[SG_T];
                const TensorDesc d = a.desc[t];
                const uint2* mid = a.mid + (size_t)t * kMultiMidCap;
                uint2 e[kWarpMid / 32];
#pragma unroll
                for (uint32_t u = 0; u < kWarpMid / 32; ++u)
                    e[u] = u * 32u + lane < m ? ld_cg(mid + u * 32u + lane) : make_uint2(0xFFFFFFFFu, 0u);
                // candidates above the band bin in the tensor's tiles before this segment
                const uint32_t nbefore = first + s[SG_TILE0] - d.tile0;
                uint32_t part = 0;
                for (uint32_t q = lane; q < nbefore; q += 32u) part += ld_cg(a.tile_cnt + d.tile0 + q);
                part = __reduce_add_sync(0xFFFFFFFFu, part);
                const uint32_t krem = s[SG_K] - s[SG_ABOVE];             // entries of the short list that are sent (1 .. m)
                // place of every own entry: entries that come before it in the order
                uint32_t place[kWarpMid / 32];
#pragma unroll
                for (uint32_t u = 0; u < kWarpMid / 32; ++u) place[u] = 0u;
#pragma unroll
                for (uint32_t uo = 0; uo < kWarpMid / 32; ++uo) {
                    if (uo * 32u >= m) break;                            // (uniform)
                    const uint32_t lim = min(32u, m - uo * 32u);
                    for (uint32_t l = 0; l < lim; ++l) {
                        const uint32_t ox = __shfl_sync(0xFFFFFFFFu, e[uo].x, (int)l);
                        const uint32_t ok = __shfl_sync(0xFFFFFFFFu, e[uo].y, (int)l) & kKeyMask;
#pragma unroll
                        for (uint32_t u = 0; u < kWarpMid / 32; ++u) {
                            const uint32_t key = e[u].y & kKeyMask;
                            place[u] += (ok > key || (ok == key && ox < e[u].x)) ? 1u : 0u;
                        }
                    }
                }
                // the last entry that is sent gives the threshold key and the tie cut; sent entries before
                // the segment shift its first slot, inside it they join the count of their chunk
                const uint32_t seg_end = s[SG_BASE0] + s[SG_NTILE] * (uint32_t)kTile;
                uint32_t before = 0, tk = 0, cut = 0;
                bool have = false;
#pragma unroll
                for (uint32_t u = 0; u < kWarpMid / 32; ++u) {
                    if (u * 32u + lane >= m) continue;
                    if (place[u] == krem - 1u) { have = true; tk = e[u].y & kKeyMask; cut = e[u].x; }
                    if (place[u] < krem) {
                        if (e[u].x < s[SG_BEGIN]) ++before;
                        else if (e[u].x < seg_end) atomicAdd(&rec2[chunk_of(s, e[u].x)], 1u);
                    }
                }
                before = __reduce_add_sync(0xFFFFFFFFu, before);
                const unsigned who = __ballot_sync(0xFFFFFFFFu, have);
                const bool good = who != 0u;                             // (the list holds at least krem entries)
                const int src = good ? __ffs(who) - 1 : 0;
                tk = __shfl_sync(0xFFFFFFFFu, tk, src); cut = __shfl_sync(0xFFFFFFFFu, cut, src);
                __syncwarp();
                if (lane == 0) {
                    s[SG_TKEY] = tk; s[SG_CUT] = cut;
                    s[SG_OUT] = d.out_off + part + before;             // slot of the segment's first sent entry
                    if (!good) {        // cannot happen unless the list changed under us: report, send nothing
                        s[SG_OK] = 0u;
                        record_status(hdr, -1 /*GC_E_INVALID*/, 0xE0000000ull + t);
                    } else if (a.out_count != nullptr && first + s[SG_TILE0] == d.tile0) {
                        a.out_count[t] = d.k; a.out_count[a.T + t] = d.k;
                    }
                }
            }
            __syncthreads();
            // longer short lists: the whole CTA, one segment after the other
            for (uint32_t sidx = 0; sidx < nseg; ++sidx) {
                uint32_t* s = seg + (size_t)sidx * kSegWords;
                const uint32_t m = s[SG_M];
                if (s[SG_OK] == 0u || m <= kWarpMid || m > kRankMid) continue;
                const uint32_t t = s[SG_T];
                const TensorDesc d = a.desc[t];
                const uint2* mid = a.mid + (size_t)t * kMultiMidCap;
                uint2* const list = reinterpret_cast<uint2*>(sm.hist);
                static_assert(kRankMid <= 1024u, "the list fits in the histogram");
                for (uint32_t i = tid; i < m; i += kBlock) { const uint2 pr = ld_cg(mid + i); list[i] = make_uint2(pr.x, pr.y & kKeyMask); }
                // candidates above the band bin in the tensor's tiles before this segment
                const uint32_t nbefore = first + s[SG_TILE0] - d.tile0;
                uint32_t before = 0;
                for (uint32_t q = tid; q < nbefore; q += kBlock) before += ld_cg(a.tile_cnt + d.tile0 + q);
                if (tid == 0) { s_cnt = 0u; sm.scratch[2] = 0u; }
                __syncthreads();
                const uint32_t krem = s[SG_K] - s[SG_ABOVE];             // entries of the short list that are sent (1 .. m)
                const uint32_t seg_end = s[SG_BASE0] + s[SG_NTILE] * (uint32_t)kTile;
                for (uint32_t i = tid; i < m; i += kBlock) {
                    const uint2 mine = list[i];
                    uint32_t place = 0;                                  // entries in front: key descending, index ascending
#pragma unroll 4
                    for (uint32_t j = 0; j < m; ++j) {
                        const uint2 o = list[j];
                        place += (o.y > mine.y || (o.y == mine.y && o.x < mine.x)) ? 1u : 0u;
                    }
                    if (place == krem - 1u) { sm.scratch[0] = mine.y; sm.scratch[1] = mine.x; sm.scratch[2] = 1u; }
                    if (place < krem) {
                        if (mine.x < s[SG_BEGIN]) ++before;
                        else if (mine.x < seg_end) atomicAdd(&rec2[chunk_of(s, mine.x)], 1u);
                    }
                }
                before = __reduce_add_sync(0xFFFFFFFFu, before);
                if (lane == 0 && before) atomicAdd(&s_cnt, before);
                __syncthreads();
                if (tid == 0) {
                    s[SG_TKEY] = sm.scratch[0]; s[SG_CUT] = sm.scratch[1];
                    s[SG_OUT] = d.out_off + s_cnt;                     // slot of the segment's first sent entry
                    if (sm.scratch[2] == 0u) {  // cannot happen unless the list changed under us: report, send nothing
                        s[SG_OK] = 0u;
                        record_status(hdr, -1 /*GC_E_INVALID*/, 0xE0000000ull + t);
                    } else if (a.out_count != nullptr && first + s[SG_TILE0] == d.tile0) {
                        a.out_count[t] = d.k; a.out_count[a.T + t] = d.k;
                    }
                }
                for (uint32_t i = tid; i < 2u * m; i += kBlock) sm.hist[i] = 0u;
                __syncthreads();
            }
            // (radix select in shared memory)
            for (uint32_t sidx = 0; sidx < nseg; ++sidx) {
                uint32_t* s = seg + (size_t)sidx * kSegWords;
                if (s[SG_OK] == 0u || s[SG_M] <= kRankMid) continue;
                const uint32_t t = s[SG_T], m = s[SG_M];
                const TensorDesc d = a.desc[t];
                const uint2* mid = a.mid + (size_t)t * kMultiMidCap;
                uint2 e[kMidRegs];
#pragma unroll
                for (uint32_t u = 0; u < kMidRegs; ++u)
                    e[u] = u * kBlock + tid < m ? ld_cg(mid + u * kBlock + tid) : make_uint2(0u, 0u);
                // candidates above the band bin in the tensor's tiles before this segment
                const uint32_t nbefore = first + s[SG_TILE0] - d.tile0;
                uint32_t part = 0;
                for (uint32_t q = tid; q < nbefore; q += kBlock) part += ld_cg(a.tile_cnt + d.tile0 + q);
                part = __reduce_add_sync(0xFFFFFFFFu, part);
                if (tid == 0) s_cnt = 0u;
                __syncthreads();
                if (lane == 0 && part) atomicAdd(&s_cnt, part);
                const uint32_t shift = s[SG_SHIFT], A = s[SG_A];
                const uint32_t binlo = s[SG_TAU] + (A << shift);
                uint32_t v_sel, mid_gt, n_eq, idx_cut = 0xFFFFFFFFu;
                const uint32_t krem = s[SG_K] - s[SG_ABOVE];
                bool good = short_list_select(sm, e, mid, m, A == 2047u ? 31 : max((int)shift, 1), krem,
                                              [&](const uint2& pr, uint32_t& v) { v = (pr.y & kKeyMask) - binlo; return true; },
                                              v_sel, mid_gt, n_eq);
                const uint32_t Tkey = binlo + v_sel;
                const uint32_t m_eq = krem - mid_gt;
                if (good && n_eq > m_eq) {
                    uint32_t v_idx, x0, x1;
                    good = short_list_select(sm, e, mid, m, 32, m_eq,
                                             [&](const uint2& pr, uint32_t& v) { v = ~pr.x; return (pr.y & kKeyMask) == Tkey; },
                                             v_idx, x0, x1);
                    idx_cut = ~v_idx;
                }
                // sent short-list entries: before the segment they shift its first slot, inside it
                // they join the count of their chunk
                const uint32_t seg_end = s[SG_BASE0] + s[SG_NTILE] * (uint32_t)kTile;
                auto settle = [&](const uint2& pr) {
                    const uint32_t key = pr.y & kKeyMask;
                    if (!(key > Tkey || (key == Tkey && pr.x <= idx_cut))) return;
                    if (pr.x < s[SG_BEGIN]) atomicAdd(&s_cnt, 1u);
                    else if (pr.x < seg_end) atomicAdd(&rec2[chunk_of(s, pr.x)], 1u);
                };
#pragma unroll
                for (uint32_t u = 0; u < kMidRegs; ++u)
                    if (good && u * kBlock + tid < m) settle(e[u]);
                for (uint32_t i = kMidFast + tid; good && i < m; i += kBlock) settle(ld_cg(mid + i));
                __syncthreads();
                if (tid == 0) {
                    s[SG_TKEY] = Tkey; s[SG_CUT] = idx_cut;
                    s[SG_OUT] = d.out_off + s_cnt;                     // slot of the segment's first sent entry
                    if (!good) {        // cannot happen unless the list changed under us: report, send nothing
                        s[SG_OK] = 0u;
                        record_status(hdr, -1 /*GC_E_INVALID*/, 0xE0000000ull + t);
                    } else if (a.out_count != nullptr && first + s[SG_TILE0] == d.tile0) {
                        a.out_count[t] = d.k; a.out_count[a.T + t] = d.k;
                    }
                }
                __syncthreads();
            }
            }
            // rec2[c] = output slot of the first sent candidate of chunk c (one warp walks each segment)
            for (uint32_t sidx = warp; sidx < nseg; sidx += kWarps) {
                const uint32_t* s = seg + (size_t)sidx * kSegWords;
                if (s[SG_OK] == 0u) continue;
                uint32_t run = s[SG_OUT];
                const uint32_t c0 = s[SG_TILE0] * kWarps, nc = s[SG_NTILE] * kWarps;
                for (uint32_t q0 = 0; q0 < nc; q0 += 32) {
                    const uint32_t q = q0 + lane;
                    const uint32_t v = q < nc ? rec2[c0 + q] : 0u;
                    const uint32_t inc = warp_incl_scan(v, lane);
                    if (q < nc) rec2[c0 + q] = run + inc - v;
                    run += __shfl_sync(0xFFFFFFFFu, inc, 31);
                }
            }
            __syncthreads();
        }
        phase_stamp(hdr, n_stamp, b);
        // of the segment at hand: its threshold key (none is reached where the tensor is redone), tie cut, guess
        uint32_t c_T = 0xFFFFFFFFu, c_cut = 0, c_tauz = 0, c_base0 = 0, c_chunk0 = 0, c_last = 0;      // c_last: end of its slots (THR)
        auto enter = [&](const uint32_t* s) {
            c_T = s[SG_OK] != 0u ? s[SG_TKEY] : 0xFFFFFFFFu;
            c_cut = s[SG_CUT]; c_tauz = s[SG_TAUZ]; c_base0 = s[SG_BASE0]; c_chunk0 = s[SG_TILE0] * kWarps;
            if (THR) { c_last = s[SG_END]; c_cut = 0xFFFFFFFFu; }
        };
        auto sent_key = [&](const uint2& pr) {
            const uint32_t key = pr.y & kKeyMask;
            return key > c_T || (key == c_T && pr.x <= c_cut);
        };
        auto enter_at = [&](uint32_t idx) { if (idx - cur_lo >= cur_len) enter(seg_of(idx)); };
        cur_len = 0u;
        // sent flags of the CTA's candidates in list order, one bit each
        if (by_chunk) {                        // see for_chunks
            const uint32_t* s = seg;
            uint32_t c_end = 0u;                   // end of the segment's chunks
            for_chunks(rec, ntl * kWarps, pool, warp, lane, [&](uint32_t c, uint32_t off, uint32_t cnt, const uint2 (&p)[2]) {
                if (c >= c_end) {
                    while (c >= (s[SG_TILE0] + s[SG_NTILE]) * kWarps) s += kSegWords;
                    c_end = (s[SG_TILE0] + s[SG_NTILE]) * kWarps;
                    enter(s);
                }
                uint32_t slot = rec2[c];
                for (uint32_t q0 = 0; q0 < cnt; q0 += 32u) {
                    const bool in = q0 + lane < cnt;
                    const uint2 pr = q0 == 0u ? p[0] : q0 == 32u ? p[1] : in ? pool[off + q0 + lane] : make_uint2(0u, 0u);
                    bool sent = in && sent_key(pr);
                    const bool zeroed = (pr.y & kKeyMask) >= c_tauz;
                    const unsigned sb = __ballot_sync(0xFFFFFFFFu, sent);
                    if constexpr (THR) sent = sent && slot + (uint32_t)__popc(sb & ((1u << lane) - 1u)) < c_last;      // (beyond the capacity: stays in the residual)
                    if (in && sent != zeroed) a.r[pr.x] = sent ? 0.0f : __uint_as_float(pr.y);
                    if (sent) {
                        const uint32_t at = slot + (uint32_t)__popc(sb & ((1u << lane) - 1u));
                        __stcs(a.out_idx + at, pr.x);
                        __stcs(a.out_val + at, __uint_as_float(pr.y));
                    }
                    slot += (uint32_t)__popc(sb);
                }
            });
        }
        const uint32_t nwords = by_chunk ? 0u : (used + 31u) >> 5;
        for (uint32_t i0 = 0; i0 < nwords * 32u; i0 += 4 * kBlock) {      // four loads in flight per thread
            uint2 pr[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t i = i0 + u * kBlock + tid;
                pr[u] = i < used ? pool[i] : make_uint2(0u, 0u);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t i = i0 + u * kBlock + tid;
                if (i0 + u * kBlock + (tid & ~31) >= nwords * 32u) continue;          // whole warp past the end
                if (i < used) enter_at(pr[u].x);
                const unsigned sb = __ballot_sync(0xFFFFFFFFu, i < used && sent_key(pr[u]));
                if (lane == 0) sent_bits[i >> 5] = sb;
            }
        }
        __syncthreads();
        // emission: slot = first slot of the chunk + sent candidates before this one in the chunk
        for (uint32_t i0 = by_chunk ? used : tid; i0 < used; i0 += 4 * kBlock) {
            uint2 pr[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t i = i0 + u * kBlock;
                pr[u] = i < used ? pool[i] : make_uint2(0u, 0u);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t i = i0 + u * kBlock;
                if (i >= used) continue;
                enter_at(pr[u].x);
                // the fold pass left +0 in the residual iff the key reached tau_z
                const bool zeroed = (pr[u].y & kKeyMask) >= c_tauz;
                if (!sent_key(pr[u])) {          // also every candidate of a tensor that is redone
                    if (zeroed) a.r[pr[u].x] = __uint_as_float(pr[u].y);     // value goes back
                    continue;
                }
                if (!THR && !zeroed) a.r[pr[u].x] = 0.0f;
                const uint32_t c = c_chunk0 + ((pr[u].x - c_base0) >> 9);
                const uint32_t p0 = rec[c] >> 10;                  // first list position of the chunk
                uint32_t before;
                if ((p0 >> 5) == (i >> 5)) {
                    before = __popc((sent_bits[i >> 5] & ((1u << (i & 31u)) - 1u)) >> (p0 & 31u));
                } else {
                    before = __popc(sent_bits[p0 >> 5] >> (p0 & 31u)) + __popc(sent_bits[i >> 5] & ((1u << (i & 31u)) - 1u));
                    for (uint32_t w = (p0 >> 5) + 1u; w < (i >> 5); ++w) before += __popc(sent_bits[w]);
                }
                const uint32_t slot = rec2[c] + before;
                if (THR) {
                    const bool goes = slot < c_last;                 // (beyond the capacity: stays in the residual)
                    if (goes != zeroed) a.r[pr[u].x] = goes ? 0.0f : __uint_as_float(pr[u].y);
                    if (!goes) continue;
                }
                a.out_idx[slot] = pr[u].x;
                a.out_val[slot] = __uint_as_float(pr[u].y);
            }
        }
        __syncthreads();
        phase_stamp(hdr, n_stamp, b);
        exit_stamp(hdr);
        if (ld_cg(&hdr->n_failed) == 0u) { leave_clean(a.cl, hdr, G, tid); return; }
    } else {
        // a candidate region overflowed: every recorded candidate gets its value back
        for (uint32_t c = tid; c < ntl * kWarps; c += kBlock) {
            const uint32_t rc = rec[c], off = rc >> 10, cnt = rc & 1023u;
            for (uint32_t j = 0; j < cnt; ++j) {
                const uint2 pr = pool[off + j];
                a.r[pr.x] = __uint_as_float(pr.y);
            }
        }
    }

    // ---------------------------------------------------------------- exact redo (rare)
    // of the flagged tensors, or of all of them after an overflow: r holds a = g + r for them again
    clean_redo(a.cl, G, b, tid);
    if (!grid_barrier(hdr, passed, &sm.ok, G)) return;
    phase_stamp(hdr, n_stamp, b);
    if constexpr (THR) {
        const TensorDesc* const def = a.desc - a.T;
        hist_body<0, SRC_RSAMPLE>(sm, def, a.T, a.nstiles_def, nullptr, a.r, a.gws, G, b);
        if (!grid_barrier(hdr, passed, &sm.ok, G)) return;
        hist_body<1, SRC_RSAMPLE>(sm, def, a.T, a.nstiles_def, nullptr, a.r, a.gws, G, b);
        if (!grid_barrier(hdr, passed, &sm.ok, G)) return;
        hist_body<2, SRC_RSAMPLE>(sm, def, a.T, a.nstiles_def, nullptr, a.r, a.gws, G, b);
        if (!grid_barrier(hdr, passed, &sm.ok, G)) return;
        WsView ws = a.ws;
        ws.gate = a.ws.sel;
        threshold_emit_body<false, true>(def, a.T, a.ntiles, nullptr, a.r, a.out_idx, a.out_val, a.out_count, ws, a.gws.sel, 0u, 0);
        return;
    }
    hist_body<0, SRC_RESID>(sm, a.desc, a.T, a.ntiles, nullptr, a.r, a.gws, G, b);
    if (!grid_barrier(hdr, passed, &sm.ok, G)) return;
    hist_body<1, SRC_RESID>(sm, a.desc, a.T, a.ntiles, nullptr, a.r, a.gws, G, b);
    if (!grid_barrier(hdr, passed, &sm.ok, G)) return;
    hist_body<2, SRC_RESID>(sm, a.desc, a.T, a.ntiles, nullptr, a.r, a.gws, G, b);
    if (!grid_barrier(hdr, passed, &sm.ok, G)) return;
    compact_body(sm, a.desc, a.T, a.ntiles, a.r, a.out_idx, a.out_val, a.out_count, a.gws, 0);
    __syncthreads();
    leave_clean(a.cl, hdr, G, tid);
}

// Votes: 25.6M elements in 161 tensors at 0.1 % 99 -> 97 us, 110M in 199 at 1 % 302 -> 289 us.
template <typename GL, bool DENSE, bool VOTES, bool THR = false>
// (three CTAs per SM: 80 registers and no spills beat four at 64 registers, see k_topk_single)
static __global__ void __launch_bounds__(kBlock, 3)
k_topk_multi(const __grid_constant__ MultiArgs a) {
    __shared__ BlockSmem sm;
    __shared__ uint32_t s_used, s_cnt;
    extern __shared__ __align__(16) unsigned char s_dyn[];
    topk_multi_body<GL, DENSE, VOTES, THR>(a, gridDim.x, blockIdx.x, sm, s_used, s_cnt, s_dyn);
}

// Several workers' compress calls in ONE cooperative launch: the grid is cut into one group of
// CTAs per worker (CTA x serves worker x mod W as number x / W of its group, so every worker's
// CTAs are spread over all SMs), and each group runs the kernel above on its own gradient,
// residual, outputs and workspace.  Nothing is shared between the groups, not even a barrier:
// a group's phases wait only for that worker's CTAs, so while one worker's CTAs sit in a
// barrier the SMs stream another worker's tiles.
constexpr uint32_t kWorkersPerLaunch = 12;       // per-worker argument blocks travel as kernel parameters
struct WorkersArgs {
    uint32_t W, G;                               // workers in this launch, CTAs per worker
    MultiArgs per[kWorkersPerLaunch];
};
static_assert(sizeof(WorkersArgs) <= 4000, "kernel parameters stay below 4 KB");

// (The scan stays here: with votes eight 161-tensor workers at 0.1 % take 544 us instead of 532, decode included, four at 1 % 276
// instead of 266.)
template <typename GL, bool DENSE, bool THR = false>
static __global__ void __launch_bounds__(kBlock, 3)
k_topk_workers(const __grid_constant__ WorkersArgs wa) {
    __shared__ BlockSmem sm;
    __shared__ uint32_t s_used, s_cnt;
    __shared__ MultiArgs s_args;                  // this CTA's worker (dynamic indexing of the parameters happens once)
    extern __shared__ __align__(16) unsigned char s_dyn[];
    const uint32_t w = blockIdx.x % wa.W, b = blockIdx.x / wa.W;
    {
        const uint32_t* src = reinterpret_cast<const uint32_t*>(&wa.per[w]);
        uint32_t* dst = reinterpret_cast<uint32_t*>(&s_args);
        for (uint32_t i = threadIdx.x; i < sizeof(MultiArgs) / 4; i += kBlock) dst[i] = src[i];
    }
    __syncthreads();
    topk_multi_body<GL, DENSE, false, THR>(s_args, wa.G, b, sm, s_used, s_cnt, s_dyn);
}

}  // namespace gc
