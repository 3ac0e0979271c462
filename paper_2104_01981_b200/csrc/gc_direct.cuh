// Exact top-k of ONE small or medium tensor in one cooperative launch, straight radix select.
//
// Tensors of a few million elements are all latency: what counts is the number of grid-wide steps, not
// the bytes.  Here every CTA folds its contiguous share of the tensor once and keeps a = g + r in shared
// memory (or, beyond what fits, reads it back from L2), so the levels of the select cost a microsecond
// or two each: histogram of the top 11 key bits | grid barrier | histogram of the next 10 bits inside the
// bin of the k-th key | barrier | the few entries that share those 21 bits go to a list, the others above
// them are counted | barrier | every CTA takes the threshold key from the list and emits its share.  No
// sample, no candidate list, no capacity that data could overflow: if more entries share the 21 bits than
// the list takes, the last 10 bits get a global histogram and the shares are counted (one more barrier),
// and nothing is ever redone.  The scratch is 29 KB; on a private workspace the launch leaves it clean,
// otherwise it clears it itself.  Without a plan, six launches over the whole tensor took 55 us at 2.4M elements; this takes
// 26.7, and 16.4 us at 200,000.
#pragma once
#include <cstddef>

#include "gc_kernels.cuh"

namespace gc {

constexpr uint32_t kDirectList = 1024;           // entries sharing 21 key bits that travel as a list
constexpr uint32_t kDirectMaxG = 512;            // most CTAs

struct DirectScratch {                           // zero before a launch (see SELF), except `list` and `tot`
    WsHeader hdr;
    uint32_t hist0[2048], hist1[1024], hist2[1024];
    uint32_t list_n, pad[63];
    uint2 list[kDirectList];
    unsigned long long tot[kDirectMaxG];         // per CTA: entries that are sent for sure | ties << 32
};

struct DirectArgs {
    const void* g;                               // fp32 or bf16, see the kernel's template argument
    float* r;
    uint32_t n, k;
    uint32_t* out_idx;
    float* out_val;
    uint32_t* out_count;                         // [2] or null
    int32_t* status_out;                         // or null
    DirectScratch* s;
    unsigned long long mark;                     // what the header's mark reads after a launch that left the scratch clean
    uint32_t expect_clean;                       // the host relies on that mark (see CleanArgs)
};

// Grid barrier: release by the arrival, acquire by the poll (see grid_barrier for the bounded wait).
__device__ __forceinline__ bool direct_barrier(WsHeader* hdr, uint32_t& passed, int* s_ok) {
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        const uint32_t target = (passed + 1u) * gridDim.x;
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&hdr->barrier) : "memory");
        uint32_t spins = 0, v;
        while (true) {
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&hdr->barrier) : "memory");
            if (v >= target) break;
            if (++spins > kSpinLimit || ((spins & 15u) == 0u && ld_cg(&hdr->abort) != 0u)) { ok = 0; break; }
            if (spins > 64) __nanosleep(spins > 4096 ? 400 : 40);
        }
        if (!ok) {
            record_status(hdr, -5 /*GC_E_TIMEOUT*/, 0xB0000000ull + passed);
            atomicExch(&hdr->abort, 1u);
        }
        *s_ok = ok;
    }
    __syncthreads();
    ++passed;
    return *s_ok != 0;
}

struct DirectSmem {
    uint32_t hist[2048];
    uint32_t wsum[kWarps], wgt[kWarps], weq[kWarps];
    uint32_t bin, above, count;
    unsigned long long part[kWarps];
    uint32_t last;
    int ok;
};

// Rank `k` (1 = largest) in a histogram of NB bins: the bin, the count above it and in it.  Returns the number
// of entries in the histogram.
template <int NB, bool IN_SMEM = false>
__device__ __forceinline__ uint32_t direct_select(DirectSmem& sm, const uint32_t* hist, uint32_t k, int tid, int lane, int warp) {
    constexpr int PER = NB / kBlock;
    uint32_t c[PER], sum = 0;
#pragma unroll
    for (int q = 0; q < PER / 4; ++q) {
        const uint4 v = IN_SMEM ? reinterpret_cast<const uint4*>(hist + tid * PER)[q] : ld_cg(reinterpret_cast<const uint4*>(hist + tid * PER) + q);
        c[4 * q] = v.x; c[4 * q + 1] = v.y; c[4 * q + 2] = v.z; c[4 * q + 3] = v.w;
    }
#pragma unroll
    for (int q = 0; q < PER; ++q) sum += c[q];
    const uint32_t inc = warp_incl_scan(sum, lane);
    if (lane == 31) sm.wsum[warp] = inc;
    __syncthreads();
    uint32_t above = 0, total = 0;                         // entries in higher bins than this thread's, in all
#pragma unroll
    for (int w = 0; w < kWarps; ++w) { above += w >= warp ? sm.wsum[w] : 0u; total += sm.wsum[w]; }
    above -= inc;
#pragma unroll
    for (int q = PER - 1; q >= 0; --q) {
        if (above < k && k <= above + c[q]) { sm.bin = (uint32_t)(tid * PER + q); sm.above = above; sm.count = c[q]; }
        above += c[q];
    }
    __syncthreads();
    return total;
}

// RES: the share of a CTA stays in (dynamic) shared memory; otherwise it is read back from r.
// SELF: the launch clears the scratch itself, whatever is in it, and leaves it as it is.  A form of its own: with
// both in one, chosen by an argument, each paid for the other's code (us, in one / apart: workspace left clean 0.3M elements 17.3 /
// 16.6, 3.9M 36.8 / 35.6, 0.5M 18.5 / 18.5; cleared by the launch 0.5M 18.4 / 17.4, 3.9M 34.6 / 32.8).
template <typename GL, bool RES, bool SELF>
static __global__ void __launch_bounds__(kBlock, 3)
k_topk_direct(const __grid_constant__ DirectArgs a) {
    __shared__ DirectSmem sm;
    extern __shared__ __align__(16) float4 s_share[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t G = gridDim.x, b = blockIdx.x;
    WsHeader* const hdr = &a.s->hdr;
    if (!SELF && a.expect_clean != 0u && ld_cg(reinterpret_cast<const unsigned long long*>(&hdr->clean_mark)) != a.mark) {
        if (b == 0 && tid == 0) record_status(hdr, -1 /*GC_E_INVALID*/, 0xC1EA0000ull);
        return;                                            // every CTA sees the same word
    }
    uint32_t passed = 0, n_stamp = 0;
    // this CTA's share and the warps' parts of it, in 4-element vectors
    const uint32_t nv = (a.n + 3u) >> 2;
    const uint32_t v0 = (uint32_t)(((unsigned long long)b * nv) / G), len = (uint32_t)(((unsigned long long)(b + 1u) * nv) / G) - v0;
    const uint32_t w0 = (uint32_t)(((unsigned long long)warp * len) / kWarps), w1 = (uint32_t)(((unsigned long long)(warp + 1) * len) / kWarps);
    for (int i = tid; i < 2048; i += kBlock) sm.hist[i] = 0u;
    // A launch that clears for itself: the clearing ends at a barrier of the launch, since the scratch's own
    // counter is among what is cleared.  Arrival here, wait behind the fold (2.4M elements, still with an exit count:
    // 28.7 us; 29.1 with the whole barrier behind the fold, 30.1 with a clearing launch in front).
    const auto grid = cooperative_groups::this_grid();
    [[maybe_unused]] cooperative_groups::grid_group::arrival_token cleared{};
    if constexpr (SELF) {
        uint4* const w = reinterpret_cast<uint4*>(a.s);
        for (uint32_t i = b * kBlock + tid; i < (uint32_t)(offsetof(DirectScratch, list) / 16); i += G * kBlock) w[i] = make_uint4(0u, 0u, 0u, 0u);
        cleared = grid.barrier_arrive();                   // (a barrier of the block as well)
    } else {
        // the header: all but the barrier's, the exit counter's and the mark's words start at zero
        if (b == 0 && tid < 62 && tid != (int)kHdrBarrierWord && tid != (int)kHdrExitWord) reinterpret_cast<uint32_t*>(hdr)[tid] = 0u;
        __syncthreads();
    }
    if (b == 0 && tid == 0) hdr->cand_total = a.k;
    phase_stamp(hdr, n_stamp);
    auto flush = [&](uint32_t* dst, int nb) {
        __syncthreads();
        for (int i = tid; i < nb; i += kBlock) {
            const uint32_t c = sm.hist[i];
            if (c) { atomicAdd(dst + i, c); sm.hist[i] = 0u; }
        }
    };
    // elements of vector v that exist (the last one may be ragged)
    auto alive = [&](uint32_t v) { return min(4u, a.n - 4u * v); };
    auto value = [&](uint32_t q) -> float4 {               // vector q of the share
        if (RES) return s_share[q];
        const uint32_t v = v0 + q;
        if (4u * v + 4u <= a.n) return ld_cg(reinterpret_cast<const float4*>(a.r) + v);
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
        o.x = ld_cg(a.r + 4u * v);
        if (4u * v + 1u < a.n) o.y = ld_cg(a.r + 4u * v + 1u);
        if (4u * v + 2u < a.n) o.z = ld_cg(a.r + 4u * v + 2u);
        return o;
    };
    // f(key, element) for every element of the share, four vectors in flight per thread
    auto for_keys = [&](auto f) {
        for (uint32_t q0 = w0; q0 < w1; q0 += 128u) {
            float4 x[4];
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u) {
                const uint32_t q = q0 + 32u * u + lane;
                x[u] = q < w1 ? value(q) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
            for (uint32_t u = 0; u < 4; ++u) {
                const uint32_t q = q0 + 32u * u + lane;
                if (q >= w1) continue;
                const uint32_t i = 4u * (v0 + q);
                f(key_of(x[u].x), i, x[u].x);
                if (i + 4u <= a.n) {
                    f(key_of(x[u].y), i + 1u, x[u].y); f(key_of(x[u].z), i + 2u, x[u].z); f(key_of(x[u].w), i + 3u, x[u].w);
                } else {
                    if (i + 1u < a.n) f(key_of(x[u].y), i + 1u, x[u].y);
                    if (i + 2u < a.n) f(key_of(x[u].z), i + 2u, x[u].z);
                }
            }
        }
    };

    // ---------------------------------------------------------------- fold, top 11 bits
    for (uint32_t q0 = w0; q0 < w1; q0 += 128u) {
        float4 gv[4], rv[4];
        uint32_t ne[4];
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) {
            const uint32_t q = q0 + 32u * u + lane, v = v0 + q;
            ne[u] = q < w1 ? alive(v) : 0u;
            gv[u] = rv[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (ne[u] == 4u) {
                gv[u] = GL::ld4(a.g, 4u * v);
                rv[u] = __ldcs(reinterpret_cast<const float4*>(a.r) + v);
            } else if (ne[u] != 0u) {
                gv[u].x = GL::ld1(a.g, 4u * v); rv[u].x = a.r[4u * v];
                if (ne[u] > 1u) { gv[u].y = GL::ld1(a.g, 4u * v + 1u); rv[u].y = a.r[4u * v + 1u]; }
                if (ne[u] > 2u) { gv[u].z = GL::ld1(a.g, 4u * v + 2u); rv[u].z = a.r[4u * v + 2u]; }
            }
        }
#pragma unroll
        for (uint32_t u = 0; u < 4; ++u) {
            const uint32_t q = q0 + 32u * u + lane, v = v0 + q;
            if (ne[u] == 0u) continue;
            const float4 s = make_float4(__fadd_rn(gv[u].x, rv[u].x), __fadd_rn(gv[u].y, rv[u].y),
                                         __fadd_rn(gv[u].z, rv[u].z), __fadd_rn(gv[u].w, rv[u].w));
            if (RES) s_share[q] = s;
            const float se[4] = {s.x, s.y, s.z, s.w};
            if (ne[u] == 4u) reinterpret_cast<float4*>(a.r)[v] = s;
            else for (uint32_t e = 0; e < ne[u]; ++e) a.r[4u * v + e] = e == 0u ? s.x : e == 1u ? s.y : s.z;
#pragma unroll
            for (uint32_t e = 0; e < 4; ++e)
                if (e < ne[u]) atomicAdd(&sm.hist[key_of(se[e]) >> 20], 1u);
        }
    }
    if constexpr (SELF) grid.barrier_wait(std::move(cleared));
    flush(a.s->hist0, 2048);
    bool live = direct_barrier(hdr, passed, &sm.ok);
    uint32_t prefix = 0, krem = 0, T = 0, m_eq = 0, gt_before = 0, eq_before = 0;
    if (live) {
        phase_stamp(hdr, n_stamp);
        if (b == 0 && tid == 0) hdr->clean_mark = 0ull;    // (every CTA has read it)
        // ------------------------------------------------------------ next 10 bits
        // Somebody else's counts in the scratch: nothing is sent (the residual keeps g + r), the scratch is
        // cleaned on the way out.  Every CTA sees the same sum.
        if (direct_select<2048>(sm, a.s->hist0, a.k, tid, lane, warp) != a.n) {
            if (b == 0 && tid == 0) { record_status(hdr, -1 /*GC_E_INVALID*/, 0xC1EA0001ull); atomicExch(&hdr->abort, 1u); }
            live = false;
        }
    }
    if (live) {
        prefix = sm.bin; krem = a.k - sm.above;
        for_keys([&](uint32_t key, uint32_t, float) { if ((key >> 20) == prefix) atomicAdd(&sm.hist[(key >> 10) & 1023u], 1u); });
        flush(a.s->hist1, 1024);
        live = direct_barrier(hdr, passed, &sm.ok);
    }
    uint32_t m = 0;
    if (live) {
        phase_stamp(hdr, n_stamp);
        direct_select<1024>(sm, a.s->hist1, krem, tid, lane, warp);
        prefix = (prefix << 10) | sm.bin; krem -= sm.above; m = sm.count;
        // ------------------------------------------------------------ list of those that share 21 bits, the others counted
        const bool listed = m <= kDirectList;
        uint32_t sure = 0;
        for_keys([&](uint32_t key, uint32_t i, float x) {
            const uint32_t p = key >> 10;
            if (p > prefix) ++sure;
            else if (p == prefix) {
                if (listed) { const uint32_t at = atomicAdd(&a.s->list_n, 1u); if (at < kDirectList) a.s->list[at] = make_uint2(i, __float_as_uint(x)); }
                else atomicAdd(&sm.hist[key & 1023u], 1u);
            }
        });
        sure = __reduce_add_sync(0xFFFFFFFFu, sure);
        if (lane == 0) { sm.wsum[warp] = sure; sm.wgt[warp] = sure; sm.weq[warp] = 0u; }
        __syncthreads();
        if (tid == 0) {
            uint32_t t = 0;
            for (int w = 0; w < kWarps; ++w) t += sm.wsum[w];
            a.s->tot[b] = t;
        }
        if (!listed) flush(a.s->hist2, 1024);
        live = direct_barrier(hdr, passed, &sm.ok);
        if (live) {
            phase_stamp(hdr, n_stamp);
            if (listed) {
                // every CTA finds the threshold key from the list: the last 10 bits of its keys
                uint2 mine[kDirectList / kBlock];
#pragma unroll
                for (uint32_t u = 0; u < kDirectList / kBlock; ++u) {
                    const uint32_t i = u * kBlock + tid;
                    mine[u] = i < m ? ld_cg(&a.s->list[i]) : make_uint2(0u, 0u);
                }
#pragma unroll
                for (uint32_t u = 0; u < kDirectList / kBlock; ++u)
                    if (u * kBlock + tid < m) atomicAdd(&sm.hist[mine[u].y & 1023u], 1u);
                __syncthreads();
                direct_select<1024, true>(sm, sm.hist, krem, tid, lane, warp);
                T = (prefix << 10) | sm.bin; m_eq = krem - sm.above;
                uint32_t gt = 0, eq = 0;                   // list entries before this CTA's share
#pragma unroll
                for (uint32_t u = 0; u < kDirectList / kBlock; ++u) {
                    const uint32_t key = mine[u].y & kKeyMask, q = (mine[u].x >> 2) - v0;
                    if (u * kBlock + tid >= m || key < T) continue;
                    if (mine[u].x < 4u * v0) { gt += key > T ? 1u : 0u; eq += key == T ? 1u : 0u; }
                    else if (q < len) {                    // one of this CTA's own: it joins its warp's count
                        int w = 0;
                        while (w + 1 < kWarps && q >= (uint32_t)(((unsigned long long)(w + 1) * len) / kWarps)) ++w;
                        atomicAdd(key > T ? &sm.wgt[w] : &sm.weq[w], 1u);
                    }
                }
                gt_before = gt; eq_before = eq;            // (summed over the CTA below)
                __syncthreads();
            } else {
                direct_select<1024>(sm, a.s->hist2, krem, tid, lane, warp);
                T = (prefix << 10) | sm.bin; m_eq = krem - sm.above;
                uint32_t gt = 0, eq = 0;
                for_keys([&](uint32_t key, uint32_t, float) { gt += key > T ? 1u : 0u; eq += key == T ? 1u : 0u; });
                gt = __reduce_add_sync(0xFFFFFFFFu, gt); eq = __reduce_add_sync(0xFFFFFFFFu, eq);
                if (lane == 0) { sm.wgt[warp] = gt; sm.weq[warp] = eq; }
                __syncthreads();
                if (tid == 0) {
                    unsigned long long t = 0;
                    for (int w = 0; w < kWarps; ++w) t += (unsigned long long)sm.weq[w] << 32 | sm.wgt[w];
                    a.s->tot[b] = t;
                }
                live = direct_barrier(hdr, passed, &sm.ok);
            }
        }
    }
    if (live) {
        // ------------------------------------------------------------ emission
        // the histograms have had their last readers (of hist2: before the barrier that followed)
        if constexpr (!SELF)
            for (uint32_t i = b * kBlock + tid; i < 4096u; i += G * kBlock) a.s->hist0[i] = 0u;    // (hist0, hist1, hist2 in a row)
        unsigned long long before = (unsigned long long)eq_before << 32 | gt_before;
        for (uint32_t c = tid; c < b; c += kBlock) before += ld_cg(&a.s->tot[c]);
        before = warp_sum64(before);
        if (lane == 0) sm.part[warp] = before;
        __syncthreads();
        unsigned long long at = 0;
        for (int w = 0; w < kWarps; ++w) { at += sm.part[w]; if (w < warp) at += (unsigned long long)sm.weq[w] << 32 | sm.wgt[w]; }
        uint32_t gt_at = (uint32_t)at, eq_at = (uint32_t)(at >> 32);
        const uint32_t lt = (1u << lane) - 1u, gt_end = gt_at + sm.wgt[warp], eq_end = eq_at + sm.weq[warp];
        if (gt_at != gt_end || eq_at != eq_end) {
            for (uint32_t q0 = w0; q0 < w1; q0 += 32u) {
                const uint32_t q = q0 + lane;
                const float4 x = q < w1 ? value(q) : make_float4(0.f, 0.f, 0.f, 0.f);
                const uint32_t top = max(max(key_of(x.x), key_of(x.y)), max(key_of(x.z), key_of(x.w)));
                if (!__any_sync(0xFFFFFFFFu, top >= T)) continue;
                const uint32_t ne = q < w1 ? alive(v0 + q) : 0u;
                const float xe[4] = {x.x, x.y, x.z, x.w};
                uint32_t gm = 0, em = 0;                   // elements above the threshold key, at it
#pragma unroll
                for (uint32_t e = 0; e < 4; ++e) {
                    const uint32_t key = key_of(xe[e]);
                    gm |= (e < ne && key > T) ? 1u << e : 0u;
                    em |= (e < ne && key == T) ? 1u << e : 0u;
                }
                uint32_t gb = 0, eb = 0, gall = 0, eall = 0;      // of the lanes before this one; of all
#pragma unroll
                for (uint32_t e = 0; e < 4; ++e) {
                    const unsigned bg = __ballot_sync(0xFFFFFFFFu, (gm >> e) & 1u), be = __ballot_sync(0xFFFFFFFFu, (em >> e) & 1u);
                    gb += (uint32_t)__popc(bg & lt); eb += (uint32_t)__popc(be & lt);
                    gall += (uint32_t)__popc(bg); eall += (uint32_t)__popc(be);
                }
#pragma unroll
                for (uint32_t e = 0; e < 4; ++e) {
                    const uint32_t low = (1u << e) - 1u, ge = gt_at + gb + (uint32_t)__popc(gm & low), ee = eq_at + eb + (uint32_t)__popc(em & low);
                    const bool sent = ((gm >> e) & 1u) || (((em >> e) & 1u) && ee < m_eq);
                    if (sent) {
                        const uint32_t slot = ge + min(ee, m_eq), i = 4u * (v0 + q) + e;
                        if (slot < a.k) {
                            a.out_idx[slot] = i;
                            a.out_val[slot] = xe[e];
                            a.r[i] = 0.0f;
                        } else {
                            record_status(hdr, -1 /*GC_E_INVALID*/, i);
                        }
                    }
                }
                gt_at += gall; eq_at += eall;
            }
        }
        // (counted and emitted entries agree and add up to k, unless others wrote to the scratch)
        if (lane == 0 && (gt_at != gt_end || eq_at != eq_end ||
                          (b == G - 1u && warp == kWarps - 1 && gt_at + min(eq_at, m_eq) != a.k)))
            record_status(hdr, -1 /*GC_E_INVALID*/, 0xC1EA0002ull);
        if (a.out_count != nullptr && b == 0 && tid == 0) { a.out_count[0] = a.k; a.out_count[1] = a.k; }
        phase_stamp(hdr, n_stamp);
    }
    if constexpr (SELF) {
        // Nothing to be left clean; the caller's status word is written when the work is done, by the CTA that leaves last.
        if (a.status_out == nullptr) return;
        __syncthreads();
        if (tid == 0) {
            uint32_t gone;                                 // (the CTAs that left before, their writes done)
            asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(gone) : "l"(&hdr->exit_count) : "memory");
            if (gone == G - 1u) {
                const int32_t st = *reinterpret_cast<volatile int32_t*>(&hdr->status);
                asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(a.status_out), "r"(st) : "memory");
            }
        }
        return;
    }
    // The CTA that leaves last resets what the others may still have been reading; after a wait that ran
    // out, or counts that do not add up, it cleans everything and sets no mark (the next call on a private
    // workspace ends with GC_E_INVALID until the status has been read, see CleanArgs).
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        sm.last = atomicAdd(&hdr->exit_count, 1u) == G - 1u ? 1u : 0u;
        __threadfence();
    }
    __syncthreads();
    if (sm.last != 0u) {
        const bool failed = ld_cg(&hdr->abort) != 0u;
        if (failed) for (uint32_t i = tid; i < 4096u; i += kBlock) a.s->hist0[i] = 0u;
        if (tid == 0) {
            a.s->list_n = 0u; hdr->barrier = 0u; hdr->exit_count = 0u; hdr->abort = 0u;
            __threadfence();
            if (!failed) hdr->clean_mark = a.mark;
        }
    }
}

// Launch geometry for n elements on a device with `sms` SMs.  A CTA has at least 2048 elements.  Up to two
// CTAs per SM as long as their shares fit kDirectResident bytes of shared memory (7.2M elements); beyond
// that three CTAs per SM read theirs back from L2 (16M elements: 100 us against 121 us with two).  Three
// with the shares in shared memory are slower up to 4M elements (1M: 24.6 against 22.4 us) and equal at 7M.
constexpr size_t kDirectResident = 96 * 1024;
struct DirectGeom { uint32_t G; size_t smem; bool resident; };
inline DirectGeom direct_geometry(uint32_t n, int sms) {
    DirectGeom d;
    const uint32_t nv = (n + 3u) / 4u;
    auto ctas = [&](uint32_t per_sm) {
        uint32_t G = (nv + 511u) / 512u;
        if (G > per_sm * (uint32_t)sms) G = per_sm * (uint32_t)sms;
        return G > kDirectMaxG ? kDirectMaxG : G < 1u ? 1u : G;
    };
    d.G = ctas(2u);
    d.smem = 16 * (size_t)((nv + d.G - 1) / d.G + 1);
    d.resident = d.smem <= kDirectResident;
    if (!d.resident) { d.G = ctas(3u); d.smem = 0; }
    return d;
}
// One-tensor plans of up to this many elements take this kernel instead of the candidate path of
// k_topk_single (workspace cleared before the call, 1 % density: 1M 24 against 31 us, 2.4M 28.8 against
// 34.4, 4M 35.3 against 37.2, 5M 39.7 against 39).
constexpr uint32_t kDirectMaxPlan = 1u << 22;

}  // namespace gc
