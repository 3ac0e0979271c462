// Tiled decode: lists through rings in shared memory, every warp adds its own part of the tile.
//
// A CTA builds eight sub-tiles at a time, one per warp.  The workers' entries come into per-worker
// rings with 16-byte asynchronous copies, each entry once; a warp finds its sub-tile's range in every
// ring by a binary search (a lane per worker) and adds the ranges one worker after the other, on its
// own: a worker's indices are distinct, so the 32 lanes never collide, and a warp's shared-memory
// accesses happen in program order, so the fixed worker order needs no barrier between workers.
//
// What bounds it: shared-memory round trips per (sub-tile, worker) pair, whatever the number of entries in
// it, with 16 to 24 warps per SM (32 lists at 1 % of 50M elements: 0.6 eligible warps per scheduler, issue
// slots 42 %, shared-memory pipe 59 %, DRAM 33 % busy).  Why rings: formulations that read the lists with
// plain loads (window in registers, per warp or per CTA, with or without conflict detection between
// workers) all ended near 330 us on 32 lists at 1 % of 110M elements, because a carve-out of 200 KB
// leaves L1 room for a few hundred lines in flight; cp.async needs none.  Measured, 110M elements at
// 1 %, lists that agree on a fifth of their entries: W = 8 / 16 / 32 in 113 / 150 / 217 us against
// 141 / 443 / 470 us before (block-wide steps per worker; a colliding-entries list that overflowed);
// 50M elements: W = 64 at 1 % 226 against 774 us, W = 16 / 32 at 5 % 180 / 389 against 258 / 864 us.
// With the optimizer behind it (parameters and velocities fetched asynchronously under the additions)
// 110M elements, W = 8: 304 against 388 us; 25.6M elements at 0.1 %, W = 8: 79 against 111 us.
#pragma once
#include "gc_decode.cuh"

namespace gc {

// 16-byte asynchronous copy global -> shared of `bytes` <= 16 (the rest is filled with zeros)
__device__ __forceinline__ void cp_async_16(void* sdst, const void* gsrc, uint32_t bytes = 16u) {
    const uint32_t sa = (uint32_t)__cvta_generic_to_shared(sdst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sa), "l"(gsrc), "r"(bytes) : "memory");
}

// Where Q lists enter the run that starts at flat index `key`: Q searches of one warp side by side
// (their probes are in flight together, so Q lists cost the round trips of one).
template <int Q>
__device__ __forceinline__ void warp_lower_bounds(const uint32_t* const (&idx)[Q], const uint32_t (&cnt)[Q], uint32_t key,
                                                  int lane, uint32_t (&lo)[Q]) {
    uint32_t hi[Q];
    bool more = false;
#pragma unroll
    for (int q = 0; q < Q; ++q) { lo[q] = 0u; hi[q] = cnt[q]; more = more || cnt[q] != 0u; }
    while (more) {
        bool ge[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const uint32_t span = hi[q] - lo[q];
            const uint32_t p = lo[q] + (uint32_t)(((unsigned long long)span * (uint32_t)(lane + 1)) / 33u);
            ge[q] = span == 0u || __ldcg(idx[q] + p) >= key;
        }
        more = false;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const uint32_t span = hi[q] - lo[q];
            const unsigned b = __ballot_sync(0xFFFFFFFFu, ge[q]);
            if (span == 0u) continue;
            const int f = b ? (__ffs(b) - 1) : 32;       // first lane that saw >= key bounds hi, the lane before it lo
            const uint32_t pf = lo[q] + (uint32_t)(((unsigned long long)span * (uint32_t)(f + 1)) / 33u);
            const uint32_t pl = lo[q] + (uint32_t)(((unsigned long long)span * (uint32_t)f) / 33u);
            const uint32_t nlo = f > 0 ? pl + 1u : lo[q];
            const uint32_t nhi = f < 32 ? pf : hi[q];
            lo[q] = nlo; hi[q] = nhi < nlo ? nlo : nhi;
            more = more || hi[q] > lo[q];
        }
    }
}

constexpr uint32_t kRingBatch = 4u;          // workers whose entries are read ahead of the additions
constexpr uint32_t kRingPad = 32u;           // words behind a warp's sub-tile that swallow what lies outside of it

// T = elements of a sub-tile (a multiple of 128), RS = slots of a ring (a multiple of 4).  ADD: the sums
// continue what the dense buffer holds.  WIDE: more than 32 workers, two per lane.
template <bool APPLY, bool ADD, bool WIDE>
static __global__ void __launch_bounds__(kDecBlock, 3)
k_decode_rings(const __grid_constant__ DecodeLists ls, uint32_t W, uint32_t cnt, uint32_t total_n, uint32_t T, uint32_t RS,
               float* __restrict__ out, int aligned, WsHeader* hdr, ApplyArgs ap) {
    static_assert(!(APPLY && ADD), "the optimizer step always starts from a sum of its own");
    constexpr int kW8 = kDecBlock / 32, U = WIDE ? 2 : 1;
    extern __shared__ __align__(128) float s_dyn_rings[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    launch_wait();
    // rings [W][2][RS] (indices, values), then the sub-tiles
    const uint32_t Wb = (W + kRingBatch - 1u) / kRingBatch * kRingBatch;
    uint32_t* const rings = reinterpret_cast<uint32_t*>(s_dyn_rings);
    float* const s_tiles = s_dyn_rings + 2u * W * RS;
    float* const s_tile = s_tiles + warp * (T + kRingPad);               // this warp's sub-tile
    float* const s_par = s_tiles + kW8 * (T + kRingPad) + warp * 2u * T;          // APPLY: its parameters and velocities
    uint2* const s_rng = reinterpret_cast<uint2*>(s_tiles + kW8 * (T + kRingPad) + (APPLY ? kW8 * 2u * T : 0u)) + warp * (32 * U);
    __shared__ uint32_t s_cur[2][64], s_slot[2][64], s_fill[64], s_len[64];      // list position the ring starts at, its slot
    const uint32_t tile = kW8 * T;
    auto wrap = [&](uint32_t s) { return min(s, s - RS); };              // slot s < 2 RS of a ring
    const uint32_t ntl = (total_n + tile - 1) / tile;
    const uint32_t t0 = (uint32_t)(((unsigned long long)blockIdx.x * ntl) / gridDim.x);
    const uint32_t t1 = (uint32_t)(((unsigned long long)(blockIdx.x + 1u) * ntl) / gridDim.x);
    if (t0 >= t1) return;

    auto fetch = [&](uint32_t tl) {                        // what this warp's sub-tile of tile tl needs besides the lists
        const uint32_t a = tl * tile + warp * T, span = a < total_n ? min(T, total_n - a) : 0u;
        if (APPLY) {                                       // (the buffer's last words with zeros behind them)
            for (uint32_t q = lane; 4 * q < span; q += 32) {
                const uint32_t bytes = min(4u, span - 4 * q) * 4u;
                cp_async_16(s_par + 4 * q, ap.param + a + 4 * q, bytes);
                cp_async_16(s_par + T + 4 * q, ap.vel + a + 4 * q, bytes);
            }
        }
        if (ADD) {
            if (span == T && aligned) for (uint32_t q = lane; q < T / 4; q += 32) cp_async_16(s_tile + 4 * q, out + a + 4 * q);
            else for (uint32_t q = lane; q < span; q += 32) cp_async_4(s_tile + q, out + a + q);
        }
    };
    fetch(t0);                                             // (under the search below)
    if (!ADD)
        for (uint32_t q = lane; q < T / 4; q += 32) reinterpret_cast<float4*>(s_tile)[q] = make_float4(0.f, 0.f, 0.f, 0.f);

    // where every list enters this CTA's run of tiles
    if (tid < 64) s_len[tid] = (uint32_t)tid >= W ? 0u : ls.len[tid] != nullptr ? min(__ldcg(ls.len[tid]), cnt) : cnt;
    __syncthreads();
    for (uint32_t w0 = (uint32_t)warp; w0 < W; w0 += 4u * kW8) {
        const uint32_t* ip[4];
        uint32_t cn[4], lo4[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t w = w0 + q * kW8;
            ip[q] = ls.idx[min(w, 63u)]; cn[q] = w < W ? s_len[min(w, 63u)] : 0u;
        }
        warp_lower_bounds<4>(ip, cn, t0 * tile, lane, lo4);
        if (lane == 0) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (w0 + q * kW8 < W) { s_cur[0][w0 + q * kW8] = lo4[q]; s_slot[0][w0 + q * kW8] = lo4[q] & 3u; }
        }
    }
    __syncthreads();

    // E consecutive threads top up one worker's ring: list positions [fill, (cur & ~3) + RS)
    uint32_t Wp = 1;
    while (Wp < W) Wp <<= 1;
    const uint32_t E = kDecBlock / Wp, my_w = (uint32_t)tid / E, sub = (uint32_t)tid % E;
    const bool top = my_w < W;
    const uint32_t* const my_idx = ls.idx[top ? my_w : 0u];
    const float* const my_val = ls.val[top ? my_w : 0u];
    const uint32_t my_len = top ? s_len[my_w] : 0u;
    const bool by16 = ((reinterpret_cast<uintptr_t>(my_idx) | reinterpret_cast<uintptr_t>(my_val)) & 15u) == 0u;
    uint32_t my_fill = top ? s_cur[0][my_w] & ~3u : 0u, my_slot = 0u;      // first position that is not in the ring, its slot
    auto top_up = [&](uint32_t cur) {
        const uint32_t to = min((my_len + 3u) & ~3u, (cur & ~3u) + RS);
        for (uint32_t p = my_fill + 4u * sub; p < to; p += 4u * E) {
            uint32_t* const di = rings + 2u * my_w * RS + wrap(my_slot + (p - my_fill));
            uint32_t* const dv = di + RS;
            if (by16) {
                const uint32_t bytes = min(4u, my_len - p) * 4u;
                cp_async_16(di, my_idx + p, bytes);
                cp_async_16(dv, my_val + p, bytes);
            } else {
                for (uint32_t q = 0; q < 4u && p + q < my_len; ++q) { cp_async_4(di + q, my_idx + p + q); cp_async_4(dv + q, my_val + p + q); }
            }
        }
        if (to > my_fill) { my_slot = wrap(my_slot + (to - my_fill)); my_fill = to; }
        if (top && sub == 0u) s_fill[my_w] = min(my_fill, my_len);
    };
    if (top) top_up(s_cur[0][my_w]);

    uint32_t top_step = 1;                                 // largest power of two <= RS
    while (2u * top_step <= RS) top_step *= 2u;
    uint32_t tl = t0, par = 0, sub_lo = t0 * tile;
    bool disorder = false;
    while (true) {
        const uint32_t lo = tl * tile, hi = min(total_n, lo + tile);
        cp_async_wait_all();
        __syncthreads();                                   // rings and cursors are complete
        // a ring that ends inside the tile while its list goes on: this step ends at the smallest
        // index up to which every ring is complete (every warp finds the same)
        uint32_t bound = hi, cur[U], have[U], slot[U];      // list position, entries, first slot of the ring
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t w = 32u * u + lane;
            cur[u] = have[u] = slot[u] = 0u;
            if (w < W) {
                const uint32_t fill = s_fill[w];
                cur[u] = s_cur[par][w]; slot[u] = s_slot[par][w]; have[u] = fill - cur[u];
                // (a ring that ends below this step, or with an index no buffer has, belongs to a list that is
                //  not ascending: it must not hold up the others)
                const uint32_t end = fill < s_len[w] ? rings[2u * w * RS + wrap(slot[u] + have[u] - 1u)] : hi;
                if (end >= sub_lo && end < hi) bound = min(bound, end + 1u);
            }
        }
        bound = __reduce_min_sync(0xFFFFFFFFu, bound);     // (above sub_lo: every step makes progress)
        // this warp's range of every ring
        const uint32_t a = lo + warp * T;
        const uint32_t k0 = min(max(a, sub_lo), bound), k1 = min(max(a + T, sub_lo), bound), span = k1 - k0;
        uint32_t longest = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t w = 32u * u + lane;
            const uint32_t* const ring = rings + 2u * w * RS;
            uint32_t b0 = 0u, b1 = 0u;
            for (uint32_t d = top_step; d != 0u; d >>= 1) {
                const uint32_t m0 = b0 + d, m1 = b1 + d;
                if (m0 <= have[u] && ring[wrap(slot[u] + m0 - 1u)] < k0) b0 = m0;
                if (m1 <= have[u] && ring[wrap(slot[u] + m1 - 1u)] < k1) b1 = m1;
            }
            // (an ascending list has nothing in front of the first sub-tile's range; what another list has
            //  there is looked at all the same, so that no entry goes by unreported)
            if (warp == 0) b0 = 0u;
            const uint32_t n = b1 > b0 ? b1 - b0 : 0u;
            s_rng[w] = make_uint2(wrap(slot[u] + b0), n);
            longest = max(longest, n);
            if (warp == kW8 - 1 && w < W) {                // (k1 = the bound)
                s_cur[par ^ 1u][w] = cur[u] + b1; s_slot[par ^ 1u][w] = wrap(slot[u] + b1);
                // two entries that changed places across the bound: the next CTA's search may step over both
                disorder = disorder || (b1 + 1u < have[u] && ring[wrap(slot[u] + b1 + 1u)] < bound);
            }
        }
        const bool small = __reduce_max_sync(0xFFFFFFFFu, longest) <= 32u;
        __syncwarp();
        // what lies outside the range (a list that is not ascending), or lanes without an entry, go to
        // this lane's own word behind the sub-tile
        const uint32_t at0 = k0 - a;
        auto place = [&](uint32_t x, bool live) {
            const bool ok = live && x - k0 < span;
            disorder = disorder || (live && !ok);
            return s_tile + (ok ? x - k0 + at0 : T + lane);
        };
        if (small) {
            for (uint32_t w0 = 0; w0 < Wb; w0 += kRingBatch) {
                uint32_t x[kRingBatch], n[kRingBatch];
                float v[kRingBatch];
#pragma unroll
                for (uint32_t j = 0; j < kRingBatch; ++j) {
                    const uint2 r = s_rng[w0 + j];
                    const uint32_t* const e = rings + 2u * min(w0 + j, W - 1u) * RS + wrap(r.x + lane);
                    n[j] = r.y; x[j] = e[0]; v[j] = __uint_as_float(e[RS]);
                }
#pragma unroll
                for (uint32_t j = 0; j < kRingBatch; ++j) {
                    float* const p = place(x[j], (uint32_t)lane < n[j]);
                    *p = __fadd_rn(*p, v[j]);
                    __syncwarp();
                }
            }
        } else {
            for (uint32_t w = 0; w < W; ++w) {
                const uint2 r = s_rng[w];
                for (uint32_t i = lane; i - lane < r.y; i += 64) {           // two rounds at a time: distinct elements
                    const uint32_t* const e0 = rings + 2u * w * RS + wrap(r.x + i);
                    const uint32_t* const e1 = rings + 2u * w * RS + wrap(min(r.x + i + 32u, 2u * RS - 1u));
                    const uint32_t x0 = e0[0], x1 = e1[0];
                    const float v0 = __uint_as_float(e0[RS]), v1 = __uint_as_float(e1[RS]);
                    float* const p0 = place(x0, i < r.y);
                    float* const p1 = place(x1, i + 32u < r.y);
                    const float s0 = *p0, s1 = *p1;
                    *p0 = __fadd_rn(s0, v0);
                    *p1 = __fadd_rn(s1, v1);
                }
                __syncwarp();
            }
        }
        __syncthreads();                                   // the rings have been read, the new cursors are there
        par ^= 1u;
        if (top) top_up(s_cur[par][my_w]);
        sub_lo = bound;
        if (bound < hi) continue;
        // the sub-tile leaves; its words are zero again
        const uint32_t n_out = a < total_n ? min(T, total_n - a) : 0u;
        if (APPLY) {
            // (the sub-tile at the buffer's end as well: its loads one after the other from global memory took
            //  longer than all the rest of a 1.5M-element call)
#pragma unroll 2
            for (uint32_t q = lane; 4 * q < n_out; q += 32) {
                float4 vv = reinterpret_cast<const float4*>(s_par + T)[q];
                float4 pp = reinterpret_cast<const float4*>(s_par)[q];
                const float4 gs = reinterpret_cast<const float4*>(s_tile)[q];
                reinterpret_cast<float4*>(s_tile)[q] = make_float4(0.f, 0.f, 0.f, 0.f);
                vv.x = __fadd_rn(__fmul_rn(ap.mu, vv.x), __fmul_rn(ap.scale, gs.x));
                vv.y = __fadd_rn(__fmul_rn(ap.mu, vv.y), __fmul_rn(ap.scale, gs.y));
                vv.z = __fadd_rn(__fmul_rn(ap.mu, vv.z), __fmul_rn(ap.scale, gs.z));
                vv.w = __fadd_rn(__fmul_rn(ap.mu, vv.w), __fmul_rn(ap.scale, gs.w));
                pp.x = __fsub_rn(pp.x, __fmul_rn(ap.lr, vv.x)); pp.y = __fsub_rn(pp.y, __fmul_rn(ap.lr, vv.y));
                pp.z = __fsub_rn(pp.z, __fmul_rn(ap.lr, vv.z)); pp.w = __fsub_rn(pp.w, __fmul_rn(ap.lr, vv.w));
                if (4 * q + 4u <= n_out) {
                    __stcs(reinterpret_cast<float4*>(ap.vel + a) + q, vv);
                    __stcs(reinterpret_cast<float4*>(ap.param + a) + q, pp);
                } else {
                    const float ve[3] = {vv.x, vv.y, vv.z}, pe[3] = {pp.x, pp.y, pp.z};
#pragma unroll
                    for (uint32_t e = 0; e < 3u; ++e)
                        if (4 * q + e < n_out) { ap.vel[a + 4 * q + e] = ve[e]; ap.param[a + 4 * q + e] = pe[e]; }
                }
            }
        } else if (n_out == T && aligned) {
#pragma unroll 4
            for (uint32_t q = lane; q < T / 4; q += 32) {
                const float4 o = reinterpret_cast<const float4*>(s_tile)[q];
                if (!ADD) reinterpret_cast<float4*>(s_tile)[q] = make_float4(0.f, 0.f, 0.f, 0.f);
                __stcs(reinterpret_cast<float4*>(out + a) + q, o);
            }
        } else {
            for (uint32_t q = lane; q < n_out; q += 32) { out[a + q] = s_tile[q]; if (!ADD) s_tile[q] = 0.0f; }
        }
        if (++tl >= t1) break;
        if (APPLY || ADD) { __syncwarp(); fetch(tl); }
    }
    cp_async_wait_all();
    if (disorder) record_status(hdr, -1 /*GC_E_INVALID*/, sub_lo);
    if (t1 == ntl && tid < (int)W && s_cur[par][tid] < s_len[tid])
        record_status(hdr, -1 /*GC_E_INVALID*/, s_cur[par][tid]);          // leftovers point at or beyond total_n
}

}  // namespace gc
