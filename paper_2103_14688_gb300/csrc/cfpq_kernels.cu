// cfpq_kernels.cu -- CUDA kernels of libcfpq for sm_103a.
//
// The index-creation loop of Listing 1 (arXiv 2103.14688, Sec. 3.1) runs as
// passes of three kernels, all driven by per-query control words in device
// memory (QCtl):
//   k_gather   one closure pass.  For every output block C[s,t] and row x it
//              ORs, over the product edges (s,x) -> (u,y) generated on the fly
//              from the RSM transitions s -l-> u and the graph edges (x,y) of
//              M2^l (the Kronecker product M1 (x) M2, never materialised), the
//              row (I + C)[u,t][y].  The first pass of an iteration uses only
//              the new edges A2 (left-distributivity, Sec. 3.1.1) with whole
//              source rows; later passes use all edges but only source rows
//              whose dirty stamp says they changed in the previous pass (the
//              incremental closure of Sec. 3.1.1 recomputes only what the new
//              edges reach).
//   k_extract  after a pass that changed nothing: for every box b and final f
//              of b, new = C[q0_b, f] & ~M2^b on the rows changed in this
//              iteration; M2^b |= new; A2^b = new (Listing 1, extraction via
//              getStates/getCoordinates).
//   k_control  advances each query's loop state and sets the CUDA-graph
//              conditional (Listing 1: "while M2 is changing").
#include <cuda_runtime.h>

#include <algorithm>
#include <stdint.h>

#include "cfpq_dev.cuh"

namespace cfpq {

#define FULLMASK 0xffffffffu

__device__ __forceinline__ bool nz4(const uint4 &v) { return (v.x | v.y | v.z | v.w) != 0u; }
__device__ __forceinline__ void or4(uint4 &a, const uint4 &b) {
    a.x |= b.x; a.y |= b.y; a.z |= b.z; a.w |= b.w;
}
__device__ __forceinline__ uint4 andnot4(const uint4 &a, const uint4 &b) {
    return make_uint4(a.x & ~b.x, a.y & ~b.y, a.z & ~b.z, a.w & ~b.w);
}
__device__ __forceinline__ int popc4(const uint4 &v) {
    return __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
}

// Set bit `pos` (0..127) of a 128-bit vector.
__device__ __forceinline__ void setbit4(uint4 &v, uint32_t pos) {
    const uint32_t m = 1u << (pos & 31);
    switch ((pos >> 5) & 3) {
        case 0: v.x |= m; break;
        case 1: v.y |= m; break;
        case 2: v.z |= m; break;
        default: v.w |= m; break;
    }
}

// Set bit z of a row held by a group of lpr lanes (lane gl holds the 128-bit
// vectors gl, gl + lpr, ...).
template <int VPL>
__device__ __forceinline__ void set_row_bit(uint4 (&acc)[VPL], uint32_t z, int lpr, int gl) {
    const uint32_t v = z >> 7;
    if ((int)(v % (uint32_t)lpr) == gl) {
        const int j = (int)(v / (uint32_t)lpr);
#pragma unroll
        for (int jj = 0; jj < VPL; ++jj)
            if (jj == j) setbit4(acc[jj], z & 127u);
    }
}

// OR rows of a pure-terminal block (see SrcDesc::pure_n) into the group's
// row: every lane with keep_l expands its own source row y_l (the columns of
// y_l's CSR rows under the block's labels, all lanes' loads in flight at
// once), and each column found is passed by shuffle to the lane that holds
// its bit.  Called by all lanes of the warp.
template <int VPL>
__device__ __forceinline__ void or_pure_rows(uint4 (&acc)[VPL], const SrcDesc &d, uint32_t y_l, bool keep_l,
                                             int lpr, int gl, int grp, unsigned gmask) {
    uint32_t e0 = 0, e1 = 0, f0 = 0, f1 = 0;
    if (keep_l) {
        e0 = d.pure_off[0][y_l];
        e1 = d.pure_off[0][y_l + 1];
        if (d.pure_n > 1) {
            f0 = d.pure_off[1][y_l];
            f1 = d.pure_off[1][y_l + 1];
        }
    }
    while (true) {
        bool has = false;
        uint32_t z = 0;
        if (e0 < e1) {
            z = d.pure_col[e0++];
            has = true;
        } else if (f0 < f1) {
            z = d.pure_col[f0++];
            has = true;
        }
        const unsigned bal = __ballot_sync(FULLMASK, has);
        if (!bal) break;
        unsigned mine = (bal & gmask) >> (grp * lpr);
        while (__any_sync(FULLMASK, mine != 0u)) {
            const bool h = mine != 0u;
            const int src = h ? __ffs(mine) - 1 : 0;
            if (h) mine &= mine - 1u;
            const uint32_t zz = __shfl_sync(FULLMASK, z, src, lpr);
            if (h) set_row_bit<VPL>(acc, zz, lpr, gl);
        }
    }
}

// Asynchronous 16-byte global -> shared copy (zero-filled when !valid); the
// copies of a thread form groups it can wait for.
__device__ __forceinline__ void cp_async16(uint4 *dst, const void *src, bool valid) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Source rows a warp of the general gather keeps in flight (shared-memory
// ring), for rows of 4+ vectors per lane where registers allow only one row
// load at a time; narrower rows batch their loads in registers.
template <int VPL>
struct GatherRing {
    static constexpr bool on = VPL >= 4;
    static constexpr int depth = VPL <= 8 ? 4 : 3;
    // narrower rows keep one row-sized slot per warp: the bitmap of
    // pure-terminal reads (pure_bitmap_*)
    static constexpr int slots = on ? depth : 1;
    static constexpr size_t bytes = (size_t)8 * slots * 32 * VPL * 16;  // 8 warps
};

// The same for a warp that owns one row (lpr = 32, rows of 4+ vectors per
// lane), with a row-sized shared-memory bitmap `bm` (uint4-aligned, the
// vectors in row order): the bitmap is cleared once per row and source, every
// lane sets the columns it finds with a shared atomic -- no broadcast -- for
// every candidate of the enumeration, and the bitmap is ORed into the
// accumulators once at the end.
template <int VPL>
__device__ __forceinline__ void pure_bitmap_clear(uint32_t nvec, int lane, uint4 *bm) {
#pragma unroll
    for (int j = 0; j < VPL; ++j) {
        const uint32_t v = (uint32_t)lane + 32u * (uint32_t)j;
        if (v < nvec) bm[v] = make_uint4(0, 0, 0, 0);
    }
    __syncwarp();
}

__device__ __forceinline__ void pure_bitmap_set(const SrcDesc &d, uint32_t y_l, bool keep_l, uint4 *bm) {
    if (!keep_l) return;
    unsigned int *w = reinterpret_cast<unsigned int *>(bm);
    for (uint32_t p = 0; p < d.pure_n; ++p) {
        const uint32_t *off = d.pure_off[p];
        const uint32_t e1 = off[y_l + 1];
        for (uint32_t e = off[y_l]; e < e1; ++e) {
            const uint32_t z = d.pure_col[e];
            atomicOr(w + (z >> 5), 1u << (z & 31u));
        }
    }
}

template <int VPL>
__device__ __forceinline__ void pure_bitmap_or(uint4 (&acc)[VPL], uint32_t nvec, int lane, const uint4 *bm) {
    __syncwarp();
#pragma unroll
    for (int j = 0; j < VPL; ++j) {
        const uint32_t v = (uint32_t)lane + 32u * (uint32_t)j;
        if (v < nvec) or4(acc[j], bm[v]);
    }
    __syncwarp();  // the bitmap (a ring slot) is reused afterwards
}

// Lowest set bit of a 128-bit vector, -1 if none; clears it when `clear`.
__device__ __forceinline__ int lowbit4(uint4 &v, bool clear) {
    if (v.x) { int b = __ffs(v.x) - 1; if (clear) v.x &= v.x - 1; return b; }
    if (v.y) { int b = __ffs(v.y) - 1; if (clear) v.y &= v.y - 1; return 32 + b; }
    if (v.z) { int b = __ffs(v.z) - 1; if (clear) v.z &= v.z - 1; return 64 + b; }
    if (v.w) { int b = __ffs(v.w) - 1; if (clear) v.w &= v.w - 1; return 96 + b; }
    return -1;
}

// Which edges of a source take part in this pass (bit mask):
//   1  new edges of the iteration, whole source rows (FIRST pass): terminal
//      edges in iteration 1, A2 rows afterwards (left-distributivity);
//   2  all edges, source rows of a lower level changed in this iteration
//      (FIRST pass; those levels are final for the iteration);
//   4  all edges, source rows of this level changed in the previous pass
//      (REPEAT pass of a cyclic level).
// Channels 2 and 4 of a tensor-core source (and of a switchable source while
// its box is dense) run as tile products over the dirty rows instead.  When
// the source's channel-1 tile job (SrcDesc::tile_new) runs in this pass,
// channel 1's row ORs go to the tiles too: the result keeps channel 1 only
// for the product edges themselves (ident), flagged by bit 8 (channel 1 reads
// no closure rows).  That job does not wait for the box to be dense: the
// iteration in which Dyck-4's answer turns dense adds a quarter of its edges to a box that
// was sparse at its start, and the hub rows of its row gather took 30 ms
// of the n = 65536 query (4 ms of 16384's); see new_tiles_pay.
template <bool NT>
__device__ __forceinline__ uint32_t src_channels(const SrcDesc &d, uint32_t mode, uint32_t iter, uint32_t g,
                                                 uint32_t g0, uint32_t dense_mask) {
    const bool tiles = d.dense || (d.box_switch && d.csr_off == nullptr && d.label_box < 32u &&
                                   ((dense_mask >> d.label_box) & 1u));
    uint32_t ch = 0u;
    if (mode == kModeNew) {
        const bool term1 = d.csr_off != nullptr && iter == 1;
        if (term1 || (d.csr_off == nullptr && *d.box_new_it == iter)) ch |= 1u;
        if (d.rblk && !d.same_level && !term1 && *d.rlast >= g0) ch |= 2u;
    } else {
        if (d.rblk && d.same_level && *d.rlast + 1u >= g) ch |= 4u;
    }
    if (tiles) ch &= 1u;
    if (NT && (ch & 1u) && d.tile_new && d.tc_kcount) {
        const unsigned long long kc = *reinterpret_cast<const volatile unsigned long long *>(d.tc_kcount);
        const uint32_t listed = ((uint32_t)(kc >> 32) == g) ? (uint32_t)kc : 0u;
        if (new_tiles_pay(listed, d.tc_kcap, *d.tc_mcount, *d.tc_ecount, d.tc_ratio))
            ch = (ch & ~1u) | (d.ident ? 9u : 0u);
    }
    return ch;
}

// Does row x have an edge of source d that takes part (channels `chans`, not
// zero)?  Called by one lane per row, 32 rows of a warp side by side: a pass
// changes few of the rows it could (one in nine on the regular query at n = 30011), and a
// warp that owns a row finds that out behind four dependent loads.  Loop time, visiting
// every row -> only these: regular query n = 30011 7.27 -> 3.05 ms, Dyck-4 n = 3001
// 4.84 -> 4.07, n = 65536 209 -> 186, 16 sources at n = 65536 5.0 -> 2.8.
// A row of more than kTestEdges edges is taken untested: its lane would walk it alone, two
// dependent loads an edge, where the gather reads the row with a warp.  a+ over a path of
// 200 vertices and four vertices with edges to all others, on the gather: n = 8000 37.9 ->
// 26.9 ms, n = 16000 78.3 -> 53.0, n = 30000 169 -> 108.
constexpr uint32_t kTestEdges = 32;
template <bool NT>
__device__ __forceinline__ bool row_has_work(const SrcDesc &d, uint32_t chans, uint32_t x, uint32_t iter, uint32_t g,
                                             uint32_t g0) {
    if (d.csr_off) {
        const uint32_t e1 = d.csr_off[x + 1];
        uint32_t e = d.csr_off[x];
        if (e >= e1) return false;
        if ((chans & 1u) || e1 - e > kTestEdges) return true;
        const uint32_t thr = (chans & 2u) ? g0 : g - 1u;
        for (; e < e1; ++e)
            if (d.rstamp[d.csr_col[e]] >= thr) return true;
        return false;
    }
    if (!NT) return false;
    return (chans & 6u) ? d.nt_new_it[x] != 0u : d.nt_new_it[x] == iter;  // (0: the row has no edge)
}

// --------------------------------------------------------------------------
// Closure pass (bit-packed rows).  One CTA of 8 warps per work item; a row is
// handled by a group of `lpr` lanes, each lane holding VPL 128-bit vectors
// (words 2v, 2v+1 for v = lane_in_group + j * lpr).  NT selects the general
// variant (nonterminal adjacency rows, pure-terminal blocks); without it the
// kernel holds only the CSR paths, which keeps its registers for the rows.
// --------------------------------------------------------------------------
// Occupancy target per row width: narrow rows keep 4 CTAs (32 warps) per SM, for
// which the general variants of widths 1 and 2 spill 160 and 224 bytes and the CSR
// one of width 1 spills 48.
template <int VPL>
struct GatherOcc {
    static constexpr int value = VPL <= 2 ? 4 : (VPL == 4 ? 2 : 1);
};
// CSR variant of wide rows: one source row in registers beside the output row
// leaves room for two CTAs (it was one CTA with two source rows in flight); at
// width 16 it spills 72 bytes.  Width 2 takes three CTAs (80 registers): four spilled
// 116 bytes in its inner loop.  With them and the item's channels in shared memory
// (ab)*c|a*b* on the gather alone, n = 8192, went from 1.43 to 1.28 ms with 48 edges a
// vertex, from 2.03 to 1.78 with 100.
template <int VPL, bool NT>
struct GatherCtas {
    static constexpr int value = NT ? GatherOcc<VPL>::value : VPL >= 8 ? 2 : VPL == 2 ? 3 : GatherOcc<VPL>::value;
};

// Scheduling.  Narrow rows: one CTA per live item (the grid covers every
// item of the class; CTAs past the live count exit at once).  Wide rows of
// the general variant (one warp per row, VPL >= 4, at most one or two CTAs
// per SM for the shared-memory ring): the grid is persistent and each warp
// takes units of kGatherParts row ranges of a live item from a counter of the
// pass (ExecTables::g_next, zeroed by the loop control), so that a warp held
// by a row with thousands of new edges leaves the other warps of its CTA free
// to take more work instead of waiting for it at a barrier.
template <int VPL, bool NT>
struct GatherDyn {
    static constexpr bool on = NT && VPL >= 4;
};
// Units per item: measured on Dyck-4 (AUTO / bit-packed, ms) at n = 65536:
// 4: 1545 / 2707, 8: 1543 / 2589, 16: 1560 / 2564, 32: 1585 / 2531; at
// n = 16384: 4: 58 / 84, 8: 50 / 71, 32: 50 / 62.  (Leaving rows with more
// than 256-4096 bits to enumerate to a second launch split over 16 warps
// gained 1-2% in AUTO and cost 10-20% bit-packed: not kept.)
constexpr uint32_t kGatherParts = 8;
constexpr uint32_t kStrideWaves = 8;  // launch_gather: waves of resident CTAs at most

// Row `at` of a CSR item, source k of more than kHubEdges edges, by the whole CTA: its warps
// take 32 edges in turn and merge what they found with atomics.  Such a row's one warp was
// the pass, bound by the latency of a source row after another, and the widest rows, which
// gave up half their loads in flight for a second CTA, took 2.5 times what they had taken before.
// a+ on the gather, a path of 200 vertices and four with edges to all others: n = 8000 26.7 ->
// 6.6 ms, 30000 105 -> 21, 60000 463 -> 63.  Not inlined, and the main loop only leaves the
// row's source out: inlined, or listed before the loop, sparse graphs lost up to 7% to
// spills and extra loads.  As it is they lost 1.5% (the regular query at n = 30011), so graphs
// without such rows take a variant without it (GraphDev::hub_rows).
constexpr uint32_t kHubEdges = 512, kHubs = 64;  // (kHubs: listed by an item at most)
template <int VPL>
__device__ __noinline__ void gather_hub(const GItem *__restrict__ item, const SrcDesc *__restrict__ srcs, uint32_t at,
                                        uint32_t k, unsigned long long *s_changed, unsigned long long *s_ors) {
    const GItem &it = *item;
    const QCtl *c = it.ctl;
    const uint32_t row = it.row0 + at;
    const uint32_t g = c->g, iter = c->iter, mode = c->mode, g0 = c->g_iter_start, dmask = c->dense_mask;
    const int lane = threadIdx.x & 31, lpr = (int)it.lpr, grp = lane / lpr, gl = lane % lpr;
    const unsigned gmask = (lpr == 32 ? FULLMASK : ((1u << lpr) - 1u)) << (grp * lpr);
    const uint32_t W = it.W, cv0 = c->col_v0, cv1 = min(c->col_v1, W / 2u);
    uint64_t *const out = it.out + (size_t)row * W;
    uint4 acc[VPL];
#pragma unroll
    for (int j = 0; j < VPL; ++j) acc[j] = make_uint4(0, 0, 0, 0);
    uint32_t ors = 0u;
    bool ch = false;
    const SrcDesc &d = srcs[it.src0 + k];
    const uint32_t chans = src_channels<false>(d, mode, iter, g, g0, dmask);
    const uint32_t *const col = d.csr_col, *const rstamp = d.rstamp;
    const uint64_t *const rblk = d.rblk;
    const uint32_t e1 = d.csr_off[row + 1];
    const bool ident = (chans & 1u) && d.ident;
    // (one channel a pass: new edges only in iteration 1, whole rows then)
    const uint32_t thr = (chans & 1u) ? 0u : (chans & 2u) ? g0 : g - 1u;
    for (uint32_t b = d.csr_off[row] + (threadIdx.x & ~31u); b < e1; b += 256u) {
        const bool has = b + (uint32_t)lane < e1;
        const uint32_t yl = has ? col[b + (uint32_t)lane] : 0u;
        if (ident && has && (yl >> 7) >= cv0 && (yl >> 7) < cv1) {
            unsigned int *const w = reinterpret_cast<unsigned int *>(out) + (yl >> 5);
            const unsigned int bit = 1u << (yl & 31u);
            if (!(*w & bit) && !(atomicOr(w, bit) & bit)) ch = true;
        }
        if (!rblk) continue;
        const unsigned bal = __ballot_sync(FULLMASK, has && (thr == 0u || rstamp[yl] >= thr));
        unsigned mine = (bal & gmask) >> (grp * lpr);
        constexpr int U = VPL >= 8 ? 1 : VPL == 4 ? 2 : 4, J = VPL < 8 ? VPL : 8;
        while (__any_sync(FULLMASK, mine != 0u)) {
            const uint4 *r[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const bool h = mine != 0u;
                const uint32_t y = __shfl_sync(FULLMASK, yl, h ? __ffs(mine) - 1 : 0, lpr);
                r[u] = h ? reinterpret_cast<const uint4 *>(rblk + (size_t)y * W) : nullptr;
                if (h && gl == 0) ++ors;
                mine &= mine - 1u;
            }
#pragma unroll
            for (int j0 = 0; j0 < VPL; j0 += J) {
                uint4 a[U][J];
#pragma unroll
                for (int u = 0; u < U; ++u)
#pragma unroll
                    for (int j = 0; j < J; ++j) {
                        const uint32_t v = (uint32_t)gl + (uint32_t)(j0 + j) * lpr;
                        a[u][j] = r[u] && v >= cv0 && v < cv1 ? r[u][v] : make_uint4(0, 0, 0, 0);
                    }
#pragma unroll
                for (int u = 0; u < U; ++u)
#pragma unroll
                    for (int j = 0; j < J; ++j) or4(acc[j0 + j], a[u][j]);
            }
        }
    }
    unsigned long long *const o = reinterpret_cast<unsigned long long *>(out);
#pragma unroll
    for (int j = 0; j < VPL; ++j) {
        if (!nz4(acc[j])) continue;
        const uint32_t v = (uint32_t)gl + (uint32_t)j * lpr;
        const unsigned long long lo = ((unsigned long long)acc[j].y << 32) | acc[j].x;
        const unsigned long long hi = ((unsigned long long)acc[j].w << 32) | acc[j].z;
        if ((lo & ~o[2u * v]) && (lo & ~atomicOr(o + 2u * v, lo))) ch = true;
        if ((hi & ~o[2u * v + 1u]) && (hi & ~atomicOr(o + 2u * v + 1u, hi))) ch = true;
    }
    // (a pass counts the row once)
    if (__any_sync(FULLMASK, ch) && lane == 0 && atomicExch(it.out_stamp + row, g) != g) atomicAdd(s_changed, 1ull);
    if (ors) atomicAdd(s_ors, (unsigned long long)ors);
}

template <int VPL, bool NT, bool HUB>
__global__ void __launch_bounds__(256, GatherCtas<VPL, NT>::value)
    k_gather(const GItem *__restrict__ items, const SrcDesc *__restrict__ srcs, ExecTables T, int cls) {
    constexpr bool kDyn = GatherDyn<VPL, NT>::on;
    __shared__ unsigned long long s_changed, s_ors;
    // rows of the item with work: their bits, then the list (an item has at most 1024 rows)
    __shared__ uint32_t s_rowbits[32];
    __shared__ uint16_t s_rows[1024];
    __shared__ uint8_t s_chans[16];  // channels of the item's first sources (one CTA per item)
    __shared__ uint32_t s_hubs[kHubs], s_nhubs;  // HUB: rows (k << 10 | row) left to gather_hub
    // general variant: per-warp ring of source rows loaded with cp.async
    extern __shared__ uint4 s_ring[];
    constexpr int P = GatherRing<VPL>::depth;
    uint4 *ring = s_ring + (size_t)(threadIdx.x >> 5) * GatherRing<VPL>::slots * 32 * VPL;
    const uint32_t total = T.g_total[cls];
    uint32_t li = blockIdx.x;
    if (kDyn) li = 0u;
    for (bool first = true;; first = false) {
    uint32_t part = 0u;
    if constexpr (kDyn) {
        uint32_t u = 0u;
        if ((threadIdx.x & 31) == 0) u = atomicAdd(T.g_next + cls, 1u);
        u = __shfl_sync(FULLMASK, u, 0);
        if (u >= total * kGatherParts) break;
        li = u / kGatherParts;
        part = u % kGatherParts;
    } else {
        if (!first) li += gridDim.x;
        if (li >= total) break;
    }
    const GItem it = items[live_item(T.g_pre[cls], T.g_beg[cls], T.nq, li)];
    const QCtl *c = it.ctl;
    if (c->phase != kPhaseRun || c->level != it.level) continue;
    const uint32_t g = c->g, iter = c->iter, mode = c->mode, g0 = c->g_iter_start, dmask = c->dense_mask;

    if constexpr (kDyn) {
        bool act = false;
        for (uint32_t k = threadIdx.x & 31; k < it.nsrc; k += 32u)
            act |= src_channels<NT>(srcs[it.src0 + k], mode, iter, g, g0, dmask) != 0u;
        if (!__any_sync(FULLMASK, act)) continue;
    } else {
        if (it.rmask) {  // multiple-source runs: no row of the item is reached
            const uint32_t w = (it.row0 >> 6) + threadIdx.x;
            if (!__syncthreads_or(w * 64u < it.row1 && it.rmask[w] != 0ull)) continue;
        }
        int act = 0;
        for (uint32_t k = threadIdx.x; k < it.nsrc; k += blockDim.x)
            act |= src_channels<NT>(srcs[it.src0 + k], mode, iter, g, g0, dmask) != 0u;
        if (!__syncthreads_or(act)) continue;

        for (uint32_t k = threadIdx.x; k < it.nsrc && k < 16u; k += blockDim.x)
            s_chans[k] = (uint8_t)src_channels<NT>(srcs[it.src0 + k], mode, iter, g, g0, dmask);
        if (threadIdx.x == 0) { s_changed = 0; s_ors = 0; s_nhubs = 0u; }
        if (threadIdx.x < 32u) s_rowbits[threadIdx.x] = 0u;
        __syncthreads();
    }

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lpr = (int)it.lpr, grp = lane / lpr, gl = lane % lpr, rpw = 32 / lpr;
    const unsigned gmask = (lpr == 32 ? FULLMASK : ((1u << lpr) - 1u)) << (grp * lpr);
    const uint32_t W = it.W, nvec = W / 2;
    // the columns of the output this rank computes (column sharding; else
    // all): closure rows are read and written only there
    // (bit j of winmask: the lane's vector j lies in [col_v0, col_v1) and in the row)
    uint32_t winmask = 0u;
    {
        const uint32_t cv0 = c->col_v0, cv1 = min(c->col_v1, nvec);
#pragma unroll
        for (int j = 0; j < VPL; ++j) {
            const uint32_t v = (uint32_t)gl + (uint32_t)j * lpr;
            if (v >= cv0 && v < cv1) winmask |= 1u << j;
        }
    }
    // column slice of the nonterminal adjacency (general variant, rows of 2+
    // vectors per lane: the engine slices only rows of 8192+ bits)
    constexpr bool kSlices = NT && VPL >= 2;
    const bool slices_on = kSlices && (dmask & it.nt_boxes) != 0u;  // a box the block reads is dense
    uint32_t sv0 = kSlices ? (it.slice & 0xFFFFu) : 0u, sv1 = kSlices ? (it.slice >> 16) : nvec;
    if (kSlices && !slices_on) {
        if (sv0 != 0u) continue;  // the first slice covers every column
        sv1 = nvec;
    }
    const bool sliced = slices_on && (sv0 != 0u || sv1 < nvec);
    uint32_t my_changed = 0, my_ors = 0;
    // channels of the item's first 16 sources in this pass: the same for every row.
    // A warp unit packs them into a register pair (4 bits each), a CTA has them in s_chans.
    unsigned long long chpack = 0ull;
    if constexpr (kDyn)
        for (uint32_t k = 0; k < it.nsrc && k < 16u; ++k)
            chpack |= (unsigned long long)src_channels<NT>(srcs[it.src0 + k], mode, iter, g, g0, dmask) << (4u * k);
    auto chans_of = [&](uint32_t k) -> uint32_t {
        if (k >= 16u) return src_channels<NT>(srcs[it.src0 + k], mode, iter, g, g0, dmask);
        return kDyn ? (uint32_t)(chpack >> (4u * k)) & 15u : (uint32_t)s_chans[k];
    };
    auto wanted = [&](uint32_t r) { return !it.rmask || ((it.rmask[r >> 6] >> (r & 63u)) & 1ull) != 0ull; };

    // Rows with work, found a lane a row.  Dynamic units: the warp tests its
    // range of rows 32 at a time and takes them in turn.  One CTA per item: up to
    // four threads a row share its sources, and the rows found are listed for the
    // groups of all warps.
    uint32_t r_next = 0u, r_end = 0u, nrows = 0u;
    unsigned r_mask = 0u;  // rows of the window [r_next - 32, r_next) still to take
    if constexpr (kDyn) {
        const uint32_t per = (it.row1 - it.row0 + kGatherParts - 1u) / kGatherParts;
        r_next = it.row0 + part * per;
        r_end = min(it.row1, r_next + per);
    } else {
        const uint32_t nr = it.row1 - it.row0;
        const uint32_t step = nr > 128u ? 256u : nr > 64u ? 128u : 64u, parts = 256u / step;
        for (uint32_t r0 = 0; r0 < nr; r0 += step) {
            const uint32_t r = r0 + threadIdx.x % step;
            bool has = false;
            if (r < nr && wanted(it.row0 + r))
                for (uint32_t k = threadIdx.x / step; k < it.nsrc && !has; k += parts) {
                    const uint32_t chans = chans_of(k);
                    has = chans != 0u && row_has_work<NT>(srcs[it.src0 + k], chans, it.row0 + r, iter, g, g0);
                }
            const unsigned bal = __ballot_sync(FULLMASK, has);
            if (lane == 0 && bal) atomicOr(&s_rowbits[r >> 5], bal);
        }
        __syncthreads();
        const uint32_t nw = (nr + 31u) >> 5;
        for (uint32_t r = threadIdx.x; r < nr; r += 256u) {
            const uint32_t bits = s_rowbits[r >> 5];
            if (!((bits >> (r & 31u)) & 1u)) continue;
            uint32_t pos = (uint32_t)__popc(bits & ((1u << (r & 31u)) - 1u));
            for (uint32_t w = 0; w < (r >> 5); ++w) pos += (uint32_t)__popc(s_rowbits[w]);
            s_rows[pos] = (uint16_t)r;
        }
        for (uint32_t w = 0; w < nw; ++w) nrows += (uint32_t)__popc(s_rowbits[w]);
        __syncthreads();
    }
    for (uint32_t i0 = (uint32_t)(warp * rpw);; i0 += 8u * rpw) {
        uint32_t row;
        bool valid;
        if constexpr (kDyn) {
            while (!r_mask && r_next < r_end) {
                const uint32_t r = r_next + (uint32_t)lane;
                bool has = false;
                if (r < r_end && wanted(r))
                    for (uint32_t k = 0; k < it.nsrc && !has; ++k) {
                        const uint32_t chans = chans_of(k);
                        has = chans != 0u && row_has_work<NT>(srcs[it.src0 + k], chans, r, iter, g, g0);
                    }
                r_mask = __ballot_sync(FULLMASK, has);
                r_next += 32u;
            }
            if (!r_mask) break;
            row = r_next - 32u + (uint32_t)(__ffs(r_mask) - 1);
            r_mask &= r_mask - 1u;
            valid = true;
        } else {
            if (i0 >= nrows) break;
            valid = i0 + (uint32_t)grp < nrows;
            row = it.row0 + (valid ? s_rows[i0 + (uint32_t)grp] : 0u);
        }
        uint4 acc[VPL];
#pragma unroll
        for (int j = 0; j < VPL; ++j) acc[j] = make_uint4(0, 0, 0, 0);

        for (uint32_t k = 0; k < it.nsrc; ++k) {
            const uint32_t chans = chans_of(k);
            if (!chans) continue;  // the source takes no part in this pass
            const SrcDesc d = srcs[it.src0 + k];
            for (uint32_t cbit = 1u; cbit <= 4u; cbit <<= 1) {
                if (!(chans & cbit)) continue;
                const bool new_edges = cbit == 1u;
                // closure rows read (none for new edges whose rows the tiles OR:
                // only the product edges themselves are left here)
                const uint64_t *const rblk = (NT && new_edges && (chans & 8u)) ? nullptr : d.rblk;
                const bool use_ident = new_edges && d.ident;
                if (!use_ident && rblk == nullptr) continue;
                // a source row takes part when its stamp is >= thr; new edges
                // take whole rows: those ever written and, where channel 2
                // reads the rows changed in this iteration over all edges,
                // not those (nt_lo <= stamp < nt_hi, nonterminal sources)
                const uint32_t thr = new_edges ? 0u : (cbit == 2u ? g0 : g - 1u);
                const uint32_t nt_lo = new_edges ? 1u : thr, nt_hi = (new_edges && !d.same_level) ? g0 : 0xFFFFFFFFu;

                // Every lane proposes one candidate edge (x, y) of its group's
                // row (y_l, has_l).  The group keeps those whose source row is
                // dirty, then ORs their rows U at a time: all U rows are loaded
                // before any is combined, so several 128-bit loads per lane are
                // in flight.
                constexpr int U = VPL >= 4 ? 1 : 4 / VPL;
                const bool bitrow = NT && d.csr_off == nullptr;
                auto take_batch = [&](uint32_t y_l, bool has_l) {
                    bool keep = has_l;
                    if (has_l && rblk != nullptr) {
                        if (bitrow) {
                            const uint32_t sy = d.rstamp[y_l];
                            keep = sy >= nt_lo && sy < nt_hi;
                        } else {
                            keep = thr == 0u || d.rstamp[y_l] >= thr;
                        }
                    }
                    if constexpr (NT) {
                        if (d.pure_n && !use_ident) {
                            if (lpr == 32) {  // one row per warp: the bitmap in the warp's first slot
                                pure_bitmap_set(d, y_l, keep, ring);
                                return;
                            }
                            or_pure_rows<VPL>(acc, d, y_l, keep, lpr, gl, grp, gmask);
                            return;
                        }
                        if (GatherRing<VPL>::on && rblk && !d.pure_n) {
                            // Rows through the warp's shared-memory ring, P in
                            // flight: row i is copied into slot i % P by
                            // cp.async (each lane its own 16-byte pieces, so a
                            // lane reads back only what it copied) and ORed
                            // once P - 1 later rows have been issued.
                            const unsigned bal = __ballot_sync(FULLMASK, keep);
                            unsigned mine = (bal & gmask) >> (grp * lpr);
                            uint32_t issued = 0, done = 0, vmask = 0;
                            auto or_slot = [&](uint32_t sidx) {
                                const uint4 *sl = ring + sidx * 32u * VPL;
#pragma unroll
                                for (int j = 0; j < VPL; ++j) or4(acc[j], sl[j * 32 + lane]);
                            };
                            while (__any_sync(FULLMASK, mine != 0u)) {
                                const bool h = mine != 0u;
                                const int pl = h ? __ffs(mine) - 1 : 0;
                                if (h) mine &= mine - 1u;
                                const uint32_t y = __shfl_sync(FULLMASK, y_l, pl, lpr);
                                if (use_ident && h) set_row_bit<VPL>(acc, y, lpr, gl);
                                const uint32_t sidx = issued % (uint32_t)P;
                                if (h) {
                                    uint4 *sl = ring + sidx * 32u * VPL;
                                    const uint4 *r = reinterpret_cast<const uint4 *>(rblk + (size_t)y * W);
#pragma unroll
                                    for (int j = 0; j < VPL; ++j) {
                                        const uint32_t v = (uint32_t)gl + (uint32_t)j * lpr;
                                        cp_async16(&sl[j * 32 + lane], r + (((winmask >> j) & 1u) ? v : 0u), ((winmask >> j) & 1u));
                                    }
                                    if (gl == 0) ++my_ors;
                                    vmask |= 1u << sidx;
                                } else {
                                    vmask &= ~(1u << sidx);
                                }
                                cp_async_commit();
                                ++issued;
                                if (issued - done == (uint32_t)P) {
                                    cp_async_wait<P - 1>();
                                    const uint32_t ds = done % (uint32_t)P;
                                    if ((vmask >> ds) & 1u) or_slot(ds);
                                    ++done;
                                }
                            }
                            cp_async_wait<0>();
                            for (; done < issued; ++done) {
                                const uint32_t ds = done % (uint32_t)P;
                                if ((vmask >> ds) & 1u) or_slot(ds);
                            }
                            return;
                        }
                    }
                    const unsigned bal = __ballot_sync(FULLMASK, keep);
                    unsigned mine = (bal & gmask) >> (grp * lpr);
                    while (__any_sync(FULLMASK, mine != 0u)) {
                        uint32_t ys[U];
                        bool hs[U];
#pragma unroll
                        for (int u = 0; u < U; ++u) {
                            hs[u] = mine != 0u;
                            const int p = hs[u] ? __ffs(mine) - 1 : 0;
                            if (hs[u]) mine &= mine - 1u;
                            ys[u] = __shfl_sync(FULLMASK, y_l, p, lpr);
                        }
                        if (use_ident) {
#pragma unroll
                            for (int u = 0; u < U; ++u) {
                                if (!hs[u]) continue;
                                const uint32_t v = ys[u] >> 7;
                                if ((int)(v % lpr) == gl) {
                                    const int j = (int)(v / lpr);
#pragma unroll
                                    for (int jj = 0; jj < VPL; ++jj)
                                        if (jj == j) setbit4(acc[jj], ys[u] & 127u);
                                }
                            }
                        }
                        if constexpr (!NT && VPL > 8) {
                            if (rblk && hs[0]) {
                                const uint4 *r = reinterpret_cast<const uint4 *>(rblk + (size_t)ys[0] * W);
#pragma unroll
                                for (int j0 = 0; j0 < VPL; j0 += 8) {
                                    uint4 a[8];
#pragma unroll
                                    for (int j = 0; j < 8; ++j)
                                        a[j] = ((winmask >> (j0 + j)) & 1u) ? r[(uint32_t)gl + (uint32_t)(j0 + j) * lpr]
                                                                            : make_uint4(0, 0, 0, 0);
#pragma unroll
                                    for (int j = 0; j < 8; ++j) or4(acc[j0 + j], a[j]);
                                }
                                if (gl == 0) ++my_ors;
                            }
                        } else if (rblk && (!NT || !d.pure_n)) {
                            uint4 rv[U][VPL];
#pragma unroll
                            for (int u = 0; u < U; ++u) {
                                const uint4 *r = reinterpret_cast<const uint4 *>(rblk + (size_t)ys[u] * W);
#pragma unroll
                                for (int j = 0; j < VPL; ++j) {
                                    const uint32_t v = (uint32_t)gl + (uint32_t)j * lpr;
                                    rv[u][j] = (hs[u] && ((winmask >> j) & 1u)) ? r[v] : make_uint4(0, 0, 0, 0);
                                }
                            }
#pragma unroll
                            for (int u = 0; u < U; ++u) {
#pragma unroll
                                for (int j = 0; j < VPL; ++j) or4(acc[j], rv[u][j]);
                                if (gl == 0 && hs[u]) ++my_ors;
                            }
                        }
                    }
                };

                if (d.csr_off) {
                    if (sv0 != 0u) continue;  // CSR sources belong to the first slice
                    const uint32_t e0 = valid ? d.csr_off[row] : 0u, e1 = valid ? d.csr_off[row + 1] : 0u;
                    uint32_t cnt = e1 - e0, maxcnt = __reduce_max_sync(FULLMASK, cnt);
                    if (maxcnt <= 8u && (!NT || !d.pure_n)) {
                        // short adjacency rows (the common case on sparse
                        // graphs): no ballot; edges two at a time so that the
                        // column, stamp and row loads of both are in flight
                        auto ident_bit = [&](uint32_t y) {
                            const uint32_t v = y >> 7;
                            if ((int)(v % lpr) == gl) {
                                const int j = (int)(v / lpr);
#pragma unroll
                                for (int jj = 0; jj < VPL; ++jj)
                                    if (jj == j) setbit4(acc[jj], y & 127u);
                            }
                        };
                        if constexpr (!NT && VPL >= 8) {
                            // (a warp owns the row: e0, e1 and the stamps are the same in every lane)
                            for (uint32_t e = e0; e < e1; ++e) {
                                const uint32_t y = d.csr_col[e];
                                if (use_ident) ident_bit(y);
                                if (!rblk || (thr && d.rstamp[y] < thr)) continue;
                                const uint4 *r = reinterpret_cast<const uint4 *>(rblk + (size_t)y * W);
                                // eight vectors in flight (sixteen would spill at two CTAs)
#pragma unroll
                                for (int j0 = 0; j0 < VPL; j0 += 8) {
                                    uint4 a[8];
#pragma unroll
                                    for (int j = 0; j < 8; ++j)
                                        a[j] = ((winmask >> (j0 + j)) & 1u) ? r[(uint32_t)gl + (uint32_t)(j0 + j) * lpr]
                                                                            : make_uint4(0, 0, 0, 0);
#pragma unroll
                                    for (int j = 0; j < 8; ++j) or4(acc[j0 + j], a[j]);
                                }
                                if (gl == 0) ++my_ors;
                            }
                        } else
                        for (uint32_t e = e0; e < e1; e += 2) {
                            const bool two = e + 1 < e1;
                            const uint32_t y0 = d.csr_col[e], y1 = two ? d.csr_col[e + 1] : 0u;
                            if (use_ident) {
                                ident_bit(y0);
                                if (two) ident_bit(y1);
                            }
                            if (rblk) {
                                const bool k0 = !thr || d.rstamp[y0] >= thr;
                                const bool k1 = two && (!thr || d.rstamp[y1] >= thr);
                                const uint4 *r0 = reinterpret_cast<const uint4 *>(rblk + (size_t)y0 * W);
                                const uint4 *r1 = reinterpret_cast<const uint4 *>(rblk + (size_t)y1 * W);
                                uint4 a0[VPL], a1[VPL];
#pragma unroll
                                for (int j = 0; j < VPL; ++j) {
                                    const uint32_t v = (uint32_t)gl + (uint32_t)j * lpr;
                                    a0[j] = (k0 && ((winmask >> j) & 1u)) ? r0[v] : make_uint4(0, 0, 0, 0);
                                    a1[j] = (k1 && ((winmask >> j) & 1u)) ? r1[v] : make_uint4(0, 0, 0, 0);
                                }
#pragma unroll
                                for (int j = 0; j < VPL; ++j) {
                                    or4(acc[j], a0[j]);
                                    or4(acc[j], a1[j]);
                                }
                                if (gl == 0) my_ors += (k0 ? 1u : 0u) + (k1 ? 1u : 0u);
                            }
                        }
                    } else {
                        if (HUB && maxcnt > kHubEdges) {  // (uniform over the warp)
                            bool listed = false;
                            if (cnt > kHubEdges && gl == 0) {
                                const uint32_t h = atomicAdd(&s_nhubs, 1u);
                                listed = h < kHubs;
                                if (listed) s_hubs[h] = (k << 10) | (row - it.row0);
                            }
                            if (__shfl_sync(FULLMASK, (int)listed, 0, lpr)) cnt = 0u;
                            maxcnt = __reduce_max_sync(FULLMASK, cnt);
                        }
                        for (uint32_t base = 0; base < maxcnt; base += (uint32_t)lpr) {
                            const uint32_t k2 = base + (uint32_t)gl;
                            const bool has = k2 < cnt;
                            const uint32_t y = has ? d.csr_col[e0 + k2] : 0u;
                            take_batch(y, has);
                        }
                    }
                } else if constexpr (NT) {
                    const uint64_t *adj;
                    bool rowok;
                    if (new_edges) { adj = d.nt_new; rowok = valid && d.nt_new_it[row] == iter; }
                    else { adj = d.nt_all; rowok = valid; }
                    // no row of the warp has edges of this channel: nothing to enumerate
                    if (!__any_sync(FULLMASK, rowok)) continue;
                    uint4 a[VPL];
#pragma unroll
                    for (int j = 0; j < VPL; ++j) {
                        const uint32_t v = (uint32_t)gl + (uint32_t)j * lpr;
                        a[j] = (rowok && v >= sv0 && v < sv1 && v < nvec)
                                   ? reinterpret_cast<const uint4 *>(adj + (size_t)row * W)[v]
                                   : make_uint4(0, 0, 0, 0);
                    }
                    if (d.pure_n) {
                        // a row y of a pure-terminal block is empty unless y
                        // has an edge of one of its labels
#pragma unroll
                        for (int j = 0; j < VPL; ++j) {
                            const uint32_t v = (uint32_t)gl + (uint32_t)j * lpr;
                            if (v >= nvec) continue;
                            uint4 m = reinterpret_cast<const uint4 *>(d.pure_mask[0])[v];
                            if (d.pure_n > 1) or4(m, reinterpret_cast<const uint4 *>(d.pure_mask[1])[v]);
                            a[j] = make_uint4(a[j].x & m.x, a[j].y & m.y, a[j].z & m.z, a[j].w & m.w);
                        }
                    }
                    if (use_ident) {
                        // product edges into t itself: bit y of the adjacency
                        // row is bit y of the output row, and the lane that
                        // holds an adjacency vector holds the same vector of
                        // the output row -- no enumeration
#pragma unroll
                        for (int j = 0; j < VPL; ++j) or4(acc[j], a[j]);
                        if (rblk == nullptr) continue;
                    }
                    // a pure-terminal block read by a warp-owned row: the
                    // columns found go to the row's shared-memory bitmap
                    const bool pure_bm = d.pure_n && !use_ident && lpr == 32;
                    if (pure_bm) pure_bitmap_clear<VPL>(nvec, lane, ring);
                    // Each lane proposes the lowest set bit of its part of the
                    // adjacency row per step (ballot/ffs enumeration).
                    while (true) {
                        bool has = false;
                        uint32_t y = 0u;
#pragma unroll
                        for (int j = 0; j < VPL; ++j) {
                            if (!has && nz4(a[j])) {
                                const int bit = lowbit4(a[j], true);
                                y = ((uint32_t)gl + (uint32_t)j * lpr) * 128u + (uint32_t)bit;
                                has = true;
                            }
                        }
                        if (!__any_sync(FULLMASK, has)) break;
                        take_batch(y, has);
                    }
                    if (pure_bm) pure_bitmap_or<VPL>(acc, nvec, lane, ring);
                }
            }
        }

        bool ch = false;
        if (valid && sliced) {
            // other slices write the same rows: merge with atomics
            unsigned long long *o = reinterpret_cast<unsigned long long *>(it.out + (size_t)row * W);
#pragma unroll
            for (int j = 0; j < VPL; ++j) {
                const uint32_t v = (uint32_t)gl + (uint32_t)j * lpr;
                if (((winmask >> j) & 1u) && nz4(acc[j])) {
                    const unsigned long long lo = ((unsigned long long)acc[j].y << 32) | acc[j].x;
                    const unsigned long long hi = ((unsigned long long)acc[j].w << 32) | acc[j].z;
                    if (lo && (lo & ~atomicOr(o + 2u * v, lo))) ch = true;
                    if (hi && (hi & ~atomicOr(o + 2u * v + 1u, hi))) ch = true;
                }
            }
        } else if (valid) {
            uint4 *o = reinterpret_cast<uint4 *>(it.out + (size_t)row * W);
#pragma unroll
            for (int j = 0; j < VPL; ++j) {
                const uint32_t v = (uint32_t)gl + (uint32_t)j * lpr;
                if (((winmask >> j) & 1u) && nz4(acc[j])) {
                    const uint4 old = o[v];
                    const uint4 nw = andnot4(acc[j], old);
                    if (nz4(nw)) {
                        uint4 m = old;
                        or4(m, nw);
                        o[v] = m;
                        ch = true;
                    }
                }
            }
        }
        const unsigned chb = __ballot_sync(FULLMASK, ch);
        if ((chb & gmask) && gl == 0) {
            it.out_stamp[row] = g;
            ++my_changed;
        }
    }
    if constexpr (kDyn) {
        const uint32_t wc = __reduce_add_sync(FULLMASK, my_changed), wo = __reduce_add_sync(FULLMASK, my_ors);
        if (lane == 0) {
            QCtl *cw = it.ctl;
            if (wc) {
                *it.out_last = g;
                atomicAdd(&cw->changed_rows, (unsigned long long)wc);
            }
            if (wo) atomicAdd(&cw->row_ors, (unsigned long long)wo);
        }
    } else {
        if (my_changed) atomicAdd(&s_changed, (unsigned long long)my_changed);
        if (my_ors) atomicAdd(&s_ors, (unsigned long long)my_ors);
        __syncthreads();
        if (HUB && s_nhubs) {
            for (uint32_t h = 0; h < min(s_nhubs, kHubs); ++h)
                gather_hub<VPL>(items + live_item(T.g_pre[cls], T.g_beg[cls], T.nq, li), srcs, s_hubs[h] & 1023u,
                                s_hubs[h] >> 10, &s_changed, &s_ors);
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            QCtl *cw = it.ctl;
            if (s_changed) {
                *it.out_last = g;
                atomicAdd(&cw->changed_rows, s_changed);
            }
            if (s_ors) atomicAdd(&cw->row_ors, s_ors);
        }
        __syncthreads();
    }
    }
}

// --------------------------------------------------------------------------
// Closure pass of the blocks that read no closure row (kExpandNarrow / Wide):
// every source is a product edge into t itself (a terminal's CSR row or a
// nonterminal's adjacency row) or a nonterminal edge into a pure-terminal
// block, whose rows are read as CSR rows (SrcDesc::pure_n).  On Dyck-4 these are
// C[p, F], C[x_i, y_i], C[x_i, F] and C[q0, p]: every new S-edge (x, y) is
// expanded by the c_i edges of y, four times.
//
// Bound by the latency of that chain (adjacency word -> CSR offsets -> column
// -> shared-memory atomic) and by uneven rows (most have no new edge, hubs have
// tens of thousands).  So: no registers or shared memory for closure rows, which
// leaves 48 warps per SM; the item's rows with work are listed first, 256 marks
// at a time; a row is expanded by a whole CTA (rows of more than
// kExpandNarrowW words) or by a warp that takes rows from the list, each
// thread on its own adjacency words, into a row-sized shared-memory bitmap that is
// merged into the output row at the end.  As part of k_gather (one warp per row,
// 8 warps per SM beside the closure-row ring) this took 110 of the 190 ms of
// gather of Dyck-4 at n = 65536; the query went from 303 to 233 ms.
// --------------------------------------------------------------------------
// CTAs per SM.  48 warps leave 40 registers a thread, where the wide and the narrow
// variant spill 44 and 48 bytes (the heaviest launch of Dyck-4 at n = 16384, 0.24 ms:
// 1.35 million spill instructions of warps, 67% of warps active).  Fewer CTAs without
// spills have not been timed.
constexpr int kExpandOcc = 6;
constexpr uint32_t kExpandParts = 4;
template <bool WIDE>
__global__ void __launch_bounds__(256, kExpandOcc)
    k_expand(const GItem *__restrict__ items, const SrcDesc *__restrict__ srcs, ExecTables T, int cls) {
    extern __shared__ unsigned long long s_bitmap[];  // WIDE: one row; else one row per warp
    __shared__ uint16_t s_rows[1024];                 // (an item has at most 1024 rows)
    __shared__ uint32_t s_nrows, s_take, s_changed, s_unit;
    __shared__ uint16_t s_list[8][1024];              // per warp: columns (below 65536) to expand
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    uint16_t *const list = s_list[warp];
    const uint32_t t0 = WIDE ? tid : lane;            // this thread's place in its row's group
    constexpr uint32_t TPR = WIDE ? 256u : 32u;
    // units: a wide item's rows in kExpandParts ranges, narrow items whole; the
    // first one by block index, the others from the pass's counter (a few units
    // hold most of a pass's work)
    constexpr uint32_t kParts = WIDE ? kExpandParts : 1u;
    const uint32_t total = T.g_total[cls] * kParts;
    for (uint32_t u = blockIdx.x; u < total;) {
        const uint32_t li = u / kParts, part = u % kParts;
        __syncthreads();  // (s_unit of the last round has been read)
        if (tid == 0) s_unit = gridDim.x + atomicAdd(T.g_next + cls, 1u);
        __syncthreads();
        u = s_unit;
        const GItem &it = items[live_item(T.g_pre[cls], T.g_beg[cls], T.nq, li)];
        QCtl *const c = it.ctl;
        if (c->phase != kPhaseRun || c->level != it.level) continue;  // (uniform)
        const uint32_t g = c->g, iter = c->iter, mode = c->mode, g0 = c->g_iter_start, W = it.W;
        const uint32_t src0 = it.src0, nsrc = it.nsrc;
        const uint32_t per = (it.row1 - it.row0 + kParts - 1u) / kParts;
        const uint32_t row0 = it.row0 + part * per, row1 = min(it.row1, row0 + per);
        int act = 0;
        for (uint32_t k = tid; k < nsrc; k += 256u) act |= src_channels<true>(srcs[src0 + k], mode, iter, g, g0, 0u) != 0u;
        if (!__syncthreads_or(act)) continue;
        if (tid == 0) { s_nrows = 0u; s_take = 0u; s_changed = 0u; }
        __syncthreads();
        // rows with an edge of a source that takes part
        for (uint32_t r = row0 + tid; r - tid < row1; r += 256u) {
            bool has = false;
            if (r < row1 && (!it.rmask || ((it.rmask[r >> 6] >> (r & 63u)) & 1ull))) {
                for (uint32_t k = 0; k < nsrc && !has; ++k) {
                    const SrcDesc &d = srcs[src0 + k];
                    const uint32_t ch = src_channels<true>(d, mode, iter, g, g0, 0u);
                    if (!ch) continue;
                    if (d.csr_off) has = d.csr_off[r + 1] > d.csr_off[r];
                    else has = (ch & 6u) ? d.nt_new_it[r] != 0u : d.nt_new_it[r] == iter;  // (0: the row has no edge)
                }
            }
            const unsigned bal = __ballot_sync(FULLMASK, has);
            uint32_t base = 0u;
            if (lane == 0u && bal) base = atomicAdd(&s_nrows, (uint32_t)__popc(bal));
            base = __shfl_sync(FULLMASK, base, 0);
            if (has) s_rows[base + (uint32_t)__popc(bal & ((1u << lane) - 1u))] = (uint16_t)(r - row0);
        }
        __syncthreads();
        const uint32_t nrows = s_nrows;
        unsigned long long *const bm = s_bitmap + (WIDE ? 0u : warp * W);
        unsigned int *const bm32 = reinterpret_cast<unsigned int *>(bm);
        const uint32_t w0 = c->col_v0 * 2u, w1 = min(c->col_v1, W / 2u) * 2u;  // this rank's columns (all unless sharded)
        uint32_t my_changed = 0u;
        for (uint32_t i = 0;; ++i) {
            if (!WIDE) {
                if (lane == 0u) i = atomicAdd(&s_take, 1u);
                i = __shfl_sync(FULLMASK, i, 0);
            }
            if (i >= nrows) break;
            const uint32_t row = row0 + s_rows[i];
            for (uint32_t w = t0; w < W; w += TPR) bm[w] = 0ull;
            if (WIDE) __syncthreads();
            else __syncwarp();
            for (uint32_t k = 0; k < nsrc; ++k) {
                const SrcDesc &d = srcs[src0 + k];
                const uint32_t ch = src_channels<true>(d, mode, iter, g, g0, 0u);
                if (!ch) continue;
                if (d.csr_off) {  // the terminal's product edges (iteration 1)
                    const uint32_t e1 = d.csr_off[row + 1];
                    for (uint32_t e = d.csr_off[row] + t0; e < e1; e += TPR) {
                        const uint32_t z = d.csr_col[e];
                        atomicOr(bm32 + (z >> 5), 1u << (z & 31u));
                    }
                    continue;
                }
                for (uint32_t cb = 1u; cb <= ch; cb <<= 1) {
                    if (!(ch & cb)) continue;
                    const bool new_edges = cb == 1u;
                    if (new_edges && d.nt_new_it[row] != iter) continue;
                    const unsigned long long *adj = reinterpret_cast<const unsigned long long *>(
                        (new_edges ? d.nt_new : d.nt_all) + (size_t)row * W);
                    if (d.ident) {
                        if (new_edges)
                            for (uint32_t w = t0; w < W; w += TPR) {
                                const unsigned long long v = adj[w];
                                if (v) atomicOr(bm + w, v);
                            }
                        continue;
                    }
                    const uint32_t thr = new_edges ? 0u : (cb == 2u ? g0 : g - 1u);
                    // 1024 columns a warp and step: the set bits' columns are
                    // listed in order, then expanded a lane each, so that the
                    // lanes' CSR loads fall into a few neighbouring lines
                    // (each lane on its own word: 32 lines a load)
                    const uint32_t pn = d.pure_n;
                    const uint32_t *const a32 = reinterpret_cast<const uint32_t *>(adj);
                    const uint32_t *const m0 = reinterpret_cast<const uint32_t *>(d.pure_mask[0]);
                    const uint32_t *const m1 = reinterpret_cast<const uint32_t *>(d.pure_mask[1]);
                    for (uint32_t b0 = (WIDE ? warp : 0u) * 32u; b0 < 2u * W; b0 += WIDE ? 256u : 32u) {
                        const uint32_t wi = b0 + lane;
                        uint32_t v = wi < 2u * W ? a32[wi] : 0u;
                        if (v) v &= pn > 1u ? m0[wi] | m1[wi] : m0[wi];
                        const uint32_t cnt = (uint32_t)__popc(v);
                        uint32_t incl = cnt;
#pragma unroll
                        for (int o2 = 1; o2 < 32; o2 <<= 1) {
                            const uint32_t u = __shfl_up_sync(FULLMASK, incl, o2);
                            if (lane >= (uint32_t)o2) incl += u;
                        }
                        const uint32_t n_set = __shfl_sync(FULLMASK, incl, 31);
                        if (n_set == 0u) continue;
                        for (uint32_t at = incl - cnt; v; v &= v - 1u) list[at++] = (uint16_t)(wi * 32u + (uint32_t)__ffs(v) - 1u);
                        __syncwarp();
                        for (uint32_t j = lane; j < n_set; j += 32u) {
                            const uint32_t y = list[j];
                            if (thr && d.rstamp[y] < thr) continue;
                            for (uint32_t p = 0; p < pn; ++p) {
                                const uint32_t e1 = d.pure_off[p][y + 1];
                                for (uint32_t e = d.pure_off[p][y]; e < e1; ++e) {
                                    const uint32_t z = d.pure_col[e];
                                    atomicOr(bm32 + (z >> 5), 1u << (z & 31u));
                                }
                            }
                        }
                        __syncwarp();  // the list is reused
                    }
                }
            }
            if (WIDE) __syncthreads();
            else __syncwarp();
            bool ch = false;
            unsigned long long *const o = reinterpret_cast<unsigned long long *>(it.out) + (size_t)row * W;
            for (uint32_t w = w0 + t0; w < w1; w += TPR) {
                const unsigned long long v = bm[w];
                if (!v) continue;
                const unsigned long long old = o[w];
                if (v & ~old) {
                    o[w] = old | v;
                    ch = true;
                }
            }
            // (also orders this row's bitmap reads before the next row's clearing)
            const bool any = WIDE ? __syncthreads_or(ch) != 0 : __any_sync(FULLMASK, ch) != 0;
            if (any && t0 == 0u) {
                it.out_stamp[row] = g;
                ++my_changed;
            }
        }
        if (my_changed) atomicAdd(&s_changed, my_changed);
        __syncthreads();
        if (tid == 0 && s_changed) {
            *it.out_last = g;
            atomicAdd(&c->changed_rows, (unsigned long long)s_changed);
        }
        __syncthreads();
    }
}

// --------------------------------------------------------------------------
// Closure of a cyclic component, one column word at a time (kSlice).  Word w
// of row x of C[s, t] depends only on word w of the rows it reads, so a CTA
// holds that word of every row of the component's blocks C[., t] in shared
// memory and sweeps the component's product edges until nothing changes, with
// a barrier per sweep: the level's fixpoint in one pass.
//
// The row gather needs a pass (two launches and a grid-wide wait, 22 us at
// least) per hop of the longest path: (ab)*c|a*b* took 70 passes at n = 1000 and
// 32 at n = 8192.  What bounds a sweep is instructions and shared-memory bank
// conflicts, so it runs over edges, not rows (rows of unequal degree left two
// thirds of the lanes idle: 9 us a sweep at n = 8192): 32 packed edges (x << 16 |
// y) per warp and coalesced load, eight in flight a thread; a byte per row holds
// the sweep that last changed it, and only edges from rows changed in this sweep or
// the one before read their words.  Slices of up to 2048 rows (R > 0) are bound by
// latency instead: a thread owns R rows for all sweeps and holds the places of their
// first four edges in registers, so that a row costs five independent loads and no
// atomics (further edges are listed and applied edge by edge; when they are more than a
// quarter of the rows, the slice is swept over edges instead: with a thread walking the rest
// of its row, a+ at n = 2000, a path of 200 vertices and 20 vertices with edges to all others,
// took 24.8 ms, with edge sweeps 1.25).  Regular query:
// n = 1000 1785 -> 385 us with edge sweeps (241 us of run time), 183 us of run time with
// owned rows; n = 8192 2119 -> 1369 us (owned rows: no gain, 1.07 ms of run time against
// 1.04).  Above 200 KB a slice (n = 22755 for one state) the component stays on
// the row gather, which also does less work on the sparse rows that such graphs
// have.
// --------------------------------------------------------------------------
constexpr uint32_t kSliceThreads = 1024, kSliceEdges = 4;
__device__ __forceinline__ void or64(uint64_t *p, uint64_t v) {  // (32-bit shared atomics are native)
    unsigned int *h = reinterpret_cast<unsigned int *>(p);
    if ((uint32_t)v) atomicOr(h, (uint32_t)v);
    if ((uint32_t)(v >> 32)) atomicOr(h + 1, (uint32_t)(v >> 32));
}
template <int R>
__global__ void __launch_bounds__(kSliceThreads, 1)
    k_slice(const SliceItem *__restrict__ items, const SliceGroup *__restrict__ groups,
            const SliceMem *__restrict__ mems, const SrcDesc *__restrict__ srcs, ExecTables T, int cls) {
    extern __shared__ uint64_t s_col[];  // [nmem][n] words, then [nmem][n] bytes
    __shared__ uint32_t s_e0[kSliceMaxSrc], s_e1[kSliceMaxSrc], s_to[kSliceMaxSrc], s_from[kSliceMaxSrc], s_n;
    __shared__ const uint32_t *s_off[kSliceMaxSrc], *s_adj;
    __shared__ uint32_t s_past, s_rest_n;
    __shared__ unsigned long long s_changed, s_ors;
    const uint32_t tid = threadIdx.x, NT = blockDim.x, total = T.g_total[cls];
    for (uint32_t li = blockIdx.x; li < total; li += gridDim.x) {
        const SliceItem it = items[live_item(T.g_pre[cls], T.g_beg[cls], T.nq, li)];
        const SliceGroup G = groups[it.group];
        QCtl *const c = G.ctl;
        if (c->phase != kPhaseRun || c->level != G.level || c->mode != kModeNew) continue;  // (uniform)
        const uint32_t w = it.w, n = G.n, W = G.W, g = c->g, g0 = c->g_iter_start, rows = G.nmem * n;
        const uint32_t *const coo = G.coo;
        const bool first = c->iter == 1u;
        if ((w >> 1) < c->col_v0 || (w >> 1) >= c->col_v1) continue;  // another rank's columns
        // work: the terminal edges in iteration 1, afterwards rows of lower levels that changed
        int act = first ? 1 : 0;
        for (uint32_t m = 0; m < G.nmem && !first; ++m) {
            const SliceMem M = mems[G.mem0 + m];
            for (uint32_t k = tid; k < M.nsrc; k += NT) {
                const SrcDesc &d = srcs[M.src0 + k];
                act |= d.rblk && d.slice_mem == kSliceNone && *d.rlast >= g0;
            }
        }
        if (!__syncthreads_or(act)) continue;
        uint8_t *const s_mark = reinterpret_cast<uint8_t *>(s_col + rows);
        if (tid == 0) {
            s_changed = 0ull;
            s_ors = 0ull;
            uint32_t k2 = 0u;
            for (uint32_t m = 0; m < G.nmem; ++m) {
                const SliceMem M = mems[G.mem0 + m];
                for (uint32_t k = 0; k < M.nsrc; ++k) {
                    const SrcDesc &d = srcs[M.src0 + k];
                    if (d.slice_mem == kSliceNone) continue;
                    s_off[k2] = d.csr_off;
                    s_adj = d.csr_col;
                    s_e0[k2] = d.csr_off[0];
                    s_e1[k2] = d.csr_off[n];
                    s_to[k2] = m * n;
                    s_from[k2] = d.slice_mem * n;
                    ++k2;
                }
            }
            s_n = k2;
            s_past = 0u;
            s_rest_n = 0u;
        }
        for (uint32_t m = 0; m < G.nmem; ++m) {
            const uint64_t *const o = mems[G.mem0 + m].out;
            for (uint32_t x = tid; x < n; x += NT) s_col[m * n + x] = first ? 0ull : o[(size_t)x * W + w];
        }
        __syncthreads();
        // product edges into t, and rows of lower levels
        uint32_t my_ors = 0u;
        for (uint32_t m = 0; m < G.nmem; ++m) {
            const SliceMem M = mems[G.mem0 + m];
            uint64_t *const to = s_col + m * n;
            for (uint32_t k = 0; k < M.nsrc; ++k) {
                const SrcDesc &d = srcs[M.src0 + k];
                const bool read = d.rblk && d.slice_mem == kSliceNone && (first || *d.rlast >= g0);
                const bool ident = first && d.ident;
                if (!read && !ident) continue;
                const uint64_t *const r = d.rblk + w;
                const uint32_t e1 = d.csr_off[n];
                for (uint32_t e = d.csr_off[0] + tid; e < e1; e += NT) {
                    const uint32_t xy = coo[e], x = xy >> 16, y = xy & 0xFFFFu;
                    uint64_t v = 0ull;
                    if (ident && (y >> 6) == w) v = 1ull << (y & 63u);
                    if (read && (first || d.rstamp[y] >= g0)) {
                        v |= r[(size_t)y * W];
                        ++my_ors;
                    }
                    if (v & ~to[x]) or64(to + x, v);
                }
            }
        }
        __syncthreads();
        const uint32_t ns = s_n;
        bool owned = false;
        if constexpr (R > 0) {
            uint32_t *const s_rest = reinterpret_cast<uint32_t *>(s_col + rows);  // edges past the fourth
            uint32_t past = 0u;
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const uint32_t row = tid + (uint32_t)i * NT;
                if (row >= rows) continue;
                const uint32_t m0 = row / n * n, x = row - m0;
                uint32_t deg = 0u;
                for (uint32_t k = 0; k < ns; ++k)
                    if (s_to[k] == m0) deg += s_off[k][x + 1] - s_off[k][x];
                past += deg > 4u ? deg - 4u : 0u;
            }
            past = __reduce_add_sync(FULLMASK, past);
            if ((tid & 31u) == 0u && past) atomicAdd(&s_past, past);
            __syncthreads();
            owned = s_past <= rows / 4u;
            // this thread's rows tid, tid + NT, ...: places of their first four
            // edges (where there are fewer, the row's own: four plain loads beat
            // four branches, 100 instructions a row)
            uint32_t place[R][2];
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const uint32_t row = tid + (uint32_t)i * NT;
                place[i][0] = place[i][1] = row < rows ? row | (row << 16) : 0u;
                if (!owned || row >= rows) continue;
                const uint32_t m0 = row / n * n, x = row - m0;
                uint32_t got = 0u;
                for (uint32_t k = 0; k < ns; ++k) {
                    if (s_to[k] != m0) continue;
                    const uint32_t e1 = s_off[k][x + 1];
                    for (uint32_t e = s_off[k][x]; e < e1; ++e, ++got) {
                        const uint32_t at = s_from[k] + s_adj[e];
                        if (got == 0u) place[i][0] = (place[i][0] & 0xFFFF0000u) | at;
                        else if (got == 1u) place[i][0] = (place[i][0] & 0xFFFFu) | (at << 16);
                        else if (got == 2u) place[i][1] = (place[i][1] & 0xFFFF0000u) | at;
                        else if (got == 3u) place[i][1] = (place[i][1] & 0xFFFFu) | (at << 16);
                        else s_rest[atomicAdd(&s_rest_n, 1u)] = (row << 16) | at;
                    }
                }
            }
            __syncthreads();
            const uint32_t rest = s_rest_n;
            bool ch = owned;
            while (__syncthreads_or(ch)) {
                ch = false;
                // (a row's owner may overwrite bits set here; the next sweep, which
                // this one's change causes, sets them again)
                for (uint32_t j = tid; j < rest; j += NT) {
                    const uint32_t ra = s_rest[j], row = ra >> 16;
                    const uint64_t v = s_col[ra & 0xFFFFu] & ~s_col[row];
                    if (v) {
                        or64(s_col + row, v);
                        ch = true;
                    }
                }
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    const uint32_t row = tid + (uint32_t)i * NT;
                    if (i * NT >= rows) break;  // (uniform)
                    const uint64_t old = s_col[row < rows ? row : 0u];
                    uint64_t v = s_col[place[i][0] & 0xFFFFu] | s_col[place[i][0] >> 16] | s_col[place[i][1] & 0xFFFFu] |
                                 s_col[place[i][1] >> 16];
                    // (a thread past the last row read row 0's word five times: it may have
                    // grown in between, and there is no row to store)
                    if (row < rows && (v & ~old)) {
                        ++my_ors;
                        s_col[row] = old | v;
                        ch = true;
                    }
                }
            }
        }
        if (!owned) {
        // mark: the low byte of the sweep that last changed the row (rows with bits start as
        // changed in sweep 0; 128 is no sweep within reach of the first ones)
        for (uint32_t x = tid; x < rows; x += NT) s_mark[x] = s_col[x] ? 0u : 128u;
        uint32_t sweep = 0u;
        bool ch = true;
        while (__syncthreads_or(ch)) {
            ch = false;
            ++sweep;
            for (uint32_t k = 0; k < ns; ++k) {
                uint64_t *const to = s_col + s_to[k];
                const uint64_t *const from = s_col + s_from[k];
                uint8_t *const to_mark = s_mark + s_to[k];
                const uint8_t *const from_mark = s_mark + s_from[k];
                const uint32_t e1 = s_e1[k];
                uint32_t next[kSliceEdges];
#pragma unroll
                for (uint32_t i = 0; i < kSliceEdges; ++i) {
                    const uint32_t e = s_e0[k] + tid + i * NT;
                    next[i] = e < e1 ? coo[e] : 0u;
                }
                for (uint32_t e0 = s_e0[k] + tid; e0 < e1; e0 += NT * kSliceEdges) {
                    uint32_t xy[kSliceEdges];
                    bool on[kSliceEdges];
#pragma unroll
                    for (uint32_t i = 0; i < kSliceEdges; ++i) {
                        const uint32_t e = e0 + i * NT, ne = e + NT * kSliceEdges;
                        xy[i] = next[i];
                        on[i] = e < e1 && ((sweep - from_mark[xy[i] & 0xFFFFu]) & 0xFFu) <= 1u;
                        next[i] = ne < e1 ? coo[ne] : 0u;  // (in flight while this round is applied)
                    }
#pragma unroll
                    for (uint32_t i = 0; i < kSliceEdges; ++i) {
                        if (!on[i]) continue;
                        const uint32_t x = xy[i] >> 16;
                        const uint64_t v = from[xy[i] & 0xFFFFu] & ~to[x];
                        ++my_ors;
                        if (v) {
                            or64(to + x, v);
                            to_mark[x] = (uint8_t)sweep;
                            ch = true;
                        }
                    }
                }
            }
        }
        }
        uint32_t my_changed = 0u;
        for (uint32_t m = 0; m < G.nmem; ++m) {
            const SliceMem M = mems[G.mem0 + m];
            bool any = false;
            for (uint32_t x = tid; x < n; x += NT) {
                const uint64_t v = s_col[m * n + x];
                if (!v) continue;
                uint64_t *const o = M.out + (size_t)x * W + w;
                if (first || (v & ~*o)) {
                    *o = v;
                    M.stamp[x] = g;
                    any = true;
                    ++my_changed;
                }
            }
            if (any) *M.last = g;
        }
        // counted in whole rows: W slices make a row
        my_ors = __reduce_add_sync(FULLMASK, my_ors);
        my_changed = __reduce_add_sync(FULLMASK, my_changed);
        if ((tid & 31u) == 0u) {
            if (my_ors) atomicAdd(&s_ors, (unsigned long long)my_ors);
            if (my_changed) atomicAdd(&s_changed, (unsigned long long)my_changed);
        }
        __syncthreads();  // (also: the next item overwrites s_col and the tables)
        if (tid == 0) {
            if (s_ors) atomicAdd(&c->row_ors, (s_ors + W - 1u) / W);
            if (s_changed) atomicAdd(&c->changed_rows, (s_changed + W - 1u) / W);
        }
        __syncthreads();
    }
}

// --------------------------------------------------------------------------
// Extraction: runs for a query only after a pass that changed no row.
// --------------------------------------------------------------------------
__device__ void control_body(QCtl *const *ctls, uint32_t nq, QCtl *mirror, cudaGraphConditionalHandle handle,
                             int use_handle, int *running_out, const ExecTables &T, int advance);

// Control fused into the last extraction launch of a pass: the CTA that
// finishes last (counted with an atomic after a fence) runs control_body.
struct FusedControl {
    QCtl *const *ctls;
    QCtl *mirror;
    int *running_out;
    unsigned int *done_counter;
    cudaGraphConditionalHandle handle;
    uint32_t nq;
    int use_handle;
    int enabled;
    uint64_t *zero;  // the tile jobs' scratch, zeroed here for the next pass
    size_t zero_words;
};

template <int VPL>
__global__ void __launch_bounds__(256) k_extract(const XItem *__restrict__ items, const FDesc *__restrict__ fds,
                                                 ExecTables T, int cls, FusedControl FC) {
    __shared__ unsigned long long s_new;
    __shared__ int s_last;
    const uint32_t total = T.x_total[cls];
    for (uint32_t li = blockIdx.x; li < total; li += gridDim.x) {
    const XItem it = items[live_item(T.x_pre[cls], T.x_beg[cls], T.nq, li)];
    const QCtl *c = it.ctl;
    if (c->phase != kPhaseRun) continue;
    // Extraction follows the last level's final pass: its FIRST pass when the
    // level is acyclic, else the first pass that changed no row.
    const bool cyc = (c->cyclic_mask >> c->level) & 1ull;
    if (c->level + 1 != c->n_levels || (cyc && c->changed_rows != 0ull)) continue;
    const uint32_t g0 = c->g_iter_start, iter = c->iter;
    if (threadIdx.x == 0) s_new = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lpr = (int)it.lpr, grp = lane / lpr, gl = lane % lpr, rpw = 32 / lpr;
    const unsigned gmask = (lpr == 32 ? FULLMASK : ((1u << lpr) - 1u)) << (grp * lpr);
    const uint32_t W = it.W, nvec = W / 2;
    const uint32_t cv0 = c->col_v0, cv1 = min(c->col_v1, nvec);  // this rank's columns (all unless sharded)
    uint32_t my_new = 0;
    for (uint32_t rbase = it.row0 + (uint32_t)(warp * rpw); rbase < it.row1; rbase += 8u * rpw) {
        const uint32_t row = rbase + grp;
        const bool valid = row < it.row1;
        uint4 acc[VPL];
#pragma unroll
        for (int j = 0; j < VPL; ++j) acc[j] = make_uint4(0, 0, 0, 0);
        bool any = false;
        for (uint32_t f = 0; f < it.nf; ++f) {
            const FDesc fd = fds[it.f0 + f];
            if (!valid || fd.stamp[row] < g0) continue;
            any = true;
            const uint4 *r = reinterpret_cast<const uint4 *>(fd.blk + (size_t)row * W);
#pragma unroll
            for (int j = 0; j < VPL; ++j) {
                const uint32_t v = (uint32_t)gl + (uint32_t)j * lpr;
                if (v >= cv0 && v < cv1) or4(acc[j], r[v]);
            }
        }
        bool has = false;
        if (any) {
            const uint4 *m = reinterpret_cast<const uint4 *>(it.m2 + (size_t)row * W);
#pragma unroll
            for (int j = 0; j < VPL; ++j) {
                const uint32_t v = (uint32_t)gl + (uint32_t)j * lpr;
                if (v >= cv0 && v < cv1) {
                    acc[j] = andnot4(acc[j], m[v]);
                    if (nz4(acc[j])) has = true;
                }
            }
        }
        const unsigned hb = __ballot_sync(FULLMASK, has);
        if (hb & gmask) {
            uint4 *m = reinterpret_cast<uint4 *>(it.m2 + (size_t)row * W);
            uint4 *a = reinterpret_cast<uint4 *>(it.a2 + (size_t)row * W);
#pragma unroll
            for (int j = 0; j < VPL; ++j) {
                const uint32_t v = (uint32_t)gl + (uint32_t)j * lpr;
                if (v >= cv0 && v < cv1) {
                    a[v] = acc[j];
                    if (nz4(acc[j])) {
                        uint4 mm = m[v];
                        or4(mm, acc[j]);
                        m[v] = mm;
                        my_new += (uint32_t)popc4(acc[j]);
                    }
                }
            }
            if (gl == 0) it.a2_it[row] = iter + 1;
        }
    }
    if (my_new) atomicAdd(&s_new, (unsigned long long)my_new);
    __syncthreads();
    if (threadIdx.x == 0 && s_new) {
        *it.box_new_it = iter + 1;
        atomicAdd(&it.ctl->new_edges, s_new);
        if (it.box_edges) atomicAdd(it.box_edges, s_new);
    }
    __syncthreads();
    }
    if (FC.enabled) {
        for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < FC.zero_words;
             i += (size_t)gridDim.x * blockDim.x)
            FC.zero[i] = 0ull;
        // Control rewrites what every CTA of this launch reads (x_total, the live
        // lists, the queries' state), so the CTA that finishes last runs it, in a pass
        // without extraction too: CTAs may start late (several waves, other work on the SMs).
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) {
            const unsigned int prev = atomicAdd(FC.done_counter, 1u);
            s_last = (prev == gridDim.x - 1) ? 1 : 0;
        }
        __syncthreads();
        if (s_last) {
            __threadfence();
            if (threadIdx.x == 0) *FC.done_counter = 0u;
            control_body(FC.ctls, FC.nq, FC.mirror, FC.handle, FC.use_handle, FC.running_out, T, 1);
        }
    }
}

// --------------------------------------------------------------------------
// Loop control: one CTA for all queries.
// --------------------------------------------------------------------------
// Advance one running query's state machine at the end of a pass.
__device__ __forceinline__ void advance_query(QCtl &c) {
    c.passes += 1;
    c.rounds_total += 1;
    c.rows_changed_total += c.changed_rows;
    c.rounds_in_iter += 1;
    const bool cyc = (c.cyclic_mask >> c.level) & 1ull;
    if (cyc && c.changed_rows != 0ull) {
        // a cyclic level repeats until a pass changes nothing
        c.g += 1;
        c.mode = kModeProp;
        if (c.max_rounds && c.rounds_in_iter >= c.max_rounds) {
            c.status = kStatusRoundCap;
            c.phase = kPhaseDone;
        }
    } else if (c.level + 1 < c.n_levels) {
        c.level += 1;
        c.g += 1;
        c.mode = kModeNew;
    } else {
        // extraction ran in this pass: the iteration is complete
        c.iters_done = c.iter;
        c.edges_total += c.new_edges;
        if (c.box_edges) {
            const unsigned long long dense_at = (unsigned long long)c.n * c.n / kDenseDiv;
            uint32_t m = 0;
            for (uint32_t b = 0; b < c.n_boxes && b < 32u; ++b)
                if (c.box_edges[b] >= dense_at && dense_at > 0ull) m |= 1u << b;
            c.dense_mask = m;
        }
        bool read_new = true;  // does some transition read a box that gained edges?
        if (c.box_new_it && c.n_boxes <= 63u && !((c.nt_read_mask >> 63) & 1ull)) {
            read_new = false;
            for (uint32_t b = 0; b < c.n_boxes; ++b)
                if (((c.nt_read_mask >> b) & 1ull) && c.box_new_it[b] == c.iter + 1u) read_new = true;
        }
        if (c.shard) {
            // column sharding: whether the loop goes on depends on every
            // rank's new edges; pause at the next iteration's start until
            // they are installed (k_shard_apply, k_shard_finish)
            c.shard_new = c.new_edges;
            c.iter += 1;
            c.g += 1;
            c.level = 0;
            c.mode = kModeNew;
            c.g_iter_start = c.g;
            c.rounds_in_iter = 0;
            c.phase = kPhasePause;
        } else if (c.new_edges == 0ull) {
            c.phase = kPhaseDone;
        } else if (c.max_iter && c.iter >= c.max_iter) {
            c.status = kStatusIterCap;
            c.phase = kPhaseDone;
        } else if (!read_new) {
            // the next iteration's product equals this one's: it adds no
            // edge, so it is the last one and is counted without passes
            c.iters_done = c.iter + 1u;
            c.phase = kPhaseDone;
        } else {
            c.iter += 1;
            c.g += 1;
            c.level = 0;
            c.mode = kModeNew;
            c.g_iter_start = c.g;
            c.rounds_in_iter = 0;
        }
        c.new_edges = 0;
    }
    if (c.phase == kPhaseRun && c.passes >= c.max_passes) {
        c.status = kStatusPassCap;
        c.phase = kPhaseDone;
    }
    c.changed_rows = 0;
}

// Loop control for every query of the executor, run by one whole CTA (any
// size up to 1024 threads, at least one warp): advance each running query's
// state machine (unless `advance` is 0), then build the live lists of the next
// pass.  It ends every pass, so it is one chain of memory latencies: a query's
// state is read once, changed in registers and written twice; a single query's
// lists are written by one thread a class, without the scans over queries.
// (extraction and control, Dyck-4 n = 3001, average over its passes with cold caches:
// 16.3 -> 10.3 us.)
__device__ void control_body(QCtl *const *ctls, uint32_t nq, QCtl *mirror, cudaGraphConditionalHandle handle,
                             int use_handle, int *running_out, const ExecTables &T, int advance) {
    constexpr int K = kClasses + kXClasses + 1;
    static_assert(K <= 32, "one thread per count");
    __shared__ uint32_t s_wsum[32][K];
    __shared__ uint32_t s_carry[K];
    __shared__ uint32_t s_lvl, s_last, s_aj;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (int)((blockDim.x + 31) >> 5);
    int running = 0;
    if (threadIdx.x < K) s_carry[threadIdx.x] = 0u;
    if (threadIdx.x == 0) s_aj = 0u;
    for (uint32_t c0 = 0; c0 < nq; c0 += blockDim.x) {
        const uint32_t q = c0 + threadIdx.x;
        bool run = false;
        uint32_t L = 0u, n_levels = 0u;
        if (q < nq) {
            QCtl *const p = ctls[q];
            QCtl c = *p;
            if (c.phase == kPhaseRun && advance) {
                advance_query(c);
                *p = c;
            }
            mirror[q] = c;
            run = c.phase == kPhaseRun;
            L = c.level;
            n_levels = c.n_levels;
            running |= run;
        }
        const bool last = run && (L + 1 == n_levels);
        if (nq == 1u) {
            // live work of the next pass: the items of the query's current level
            if (threadIdx.x == 0) {
                s_lvl = run ? L : 0xFFFFFFFFu;
                s_last = last ? 1u : 0u;
            }
            __syncthreads();
            const uint32_t lv = s_lvl;
            const bool r1 = lv != 0xFFFFFFFFu;
            const int k = threadIdx.x;
            if (k < kClasses) {
                const uint32_t gb = r1 ? T.g_lvl[k][lv] : 0u, ge = r1 ? T.g_lvl[k][lv + 1] : 0u;
                T.g_beg[k][0] = gb;
                T.g_pre[k][0] = 0u;
                s_carry[k] = ge - gb;
            } else if (k < kClasses + kXClasses) {
                const int v = k - kClasses;
                const uint32_t xb = s_last ? T.x_rng[v][0] : 0u, xe = s_last ? T.x_rng[v][1] : 0u;
                T.x_beg[v][0] = xb;
                T.x_pre[v][0] = 0u;
                s_carry[k] = xe - xb;
            } else if (k == K - 1) {
                T.t_job_beg[0] = r1 ? T.t_lvl[lv] : 0u;
                T.t_job_end[0] = r1 ? T.t_lvl[lv + 1] : 0u;
                T.t_pre[0] = 0u;
                s_carry[k] = r1 ? T.t_lvl_tiles[lv] : 0u;
            }
            break;
        }
        // All K counts of a query sit in registers and are scanned together
        // across the CTA (warp shuffles, then the warp totals), one chunk of
        // blockDim queries at a time.
        uint32_t cnt[K];
#pragma unroll
        for (int k = 0; k < K; ++k) cnt[k] = 0u;
        if (q < nq) {
            const uint32_t base = q * T.maxL1 + L;
#pragma unroll
            for (int v = 0; v < kClasses; ++v) {
                const uint32_t gb = run ? T.g_lvl[v][base] : 0u, ge = run ? T.g_lvl[v][base + 1] : 0u;
                T.g_beg[v][q] = gb;
                cnt[v] = ge - gb;
            }
#pragma unroll
            for (int v = 0; v < kXClasses; ++v) {
                const uint32_t xb = last ? T.x_rng[v][q] : 0u, xe = last ? T.x_rng[v][q + 1] : 0u;
                T.x_beg[v][q] = xb;
                cnt[kClasses + v] = xe - xb;
            }
            T.t_job_beg[q] = run ? T.t_lvl[base] : 0u;
            T.t_job_end[q] = run ? T.t_lvl[base + 1] : 0u;
            cnt[K - 1] = run ? T.t_lvl_tiles[base] : 0u;
        }
        uint32_t inc[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            uint32_t x = cnt[k];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            inc[k] = x;
            if (lane == 31) s_wsum[wid][k] = x;
        }
        __syncthreads();
        if (wid == 0) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                uint32_t w = lane < nw ? s_wsum[lane][k] : 0u;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
                    if (lane >= o) w += y;
                }
                if (lane < nw) s_wsum[lane][k] = w;  // inclusive prefix of warp totals
            }
        }
        __syncthreads();
        if (q < nq) {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const uint32_t pre = s_carry[k] + (wid ? s_wsum[wid - 1][k] : 0u) + inc[k] - cnt[k];
                if (k < kClasses) T.g_pre[k][q] = pre;
                else if (k < kClasses + kXClasses) T.x_pre[k - kClasses][q] = pre;
                else T.t_pre[q] = pre;
            }
        }
        __syncthreads();
        if (threadIdx.x < K) s_carry[threadIdx.x] += s_wsum[nw - 1][threadIdx.x];
        __syncthreads();
    }
    running = __syncthreads_or(running);
    // The tile jobs of the next pass: those of the live levels that take part
    // (their activity depends only on the loop state just written).  The CTA's
    // threads split a query's jobs when there are more threads than queries.
    if (T.jobs) {
        uint32_t per = 1u;  // threads per query
        while (per < 32u && 2u * per * nq <= blockDim.x) per <<= 1;
        for (uint32_t i = threadIdx.x; i < nq * per; i += blockDim.x) {
            const uint32_t q = i / per, je = T.t_job_end[q];
            for (uint32_t j = T.t_job_beg[q] + i % per; j < je; j += per) {
                uint32_t thr, it, g;
                if (tc_job_active(T.jobs[j], &thr, &it, &g)) T.aj[atomicAdd(&s_aj, 1u)] = j;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) *T.aj_n = s_aj;
    }
    if (threadIdx.x < K) {
        const int k = threadIdx.x;
        if (k < kClasses) T.g_next[k] = 0u;  // dynamic gather units of the next pass
        if (k < kClasses) T.g_total[k] = s_carry[k];
        else if (k < kClasses + kXClasses) T.x_total[k - kClasses] = s_carry[k];
        else *T.t_total = s_carry[k];
    }
    if (threadIdx.x == 0) {
        if (use_handle) cudaGraphSetConditional(handle, running ? 1u : 0u);
        if (running_out) *running_out = running;
    }
}

__global__ void __launch_bounds__(1024) k_control(QCtl *const *ctls, uint32_t nq, QCtl *mirror,
                                                  cudaGraphConditionalHandle handle, int use_handle, int *running_out,
                                                  ExecTables T, int advance) {
    control_body(ctls, nq, mirror, handle, use_handle, running_out, T, advance);
}

// Reset the loop state of queries [0, nq) (start of a run).
__global__ void k_ctl_reset(QCtl *const *ctls, uint32_t nq, uint32_t max_iter, uint32_t max_rounds,
                            uint32_t max_passes, uint32_t n_levels, unsigned long long cyclic_mask,
                            unsigned long long *box_edges, uint32_t n_boxes, uint32_t n,
                            const uint32_t *box_new_it, unsigned long long nt_read_mask) {
    for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q < nq; q += gridDim.x * blockDim.x) {
        QCtl c;
        memset(&c, 0, sizeof(c));
        c.g = 2;
        c.iter = 1;
        c.mode = kModeNew;
        c.phase = kPhaseRun;
        c.g_iter_start = 2;
        c.col_v0 = 0u;
        c.col_v1 = 0xFFFFFFFFu;
        c.max_iter = max_iter;
        c.max_rounds = max_rounds;
        c.max_passes = max_passes;
        c.level = 0;
        c.n_levels = n_levels;
        c.cyclic_mask = cyclic_mask;
        c.box_edges = box_edges;
        c.n_boxes = n_boxes;
        c.n = n;
        c.dense_mask = 0;
        c.box_new_it = box_new_it;
        c.nt_read_mask = nt_read_mask;
        *ctls[q] = c;
    }
}

// Epsilon case of Listing 1: a box whose start state is final derives the
// empty word, so M2^b[i,i] = 1 for every vertex i.  These edges are new edges
// of the first iteration (A2^b rows = e_i), so that they take part in the
// product like any other nonterminal edge.
struct EpsDesc {
    uint64_t *m2, *a2;
    uint32_t *a2_it, *box_new_it;
    QCtl *ctl;
    unsigned long long *box_edges;
    uint32_t n, W;
};
// (One warp a row and 16-byte stores, grid over all rows: bound by the A2 rows
// written -- 512 MiB at n = 65536, 299 us with a division and an 8-byte store per word.)
__global__ void __launch_bounds__(256) k_eps_init(const EpsDesc *__restrict__ eds, uint32_t ned) {
    const uint32_t lane = threadIdx.x & 31u, gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nw = (gridDim.x * blockDim.x) >> 5;
    for (uint32_t e = 0; e < ned; ++e) {
        const EpsDesc d = eds[e];
        for (uint32_t row = gw; row < d.n; row += nw) {
            ulonglong2 *a = reinterpret_cast<ulonglong2 *>(d.a2 + (size_t)row * d.W);
            const uint32_t bw = row >> 6;
            const unsigned long long bit = 1ull << (row & 63u);
            for (uint32_t v = lane; v < d.W / 2u; v += 32u)
                a[v] = make_ulonglong2(2u * v == bw ? bit : 0ull, 2u * v + 1u == bw ? bit : 0ull);
            if (lane == 0u) {
                d.m2[(size_t)row * d.W + bw] |= bit;
                d.a2_it[row] = 1;
            }
        }
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            *d.box_new_it = 1;
            atomicAdd(&d.ctl->edges_total, (unsigned long long)d.n);
            if (d.box_edges) atomicAdd(d.box_edges, (unsigned long long)d.n);
        }
    }
}

// Start of a run: zero the bit rows that hold bits and their marks.  A row that was
// ever written has a nonzero mark (closure blocks: the stamp, M2: the iteration of its last
// new edges), so buffers left by an earlier run need only those rows zeroed;
// *all (set for buffers in any other state) zeroes every row.  16 sources at n = 65536
// leave some 200 of 1.7 million rows: 2.2 ms of zeroing 13.6 GB -> 10 us.
__global__ void __launch_bounds__(256) k_clear_rows(uint64_t *rows, uint32_t *mark, size_t n_rows, uint32_t W,
                                                    const uint32_t *all) {
    const uint32_t lane = threadIdx.x & 31u;
    const size_t gw = ((size_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5, nw = ((size_t)gridDim.x * blockDim.x) >> 5;
    const bool every = *all != 0u;
    for (size_t r0 = gw * 32u; r0 < n_rows; r0 += nw * 32u) {
        const size_t r = r0 + lane;
        const bool has = r < n_rows && (every || mark[r] != 0u);
        if (has) mark[r] = 0u;
        for (unsigned m = __ballot_sync(FULLMASK, has); m; m &= m - 1u) {
            uint4 *p = reinterpret_cast<uint4 *>(rows + (r0 + (size_t)(__ffs(m) - 1)) * W);
            for (uint32_t v = lane; v < W / 2u; v += 32u) p[v] = make_uint4(0, 0, 0, 0);
        }
    }
}

// --------------------------------------------------------------------------
// Graph staging: edge list -> deduplicated CSR per used terminal label.
// --------------------------------------------------------------------------
__global__ void k_stage_count(const uint32_t *__restrict__ src, const uint32_t *__restrict__ lbl,
                              const uint32_t *__restrict__ dst, size_t m, uint32_t n, uint32_t n_term,
                              const int32_t *__restrict__ label_map, uint32_t *cnt, int *err) {
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (size_t)gridDim.x * blockDim.x) {
        const uint32_t s = src[e], l = lbl[e], d = dst[e];
        if (s >= n || d >= n || l >= n_term) { atomicOr(err, 1); continue; }
        const int32_t li = label_map[l];
        if (li >= 0) atomicAdd(&cnt[(size_t)li * n + s], 1u);
    }
}

__global__ void k_stage_fill(const uint32_t *__restrict__ src, const uint32_t *__restrict__ lbl,
                             const uint32_t *__restrict__ dst, size_t m, uint32_t n, uint32_t n_term,
                             const int32_t *__restrict__ label_map, const uint32_t *__restrict__ off,
                             uint32_t *fill, uint32_t *col) {
    for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (size_t)gridDim.x * blockDim.x) {
        const uint32_t s = src[e], l = lbl[e], d = dst[e];
        if (s >= n || d >= n || l >= n_term) continue;
        const int32_t li = label_map[l];
        if (li < 0) continue;
        const size_t r = (size_t)li * n + s;
        col[off[r] + atomicAdd(&fill[r], 1u)] = d;
    }
}

// Sort each adjacency row and drop duplicates; ucnt[r] = distinct count.
// Rows longer than kUniqueMax are left as they are: a repeated edge only
// repeats an idempotent OR of the same source row, so duplicates cost time,
// never correctness, and the per-row work stays bounded.
constexpr uint32_t kUniqueMax = 256;
__global__ void k_stage_unique(const uint32_t *__restrict__ off, uint32_t *col, uint32_t *ucnt, size_t rows) {
    for (size_t r = (size_t)blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += (size_t)gridDim.x * blockDim.x) {
        const uint32_t a = off[r], b = off[r + 1];
        if (b - a > kUniqueMax) { ucnt[r] = b - a; continue; }
        for (uint32_t i = a + 1; i < b; ++i) {
            const uint32_t v = col[i];
            uint32_t j = i;
            while (j > a && col[j - 1] > v) { col[j] = col[j - 1]; --j; }
            col[j] = v;
        }
        uint32_t k = a;
        for (uint32_t i = a; i < b; ++i)
            if (i == a || col[i] != col[k - 1]) col[k++] = col[i];
        ucnt[r] = k - a;
    }
}

// result[0] bit 1: a row of more than kHubEdges edges is kept.
__global__ void k_stage_compact(const uint32_t *__restrict__ off, const uint32_t *__restrict__ col,
                                const uint32_t *__restrict__ uoff, uint32_t *ucol, size_t rows, uint32_t n,
                                uint32_t counted, uint32_t *result) {
    if (blockIdx.x == 0) {
        if (threadIdx.x == 0) result[1] = uoff[rows];
        for (uint32_t l = threadIdx.x; l < counted; l += blockDim.x) result[2u + l] = uoff[(size_t)l * n];
    }
    for (size_t r = (size_t)blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += (size_t)gridDim.x * blockDim.x) {
        const uint32_t a = off[r], u0 = uoff[r], k = uoff[r + 1] - u0;
        if (k > kHubEdges) atomicOr(result, 2u);
        for (uint32_t i = 0; i < k; ++i) ucol[u0 + i] = col[a + i];
    }
}

// Exclusive scan of n uint32 (n < 2^32 total): out[0..n], out[n] = total.
constexpr int kScanThreads = 1024, kScanPer = 4, kScanChunk = kScanThreads * kScanPer;

__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t *total) {
    __shared__ uint32_t warp_sums[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(FULLMASK, x, o);
        if (lane >= o) x += t;
    }
    if (lane == 31) warp_sums[wid] = x;
    __syncthreads();
    if (wid == 0) {
        uint32_t s = (lane < (int)(blockDim.x >> 5)) ? warp_sums[lane] : 0u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(FULLMASK, s, o);
            if (lane >= o) s += t;
        }
        warp_sums[lane] = s;
    }
    __syncthreads();
    const uint32_t base = wid ? warp_sums[wid - 1] : 0u;
    if (total) *total = warp_sums[(blockDim.x >> 5) - 1];
    __syncthreads();
    return base + x - v;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_local(const uint32_t *__restrict__ in, uint32_t *out,
                                                             uint32_t *block_sums, size_t n) {
    const size_t base = (size_t)blockIdx.x * kScanChunk + (size_t)threadIdx.x * kScanPer;
    uint32_t v[kScanPer], s = 0;
#pragma unroll
    for (int i = 0; i < kScanPer; ++i) { v[i] = (base + i < n) ? in[base + i] : 0u; s += v[i]; }
    uint32_t tot;
    uint32_t ex = block_exclusive_scan(s, &tot);
#pragma unroll
    for (int i = 0; i < kScanPer; ++i) {
        if (base + i < n) out[base + i] = ex;
        ex += v[i];
    }
    if (threadIdx.x == 0) block_sums[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_sums(uint32_t *block_sums, uint32_t nb, uint32_t *total_out) {
    // nb <= kScanChunk
    const uint32_t base = threadIdx.x * kScanPer;
    uint32_t v[kScanPer], s = 0;
#pragma unroll
    for (int i = 0; i < kScanPer; ++i) { v[i] = (base + i < nb) ? block_sums[base + i] : 0u; s += v[i]; }
    uint32_t tot;
    uint32_t ex = block_exclusive_scan(s, &tot);
#pragma unroll
    for (int i = 0; i < kScanPer; ++i) {
        if (base + i < nb) block_sums[base + i] = ex;
        ex += v[i];
    }
    if (threadIdx.x == 0) *total_out = tot;
}

__global__ void k_scan_add(uint32_t *out, const uint32_t *__restrict__ block_sums, size_t n, const uint32_t *total,
                           uint32_t *out_total) {
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] += block_sums[i / kScanChunk];
    if (i == 0) *out_total = *total;
}

// The whole staging in one CTA for graphs whose counters and edges fit its
// shared memory (rows = n_term * n counters, m columns): a load of a small graph is a
// chain of launches otherwise, 62 us at n = 200 and 72 at n = 1000 with eleven, 21 and
// 29 with this one.  The CSR is the same (rows sorted, repeated edges dropped up
// to kUniqueMax).  result[0] = 1 on an edge out of range, | 2 on a row
// of more than kHubEdges edges, result[1] = edges kept,
// result[2 + l] = edges kept of the labels before l (l < counted).
constexpr uint32_t kStageThreads = 1024;
__global__ void __launch_bounds__(kStageThreads, 1)
    k_stage_small(const uint32_t *__restrict__ src, const uint32_t *__restrict__ lbl, const uint32_t *__restrict__ dst,
                  uint32_t m, uint32_t n, uint32_t n_term, uint32_t counted, uint32_t *csr_off, uint32_t *csr_col,
                  uint32_t *result) {
    extern __shared__ uint32_t s_stage[];  // [rows] counters, then [m] columns
    const uint32_t tid = threadIdx.x, rows = n * n_term;
    uint32_t *const cnt = s_stage, *const col = s_stage + rows;
    int bad = 0;
    for (uint32_t r = tid; r < rows; r += kStageThreads) cnt[r] = 0u;
    __syncthreads();
    for (uint32_t e = tid; e < m; e += kStageThreads) {
        const uint32_t s = src[e], l = lbl[e];
        if (s >= n || l >= n_term || dst[e] >= n) bad = 1;
        else atomicAdd(&cnt[l * n + s], 1u);
    }
    bad = __syncthreads_or(bad);
    // exclusive scan in place: thread t owns the counters [t * per, (t + 1) * per)
    const uint32_t per = (rows + kStageThreads - 1u) / kStageThreads, r0 = min(rows, tid * per), r1 = min(rows, r0 + per);
    auto scan = [&]() -> uint32_t {
        uint32_t sum = 0u, total;
        for (uint32_t r = r0; r < r1; ++r) sum += cnt[r];
        uint32_t run = block_exclusive_scan(sum, &total);
        for (uint32_t r = r0; r < r1; ++r) {
            const uint32_t c = cnt[r];
            cnt[r] = run;
            run += c;
        }
        __syncthreads();
        return total;
    };
    scan();
    for (uint32_t e = tid; e < m; e += kStageThreads) {
        const uint32_t s = src[e], l = lbl[e], d = dst[e];
        if (s < n && l < n_term && d < n) col[atomicAdd(&cnt[l * n + s], 1u)] = d;
    }
    __syncthreads();
    // cnt[r] is the row's end now (the next row's start): sort, drop repeats
    uint32_t ends_before = r0 > 0u && r0 < r1 ? cnt[r0 - 1u] : 0u;
    __syncthreads();
    const uint32_t first = ends_before;
    for (uint32_t r = r0; r < r1; ++r) {
        const uint32_t a = ends_before, b = cnt[r];
        ends_before = b;
        uint32_t k = b - a;
        if (k <= kUniqueMax) {
            for (uint32_t i = a + 1u; i < b; ++i) {
                const uint32_t v = col[i];
                uint32_t j = i;
                while (j > a && col[j - 1u] > v) { col[j] = col[j - 1u]; --j; }
                col[j] = v;
            }
            k = 0u;
            for (uint32_t i = a; i < b; ++i)
                if (i == a || col[i] != col[i - 1u]) ++k;
        }
        cnt[r] = k | ((b - a) << 16);  // (m < 65536: both fit)
    }
    __syncthreads();
    uint32_t sum = 0u, total;
    for (uint32_t r = r0; r < r1; ++r) sum += cnt[r] & 0xFFFFu;
    uint32_t out = block_exclusive_scan(sum, &total), a = first;
    bool hub = false;
    for (uint32_t r = r0; r < r1; ++r) {
        const uint32_t k = cnt[r] & 0xFFFFu, len = cnt[r] >> 16;
        csr_off[r] = out;
        hub |= k > kHubEdges;
        if (r % n == 0u && r / n < counted) result[2u + r / n] = out;
        if (k == len)
            for (uint32_t i = 0; i < len; ++i) csr_col[out + i] = col[a + i];
        else
            for (uint32_t i = 0, w = out; i < len; ++i)
                if (i == 0u || col[a + i] != col[a + i - 1u]) csr_col[w++] = col[a + i];
        out += k;
        a += len;
    }
    hub = __syncthreads_or(hub) != 0;
    if (tid == 0) {
        csr_off[rows] = total;
        result[0] = (bad ? 1u : 0u) | (hub ? 2u : 0u);
        result[1] = total;
    }
}

// Terminal adjacency as bit rows (needed when terminal sources run on the
// tensor cores): bits[l][x] has bit y for every CSR edge (x, l, y).
__global__ void k_csr_to_bits(const uint32_t *__restrict__ off, const uint32_t *__restrict__ col, size_t rows,
                              uint32_t W, uint64_t *bits) {
    for (size_t r = (size_t)blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += (size_t)gridDim.x * blockDim.x) {
        uint64_t *row = bits + r * W;
        for (uint32_t e = off[r]; e < off[r + 1]; ++e) {
            const uint32_t y = col[e];
            row[y >> 6] |= 1ull << (y & 63u);
        }
    }
}

// The CSR's edges with their row: coo[e] = row's vertex << 16 | column (both below 65536).
__global__ void k_csr_to_coo(const uint32_t *__restrict__ off, const uint32_t *__restrict__ col, size_t rows, uint32_t n,
                             uint32_t *coo) {
    for (size_t r = (size_t)blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += (size_t)gridDim.x * blockDim.x) {
        const uint32_t x = (uint32_t)(r % n) << 16;
        for (uint32_t e = off[r]; e < off[r + 1]; ++e) coo[e] = x | col[e];
    }
}

// bits[l * W + w] bit b = row (l, 64 w + b) of the CSR has an edge.
__global__ void k_nonempty_bits(const uint32_t *__restrict__ off, uint32_t n, uint32_t n_term, uint32_t W,
                                uint64_t *bits) {
    const size_t total = (size_t)n_term * W;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const uint32_t l = (uint32_t)(i / W), w = (uint32_t)(i % W);
        uint64_t word = 0;
        for (uint32_t b = 0; b < 64u; ++b) {
            const uint32_t y = w * 64u + b;
            if (y >= n) break;
            const size_t r = (size_t)l * n + y;
            if (off[r + 1] > off[r]) word |= 1ull << b;
        }
        bits[i] = word;
    }
}

// --------------------------------------------------------------------------
// Result helpers.
// --------------------------------------------------------------------------
__global__ void k_popcount(const uint64_t *__restrict__ p, size_t nwords, unsigned long long *out) {
    unsigned long long s = 0;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < nwords; i += (size_t)gridDim.x * blockDim.x)
        s += (unsigned long long)__popcll(p[i]);
#pragma unroll
    for (int o = 16; o; o >>= 1) s += __shfl_down_sync(FULLMASK, s, o);
    if ((threadIdx.x & 31) == 0 && s) atomicAdd(out, s);
}

// Copy rows of several blocks into a dense staging buffer:
// job k copies row rows[k] of block ptrs[k] (W words) to out + k * W.
__global__ void k_copy_rows(const uint64_t *const *__restrict__ ptrs, const uint32_t *__restrict__ rows, uint32_t njobs,
                            uint32_t W, uint64_t *out) {
    for (uint32_t k = blockIdx.x; k < njobs; k += gridDim.x) {
        const uint64_t *p = ptrs[k];
        for (uint32_t w = threadIdx.x; w < W; w += blockDim.x) out[(size_t)k * W + w] = p ? p[(size_t)rows[k] * W + w] : 0ull;
    }
}

// Rows [r0, r0 + rows) of a bit matrix without their padding word: wn < W words
// each, back to back (a linear write, 8 bytes a thread; bound by HBM, and two
// orders below the host copy that follows).
__global__ void k_pack_rows(const uint64_t *__restrict__ src, uint32_t W, uint32_t wn, uint32_t r0, size_t words,
                            uint64_t *__restrict__ out) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < words; i += (size_t)gridDim.x * blockDim.x) {
        const size_t r = i / wn;
        out[i] = src[(r0 + r) * W + (i - r * wn)];
    }
}

// ---------------------------------------------------------------------------
// Host launchers.
// ---------------------------------------------------------------------------
int vpl_for_words(uint32_t W) {
    if (W <= 64) return 1;
    if (W <= 128) return 2;
    if (W <= 256) return 4;
    if (W <= 512) return 8;
    if (W <= 1024) return 16;
    return 0;
}

static int g_gather_sms[64];
static int g_extract_ctas[64][kXClasses];  // CTAs of k_extract that a device holds at once, per row width

cudaError_t launch_gather(int vpl, bool nt, bool hubs, const GItem *items, uint32_t n_items, const SrcDesc *srcs,
                          const ExecTables &T, int cls, cudaStream_t st) {
    if (n_items == 0) return cudaSuccess;
    int dev = 0;
    cudaGetDevice(&dev);
    const uint32_t sms = (dev >= 0 && dev < 64 && g_gather_sms[dev]) ? (uint32_t)g_gather_sms[dev] : 0u;
    // dynamic scheduling: a persistent grid (resident CTAs), at most one warp
    // per unit; otherwise one CTA per live item, at most kStrideWaves waves of
    // resident CTAs (the CTAs stride over the live items): n_items bounds the
    // live items of any pass, and a batch's pass with few live queries would
    // otherwise launch tens of thousands of CTAs that exit at once
    auto grid_of = [&](bool dyn, int occ) -> uint32_t {
        if (!sms) return n_items;
        if (!dyn) return std::min<uint32_t>(n_items, sms * (uint32_t)occ * kStrideWaves);
        const uint32_t want = (n_items * kGatherParts + 7u) / 8u;
        return std::max<uint32_t>(1u, std::min<uint32_t>(want, sms * (uint32_t)occ));
    };
#define CFPQ_GATHER(V)                                                                                          \
    if (nt) k_gather<V, true, false><<<grid_of(GatherDyn<V, true>::on, GatherCtas<V, true>::value), 256, GatherRing<V>::bytes, \
                                st>>>(items, srcs, T, cls);                                                     \
    else if (hubs) k_gather<V, false, true><<<grid_of(false, GatherCtas<V, false>::value), 256, 0, st>>>(       \
        items, srcs, T, cls);                                                                                   \
    else k_gather<V, false, false><<<grid_of(false, GatherCtas<V, false>::value), 256, 0, st>>>(items, srcs, T, cls);
    switch (vpl) {
        case 1: CFPQ_GATHER(1) break;
        case 2: CFPQ_GATHER(2) break;
        case 4: CFPQ_GATHER(4) break;
        case 8: CFPQ_GATHER(8) break;
        case 16: CFPQ_GATHER(16) break;
        default: return cudaErrorInvalidValue;
    }
#undef CFPQ_GATHER
    return cudaGetLastError();
}

cudaError_t launch_expand(bool wide, const GItem *items, uint32_t n_items, const SrcDesc *srcs, uint32_t max_w,
                          const ExecTables &T, int cls, cudaStream_t st) {
    if (n_items == 0) return cudaSuccess;
    int dev = 0;
    cudaGetDevice(&dev);
    const uint32_t sms = (dev >= 0 && dev < 64 && g_gather_sms[dev]) ? (uint32_t)g_gather_sms[dev] : 0u;
    const uint32_t units = n_items * (wide ? kExpandParts : 1u);
    const uint32_t grid = sms ? std::min<uint32_t>(units, sms * (uint32_t)kExpandOcc) : units;  // resident CTAs take units
    if (wide) k_expand<true><<<grid, 256, (size_t)max_w * 8, st>>>(items, srcs, T, cls);
    else k_expand<false><<<grid, 256, (size_t)std::min(max_w, kExpandNarrowW) * 8 * 8, st>>>(items, srcs, T, cls);
    return cudaGetLastError();
}

cudaError_t launch_slice(const SliceItem *items, uint32_t n_items, const SliceGroup *groups, const SliceMem *mems,
                         const SrcDesc *srcs, uint32_t smem, const ExecTables &T, int cls, cudaStream_t st) {
    if (n_items == 0) return cudaSuccess;
    int dev = 0;
    cudaGetDevice(&dev);
    const uint32_t sms = (dev >= 0 && dev < 64 && g_gather_sms[dev]) ? (uint32_t)g_gather_sms[dev] : 0u;
    const uint32_t grid = sms ? std::min<uint32_t>(n_items, sms * 4u) : n_items;
    // small slices: a barrier over 16 warps costs less than their extra loads gain (n = 1000: 44 us
    // against 56 for a level; n = 8192: 115 against 98)
    const uint32_t rows = smem / 9u, threads = rows >= 4096u ? kSliceThreads : kSliceThreads / 2u;
    if (rows <= 1024u) k_slice<2><<<grid, threads, smem, st>>>(items, groups, mems, srcs, T, cls);
    else if (rows <= 2048u) k_slice<4><<<grid, threads, smem, st>>>(items, groups, mems, srcs, T, cls);
    else k_slice<0><<<grid, threads, smem, st>>>(items, groups, mems, srcs, T, cls);
    return cudaGetLastError();
}

// Shared-memory limits of the general gather variants and of the column slices
// (call outside any stream capture).
cudaError_t prepare_gather_launch() {
    {
        cudaError_t e = cudaSuccess;
        auto room = [&](auto kernel) {
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSliceMaxBytes);
        };
        room(k_slice<0>);
        room(k_slice<2>);
        room(k_slice<4>);
        if (e != cudaSuccess) return e;
    }
#define CFPQ_RING(V)                                                                                      \
    {                                                                                                     \
        const cudaError_t e = cudaFuncSetAttribute(k_gather<V, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                                                   (int)GatherRing<V>::bytes);                            \
        if (e != cudaSuccess) return e;                                                                   \
    }
    CFPQ_RING(4) CFPQ_RING(8) CFPQ_RING(16)
#undef CFPQ_RING
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    int sms = 0;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    int per_sm[kXClasses];
    const void *const extract[kXClasses] = {(const void *)k_extract<1>, (const void *)k_extract<2>,
                                            (const void *)k_extract<4>, (const void *)k_extract<8>,
                                            (const void *)k_extract<16>};
    for (int c = 0; c < kXClasses; ++c) {
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm[c], extract[c], 256, 0);
        if (e != cudaSuccess) return e;
    }
    for (int c = 0; c < kXClasses; ++c) g_extract_ctas[dev][c] = sms * std::max(1, per_sm[c]);
    g_gather_sms[dev] = sms;
    return cudaSuccess;
}

// With fused control (ctls != null) this launch also runs the pass's loop
// control in its last CTA; done_counter must be 0 before the first launch.
cudaError_t launch_extract(int vpl, const XItem *items, uint32_t n_items, const FDesc *fds, const ExecTables &T,
                           int cls, QCtl *const *ctls, uint32_t nq, QCtl *mirror, cudaGraphConditionalHandle h,
                           int use_handle, int *running_out, unsigned int *done_counter, uint64_t *zero,
                           size_t zero_words, cudaStream_t st) {
    if (n_items == 0) return cudaSuccess;
    FusedControl fc{ctls, mirror, running_out, done_counter, h, nq, use_handle, ctls != nullptr ? 1 : 0, zero,
                    zero_words};
    // resident CTAs that stride over the live items (3, 3, 2, 1 and 1 an SM by row width: registers):
    // every CTA of the fused launch is counted, and a pass without extraction is nothing but that count
    int dev = 0;
    cudaGetDevice(&dev);
    const uint32_t ctas = (dev >= 0 && dev < 64) ? (uint32_t)g_extract_ctas[dev][cls] : 0u;
    const uint32_t grid = ctas ? std::min<uint32_t>(n_items, ctas) : n_items;
    switch (vpl) {
        case 1: k_extract<1><<<grid, 256, 0, st>>>(items, fds, T, cls, fc); break;
        case 2: k_extract<2><<<grid, 256, 0, st>>>(items, fds, T, cls, fc); break;
        case 4: k_extract<4><<<grid, 256, 0, st>>>(items, fds, T, cls, fc); break;
        case 8: k_extract<8><<<grid, 256, 0, st>>>(items, fds, T, cls, fc); break;
        case 16: k_extract<16><<<grid, 256, 0, st>>>(items, fds, T, cls, fc); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_control(QCtl *const *ctls, uint32_t nq, QCtl *mirror, cudaGraphConditionalHandle h, int use_handle,
                           int *running_out, const ExecTables &T, int advance, cudaStream_t st) {
    // one thread per query up to 1024 (a single warp for small batches keeps
    // the per-pass scans to shuffles)
    uint32_t threads = ((nq + 31u) / 32u) * 32u;
    if (threads < 32u) threads = 32u;
    if (threads > 1024u) threads = 1024u;
    k_control<<<1, threads, 0, st>>>(ctls, nq, mirror, h, use_handle, running_out, T, advance);
    return cudaGetLastError();
}

cudaError_t launch_ctl_reset(QCtl *const *ctls, uint32_t nq, uint32_t max_iter, uint32_t max_rounds,
                             uint32_t max_passes, uint32_t n_levels, unsigned long long cyclic_mask,
                             unsigned long long *box_edges, uint32_t n_boxes, uint32_t n,
                             const uint32_t *box_new_it, unsigned long long nt_read_mask, cudaStream_t st) {
    k_ctl_reset<<<(nq + 255) / 256, 256, 0, st>>>(ctls, nq, max_iter, max_rounds, max_passes, n_levels, cyclic_mask,
                                                  box_edges, n_boxes, n, box_new_it, nt_read_mask);
    return cudaGetLastError();
}

cudaError_t launch_eps_init(const void *eds, uint32_t ned, uint32_t n, cudaStream_t st) {
    if (ned == 0) return cudaSuccess;
    const uint32_t grid = std::min<uint32_t>(2048u, (n + 7u) / 8u);
    k_eps_init<<<grid, 256, 0, st>>>(static_cast<const EpsDesc *>(eds), ned);
    return cudaGetLastError();
}

cudaError_t launch_clear_rows(uint64_t *rows, uint32_t *mark, size_t n_rows, uint32_t W, const uint32_t *all,
                              cudaStream_t st) {
    if (n_rows == 0) return cudaSuccess;
    const uint32_t grid = (uint32_t)std::min<size_t>(2432u, (n_rows + 255u) / 256u);  // 16 CTAs an SM at most
    k_clear_rows<<<grid, 256, 0, st>>>(rows, mark, n_rows, W, all);
    return cudaGetLastError();
}

size_t eps_desc_size() { return sizeof(EpsDesc); }
void fill_eps_desc(void *dst, uint64_t *m2, uint64_t *a2, uint32_t *a2_it, uint32_t *box_new_it, QCtl *ctl,
                   unsigned long long *box_edges, uint32_t n, uint32_t W) {
    EpsDesc d{m2, a2, a2_it, box_new_it, ctl, box_edges, n, W};
    memcpy(dst, &d, sizeof(d));
}

static uint32_t grid_for(size_t work, uint32_t threads, uint32_t cap = 4096) {
    size_t g = (work + threads - 1) / threads;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (uint32_t)g;
}

// Exclusive scan with total: out has n+1 entries.  tmp needs
// ceil(n / kScanChunk) + 1 words.
cudaError_t scan_exclusive(const uint32_t *in, uint32_t *out, size_t n, uint32_t *tmp, cudaStream_t st) {
    const size_t nb = (n + kScanChunk - 1) / kScanChunk;
    if (nb > (size_t)kScanChunk) return cudaErrorInvalidValue;
    if (n == 0) return cudaMemsetAsync(out, 0, sizeof(uint32_t), st);
    k_scan_local<<<(uint32_t)nb, kScanThreads, 0, st>>>(in, out, tmp, n);
    k_scan_sums<<<1, kScanThreads, 0, st>>>(tmp, (uint32_t)nb, tmp + nb);
    k_scan_add<<<(uint32_t)((n + 255) / 256), 256, 0, st>>>(out, tmp, n, tmp + nb, out + n);
    return cudaGetLastError();
}

cudaError_t launch_stage_count(const uint32_t *src, const uint32_t *lbl, const uint32_t *dst, size_t m, uint32_t n,
                               uint32_t n_term, const int32_t *label_map, uint32_t *cnt, int *err, cudaStream_t st) {
    if (m == 0) return cudaSuccess;
    k_stage_count<<<grid_for(m, 256), 256, 0, st>>>(src, lbl, dst, m, n, n_term, label_map, cnt, err);
    return cudaGetLastError();
}
cudaError_t launch_stage_fill(const uint32_t *src, const uint32_t *lbl, const uint32_t *dst, size_t m, uint32_t n,
                              uint32_t n_term, const int32_t *label_map, const uint32_t *off, uint32_t *fill,
                              uint32_t *col, cudaStream_t st) {
    if (m == 0) return cudaSuccess;
    k_stage_fill<<<grid_for(m, 256), 256, 0, st>>>(src, lbl, dst, m, n, n_term, label_map, off, fill, col);
    return cudaGetLastError();
}
cudaError_t launch_stage_unique(const uint32_t *off, uint32_t *col, uint32_t *ucnt, size_t rows, cudaStream_t st) {
    if (rows == 0) return cudaSuccess;
    k_stage_unique<<<grid_for(rows, 128), 128, 0, st>>>(off, col, ucnt, rows);
    return cudaGetLastError();
}
// Shared memory of k_stage_small, 0 when the graph does not fit it.
size_t stage_small_bytes(uint32_t n, uint32_t n_term, size_t m) {
    const uint64_t bytes = ((uint64_t)n * n_term + m) * 4u;
    // (24000 counters: 100 us, as long as the grid-wide kernels take)
    return m <= 16384u && (uint64_t)n * n_term <= 12288u && bytes <= (160u << 10) ? (size_t)std::max<uint64_t>(bytes, 16u) : 0;
}
cudaError_t launch_stage_small(const uint32_t *src, const uint32_t *lbl, const uint32_t *dst, size_t m, uint32_t n,
                               uint32_t n_term, uint32_t counted, uint32_t *csr_off, uint32_t *csr_col,
                               uint32_t *result, cudaStream_t st) {
    const size_t smem = stage_small_bytes(n, n_term, m);
    const cudaError_t e = cudaFuncSetAttribute(k_stage_small, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 << 10);
    if (e != cudaSuccess) return e;
    k_stage_small<<<1, kStageThreads, smem, st>>>(src, lbl, dst, (uint32_t)m, n, n_term, counted, csr_off, csr_col,
                                                  result);
    return cudaGetLastError();
}
cudaError_t launch_stage_compact(const uint32_t *off, const uint32_t *col, const uint32_t *uoff, uint32_t *ucol,
                                 size_t rows, uint32_t n, uint32_t counted, uint32_t *result, cudaStream_t st) {
    if (rows == 0) return cudaSuccess;
    k_stage_compact<<<grid_for(rows, 128), 128, 0, st>>>(off, col, uoff, ucol, rows, n, counted, result);
    return cudaGetLastError();
}
cudaError_t launch_csr_to_bits(const uint32_t *off, const uint32_t *col, size_t rows, uint32_t W, uint64_t *bits,
                               cudaStream_t st) {
    if (rows == 0) return cudaSuccess;
    k_csr_to_bits<<<grid_for(rows, 128), 128, 0, st>>>(off, col, rows, W, bits);
    return cudaGetLastError();
}
cudaError_t launch_csr_to_coo(const uint32_t *off, const uint32_t *col, size_t rows, uint32_t n, uint32_t *coo,
                              cudaStream_t st) {
    if (rows == 0) return cudaSuccess;
    k_csr_to_coo<<<grid_for(rows, 128), 128, 0, st>>>(off, col, rows, n, coo);
    return cudaGetLastError();
}
cudaError_t launch_nonempty_bits(const uint32_t *off, uint32_t n, uint32_t n_term, uint32_t W, uint64_t *bits,
                                 cudaStream_t st) {
    const size_t total = (size_t)n_term * W;
    if (total == 0) return cudaSuccess;
    k_nonempty_bits<<<grid_for(total, 256), 256, 0, st>>>(off, n, n_term, W, bits);
    return cudaGetLastError();
}
cudaError_t launch_popcount(const uint64_t *p, size_t nwords, unsigned long long *out, cudaStream_t st) {
    if (nwords == 0) return cudaSuccess;
    k_popcount<<<grid_for(nwords, 256, 2048), 256, 0, st>>>(p, nwords, out);
    return cudaGetLastError();
}
cudaError_t launch_pack_rows(const uint64_t *src, uint32_t W, uint32_t wn, uint32_t r0, uint32_t rows, uint64_t *out,
                             cudaStream_t st) {
    const size_t words = (size_t)rows * wn;
    if (words == 0) return cudaSuccess;
    k_pack_rows<<<grid_for(words, 256, 2048), 256, 0, st>>>(src, W, wn, r0, words, out);
    return cudaGetLastError();
}
cudaError_t launch_copy_rows(const uint64_t *const *ptrs, const uint32_t *rows, uint32_t njobs, uint32_t W,
                             uint64_t *out, cudaStream_t st) {
    if (njobs == 0) return cudaSuccess;
    k_copy_rows<<<njobs < 4096 ? njobs : 4096, 128, 0, st>>>(ptrs, rows, njobs, W, out);
    return cudaGetLastError();
}

}  // namespace cfpq
