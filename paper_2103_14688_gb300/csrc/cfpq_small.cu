// cfpq_small.cu -- whole fixpoint of a small query in one CTA.
//
// When a query's device state (closure blocks, M2, A2, stamps) fits in the
// shared memory of one SM, the index-creation loop of Listing 1 (arXiv
// 2103.14688, Sec. 3.1) runs inside a single CTA: the same level schedule,
// edge channels and dirty stamps as the multi-kernel path (cfpq_kernels.cu),
// with a barrier between passes instead of kernel launches.  Rows are at
// most 512 bits wide (W <= 8 words), so each thread owns one output row per
// step and keeps it in registers.  At the end the closure blocks and M2 are
// copied to the query's global buffers, where every result call reads them.
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <vector>

#include "cfpq_engine.cuh"

namespace cfpq {

constexpr uint32_t kSmallMaxW = 8;
constexpr int kSmallMaxThreads = 512;  // 128 registers a thread: 1024 threads would spill

// One source of a block (SrcDesc without the pointers), read as one 16-byte
// shared-memory load.
struct alignas(16) SmallSrc {
    uint32_t kind, label;
    uint32_t flags;  // bit 0: ident, bit 1: same level
    int32_t rblk;
};

// One level: its blocks lvl_blk[blk0 .. blk0 + nblk), and what its first pass
// of an iteration reads: the boxes of its nonterminal sources, the levels
// below that its sources read blocks of, whether it has terminal sources.
struct alignas(16) SmallLevel {
    uint32_t blk0, nblk, has_term, any_box;  // any_box: a nonterminal source of a box >= 64
    unsigned long long boxes, reads;
};

struct SmallDesc {
    uint32_t n, W, B, nblk, n_levels, max_iter, max_passes;
    uint32_t magic;           // ceil(2^32 / n): item / n = umulhi(item, magic) while item * n < 2^32; 0 for n = 1
    uint32_t meta_words;      // words of the plan's tables at `meta` (a multiple of 4)
    uint32_t o_srcs, o_blk, o_src0, o_nsrc, o_f0, o_nf, o_null, o_fb, o_box;  // word offsets in `meta` (levels at 0)
    // Every box's answer is one block, on the last level, which does not
    // repeat and reads no nonterminal: its rows are extracted by the thread that
    // computed them (o_box: block -> box or ~0).
    uint32_t fuse;
    uint32_t pad;
    unsigned long long cyclic_mask;
    const uint32_t *meta;
    const uint32_t *csr_off;  // label l, vertex x: csr_off[l * n + x] .. csr_off[l * n + x + 1]
    const uint32_t *csr_col;
    uint64_t *blk_out;        // nblk * n * W
    uint64_t *m2_out;         // B * n * W
    QCtl *ctl;                // statistics written at the end
};

// Latency-bound: a query of this size holds a few thousand row words, and its
// fixpoint is a chain of thousands of dependent passes (two coprime cycles of
// 63 and 64 vertices: 4033 iterations, 12099 passes).  So what a pass costs
// is counted in barriers and in dependent shared-memory loads:
//   - the plan's tables and the graph's CSR are copied to shared memory when
//     they fit beside the state (`meta_smem`, `csr_smem`);
//   - a level whose first pass has nothing to read in this iteration (no new
//     terminal or box edge, no lower level that changed) is counted and passed
//     over without a barrier: what decides it is the same in every thread
//     (register masks of the boxes and levels that changed);
//   - a pass has one barrier, which also carries the "some row changed" flag;
//     counters stay in registers until the end;
//   - where the last level allows it (SmallDesc::fuse) extraction is no phase of
//     its own;
//   - whether the tables and the CSR are in shared memory is known at compile
//     time (SMEM), which makes their loads 32-bit shared ones.
// Two cycles 63 / 64: 23.1 -> 9.7 ms (1.9 us a pass before, with four barriers,
// divisions and table loads from global memory; 11.3 with extraction apart and
// generic loads); the regular query (ab)*c|a*b* at n = 200: 620 -> 142 us.
template <uint32_t W, bool SMEM>
__global__ void __launch_bounds__(kSmallMaxThreads, 1)
    k_small_fixpoint(const SmallDesc *__restrict__ desc, uint32_t meta_smem, uint32_t csr_smem, uint32_t csr_rows,
                     uint32_t csr_m) {
    if (SMEM) meta_smem = csr_smem = 1u;
    const SmallDesc &D = *desc;
    const uint32_t n = D.n, B = D.B, nblk = D.nblk;
    extern __shared__ __align__(16) uint64_t sm[];
    uint64_t *C = sm;
    uint64_t *M2 = C + (size_t)nblk * n * W;
    uint64_t *A2 = M2 + (size_t)B * n * W;
    uint32_t *stamp = reinterpret_cast<uint32_t *>(A2 + (size_t)B * n * W);
    uint32_t *last = stamp + (size_t)nblk * n;
    uint32_t *a2it = last + nblk;
    uint32_t *boxit = a2it + (size_t)B * n;
    const uint32_t words32 = nblk * n + nblk + B * n + B;
    __shared__ unsigned long long s_new, s_ors, s_rows;
    const uint32_t tid = threadIdx.x, T = blockDim.x;

    const uint32_t words64 = (nblk + 2u * B) * n * W;
    for (uint32_t i = tid; i < words64; i += T) sm[i] = 0ull;
    for (uint32_t i = tid; i < words32; i += T) stamp[i] = 0u;
    uint32_t *extra = stamp + ((words32 + 3u) & ~3u);  // 16-byte aligned: the tables, then the CSR
    uint32_t *const s_csr = extra + (meta_smem ? D.meta_words : 0u);
    if (meta_smem)
        for (uint32_t i = tid; i < D.meta_words; i += T) extra[i] = D.meta[i];
    if (csr_smem) {
        for (uint32_t i = tid; i <= csr_rows; i += T) s_csr[i] = D.csr_off[i];
        for (uint32_t i = tid; i < csr_m; i += T) s_csr[csr_rows + 1u + i] = D.csr_col[i];
    }
    const uint32_t *const meta = SMEM ? extra : meta_smem ? extra : D.meta;
    const uint32_t *const csr_off = SMEM ? s_csr : csr_smem ? s_csr : D.csr_off;
    const uint32_t *const csr_col = SMEM ? s_csr + csr_rows + 1u : csr_smem ? s_csr + csr_rows + 1u : D.csr_col;
    if (tid == 0) { s_new = 0; s_ors = 0; s_rows = 0; }
    __syncthreads();
    const SmallLevel *levels = reinterpret_cast<const SmallLevel *>(meta);
    const SmallSrc *srcs = reinterpret_cast<const SmallSrc *>(meta + D.o_srcs);
    const uint32_t *lvl_blk = meta + D.o_blk, *blk_src0 = meta + D.o_src0, *blk_nsrc = meta + D.o_nsrc;
    const uint32_t *box_f0 = meta + D.o_f0, *box_nf = meta + D.o_nf, *nullable = meta + D.o_null;
    const uint32_t *fblocks = meta + D.o_fb, *blk_box = meta + D.o_box;
    const bool fuse = D.fuse != 0u;
    const uint32_t n_levels = D.n_levels, magic = D.magic, max_passes = D.max_passes;
    const unsigned long long cyclic_mask = D.cyclic_mask;

    unsigned long long edges_eps = 0, my_new = 0;
    unsigned long long new_boxes = 0;  // boxes (< 64) with edges new in this iteration
    bool new_any = false;              // some box has
    uint32_t my_ors = 0, my_rows = 0;
    // epsilon rows: M2^b[i,i] = A2^b[i,i] = 1 for boxes whose start state is final
    for (uint32_t b = 0; b < B; ++b) {
        if (!nullable[b]) continue;
        for (uint32_t x = tid; x < n; x += T) {
            M2[(b * n + x) * W + (x >> 6)] = 1ull << (x & 63);
            A2[(b * n + x) * W + (x >> 6)] = 1ull << (x & 63);
            a2it[b * n + x] = 1;
        }
        if (tid == 0) boxit[b] = 1;
        edges_eps += n;
        new_any = true;
        if (b < 64u) new_boxes |= 1ull << b;
    }
    __syncthreads();

    uint32_t g = 2, iter = 1, passes = 0, iters_done = 0, status = kStatusOk;
    bool done = false;
    while (!done) {
        const uint32_t g0 = g;
        unsigned long long lvl_changed = 0;  // levels that changed in this iteration
        bool added = false;
        for (uint32_t L = 0; L < n_levels && !done; ++L) {
            const SmallLevel lv = levels[L];
            const bool cyc = (cyclic_mask >> L) & 1ull;
            const bool fused = fuse && L + 1u == n_levels;
            bool active = (iter == 1u && lv.has_term) || (lv.boxes & new_boxes) != 0ull || (lv.any_box && new_any) ||
                          (lv.reads & lvl_changed) != 0ull;
            uint32_t mode = kModeNew;
            while (true) {
                bool ch_any = false;
                const uint32_t items = active ? lv.nblk * n : 0u;
                for (uint32_t item = tid; item < items; item += T) {
                    const uint32_t bi = magic ? __umulhi(item, magic) : item, x = item - bi * n;
                    const uint32_t b = lvl_blk[lv.blk0 + bi];
                    uint64_t acc[W];
#pragma unroll
                    for (uint32_t w = 0; w < W; ++w) acc[w] = 0ull;
                    bool any = false;
                    const uint32_t k0 = blk_src0[b], k1 = k0 + blk_nsrc[b];
                    for (uint32_t k = k0; k < k1; ++k) {
                        const SmallSrc s = srcs[k];
                        uint32_t chans = 0;
                        if (mode == kModeNew) {
                            const bool term1 = s.kind == 0 && iter == 1;
                            if (term1 || (s.kind == 1 && boxit[s.label] == iter)) chans |= 1u;
                            if (s.rblk >= 0 && !(s.flags & 2u) && !term1 && last[s.rblk] >= g0) chans |= 2u;
                        } else if (s.rblk >= 0 && (s.flags & 2u) && last[s.rblk] + 1u >= g) {
                            chans |= 4u;
                        }
                        for (uint32_t cb = 1u; cb <= chans; cb <<= 1) {
                            if (!(chans & cb)) continue;
                            const bool new_edges = cb == 1u;
                            const bool ident = new_edges && (s.flags & 1u);
                            if (!ident && s.rblk < 0) continue;
                            const uint32_t thr = new_edges ? 0u : (cb == 2u ? g0 : g - 1u);
                            const uint32_t *rstamp = stamp + (s.rblk >= 0 ? (uint32_t)s.rblk * n : 0u);
                            const uint64_t *rrow = C + (s.rblk >= 0 ? (uint32_t)s.rblk * n * W : 0u);
                            auto take = [&](uint32_t y) __attribute__((always_inline)) {
                                if (ident && s.kind == 0) {
                                    const uint64_t bit = 1ull << (y & 63);
#pragma unroll
                                    for (uint32_t w = 0; w < W; ++w) acc[w] |= (y >> 6) == w ? bit : 0ull;
                                    any = true;
                                }
                                if (s.rblk >= 0 && (thr == 0u || rstamp[y] >= thr)) {
                                    const ulonglong2 *r = reinterpret_cast<const ulonglong2 *>(rrow + y * W);
#pragma unroll
                                    for (uint32_t w = 0; w < W / 2; ++w) {
                                        const ulonglong2 v = r[w];
                                        acc[2 * w] |= v.x;
                                        acc[2 * w + 1] |= v.y;
                                    }
                                    any = true;
                                    ++my_ors;
                                }
                            };
                            if (s.kind == 0) {
                                const uint32_t *off = csr_off + s.label * n + x;
                                const uint32_t e1 = off[1];
                                for (uint32_t e = off[0]; e < e1; ++e) take(csr_col[e]);
                            } else {
                                if (new_edges && a2it[s.label * n + x] != iter) continue;
                                const uint64_t *adj = (new_edges ? A2 : M2) + (s.label * n + x) * W;
                                if (ident) {  // the row's product edges into t are the row itself
#pragma unroll
                                    for (uint32_t w = 0; w < W; ++w) acc[w] |= adj[w];
                                    any = true;
                                    if (s.rblk < 0) continue;
                                }
#pragma unroll 1
                                for (uint32_t w = 0; w < W; ++w) {
                                    uint64_t bits = adj[w];
                                    while (bits) {
                                        const uint32_t y = w * 64u + (uint32_t)__ffsll((long long)bits) - 1u;
                                        bits &= bits - 1;
                                        take(y);
                                    }
                                }
                            }
                        }
                    }
                    if (!any) continue;
                    uint64_t *o = C + (b * n + x) * W;
                    bool ch = false;
#pragma unroll
                    for (uint32_t w = 0; w < W; ++w) {
                        const uint64_t old = o[w];
                        if (acc[w] & ~old) {
                            o[w] = old | acc[w];
                            ch = true;
                        }
                    }
                    if (ch) {
                        stamp[b * n + x] = g;
                        last[b] = g;
                        ++my_rows;
                        if (!fused) ch_any = true;
                        const uint32_t box = fused ? blk_box[b] : 0xFFFFFFFFu;
                        if (box != 0xFFFFFFFFu) {  // the row's new pairs
                            uint64_t *m = M2 + (box * n + x) * W, *a = A2 + (box * n + x) * W;
                            bool has = false;
#pragma unroll
                            for (uint32_t w = 0; w < W; ++w) {
                                acc[w] = o[w] & ~m[w];
                                has |= acc[w] != 0ull;
                            }
                            if (has) {
#pragma unroll
                                for (uint32_t w = 0; w < W; ++w) {
                                    a[w] = acc[w];
                                    m[w] |= acc[w];
                                    my_new += (unsigned long long)__popcll(acc[w]);
                                }
                                a2it[box * n + x] = iter + 1;
                                boxit[box] = iter + 1;
                                ch_any = true;
                            }
                        }
                    }
                }
                // (a fused level's flag says whether pairs were added)
                const bool changed = active && __syncthreads_or(ch_any) != 0;
                if (fused) added = changed;
                if (changed) lvl_changed |= 1ull << L;
                ++passes;
                g += 1;
                if (passes >= max_passes) {
                    status = kStatusPassCap;
                    done = true;
                    break;
                }
                if (cyc && changed) {
                    mode = kModeProp;
                    continue;
                }
                break;
            }
        }
        if (done) break;
        // extraction: new = OR_f C[q0, f] & ~M2 on rows changed this iteration
        bool has_new = false;
        for (uint32_t item = tid; item < B * n && !fuse; item += T) {
            const uint32_t b = magic ? __umulhi(item, magic) : item, x = item - b * n;
            const uint32_t f0 = box_f0[b], f1 = f0 + box_nf[b];
            uint64_t cand[W];
#pragma unroll
            for (uint32_t w = 0; w < W; ++w) cand[w] = 0ull;
            bool any = false;
            for (uint32_t f = f0; f < f1; ++f) {
                const uint32_t fb = fblocks[f];
                if (stamp[fb * n + x] < g0) continue;
                any = true;
                const uint64_t *r = C + (fb * n + x) * W;
#pragma unroll
                for (uint32_t w = 0; w < W; ++w) cand[w] |= r[w];
            }
            if (!any) continue;
            uint64_t *m = M2 + item * W;
            uint64_t *a = A2 + item * W;
            bool has = false;
#pragma unroll
            for (uint32_t w = 0; w < W; ++w) {
                cand[w] &= ~m[w];
                has |= cand[w] != 0ull;
            }
            if (!has) continue;
#pragma unroll
            for (uint32_t w = 0; w < W; ++w) {
                a[w] = cand[w];
                m[w] |= cand[w];
                my_new += (unsigned long long)__popcll(cand[w]);
            }
            a2it[item] = iter + 1;
            boxit[b] = iter + 1;
            has_new = true;
        }
        if (!fuse) added = __syncthreads_or(has_new) != 0;
        iters_done = iter;
        if (!added) break;
        if (D.max_iter && iter >= D.max_iter) {
            status = kStatusIterCap;
            break;
        }
        ++iter;
        new_any = true;
        new_boxes = 0ull;
        for (uint32_t b = 0; b < B && b < 64u; ++b)
            if (boxit[b] == iter) new_boxes |= 1ull << b;
    }
    if (my_new) atomicAdd(&s_new, my_new);
    if (my_ors) atomicAdd(&s_ors, (unsigned long long)my_ors);
    if (my_rows) atomicAdd(&s_rows, (unsigned long long)my_rows);
    __syncthreads();
    for (uint32_t i = tid; i < nblk * n * W; i += T) D.blk_out[i] = C[i];
    for (uint32_t i = tid; i < B * n * W; i += T) D.m2_out[i] = M2[i];
    if (tid == 0) {
        QCtl c;
        memset(&c, 0, sizeof(c));
        c.g = g;
        c.iter = iter;
        c.phase = kPhaseDone;
        c.status = status;
        c.iters_done = iters_done;
        c.passes = passes;
        c.edges_total = edges_eps + s_new;
        c.row_ors = s_ors;
        c.rounds_total = passes;
        c.rows_changed_total = s_rows;
        c.n_levels = D.n_levels;
        c.cyclic_mask = D.cyclic_mask;
        *D.ctl = c;
    }
}

size_t small_smem_bytes(uint32_t n, uint32_t W, uint32_t B, uint32_t nblk) {
    return (size_t)(nblk + 2 * B) * n * W * 8 + ((size_t)nblk * n + nblk + (size_t)B * n + B) * 4;
}

size_t small_desc_size() { return sizeof(SmallDesc); }

// Largest dynamic shared memory a CTA may use on the current device.
size_t small_smem_limit() {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) return 0;
    return (size_t)v > 2048 ? (size_t)v - 2048 : 0;  // room for the static shared variables
}

// The query's tables go to shared memory when they fit beside the state, and
// then the graph's CSR (csr_rows offsets and csr_m columns).  threads: the
// items of the largest level (one row each), at most 512 -- a barrier over
// fewer warps is cheaper.
cudaError_t launch_small_fixpoint(const void *desc, uint32_t W, size_t state_smem, size_t meta_bytes, uint64_t csr_rows,
                                  uint64_t csr_m, uint32_t max_items, cudaStream_t st) {
    size_t smem = (state_smem + 15) & ~(size_t)15;
    const size_t limit = small_smem_limit();
    const uint32_t meta_smem = smem + meta_bytes <= limit ? 1u : 0u;
    if (meta_smem) smem += meta_bytes;
    const uint64_t csr_bytes = (csr_rows + 1 + csr_m) * 4;
    const uint32_t csr_smem = smem + csr_bytes <= limit ? 1u : 0u;
    if (csr_smem) smem += csr_bytes;
    const uint32_t threads = max_items >= (uint32_t)kSmallMaxThreads ? (uint32_t)kSmallMaxThreads
                                                                     : (max_items < 64u ? 64u : (max_items + 31u) & ~31u);
    auto run = [&](auto kernel) -> cudaError_t {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        kernel<<<1, threads, smem, st>>>(static_cast<const SmallDesc *>(desc), meta_smem, csr_smem, (uint32_t)csr_rows,
                                         (uint32_t)csr_m);
        return cudaGetLastError();
    };
    const bool both = meta_smem && csr_smem;
    switch (W) {
        case 2: return both ? run(k_small_fixpoint<2, true>) : run(k_small_fixpoint<2, false>);
        case 4: return both ? run(k_small_fixpoint<4, true>) : run(k_small_fixpoint<4, false>);
        case 6: return both ? run(k_small_fixpoint<6, true>) : run(k_small_fixpoint<6, false>);
        case 8: return both ? run(k_small_fixpoint<8, true>) : run(k_small_fixpoint<8, false>);
        default: return cudaErrorInvalidValue;
    }
}

// Host-side packing of one query's plan: the tables the kernel reads (levels,
// sources, blocks by level, boxes) as words, and the descriptor.
std::vector<uint32_t> build_small_plan(const QueryDev &q, void *desc_out) {
    const uint32_t nblk = (uint32_t)q.blocks.size();
    std::vector<SmallLevel> lv(q.n_levels);
    std::vector<SmallSrc> src;
    std::vector<uint32_t> by_level;
    for (uint32_t L = 0; L < q.n_levels; ++L) {
        memset(&lv[L], 0, sizeof(SmallLevel));
        lv[L].blk0 = (uint32_t)by_level.size();
        for (uint32_t b = 0; b < nblk; ++b) {
            if (q.blk_level[b] != L) continue;
            by_level.push_back(b);
            for (uint32_t k = 0; k < q.blk_nsrc[b]; ++k) {
                const auto &s = q.srcs[q.blk_src0[b] + k];
                if (s.label_kind == 0) lv[L].has_term = 1u;
                else if (s.label < 64u) lv[L].boxes |= 1ull << s.label;
                else lv[L].any_box = 1u;
                if (s.rblk >= 0 && !s.same_level) lv[L].reads |= 1ull << q.blk_level[(size_t)s.rblk];
            }
        }
        lv[L].nblk = (uint32_t)by_level.size() - lv[L].blk0;
    }
    for (const auto &s : q.srcs)
        src.push_back(SmallSrc{s.label_kind, s.label, (s.ident ? 1u : 0u) | (s.same_level ? 2u : 0u), s.rblk});
    std::vector<uint32_t> m;
    auto put = [&](const void *p, size_t bytes) {
        const uint32_t at = (uint32_t)m.size();
        m.resize(at + bytes / 4);
        if (bytes) memcpy(m.data() + at, p, bytes);
        return at;
    };
    SmallDesc d;
    memset(&d, 0, sizeof(d));
    put(lv.data(), lv.size() * sizeof(SmallLevel));
    d.o_srcs = put(src.data(), src.size() * sizeof(SmallSrc));  // (16-byte records up to here)
    d.o_blk = put(by_level.data(), by_level.size() * 4);
    d.o_src0 = put(q.blk_src0.data(), q.blk_src0.size() * 4);
    d.o_nsrc = put(q.blk_nsrc.data(), q.blk_nsrc.size() * 4);
    d.o_f0 = put(q.box_f0.data(), q.box_f0.size() * 4);
    d.o_nf = put(q.box_nf.data(), q.box_nf.size() * 4);
    std::vector<uint32_t> null_box(q.B);
    for (uint32_t b = 0; b < q.B; ++b) null_box[b] = q.rsm.final_[q.rsm.box_start[b]] ? 1u : 0u;
    d.o_null = put(null_box.data(), null_box.size() * 4);
    d.o_fb = put(q.fblocks.data(), q.fblocks.size() * 4);
    std::vector<uint32_t> box_of(nblk, 0xFFFFFFFFu);
    bool fuse = q.n_levels > 0 && !((q.cyclic_mask >> (q.n_levels - 1u)) & 1ull);
    for (uint32_t b = 0; b < q.B; ++b) {
        if (q.box_nf[b] == 0) continue;
        const uint32_t fb = q.fblocks[q.box_f0[b]];
        fuse = fuse && q.box_nf[b] == 1u && q.blk_level[fb] + 1u == q.n_levels;
        box_of[fb] = b;
    }
    for (uint32_t b = 0; b < nblk && fuse; ++b)
        for (uint32_t k = 0; k < q.blk_nsrc[b] && q.blk_level[b] + 1u == q.n_levels; ++k)
            fuse = fuse && q.srcs[q.blk_src0[b] + k].label_kind == 0;
    d.o_box = put(box_of.data(), box_of.size() * 4);
    d.fuse = fuse ? 1u : 0u;
    while (m.size() % 4) m.push_back(0u);
    d.n = q.n;
    d.W = q.W;
    d.B = q.B;
    d.nblk = nblk;
    d.n_levels = q.n_levels;
    d.magic = (uint32_t)((0x100000000ull + q.n - 1) / q.n);  // (n = 1: wraps to 0)
    d.meta_words = (uint32_t)m.size();
    d.cyclic_mask = q.cyclic_mask;
    memcpy(desc_out, &d, sizeof(d));
    return m;
}

void finish_small_desc(void *desc, const uint32_t *meta, uint32_t max_iter, uint32_t max_passes,
                       const uint32_t *csr_off, const uint32_t *csr_col, uint64_t *blk_out, uint64_t *m2_out,
                       QCtl *ctl) {
    SmallDesc *d = static_cast<SmallDesc *>(desc);
    d->meta = meta;
    d->max_iter = max_iter;
    d->max_passes = max_passes;
    d->csr_off = csr_off;
    d->csr_col = csr_col;
    d->blk_out = blk_out;
    d->m2_out = m2_out;
    d->ctl = ctl;
}

}  // namespace cfpq
