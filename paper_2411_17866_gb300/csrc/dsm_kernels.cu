// CUDA kernels (sm_103a) for one global round of distributed sign momentum
// with local steps (arXiv 2411.17866, Algorithm 1): initialisation, the
// synthetic gradients (K1), the global step (K4) and its statistics (K5).
// The local steps are in dsm_local.cu, the fused round in dsm_fused.cuh.
//
// Every kernel is a grid-stride loop over work items, persistent but for K1
// (whose grid has more CTAs than are resident): tiles of at most kTile = 1024
// elements that lie inside one tensor (for the local steps, a tile of one
// worker).  A CTA of 256 threads takes one item at a time; each thread owns 4
// consecutive elements and moves them with one 16-byte load or store per fp32
// stream (8 bytes per bf16 stream), so every warp instruction covers 512
// contiguous bytes.  (K1 instead runs 64-thread CTAs whose threads own four
// such groups of a tile.)  The local and global steps double-buffer in
// registers: a thread issues the loads of its next item before it computes the
// current one, so the HBM requests of one item are in flight during the
// arithmetic of the previous one.  The work is streaming and elementwise,
// bound by HBM bandwidth (K1: by instruction issue); nothing is a contraction,
// and no tensor core is used.
//
// All method arithmetic uses the explicit round-to-nearest intrinsics
// (__fadd_rn, __fmul_rn, __fdiv_rn, __fsqrt_rn, ...), which the compiler
// never contracts into FMAs, so each result is the fp32 value of the
// paper's expression evaluated one operation at a time (AdamW's divisions use
// fused multiply-adds for the same correctly rounded quotients).

#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "dsm_device.cuh"

namespace dsm {
namespace {

// ---------------------------------------------------------------------------
// Kernels
// ---------------------------------------------------------------------------

// Initial value of element gi (hash init by tensor kind).
__device__ __forceinline__ float init_value(uint32_t kind, float u) {
    if (kind == 0) return __fmul_rn(0.02f, __fsub_rn(__fmul_rn(2.0f, u), 1.0f));
    return kind == 2 ? 1.0f : 0.0f;
}

// Initial state: x (hash init by tensor kind, or as already copied) and every replica = x.  Also the reset of
// the replicas that a lazy round left pending.  Bound by its writes: n 16-byte stores per group of 4 elements
// (with 4-byte accesses, 16 bytes apart between threads, it took 1.26 ms on GPT-2 S with n = 4, 2.5 GB).
__global__ void __launch_bounds__(kThreads) k_init(Problem p, uint64_t key_init, int from_hash) {
    const uint32_t e0 = threadIdx.x * kElemsPerThread;
    wait_previous();
    for (uint32_t ti = blockIdx.x; ti < p.num_tiles; ti += gridDim.x) {
        const TileDesc td = p.tiles[ti];
        const uint32_t kind = p.tensors[td.tensor].kind;
        if (vector_ok(td, e0)) {
            const uint64_t gi = td.start + e0;
            float v[4];
            if (from_hash) {
                const uint64_t h0 = sm64_output(key_init, (gi >> 1) + 1), h1 = sm64_output(key_init, (gi >> 1) + 2);
                v[0] = init_value(kind, draw_even(h0)); v[1] = init_value(kind, draw_odd(h0));
                v[2] = init_value(kind, draw_even(h1)); v[3] = init_value(kind, draw_odd(h1));
                store4(p.x + gi, v);
            } else {
                load4(p.x + gi, v);
            }
            for (uint32_t w = 0; w < p.n; ++w) store4(p.X + w * p.d_stride + gi, v);
        }
        if (uint32_t e; edge_element(td, e)) {
            const uint64_t gi = td.start + e;
            const float v = from_hash ? init_value(kind, hash_uniform(key_init, gi)) : p.x[gi];
            if (from_hash) p.x[gi] = v;
            for (uint32_t w = 0; w < p.n; ++w) p.X[w * p.d_stride + gi] = v;
        }
    }
}

// K1: synthetic gradients of one local step for every worker.  Bound by the
// integer work of the hash (one 64-bit SplitMix64 output per two elements
// and per draw family), not by its write stream.  A CTA of kFillThreads
// threads fills one tile; a thread owns kFillGroups groups of 4 elements
// (group q at 4*thread + q*4*kFillThreads), so it carries 2*kFillGroups
// independent hash chains per family, and every warp store covers 512
// contiguous bytes of fp32 (256 of bf16).
constexpr uint32_t kFillThreads = 64;
constexpr uint32_t kFillGroups = kTile / (4 * kFillThreads);  // 4

// Output j of any family is finalise(key + j*gamma); the j*gamma of a
// group (j = e/2 + 1 and e/2 + 2 for its even first element e) is shared by
// the step family and every worker family.
template <bool kBf16, bool kPrescaled, int kGroups, uint32_t kGroupStride>
__device__ __forceinline__ void grad_fill_groups(const Problem& p, const GradKeys& k, uint64_t gi0, float s,
                                                 float s2) {
    uint64_t jg0[kGroups], jg1[kGroups];
    float a[kGroups][4];
#pragma unroll
    for (int q = 0; q < kGroups; ++q) {
        const uint64_t gi = gi0 + q * kGroupStride;
        jg0[q] = ((gi >> 1) + 1) * kGoldenGamma;
        jg1[q] = jg0[q] + kGoldenGamma;
        const uint64_t h0 = sm64_finalise(k.step + jg0[q]), h1 = sm64_finalise(k.step + jg1[q]);
        if (kPrescaled) {
            a[q][0] = __fmul_rn(s, centred_even(h0)); a[q][1] = __fmul_rn(s, centred_odd(h0));
            a[q][2] = __fmul_rn(s, centred_even(h1)); a[q][3] = __fmul_rn(s, centred_odd(h1));
        } else {
            a[q][0] = step_term(s, draw_even(h0)); a[q][1] = step_term(s, draw_odd(h0));
            a[q][2] = step_term(s, draw_even(h1)); a[q][3] = step_term(s, draw_odd(h1));
        }
    }
    using Elem = typename std::conditional<kBf16, __nv_bfloat16, float>::type;
    Elem* out = reinterpret_cast<Elem*>(p.grad) + gi0;
    for (uint32_t w = 0; w < p.n; ++w, out += p.d_stride) {
#pragma unroll
        for (int q = 0; q < kGroups; ++q) {
            const uint64_t q0 = sm64_finalise(k.worker[w] + jg0[q]), q1 = sm64_finalise(k.worker[w] + jg1[q]);
            float g[4];
            if (kPrescaled) {
                g[0] = __fadd_rn(a[q][0], __fmul_rn(s2, centred_even(q0)));
                g[1] = __fadd_rn(a[q][1], __fmul_rn(s2, centred_odd(q0)));
                g[2] = __fadd_rn(a[q][2], __fmul_rn(s2, centred_even(q1)));
                g[3] = __fadd_rn(a[q][3], __fmul_rn(s2, centred_odd(q1)));
            } else {
                g[0] = grad_value(a[q][0], s2, draw_even(q0)); g[1] = grad_value(a[q][1], s2, draw_odd(q0));
                g[2] = grad_value(a[q][2], s2, draw_even(q1)); g[3] = grad_value(a[q][3], s2, draw_odd(q1));
            }
            if (kBf16) store4_bf16(reinterpret_cast<__nv_bfloat16*>(out) + q * kGroupStride, g);
            else store4(reinterpret_cast<float*>(out) + q * kGroupStride, g);
        }
    }
}

// Element-by-element fill (a tensor's partial groups).
template <bool kBf16>
__device__ __forceinline__ void grad_fill_elem(const Problem& p, const GradKeys& k, uint64_t gi, float s, float s2) {
    const float a = step_term(s, hash_uniform(k.step, gi));
    for (uint32_t w = 0; w < p.n; ++w) {
        const float g = grad_value(a, s2, hash_uniform(k.worker[w], gi));
        const uint64_t o = w * p.d_stride + gi;
        if (kBf16) reinterpret_cast<__nv_bfloat16*>(p.grad)[o] = __float2bfloat16_rn(g);
        else reinterpret_cast<float*>(p.grad)[o] = g;
    }
}

template <bool kBf16>
__global__ void __launch_bounds__(kFillThreads) k_grad_fill(Problem p, GradKeys k) {
    constexpr uint32_t kStride = 4 * kFillThreads;  // elements between a thread's groups
    wait_previous();
    for (uint32_t ti = blockIdx.x; ti < p.num_tiles; ti += gridDim.x) {
        const TileDesc td = p.tiles[ti];
        const TensorDesc& T = p.tensors[td.tensor];
        const float s = T.scale, s2 = T.scale2;
        // one multiplication per draw where both scales allow it (see centred_even)
        const bool pre = fabsf(s) >= kMinPrescaled && fabsf(s2) >= kMinPrescaled;
        const float sp = __fmul_rn(s, kTwoPowM24), sp2 = __fmul_rn(s2, kTwoPowM24);
        if (td.skip() == 0 && td.end() == kTile) {  // a full tile (uniform across the CTA)
            const uint64_t gi0 = td.start + threadIdx.x * 4;
            if (pre) grad_fill_groups<kBf16, true, kFillGroups, kStride>(p, k, gi0, sp, sp2);
            else grad_fill_groups<kBf16, false, kFillGroups, kStride>(p, k, gi0, s, s2);
            continue;
        }
        for (uint32_t e0 = threadIdx.x * 4; e0 < td.end(); e0 += kStride) {  // a ragged tile, group by group
            if (vector_ok(td, e0)) {
                if (pre) grad_fill_groups<kBf16, true, 1, kStride>(p, k, td.start + e0, sp, sp2);
                else grad_fill_groups<kBf16, false, 1, kStride>(p, k, td.start + e0, s, s2);
            } else {
                const uint32_t e1 = min(e0 + 4u, td.end());
                for (uint32_t e = max(e0, td.skip()); e < e1; ++e)
                    grad_fill_elem<kBf16>(p, k, td.start + e, s, s2);
            }
        }
    }
}

// Global step on one element of a partial group, more than 8 workers, by a warp:
// lane l reads workers l and l + 32, and the sums take them in worker order by
// shuffles.  (One thread reading one replica after the other made a tensor's
// partial groups take longer than its tile: 20 us for 64 workers.)
template <int MODE>
__device__ __forceinline__ void global_elem_warp(const Problem& p, const GlobalScalars& g, float lam, uint64_t gi,
                                                 ThreadStats& st) {
    const uint32_t lane = threadIdx.x & 31u;
    float x = p.x[gi], m = p.m[gi], v = MODE == 4 ? p.gv[gi] : 0.f;
    float d[2] = {0.f, 0.f};
#pragma unroll
    for (int k = 0; k < 2; ++k)
        if (lane + 32 * k < p.n) d[k] = __fsub_rn(x, p.X[(lane + 32 * k) * p.d_stride + gi]);
    float r = 0.f;
    if (MODE == 0 && g.sign_mode != 0)
        r = philox_unit(word_of(philox_block((gi >> 2) + g.philox_q0, g.philox_k0, g.philox_k1), gi & 3));
    float acc = 0.f;
#pragma unroll 1
    for (uint32_t i = 0; i < p.n; ++i) acc = __fadd_rn(acc, __shfl_sync(0xffffffffu, i < 32 ? d[0] : d[1], i & 31));
    const float D = __fdiv_rn(acc, g.n_f);
    float u, s;
    global_update<MODE>(D, x, m, v, g, lam, r, u, s);
    bool unan = true;
    float sq[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const float e = __fsub_rn(d[k], D);
        sq[k] = __fmul_rn(e, e);
        if (lane + 32 * k < p.n) unan = unan && sgn(d[k]) == sgn(D);
    }
    unan = __all_sync(0xffffffffu, unan);
    float dr = 0.f;
#pragma unroll 1
    for (uint32_t i = 0; i < p.n; ++i) dr = __fadd_rn(dr, __shfl_sync(0xffffffffu, i < 32 ? sq[0] : sq[1], i & 31));
    if (lane == 0) {
        count_elem<MODE>(D, u, s, unan, g, st);
        csum_add(st.drift, dr);
        p.x[gi] = x;
        p.m[gi] = m;
        if (MODE == 4) p.gv[gi] = v;
    }
    if (!g.skip_reset)
#pragma unroll
        for (int k = 0; k < 2; ++k)
            if (lane + 32 * k < p.n) p.X[(lane + 32 * k) * p.d_stride + gi] = x;
}

// K4: the fused global step (average over the replicas, sign-momentum update,
// momentum update, reset of every replica unless g.skip_reset) with statistics.
// Exactly NW replicas (up to 8), held in registers and double-buffered.
// Statistics: a CTA keeps per-thread sums while its successive tiles belong
// to one tensor and reduces them only when the tensor changes (or at its last
// tile), writing the segment's partial at the segment's last tile.  With a
// grid of G CTAs, tile t is a CTA's last tile of its tensor exactly when
// t + G lies beyond the tensor, so the partials of a tensor are its last
// min(G, tiles) tiles, which K5 sums.
// CTAs per SM: what the double-buffered replicas leave room for (4 for n = 1, 3 up to n = 4, 2 above).
template <int NW, int MODE>
__global__ void __launch_bounds__(kThreads, NW > 4 ? 2 : (NW == 1 ? 4 : 3)) k_global(Problem p, GlobalScalars g) {
    const uint32_t e0 = threadIdx.x * kElemsPerThread;
    constexpr int W = NW;
    uint32_t ti = blockIdx.x;
    if (p.fresh_tables) wait_previous();
    TileDesc nt = p.tiles[ti];
    bool nvec = vector_ok(nt, e0);
    wait_previous();
    float x[4], m[4], v[4] = {0.f, 0.f, 0.f, 0.f}, r[W][4];
    ThreadStats st;
    if (nvec) {
        load4(p.x + nt.start + e0, x);
        load4(p.m + nt.start + e0, m);
        if (MODE == 4) load4(p.gv + nt.start + e0, v);
#pragma unroll
        for (int i = 0; i < W; ++i) load4(p.X + i * p.d_stride + nt.start + e0, r[i]);
    }
    for (; ti < p.num_tiles; ti += gridDim.x) {
        const TileDesc td = nt;
        const bool vec = nvec;
        float cx[4], cm[4], cv[4], cr[W][4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            cx[j] = x[j];
            cm[j] = m[j];
            cv[j] = v[j];
#pragma unroll
            for (int i = 0; i < W; ++i) cr[i][j] = r[i][j];
        }
        const uint32_t next = ti + gridDim.x;
        if (next < p.num_tiles) {
            nt = p.tiles[next];
            nvec = vector_ok(nt, e0);
            if (nvec) {
                load4(p.x + nt.start + e0, x);
                load4(p.m + nt.start + e0, m);
                if (MODE == 4) load4(p.gv + nt.start + e0, v);
#pragma unroll
                for (int i = 0; i < W; ++i) load4(p.X + i * p.d_stride + nt.start + e0, r[i]);
            }
        }
        const float lam = p.tensors[td.tensor].lam_global;
        if (vec) {
            const uint64_t gi = td.start + e0;  // a multiple of 4: the four words of one Philox block
            float ru[4] = {0.f, 0.f, 0.f, 0.f};
            if (MODE == 0 && g.sign_mode != 0) {
                const uint4 b = philox_block((gi >> 2) + g.philox_q0, g.philox_k0, g.philox_k1);
                ru[0] = philox_unit(b.x); ru[1] = philox_unit(b.y); ru[2] = philox_unit(b.z); ru[3] = philox_unit(b.w);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float dif[W];
#pragma unroll
                for (int i = 0; i < W; ++i) dif[i] = __fsub_rn(cx[j], cr[i][j]);
                global_elem<W, MODE>(cx[j], cm[j], cv[j], dif, g, lam, ru[j], st);
            }
            store4(p.x + gi, cx);
            store4(p.m + gi, cm);
            if (MODE == 4) store4(p.gv + gi, cv);
            if (!g.skip_reset) {
#pragma unroll
                for (int i = 0; i < W; ++i) store4(p.X + i * p.d_stride + gi, cx);
            }
        }
        if (uint32_t e; edge_element(td, e)) {
            const uint64_t gj = td.start + e;
            float xs = p.x[gj], ms = p.m[gj], vs = MODE == 4 ? p.gv[gj] : 0.f, dif[W];
#pragma unroll
            for (int i = 0; i < W; ++i) dif[i] = __fsub_rn(xs, p.X[i * p.d_stride + gj]);
            float r = 0.f;
            if (MODE == 0 && g.sign_mode != 0)
                r = philox_unit(word_of(philox_block((gj >> 2) + g.philox_q0, g.philox_k0, g.philox_k1), gj & 3));
            global_elem<W, MODE>(xs, ms, vs, dif, g, lam, r, st);
            p.x[gj] = xs;
            p.m[gj] = ms;
            if (MODE == 4) p.gv[gj] = vs;
            if (!g.skip_reset) {
#pragma unroll
                for (int i = 0; i < W; ++i) p.X[i * p.d_stride + gj] = xs;
            }
        }
        if (next >= p.num_tiles || nt.tensor != td.tensor) {  // uniform across the CTA
            reduce_stats(st, p.partials + ti);
            st = ThreadStats();
        }
    }
    if (p.sum_stats) sum_stats(p, gridDim.x);
}

// reduce_stats() over the CTAs of a cluster: each one's sums in its shared memory, added in rank order by the first.
__device__ __forceinline__ void reduce_stats_cluster(const ThreadStats& st, StatPartial* out) {
    __shared__ StatPartial s_part;
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    reduce_stats(st, &s_part);
    cluster.sync();
    if (cluster.block_rank() == 0 && threadIdx.x == 0) {
        StatPartial o = s_part;
        for (uint32_t r = 1; r < cluster.num_blocks(); ++r) {
            const StatPartial q = *cluster.map_shared_rank(&s_part, r);
            o.delta_sq += q.delta_sq; o.drift += q.drift;
            o.zero_sign += q.zero_sign; o.flips += q.flips; o.unanimous += q.unanimous; o.clamped += q.clamped;
        }
        *out = o;
    }
    cluster.sync();  // no CTA ends, or writes its sums again, before they are read
}

// K4 for more than 8 workers (up to NW): the replicas of a thread's E elements in registers, all of their loads in
// flight at once, no second read for the statistics.  NW * E is 64: 4 elements a thread up to 16 workers, 2 up to 32,
// 1 up to 64, a tile by a cluster of 4 / E CTAs that add up their statistics through distributed shared memory, or by
// one CTA in as many passes.  Bound by HBM bandwidth; 2 CTAs per SM hold 128 KB of loads in flight.  16
// workers of 16 M parameters, reset deferred (1.28 GB): 223 us, against 330 us with 8 replicas at a time and a second
// read from L2 for the statistics; 2 elements a thread in 4 CTAs per SM spill and are slower, in 3 the same.
template <int NW, int E, int MODE, bool kCluster>
__global__ void __launch_bounds__(kThreads, 2) k_global_many(Problem p, GlobalScalars g) {
    constexpr uint32_t parts = kCluster ? 4 / E : 1;
    const uint32_t part = blockIdx.x % parts, clusters = gridDim.x / parts;
    uint32_t ti = blockIdx.x / parts;
    if (p.fresh_tables) wait_previous();
    TileDesc nt = p.tiles[ti];
    wait_previous();
    ThreadStats st;
    for (; ti < p.num_tiles; ti += clusters) {
        const TileDesc td = nt;
        const uint32_t next = ti + clusters;
        if (next < p.num_tiles) nt = p.tiles[next];
        const float lam = p.tensors[td.tensor].lam_global;
#pragma unroll 1
        for (uint32_t e = (part * kThreads + threadIdx.x) * E; e < kTile && e < td.end(); e += parts * kThreads * E) {
            if (!vector_ok(td, e & ~3u)) continue;
            const uint64_t gi = td.start + e;
            float x[E], m[E], v[E], r[NW][E];
            load_elems(p.x + gi, x);
            // eight workers at a time, the last one again in the place of any beyond it, so that the loads are straight-
            // line code: with a test of i for each, global AdamW for 64 workers waited for one load after the other
            // (283 k parameters: 58 instead of 35 us)
#pragma unroll
            for (int i = 0; i < NW; i += 8) {
                if (i < p.n) {
#pragma unroll
                    for (int k = 0; k < 8; ++k) load_elems(p.X + min(i + k, int(p.n) - 1) * p.d_stride + gi, r[i + k]);
                }
            }
            load_elems(p.m + gi, m);
            if (MODE == 4) load_elems(p.gv + gi, v);
            float ru[E];
#pragma unroll
            for (int j = 0; j < E; ++j) ru[j] = 0.f;
            if (MODE == 0 && g.sign_mode != 0) {
                const uint4 b = philox_block((gi >> 2) + g.philox_q0, g.philox_k0, g.philox_k1);
#pragma unroll
                for (int j = 0; j < E; ++j) ru[j] = philox_unit(word_of(b, (e + j) & 3u));
            }
            // the differences x - x_i, their sum in worker order, their extremes
            float acc[E], lo[E], hi[E];
#pragma unroll
            for (int j = 0; j < E; ++j) { acc[j] = 0.f; lo[j] = INFINITY; hi[j] = -INFINITY; }
#pragma unroll
            for (int i = 0; i < NW; ++i) {
                if (i < p.n) {
#pragma unroll
                    for (int j = 0; j < E; ++j) {
                        r[i][j] = __fsub_rn(x[j], r[i][j]);
                        acc[j] = __fadd_rn(acc[j], r[i][j]);
                        lo[j] = fminf(lo[j], r[i][j]);
                        hi[j] = fmaxf(hi[j], r[i][j]);
                    }
                }
            }
            float D[E], dr[E];
#pragma unroll
            for (int j = 0; j < E; ++j) {
                D[j] = __fdiv_rn(acc[j], g.n_f);
                float u, s;
                global_update<MODE>(D[j], x[j], m[j], v[j], g, lam, ru[j], u, s);
                count_elem<MODE>(D[j], u, s, same_signs(D[j], lo[j], hi[j]), g, st);
                dr[j] = 0.f;
            }
            store_elems(p.x + gi, x);
            store_elems(p.m + gi, m);
            if (MODE == 4) store_elems(p.gv + gi, v);
            if (!g.skip_reset) {
#pragma unroll
                for (int i = 0; i < NW; ++i)
                    if (i < p.n) store_elems(p.X + i * p.d_stride + gi, x);
            }
#pragma unroll
            for (int i = 0; i < NW; ++i) {
                if (i < p.n) {
#pragma unroll
                    for (int j = 0; j < E; ++j) {
                        const float d = __fsub_rn(r[i][j], D[j]);
                        dr[j] = __fadd_rn(dr[j], __fmul_rn(d, d));
                    }
                }
            }
#pragma unroll
            for (int j = 0; j < E; ++j) csum_add(st.drift, dr[j]);
        }
        // the last warps of the last CTA first, as edge_element()
        if (uint32_t ee; part == parts - 1 && edge_at(td, kThreads / 32 - 1 - threadIdx.x / 32, ee))
            global_elem_warp<MODE>(p, g, lam, td.start + ee, st);
        if (next >= p.num_tiles || nt.tensor != td.tensor) {  // uniform across the cluster (as in k_global)
            if (kCluster) reduce_stats_cluster(st, p.partials + ti);
            else reduce_stats(st, p.partials + ti);
            st = ThreadStats();
        }
    }
    if (p.sum_stats) sum_stats(p, clusters);
}

// K5: per-tensor statistics from the tile partials, in a fixed order: a
// tensor's partials are its last min(G, tiles) tiles for a producing grid of
// G CTAs (see K4).
__global__ void __launch_bounds__(kThreads) k_stats(Problem p, uint32_t producer_grid) {
    const uint32_t T = blockIdx.x;
    if (p.fresh_tables) wait_previous();
    const TensorDesc td = p.tensors[T];
    wait_previous();
    double a = 0.0, b = 0.0;
    unsigned long long c0 = 0, c1 = 0, c2 = 0, c3 = 0;
    const uint32_t first =
        td.tile_end - td.tile_begin > producer_grid ? td.tile_end - producer_grid : td.tile_begin;
    // each thread sums partials first + tid, first + tid + 256, ...; the loads of up to 4 of them are
    // issued before their additions (a tensor has at most producer_grid partials)
    for (uint32_t t0 = first + threadIdx.x; t0 < td.tile_end; t0 += 4 * kThreads) {
        StatPartial q[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (t0 + u * kThreads < td.tile_end) q[u] = p.partials[t0 + u * kThreads];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (t0 + u * kThreads < td.tile_end) {
                a += q[u].delta_sq; b += q[u].drift;
                c0 += q[u].zero_sign; c1 += q[u].flips; c2 += q[u].unanimous; c3 += q[u].clamped;
            }
        }
    }
    // the lanes of each warp by shuffles in a fixed pattern, then the warps in order
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, off);
        b += __shfl_down_sync(0xffffffffu, b, off);
        c0 += __shfl_down_sync(0xffffffffu, c0, off);
        c1 += __shfl_down_sync(0xffffffffu, c1, off);
        c2 += __shfl_down_sync(0xffffffffu, c2, off);
        c3 += __shfl_down_sync(0xffffffffu, c3, off);
    }
    __shared__ double s_d[kThreads / 32][2];
    __shared__ unsigned long long s_c[kThreads / 32][4];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
        s_d[warp][0] = a; s_d[warp][1] = b;
        s_c[warp][0] = c0; s_c[warp][1] = c1; s_c[warp][2] = c2; s_c[warp][3] = c3;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        TensorStats o;
        o.delta_sq = 0.0; o.drift = 0.0;
        o.zero_sign = o.flips = o.unanimous = o.clamped = 0;
        for (int w = 0; w < kThreads / 32; ++w) {
            o.delta_sq += s_d[w][0]; o.drift += s_d[w][1];
            o.zero_sign += s_c[w][0]; o.flips += s_c[w][1]; o.unanimous += s_c[w][2]; o.clamped += s_c[w][3];
        }
        p.stats[T] = o;
    }
}

using GlobalKernel = void (*)(Problem, GlobalScalars);

template <int MODE>
GlobalKernel global_kernel_mode(uint32_t n, bool cluster) {
    switch (n) {
        case 1: return k_global<1, MODE>;
        case 2: return k_global<2, MODE>;
        case 3: return k_global<3, MODE>;
        case 4: return k_global<4, MODE>;
        case 5: return k_global<5, MODE>;
        case 6: return k_global<6, MODE>;
        case 7: return k_global<7, MODE>;
        case 8: return k_global<8, MODE>;
        default: break;
    }
    if (n <= 16) return k_global_many<16, 4, MODE, false>;
    if (n <= 32) return cluster ? k_global_many<32, 2, MODE, true> : k_global_many<32, 2, MODE, false>;
    return cluster ? k_global_many<64, 1, MODE, true> : k_global_many<64, 1, MODE, false>;
}

GlobalKernel global_kernel_for(uint32_t n, int mode, bool cluster) {
    switch (mode) {
        case 1: return global_kernel_mode<1>(n, cluster);
        case 2: return global_kernel_mode<2>(n, cluster);
        case 3: return global_kernel_mode<3>(n, cluster);
        case 4: return global_kernel_mode<4>(n, cluster);
        default: return global_kernel_mode<0>(n, cluster);
    }
}

}  // namespace

cudaError_t query_global_shape(const Problem& p, LaunchShape* out) {
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    err = cudaDeviceGetAttribute(&out->sms, cudaDevAttrMultiProcessorCount, dev);
    if (err != cudaSuccess) return err;
    out->grid_global = grid_for(global_kernel_for(p.n, p.global_mode, false), out->sms);
    return cudaGetLastError();
}

cudaError_t query_launch_shape(const Problem& p, const TensorDesc* tensors, LaunchShape* out) {
    const cudaError_t err = query_global_shape(p, out);
    if (err != cudaSuccess) return err;
    const int sms = out->sms;
    out->grid_init = grid_for(k_init, sms);
    // K1 runs up to 300 CTAs per SM, of which 20 are resident: bound by
    // instruction issue, it gains when a CTA's end makes room for the next
    // (us a fill, 20 / 80 / 300 CTAs per SM / one CTA a tile: GPT-2 S, n = 4,
    // fp32 339 / 328 / 325 / 325; n = 1 141.6 / 135.6 / 134.1 / 135.2; GPT-2 M,
    // n = 4, bf16 1018 / 979 / 970 / 969; 1 M, n = 4 4.9 for 20 as for 300).
    constexpr int kFillCtasPerSm = 300;
    out->grid_grad = kFillCtasPerSm * sms;
    cudaError_t e = query_local_shape(p, out);
    if (e != cudaSuccess) return e;
    if (fused_round_available(p) && (e = query_fused_shape(p, tensors, out)) != cudaSuccess) return e;
    return cudaGetLastError();
}

cudaError_t launch_init(const Problem& p, const LaunchShape& ls, uint64_t key_init, int from_hash, cudaStream_t s) {
    const int grid = clamp_grid(ls.grid_init, p.num_tiles);
    if (grid == 0) return cudaSuccess;
    return launch(k_init, grid, kThreads, 0, s, false, p, key_init, from_hash);
}

cudaError_t launch_grad_fill(const Problem& p, const LaunchShape& ls, const GradKeys& k, cudaStream_t s) {
    const int grid = clamp_grid(ls.grid_grad, p.num_tiles);
    if (grid == 0) return cudaSuccess;
    return launch(p.grad_bf16 ? k_grad_fill<true> : k_grad_fill<false>, grid, kFillThreads, 0, s, p.early, p, k);
}

// CTAs that share a tile in the global step for more than 8 workers: a cluster of 4 / E (see k_global_many) as long as
// every tile's then runs at the same time; beyond that one CTA takes a tile in 4 / E passes, which leaves no CTA
// waiting for another's sums.  Rounds of one SGD-momentum step, 64 workers, one CTA / clusters: 3 k parameters 20.8 /
// 12.1 us, 30 k 23.5 / 14.9, 200 k (784 CTAs) 61.9 / 59.4, 283 k 85.2 / 90.8, 4 M 1100 / 1151.
static uint32_t tile_ctas(const Problem& p, const LaunchShape& ls) {
    const uint32_t parts = p.n <= 16 ? 1 : (p.n <= 32 ? 2 : 4);
    return uint64_t(p.num_tiles) * parts <= static_cast<uint64_t>(ls.grid_global) ? parts : 1;
}

cudaError_t launch_global(const Problem& p, const LaunchShape& ls, const GlobalScalars& g, cudaStream_t s,
                          uint32_t* grid_used) {
    const uint32_t parts = tile_ctas(p, ls);
    const int tiles = clamp_grid(ls.grid_global, p.num_tiles);  // (clusters of) CTAs
    *grid_used = static_cast<uint32_t>(tiles);
    if (tiles == 0) return cudaSuccess;
    // For a model so small that a round is its launches the last of K4's CTAs sums the statistics, and K5 is not
    // launched: up to 8 tiles.  Rounds of one SGD-momentum step, us, without / with K5 (n = 1, 4, 8, 16, 40): 2 tiles
    // 5.8 / 6.9, 6.4 / 7.0, 7.0 / 7.6, 9.5 / 9.6, 10.5 / 11.4; 8 tiles 5.8 / 7.0, 6.6 / 7.2, 7.2 / 7.7, 9.0 / 9.6,
    // 11.6 / 11.9; 10 tiles 6.9 / 7.0, 7.5 / 7.4, 8.6 / 7.8, 9.9 / 9.9, 12.3 / 12.1; 24 tiles 7.5 / 7.0, 7.6 / 7.4,
    // 8.2 / 8.1, 10.2 / 10.0, 13.0 / 13.1; 244 tiles, n = 4, 14.4 / 10.1.  Between, 4 and 6 tiles gain 2 to 8% but
    // for n = 8 (2% the other way).  Not so in the fused round's kernel, which runs 5% slower on large models for
    // having that code (GPT-2-shaped 184 M, n = 4: 6085 against 5778 us).
    constexpr uint32_t kSumStatsTiles = 8;
    Problem q = p;
    q.sum_stats = p.num_tiles <= kSumStatsTiles && p.num_tensors <= 4 * kSumStatsTiles;
    if (q.sum_stats) *grid_used = 0;
    return launch_clusters(global_kernel_for(p.n, p.global_mode, parts > 1), tiles * static_cast<int>(parts), parts,
                           kThreads, 0, s, p.early, q, g);
}

cudaError_t launch_stats(const Problem& p, uint32_t producer_grid, cudaStream_t s) {
    if (producer_grid == 0) return cudaSuccess;
    return launch(k_stats, static_cast<int>(p.num_tensors), kThreads, 0, s, p.early, p, producer_grid);
}

}  // namespace dsm
