// kernels_render.cu -- variants of the forward kernel for emission/absorption compositing
// (with and without gradient checkpoints), the adjoint, the longest-ray-first tile order and
// the decision trace.  The forward kernel template and its building blocks are in
// render_common.cuh.
#include "render_common.cuh"

namespace volrc {
namespace {

// ------------------------------------------------------------------ adjoint

__device__ __forceinline__ void red4(float4* p, float a, float b, float c, float d) {
    asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d));
}

// dL/dtf accumulates in 256-entry tables, one or more per warp, in global memory (L2), an entry's 4
// channels by one 16-byte reduction; k_sum_tables adds the tables up.  (Floating-point additions in shared
// memory are compare-and-swap loops, four of them per entry.)  Measured with the gradient quads
// below and the segment's values kept in shared memory, 256^3, 16 views of 512x512: the adjoint
// 7.0 -> 4.25 ms (with the pairs of the reverse sweep 3.72); 101x90x77 with 3 levels, 3 views of 203x151: 0.55 -> 0.26 ms.
__device__ __forceinline__ void flush_dtf4(float4* tab, int idx, float2 rg, float2 ba) {
    if (rg.x != 0.0f || rg.y != 0.0f || ba.x != 0.0f || ba.y != 0.0f) red4(tab + idx, rg.x, rg.y, ba.x, ba.y);
}
__device__ __forceinline__ void flush_dtf(float4* tab, int idx, float2 acc[4]) {
    if (idx >= 0) {
        flush_dtf4(tab, idx, acc[0], acc[1]);
        flush_dtf4(tab, idx + 1, acc[2], acc[3]);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[c] = f2(0.0f);
}

// Adds the corner accumulators of trilinear cell `cell` to the level's gradient quads: entry
// (x, y, z) collects the gradients of voxels (x, y), (x+1, y), (x, y+1), (x+1, y+1) of slice z, so a
// cell is two 16-byte reductions, at its lower corner's entry and the one a slice above (a slice of
// padding takes those past the last).  Corners past an edge have weight 0.  k_gather_quads adds
// the quads up per voxel.
__device__ __forceinline__ void flush_quad(float4* gq, long long cell, long long slice, float2 cacc[4]) {
    if (cell >= 0) {
        red4(gq + cell, cacc[0].x, cacc[0].y, cacc[1].x, cacc[1].y);
        red4(gq + cell + slice, cacc[2].x, cacc[2].y, cacc[3].x, cacc[3].y);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) cacc[r] = f2(0.0f);
}

// Adds the corner accumulators of trilinear cell `cell` (linear index of its lower corner;
// cacc[cy + 2 cz] holds the corners at x and x + 1; mask: which +1 corners exist) to dvox, row by row (x-neighbour
// pairs), skipping rows that do not exist or hold only zeros.  (16-byte vector atomics for the
// pairs measured 2% slower than these scalar ones on the 16 x 512^2 workload.)
__device__ __forceinline__ void flush_vox(float* dvox, long long cell, int mask, int Dx, int Dy, float2 cacc[4]) {
    if (cell >= 0) {
        const long long sy = Dx, sz = (long long)Dx * Dy;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int cy = r & 1, cz = r >> 1;
            const bool row_ok = (!cy || (mask & 2)) && (!cz || (mask & 4));
            const float v0 = cacc[r].x, v1 = (mask & 1) ? cacc[r].y : 0.0f;
            if (!row_ok || (v0 == 0.0f && v1 == 0.0f)) continue;
            const long long L = cell + cy * sy + cz * sz;
            if (v0 != 0.0f) atomicAdd(dvox + L, v0);
            if (v1 != 0.0f) atomicAdd(dvox + L + 1, v1);
        }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) cacc[r] = f2(0.0f);
}

// Samples per lane whose page-table lookups and gathers the adjoint's forward recompute issues
// together.
#ifndef VOLRC_BWD_BATCH
#define VOLRC_BWD_BATCH 4
#endif
constexpr int kBwdBatch = VOLRC_BWD_BATCH;
// Adjoint CTA size and the resident CTAs per SM its register allocation must allow (shared
// memory per CTA: 4 KiB + 256 B per thread).
// 160 threads: 49 KiB and up to 102 registers; 192 threads (57 KiB, 80 registers) leave the L1 next to
// nothing and spill (16 views of 512x512, 256^3: forward + adjoint 7.72 against 7.97 ms; 128 threads at
// 6 CTAs 8.30).
constexpr int kBwdThreads = 160;
constexpr int kBwdMinBlocks = 4;

// Adjoint, warp-synchronous by checkpoint segment: a warp takes 32 rays (a ray tile, or a
// 32-pixel part of it) and, round by round, processes segment s of every one of them that has
// it (samples 32 s .. 32 s + 31, the last one partial), s descending from the longest ray's last
// segment: first forward -- transmittance from the segment's checkpoint and the sample values
// into shared memory, kBwdBatch samples at a time -- then in reverse, accumulating dL/dtf and
// dL/dvoxel.  Neighbouring rays then sample neighbouring depths in each round, as in the forward
// march, which keeps the gathers and the dL/dvoxel reductions of a round together in the cache.
// (With checkpoints before every sample -- the store-all debug mode -- a segment is one sample
// and its transmittance is read, not recomputed.)
// LOD: samples on footprint levels; the gradient of a level-l voxel goes to P.dlev[l], which
// the host then carries down to level 0 through the box filter's adjoint.
// TAPE: the segment's sample values are read from the forward's value tape instead of being
// interpolated again from the bricks (the transmittance is recomputed from the checkpoint either way).
template <int DT, bool LOD, bool TAPE>
__global__ void __launch_bounds__(kBwdThreads, kBwdMinBlocks) k_backward(const __grid_constant__ BackwardDev P) {
    __shared__ float4 s_tf[256];
    __shared__ float4 s_tfd[255];  // tf[i+1] - tf[i], each difference rounded once
    // the lane's dL/dtf table: lane l adds to copy l mod dtf_copies of its warp's
    float4* const w_dtf = P.dtf_tabs + (((long long)blockIdx.x * (kBwdThreads / 32) + (threadIdx.x >> 5)) * P.dtf_copies +
                                        ((int)threadIdx.x & (P.dtf_copies - 1))) * 256;
    __shared__ float s_T[kCkptEvery][kBwdThreads];
    __shared__ float s_V[kCkptEvery][kBwdThreads];  // (a lane's tape values are 128 B apart from its neighbour's: read once)
    __shared__ LevelDev s_lv[LOD ? kMaxLevels : 1];
    for (int i = threadIdx.x; i < 256; i += blockDim.x) s_tf[i] = P.tf[i];
    for (int i = threadIdx.x; i < 255; i += blockDim.x) {
        const float4 a = P.tf[i], b = P.tf[i + 1];
        s_tfd[i] = make_float4(__fsub_rn(b.x, a.x), __fsub_rn(b.y, a.y), __fsub_rn(b.z, a.z), __fsub_rn(b.w, a.w));
    }
    if (LOD && threadIdx.x < P.vol.nlevels) s_lv[threadIdx.x] = P.vol.lv[threadIdx.x];
    __syncthreads();

    using VT = typename Voxel<DT>::T;
    const VT* __restrict__ atlas = (const VT*)P.vol.atlas;
    const unsigned lane = threadIdx.x & 31;
    const int tid = threadIdx.x;
    const int bshift = P.vol.bshift, bmask = P.vol.bmask, B1 = P.vol.B1;
    const bool quad = P.vol.quad != 0;
    const int row = quad ? B1 - 1 : B1;
    const unsigned long long slot_stride = quad ? P.vol.slot_entries : P.vol.slot_elems;
    LvReg L0 = load_lv(P.vol.lv[0]);  // LOD: the level of the last resolved sample
    // voxels along x and y of level l (the shared level table when LOD)
    auto dim_x = [&](int l) { return LOD ? s_lv[l].D[0] : P.vol.lv[0].D[0]; };
    auto dim_y = [&](int l) { return LOD ? s_lv[l].D[1] : P.vol.lv[0].D[1]; };
    int cur_l = 0;
    const int nlev = P.vol.nlevels;
    const float step = P.step;
    // per-lane accumulators: dL/dtf for entries acc_i, acc_i + 1; dL/dvoxel for the 8 corners
    // of cell cell_cur on level cell_lvl (cell_mask: which +1 corners exist)
    int acc_i = -1;
    float2 acc[4] = {f2(0.f), f2(0.f), f2(0.f), f2(0.f)};   // entry acc_i: red, green; blue, alpha; then acc_i + 1
    long long cell_cur = -1;
    int cell_mask = 0, cell_lvl = 0;
    float2 cacc[4] = {f2(0.f), f2(0.f), f2(0.f), f2(0.f)};  // corners (x, x + 1) of rows y + 2 z

    // lane state: the lane's ray, its sample count n and segment count nseg
    bool has = false;
    long long ray = 0;
    float o0 = 0, o1 = 0, o2 = 0, d0 = 0, d1 = 0, d2 = 0, t0 = 0, lodscale = 0;
    float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
    float2 R01 = f2(0.f), R23 = f2(0.f);  // what lies behind the sample: colour, opacity
    int n = 0, nseg = 0;
    // warp-uniform: the segment index every lane processes in this round, descending; each
    // lane's rays sample the same depths as its neighbours' (adjacent pixels), so the gathers
    // and the dL/dvoxel reductions of a round stay close together in the volume
    int s = -1;
    const int tile_px = P.tile_w * P.tile_h;
    const int chunks = (tile_px + 31) >> 5;  // work items per tile: 32 rays each

    for (;;) {
        if (s < 0) {
            // ---- the next 32 rays: one tile, or a 32-pixel part of a larger one
            int item = 0;
            if (lane == 0) item = (int)atomicAdd(&P.counters[kWork], 1u);
            item = __shfl_sync(kFull, item, 0);
            if (item >= P.nwork) break;
            const int ti = item / chunks, part = item - ti * chunks;
            const int tile = P.tile_order ? P.tile_order[ti] : ti;
            const int v = find_view_tile(P.views, P.nviews, tile);
            const ViewDev& V = P.views[v];
            const int tl = tile - V.tile_off;
            const int idx = part * 32 + (int)lane;
            const int px = (tl % V.tiles_x) * P.tile_w + idx % P.tile_w;
            const int py = (tl / V.tiles_x) * P.tile_h + idx / P.tile_w;
            has = false;
            nseg = 0;
            if (idx < tile_px && px < V.w && py < V.h) {
                ray = V.ray_off + (long long)py * V.w + px;
                n = P.ray_n[ray];
                if (n > 0) {
                    Ray R;
                    make_ray(V, P.vol.D0f, px, py, R);
                    o0 = R.o[0]; o1 = R.o[1]; o2 = R.o[2];
                    d0 = R.d[0]; d1 = R.d[1]; d2 = R.d[2];
                    t0 = R.t0;
                    lodscale = V.lodscale;
                    g = P.drgba[ray];
                    R01 = make_float2(P.bg.x, P.bg.y);
                    R23 = make_float2(P.bg.z, P.bg.w);
                    nseg = ((n - 1) >> P.ckpt_shift) + 1;
                    has = true;
                }
            }
            s = __reduce_max_sync(kFull, nseg) - 1;
            if (s < 0) continue;
        }

        // ---- one round: segment s (2^ckpt_shift <= kCkptEvery samples) of every lane's ray that has it
        const bool seg = has && s < nseg;
        const int k0 = s << P.ckpt_shift;
        const int len = seg ? min(1 << P.ckpt_shift, n - k0) : 0;
        float T = (seg && s > 0) ? P.ckpt[(long long)(s - 1) * P.nrays + ray] : 1.0f;
        const int maxlen = __reduce_max_sync(kFull, len);
        // the lane's segment on the tape: 32 values in 128 contiguous bytes
        const float* tp = TAPE ? P.tape + ((long long)s * P.nrays + (seg ? ray : 0)) * kCkptEvery : nullptr;
        if (TAPE) {
            // forward from the tape, a 32-byte sector at a time (the lanes' values lie 128 bytes apart)
            constexpr int TW = 8;
            for (int jb = 0; jb < maxlen; jb += TW) {
                float vv[TW];
#pragma unroll
                for (int q = 0; q < TW; q += 4) {
                    const float4 v4 = jb + q < len ? __ldg(reinterpret_cast<const float4*>(tp + jb + q)) : make_float4(0.f, 0.f, 0.f, 0.f);
                    vv[q] = v4.x, vv[q + 1] = v4.y, vv[q + 2] = v4.z, vv[q + 3] = v4.w;
                }
#pragma unroll
                for (int u = 0; u < TW; ++u) {
                    if (jb + u < len) {
                        int i;
                        float wt;
                        tf_index<DT>(vv[u], i, wt);
                        const float al = fmaf(wt, s_tfd[i].w, s_tf[i].w);
                        s_T[jb + u][tid] = T;
                        s_V[jb + u][tid] = vv[u];
                        T = T * (1.0f - al);
                    }
                }
            }
        }
        // forward: decisions, then the page-table lookups, then the gathers of kBwdBatch samples
        for (int jb = 0; !TAPE && jb < maxlen; jb += kBwdBatch) {
            uint32_t pti[kBwdBatch], loc[kBwdBatch];
            float wv[kBwdBatch][3];
            const float kf = (float)(k0 + jb);  // + u stays exact: indices are below 2^24
#pragma unroll
            for (int u = 0; u < kBwdBatch; ++u) {
                const float t = __fadd_rn(t0, __fmul_rn(__fadd_rn(kf, (float)u), step));
                const float p[3] = {__fadd_rn(o0, __fmul_rn(t, d0)), __fadd_rn(o1, __fmul_rn(t, d1)),
                                    __fadd_rn(o2, __fmul_rn(t, d2))};
                if (LOD) {
                    const int l = lod_level(t, lodscale, P.lod_bias, nlev);
                    if (l != cur_l) {
                        cur_l = l;
                        L0 = load_lv(s_lv[l]);
                    }
                }
                Resolved Q;
                resolve_reg(L0, bshift, bmask, row, p, Q);
                pti[u] = Q.pti;
                loc[u] = Q.local;
                wv[u][0] = Q.w[0];
                wv[u][1] = Q.w[1];
                wv[u][2] = Q.w[2];
            }
            uint32_t slot[kBwdBatch];
#pragma unroll
            for (int u = 0; u < kBwdBatch; ++u) slot[u] = __ldg(P.vol.pt + (jb + u < len ? pti[u] : 0u));
            float val[kBwdBatch];
#pragma unroll
            for (int u = 0; u < kBwdBatch; ++u) {
                const bool use = jb + u < len && slot[u] != kInvalidSlot;
                const unsigned long long base = use ? (unsigned long long)slot[u] * slot_stride + loc[u] : 0ull;
                val[u] = quad ? trilinear_quad<DT>(P.vol.atlas, base, B1 - 1, wv[u])
                              : trilinear<DT>(atlas, base, B1, wv[u]);
            }
#pragma unroll
            for (int u = 0; u < kBwdBatch; ++u) {
                if (jb + u < len) {
                    if (slot[u] == kInvalidSlot) atomicAdd(&P.counters[kDevError], 1u);
                    int i;
                    float wt;
                    tf_index<DT>(val[u], i, wt);
                    const float al = fmaf(wt, s_tfd[i].w, s_tf[i].w);
                    s_T[jb + u][tid] = T;
                    s_V[jb + u][tid] = val[u];
                    T = T * (1.0f - al);
                }
            }
        }
        float kf = (float)(k0 + maxlen - 1);  // (float)(k0 + j), stepped down exactly
        for (int j = maxlen - 1; j >= 0; --j, kf = __fsub_rn(kf, 1.0f)) {
            if (j < len) {
                // (the arithmetic goes by packed pairs: channels, axes x and y, corners x and x + 1;
                // the kernel is bound by instruction issue)
                float2 w01 = f2(0.f);  // the sample's weights and voxel: only dL/dvoxel needs them
                float w2 = 0.f;
                int i0 = 0, i1 = 0, i2 = 0;
                if (P.dvox) {
                    const float t = __fadd_rn(t0, __fmul_rn(kf, step));
                    if (LOD) {
                        const int l = lod_level(t, lodscale, P.lod_bias, nlev);
                        if (l != cur_l) {
                            cur_l = l;
                            L0 = load_lv(s_lv[l]);
                        }
                    }
                    // resolve_reg's positions and clamp (level 0: the ratio is exactly 1)
                    const float nz = P.neg_zero;
                    float2 x01 = add2(make_float2(o0, o1), mul2(f2(t), make_float2(d0, d1), nz));
                    float x2 = __fadd_rn(o2, __fmul_rn(t, d2));
                    if (LOD) {
                        x01 = mul2(x01, make_float2(L0.r[0], L0.r[1]), nz);
                        x2 = __fmul_rn(x2, L0.r[2]);
                    }
                    x01 = add2(x01, f2(-0.5f));
                    x2 = __fsub_rn(x2, 0.5f);
                    x01 = make_float2(fminf(fmaxf(x01.x, 0.0f), L0.Dm[0]), fminf(fmaxf(x01.y, 0.0f), L0.Dm[1]));
                    x2 = fminf(fmaxf(x2, 0.0f), L0.Dm[2]);
                    const float2 fl01 = make_float2(floorf(x01.x), floorf(x01.y));
                    const float fl2 = floorf(x2);
                    w01 = fma2(fl01, f2(-1.0f), x01);
                    w2 = __fsub_rn(x2, fl2);
                    i0 = (int)fl01.x;
                    i1 = (int)fl01.y;
                    i2 = (int)fl2;
                }
                const float val = s_V[j][tid];
                const float Tk = s_T[j][tid];
                int i;
                float wt;
                tf_index<DT>(val, i, wt);
                const float4 a = s_tf[i], b = s_tfd[i];
                const float2 b01 = make_float2(b.x, b.y), b23 = make_float2(b.z, b.w);
                const float2 c01 = fma2(f2(wt), b01, make_float2(a.x, a.y)), c23 = fma2(f2(wt), b23, make_float2(a.z, a.w));
                const float al = c23.y;
                const float2 e01 = fma2(R01, f2(-1.0f), c01), e23 = fma2(R23, f2(-1.0f), make_float2(c23.x, 1.0f));
                const float2 g01 = make_float2(g.x, g.y), g23 = make_float2(g.z, g.w);
                const float2 ge = fma2(g01, e01, fma2(g23, e23, f2(0.0f)));
                const float dal = Tk * (ge.x + ge.y);
                const float Ta = Tk * al;
                const float2 q01 = fma2(g01, f2(Ta), f2(0.0f));         // dL/d(red, green) of the row
                const float2 q23 = make_float2(g.z * Ta, dal);          // blue, alpha
                R01 = fma2(f2(al), e01, R01);
                R23 = fma2(f2(al), e23, R23);
                if (P.dtf) {
                    // register accumulation while the TF index stays the same
                    if (i != acc_i) {
                        // to a neighbouring index the entry both lookups share stays in registers:
                        // only the one left behind is added to the table
                        const bool up = i == acc_i + 1, down = i == acc_i - 1;
                        if (acc_i >= 0 && (up || down)) {
                            flush_dtf4(w_dtf, up ? acc_i : acc_i + 1, up ? acc[0] : acc[2], up ? acc[1] : acc[3]);
                            const float2 k0 = up ? acc[2] : acc[0], k1 = up ? acc[3] : acc[1];
                            acc[0] = up ? k0 : f2(0.0f);
                            acc[1] = up ? k1 : f2(0.0f);
                            acc[2] = up ? f2(0.0f) : k0;
                            acc[3] = up ? f2(0.0f) : k1;
                        } else {
                            flush_dtf(w_dtf, acc_i, acc);
                        }
                        acc_i = i;
                    }
                    const float w0 = 1.0f - wt;
                    acc[0] = fma2(f2(w0), q01, acc[0]);
                    acc[1] = fma2(f2(w0), q23, acc[1]);
                    acc[2] = fma2(f2(wt), q01, acc[2]);
                    acc[3] = fma2(f2(wt), q23, acc[3]);
                }
                if (P.dvox && tf_inside<DT>(val)) {
                    const float2 qb = fma2(q01, b01, fma2(q23, b23, f2(0.0f)));
                    const float dv = 255.0f * (qb.x + qb.y);
                    if (dv != 0.0f) {
                        // register accumulation while the trilinear cell (and level) stays the same
                        const int lq = LOD ? cur_l : 0;
                        const int Dx = (int)L0.Dm[0] + 1, Dy = (int)L0.Dm[1] + 1;
                        const long long cell = (long long)i0 + (long long)Dx * ((long long)i1 + (long long)Dy * i2);
                        if (cell != cell_cur || lq != cell_lvl) {
                            if (P.gq[0])
                                flush_quad(P.gq[cell_lvl], cell_cur, (long long)dim_x(cell_lvl) * dim_y(cell_lvl), cacc);
                            else
                                flush_vox(P.dlev[cell_lvl], cell_cur, cell_mask, dim_x(cell_lvl), dim_y(cell_lvl), cacc);
                            cell_cur = cell;
                            cell_lvl = lq;
                            cell_mask = ((float)i0 < L0.Dm[0] ? 1 : 0) | ((float)i1 < L0.Dm[1] ? 2 : 0) |
                                        ((float)i2 < L0.Dm[2] ? 4 : 0);
                        }
                        const float2 wx = make_float2(1.0f - w01.x, w01.x);
                        const float v0 = (1.0f - w2) * dv, v1 = w2 * dv, wy0 = 1.0f - w01.y;
                        cacc[0] = fma2(wx, f2(wy0 * v0), cacc[0]);
                        cacc[1] = fma2(wx, f2(w01.y * v0), cacc[1]);
                        cacc[2] = fma2(wx, f2(wy0 * v1), cacc[2]);
                        cacc[3] = fma2(wx, f2(w01.y * v1), cacc[3]);
                    }
                }
            }
        }
        --s;
    }
    if (P.dtf) flush_dtf(w_dtf, acc_i, acc);
    if (P.dvox) {
        if (P.gq[0]) flush_quad(P.gq[cell_lvl], cell_cur, (long long)dim_x(cell_lvl) * dim_y(cell_lvl), cacc);
        else flush_vox(P.dlev[cell_lvl], cell_cur, cell_mask, dim_x(cell_lvl), dim_y(cell_lvl), cacc);
    }
}

// dtf[entry] += the sums of the entries over the tables: a CTA takes 8 entries (a 128-byte line of
// every table) of one in kSumSlices slices of the tables and sums them in binary64.
constexpr int kSumThreads = 256, kSumSlices = 16;

__global__ void __launch_bounds__(kSumThreads) k_sum_tables(const float4* __restrict__ tabs, int n, float* dtf) {
    __shared__ double s_sum[kSumThreads / 8][8][4];
    const int q = threadIdx.x & 7, r = threadIdx.x >> 3;
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    for (int t = (int)blockIdx.y * (kSumThreads / 8) + r; t < n; t += kSumSlices * (kSumThreads / 8)) {
        const float4 a = tabs[(long long)t * 256 + blockIdx.x * 8 + q];
        v[0] += a.x;
        v[1] += a.y;
        v[2] += a.z;
        v[3] += a.w;
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) s_sum[r][q][c] = v[c];
    __syncthreads();
    if (threadIdx.x < 32) {
        double sum = 0.0;
        for (int w = 0; w < kSumThreads / 8; ++w) sum += s_sum[w][threadIdx.x >> 2][threadIdx.x & 3];
        if (sum != 0.0) atomicAdd(dtf + blockIdx.x * 32 + threadIdx.x, (float)sum);
    }
}

// dvox[voxel] += (level 0) or = the sum of the gradient quads' components that belong to it.
__global__ void __launch_bounds__(256) k_gather_quads(const float4* __restrict__ gq, float* __restrict__ dvox, int Dx, int Dy,
                                                      int Dz, int add) {
    const long long n = (long long)Dx * Dy * Dz;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(i % Dx), y = (int)(i / Dx % Dy);
        float v = gq[i].x;
        if (x > 0) v += gq[i - 1].y;
        if (y > 0) v += gq[i - Dx].z;
        if (x > 0 && y > 0) v += gq[i - Dx - 1].w;
        if (add) {
            if (v != 0.0f) dvox[i] += v;
        } else {
            dvox[i] = v;
        }
    }
}

// ------------------------------------------------------------------ scheduling

// Work order for the next frame: tiles bucketed by floor(log2(cost + 1)), buckets in descending
// order, where a tile's cost is the sample count of its longest ray.  The longest rays start
// first, so none of them begins near the end of the launch and runs on while other SMs idle
// (ordering by the tile's total samples instead left a tail: c2 0.91 -> 0.81 ms with this key).
constexpr int kOrderThreads = 256;

__device__ __forceinline__ int cost_bucket(int c) { return 31 - __clz(c + 1); }

// buckets[0..31]: tiles per bucket; one thread per tile, one global atomic per bucket per block
__global__ void __launch_bounds__(kOrderThreads) k_order_count(const int* cost, int ntiles, int* buckets) {
    __shared__ int s_count[32];
    if (threadIdx.x < 32) s_count[threadIdx.x] = 0;
    __syncthreads();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < ntiles) atomicAdd(&s_count[cost_bucket(cost[i])], 1);
    __syncthreads();
    if (threadIdx.x < 32 && s_count[threadIdx.x]) atomicAdd(&buckets[threadIdx.x], s_count[threadIdx.x]);
}

// order[] = tiles grouped by bucket, highest bucket first; each block reserves its places in
// every bucket with one atomic on the bucket's fill cursor (buckets[32 + b]).  Zeroes cost[].
__global__ void __launch_bounds__(kOrderThreads) k_order_scatter(int* cost, int* order, int ntiles, int* buckets) {
    __shared__ int s_count[32], s_base[32];
    if (threadIdx.x < 32) s_count[threadIdx.x] = 0;
    __syncthreads();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int b = i < ntiles ? cost_bucket(cost[i]) : 0;
    const int rank = i < ntiles ? atomicAdd(&s_count[b], 1) : 0;
    __syncthreads();
    if (threadIdx.x < 32) {
        int base = 0;
        for (int q = 31; q > (int)threadIdx.x; --q) base += buckets[q];
        s_base[threadIdx.x] = s_count[threadIdx.x] ? base + atomicAdd(&buckets[32 + threadIdx.x], s_count[threadIdx.x]) : 0;
    }
    __syncthreads();
    if (i < ntiles) {
        order[s_base[b] + rank] = i;
        cost[i] = 0;
    }
}

// The same in one launch of one CTA, for a few tiles: the lanes of a warp on one bucket add to it
// together.  Up to kOrderSmall tiles (a 512 x 512 view) that takes no longer than the two kernels
// above, and their launches and the zeroing of the buckets go: what a small frame's time is made of.

__global__ void __launch_bounds__(1024) k_order_small(int* cost, int* order, int ntiles) {
    __shared__ int s_count[32], s_next[32];
    if (threadIdx.x < 32) s_count[threadIdx.x] = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int i0 = 0; i0 < ntiles; i0 += 1024) {
        const int i = i0 + (int)threadIdx.x;
        const int b = i < ntiles ? cost_bucket(cost[i]) : -1;
        const unsigned m = __match_any_sync(kFull, b);
        if (b >= 0 && lane == __ffs(m) - 1) atomicAdd(&s_count[b], __popc(m));
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        int base = 0;
        for (int q = 31; q > lane; --q) base += s_count[q];
        s_next[lane] = base;
    }
    __syncthreads();
    for (int i0 = 0; i0 < ntiles; i0 += 1024) {
        const int i = i0 + (int)threadIdx.x;
        const int b = i < ntiles ? cost_bucket(cost[i]) : -1;
        const unsigned m = __match_any_sync(kFull, b);
        const int leader = __ffs(m) - 1;
        int base = 0;
        if (b >= 0 && lane == leader) base = atomicAdd(&s_next[b], __popc(m));
        base = __shfl_sync(kFull, base, leader);
        if (b >= 0) {
            order[base + __popc(m & ((1u << lane) - 1u))] = i;
            cost[i] = 0;
        }
    }
}

// ------------------------------------------------------------------ trace

__global__ void k_trace(const __grid_constant__ TraceDev P) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= P.npix) return;
    Ray R;
    make_ray(P.view, P.vol.D0f, P.pixels[2 * q], P.pixels[2 * q + 1], R);
    int k = 0;
    if (R.hit) {
        float t = R.t0;
        int l = 0;
        for (;; ++k) {
            t = P.level_step ? (k ? next_t_level_step(t, P.step, l) : R.t0) : __fadd_rn(R.t0, __fmul_rn((float)k, P.step));
            if (!(t < R.t1)) break;
            l = P.lod_mode ? lod_level(t, P.view.lodscale, P.lod_bias, P.vol.nlevels) : 0;
            if (k >= P.max_samples) continue;
            const float p[3] = {__fadd_rn(R.o[0], __fmul_rn(t, R.d[0])), __fadd_rn(R.o[1], __fmul_rn(t, R.d[1])),
                                __fadd_rn(R.o[2], __fmul_rn(t, R.d[2]))};
            const LevelDev& L = P.vol.lv[l];
            Resolved Q;
            resolve(L, P.vol.bshift, P.vol.bmask, P.vol.quad ? P.vol.B1 - 1 : P.vol.B1, p, Q);
            vol_trace_rec rec;
            rec.k = k;
            rec.t_bits = __float_as_uint(t);
            rec.level = l;
            for (int a = 0; a < 3; ++a) {
                rec.i0[a] = Q.i0[a];
                rec.local[a] = Q.i0[a] & P.vol.bmask;
            }
            rec.pad = 0;
            if (P.vol.sparse) {
                const int h0 = Q.i0[0] >> P.vol.bshift, h1 = Q.i0[1] >> P.vol.bshift, h2 = Q.i0[2] >> P.vol.bshift;
                rec.brick_id = (int64_t)h0 + (int64_t)L.nb[0] * ((int64_t)h1 + (int64_t)L.nb[1] * h2);
                uint32_t leaf;
                rec.slot = sparse_walk(P.vol.pt, load_lv(L), h0, h1, h2, leaf);
            } else {
                rec.brick_id = (int64_t)(Q.pti - L.pt_off);
                rec.slot = P.vol.pt[Q.pti];
            }
            rec.pad2 = 0;
            P.out[(long long)q * P.max_samples + k] = rec;
        }
    }
    P.counts[q] = k;
}

template <int DT, int BS, bool Q>
const void* pick_render_b(bool lod, bool grad) {
    if (grad) return lod ? (const void*)k_render<DT, true, kDvrGrad, BS, Q> : (const void*)k_render<DT, false, kDvrGrad, BS, Q>;
    return lod ? (const void*)k_render<DT, true, kDvr, BS, Q> : (const void*)k_render<DT, false, kDvr, BS, Q>;
}

// quad layout: specialised for bricks of 32 and 64; compact layout: any brick size
template <int DT>
const void* pick_render_d(int brick, bool quad, bool lod, bool grad) {
    if (!quad) return pick_render_b<DT, 0, false>(lod, grad);
    if (brick == 32) return pick_render_b<DT, 32, true>(lod, grad);
    if (brick == 64) return pick_render_b<DT, 64, true>(lod, grad);
    return pick_render_b<DT, 0, true>(lod, grad);
}

const void* pick_render(int dtype, int brick, bool quad, bool lod, bool grad) {
    switch (dtype) {
    case VOL_U8: return pick_render_d<VOL_U8>(brick, quad, lod, grad);
    case VOL_U16: return pick_render_d<VOL_U16>(brick, quad, lod, grad);
    case VOL_F16: return pick_render_d<VOL_F16>(brick, quad, lod, grad);
    case VOL_F32: return pick_render_d<VOL_F32>(brick, quad, lod, grad);
    }
    return nullptr;
}

template <bool LOD, bool TAPE>
const void* pick_backward_l(int dtype) {
    switch (dtype) {
    case VOL_U8: return (const void*)k_backward<VOL_U8, LOD, TAPE>;
    case VOL_U16: return (const void*)k_backward<VOL_U16, LOD, TAPE>;
    case VOL_F16: return (const void*)k_backward<VOL_F16, LOD, TAPE>;
    case VOL_F32: return (const void*)k_backward<VOL_F32, LOD, TAPE>;
    }
    return nullptr;
}

const void* pick_backward(int dtype, bool lod, bool tape) {
    if (tape) return lod ? pick_backward_l<true, true>(dtype) : pick_backward_l<false, true>(dtype);
    return lod ? pick_backward_l<true, false>(dtype) : pick_backward_l<false, false>(dtype);
}

}  // namespace

cudaError_t launch_render(int dtype, int mode, const RenderDev& p, int grid, cudaStream_t s) {
    const void* fn = nullptr;
    // empty-space skipping: flat page table, uniform steps (a quad layout with bricks other than
    // 32 or 64 has no such variant and renders without it; the image is the same)
    if (p.skip_empty && !p.vol.sparse && !p.level_step)
        fn = (mode == kMop || mode == kMip) ? pick_render_skip_projection(dtype, p.vol.B1 - 1, p.vol.quad != 0,
                                                                          p.lod_mode != 0, mode)
                                            : pick_render_skip(dtype, p.vol.B1 - 1, p.vol.quad != 0, p.lod_mode != 0,
                                                               mode);
    if (fn) {
    } else if (mode == kMop || mode == kMip)
        fn = pick_render_projection(dtype, p.vol.B1 - 1, p.vol.quad != 0, p.lod_mode != 0, mode);
    else if (p.vol.sparse && mode == kDvr && !p.level_step)
        fn = pick_render_sparse(dtype, p.vol.B1 - 1, p.vol.quad != 0, p.lod_mode != 0);
    else if (p.vol.sparse)
        fn = nullptr;  // the sparse table has only the emission/absorption variant
    else if (p.level_step && mode == kDvr)
        fn = pick_render_level_step(dtype, p.vol.B1 - 1, p.vol.quad != 0, p.lod_mode != 0);
    else if (!p.level_step)
        fn = pick_render(dtype, p.vol.B1 - 1, p.vol.quad != 0, p.lod_mode != 0, mode == kDvrGrad);
    if (!fn) return cudaErrorInvalidValue;
    void* args[] = {(void*)&p};
    return cudaLaunchKernel(fn, dim3(grid), dim3(kRenderThreads), args, 0, s);
}

cudaError_t launch_backward(int dtype, const BackwardDev& p, int grid, cudaStream_t s) {
    const void* fn = pick_backward(dtype, p.lod_mode != 0, p.tape != nullptr);
    if (!fn) return cudaErrorInvalidValue;
    void* args[] = {(void*)&p};
    return cudaLaunchKernel(fn, dim3(grid), dim3(kBwdThreads), args, 0, s);
}

cudaError_t launch_sum_tables(const float4* tabs, int n, float* dtf, cudaStream_t s) {
    k_sum_tables<<<dim3(32, kSumSlices), kSumThreads, 0, s>>>(tabs, n, dtf);
    return cudaGetLastError();
}

cudaError_t launch_gather_quads(const float4* gq, float* dvox, const int D[3], bool add, cudaStream_t s) {
    const long long n = (long long)D[0] * D[1] * D[2];
    const unsigned blocks = (unsigned)(n / 256 + 1 < 65536 ? n / 256 + 1 : 65536);
    k_gather_quads<<<blocks, 256, 0, s>>>(gq, dvox, D[0], D[1], D[2], add ? 1 : 0);
    return cudaGetLastError();
}

cudaError_t launch_tile_order(int* cost, int* order, int ntiles, int* buckets, cudaStream_t s) {
    if (ntiles <= 0) return cudaSuccess;
    if (ntiles <= kOrderSmall) {
        k_order_small<<<1, 1024, 0, s>>>(cost, order, ntiles);
        return cudaGetLastError();
    }
    cudaError_t e = cudaMemsetAsync(buckets, 0, sizeof(int) * 64, s);
    if (e != cudaSuccess) return e;
    const int grid = (ntiles + kOrderThreads - 1) / kOrderThreads;
    k_order_count<<<grid, kOrderThreads, 0, s>>>(cost, ntiles, buckets);
    k_order_scatter<<<grid, kOrderThreads, 0, s>>>(cost, order, ntiles, buckets);
    return cudaGetLastError();
}

cudaError_t launch_trace(const TraceDev& p, cudaStream_t s) {
    const int threads = 64;
    k_trace<<<(p.npix + threads - 1) / threads, threads, 0, s>>>(p);
    return cudaGetLastError();
}

int backward_warps_per_cta() { return kBwdThreads / 32; }

// (what the launch bounds allot registers for; the shared memory allows 4 as well)
int backward_blocks_per_sm() { return kBwdMinBlocks; }

}  // namespace volrc
