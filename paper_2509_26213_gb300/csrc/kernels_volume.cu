// kernels_volume.cu -- brick upload/transcode with apron, LOD downsample, page-table update.
//
// Slot layouts (include/vol.h): compact slots hold the (B+1)^3 voxels of a brick and its
// +x/+y/+z apron; quad slots hold B x B x (B+1) entries of four voxels each, entry (x, y, z)
// = voxels (x, y), (x+1, y), (x, y+1), (x+1, y+1) of slice z of that region.
#include <algorithm>

#include "internal.cuh"

namespace volrc {
namespace {

// ---- storage conversions (normalised value -> stored type) ----
// u16 -> f16: binary16 (round to nearest even) of the binary32 quotient u / 65535.
template <int SRC, int DST>
struct Convert;
template <> struct Convert<VOL_U8, VOL_U8> {
    static __device__ __forceinline__ uint8_t run(uint8_t v) { return v; }
};
template <> struct Convert<VOL_U16, VOL_U16> {
    static __device__ __forceinline__ uint16_t run(uint16_t v) { return v; }
};
template <> struct Convert<VOL_F16, VOL_F16> {
    static __device__ __forceinline__ __half run(__half v) { return v; }
};
template <> struct Convert<VOL_F32, VOL_F32> {
    static __device__ __forceinline__ float run(float v) { return v; }
};
template <> struct Convert<VOL_U16, VOL_F16> {
    static __device__ __forceinline__ __half run(uint16_t v) { return __float2half_rn(__fdiv_rn((float)v, 65535.0f)); }
};
template <> struct Convert<VOL_U8, VOL_F32> {
    static __device__ __forceinline__ float run(uint8_t v) { return __fdiv_rn((float)v, 255.0f); }
};
template <> struct Convert<VOL_U16, VOL_F32> {
    static __device__ __forceinline__ float run(uint16_t v) { return __fdiv_rn((float)v, 65535.0f); }
};

template <int DT> struct Stored;
template <> struct Stored<VOL_U8> { using T = uint8_t; };
template <> struct Stored<VOL_U16> { using T = uint16_t; };
template <> struct Stored<VOL_F16> { using T = __half; };
template <> struct Stored<VOL_F32> { using T = float; };

// one quad entry written with a single vector store
template <int DT>
__device__ __forceinline__ void store4(typename Stored<DT>::T* p, typename Stored<DT>::T a, typename Stored<DT>::T b,
                                       typename Stored<DT>::T c, typename Stored<DT>::T d) {
    if constexpr (DT == VOL_U8) {
        *(uchar4*)p = make_uchar4(a, b, c, d);
    } else if constexpr (DT == VOL_U16) {
        *(ushort4*)p = make_ushort4(a, b, c, d);
    } else if constexpr (DT == VOL_F16) {
        *(ushort4*)p = make_ushort4(__half_as_ushort(a), __half_as_ushort(b), __half_as_ushort(c), __half_as_ushort(d));
    } else {
        *(float4*)p = make_float4(a, b, c, d);
    }
}

// Transfer-function coordinate x = 255 clamp(v, 0, 1) of a stored value (u8: v; u16: v / 65535;
// floats: v), with the arithmetic the render kernels use.
template <int DT>
__device__ __forceinline__ float stored_coord(float v) {
    if (DT == VOL_U8) return v;
    if (DT == VOL_U16) return v * (255.0f / 65535.0f);
    return fminf(fmaxf(v, 0.0f), 1.0f) * 255.0f;
}

// A stored value as a 32-bit word (shuffled between lanes) and as a float.
template <int DT>
__device__ __forceinline__ uint32_t to_word(typename Stored<DT>::T v) {
    if constexpr (DT == VOL_F16) return __half_as_ushort(v);
    else if constexpr (DT == VOL_F32) return __float_as_uint(v);
    else return v;
}
template <int DT>
__device__ __forceinline__ typename Stored<DT>::T from_word(uint32_t w) {
    if constexpr (DT == VOL_F16) return __ushort_as_half((unsigned short)w);
    else if constexpr (DT == VOL_F32) return __uint_as_float(w);
    else return (typename Stored<DT>::T)w;
}
template <int DT>
__device__ __forceinline__ float word_value(uint32_t w) {
    if constexpr (DT == VOL_F16) return __half2float(__ushort_as_half((unsigned short)w));
    else if constexpr (DT == VOL_F32) return __uint_as_float(w);
    else return (float)w;
}

struct BrickAt {
    int x, y, z;  // first voxel of the brick on its level
};
__device__ __forceinline__ BrickAt brick_at(const LevelDev& L, long long b, int bshift) {
    const unsigned nb0 = (unsigned)L.nb[0], nb1 = (unsigned)L.nb[1], i = (unsigned)b;  // (fewer than 2^32 bricks)
    return BrickAt{(int)(i % nb0) << bshift, (int)(i / nb0 % nb1) << bshift, (int)(i / nb0 / nb1) << bshift};
}

// ---- where the (B+1)^3 voxels of a brick come from: words at local (x, y, z), 0 <= x, y, z <= B ----

// a dense level (clamped to its edge)
template <int SRC, int DST>
struct LevelSource {
    const typename Stored<SRC>::T* src;
    BrickAt at;
    int X, Y, Z;  // last voxel per axis
    __device__ __forceinline__ uint32_t word(int x, int y, int z) const {
        const long long row = (long long)min(at.z + z, Z) * (Y + 1) + min(at.y + y, Y);
        return to_word<DST>(Convert<SRC, DST>::run(__ldg(src + row * (X + 1) + min(at.x + x, X))));
    }
};

// the level below through the 2x2x2 box filter (Sec. III-D): children 2g and 2g+1 per axis, an index
// past the edge replaced by the last fine voxel; integer types (sum + 4) >> 3, float types a
// binary32 sum in (dz, dy, dx) order times 0.125.  The 8 children lie in one brick (its edge is
// even): one page-table word, and in a quad slot the 4 children of a slice are one entry.
// (Q: quad slots.  A branch on the layout per voxel would keep a slice's loads from being issued
// together.)
template <int DT, bool Q>
struct CoarseSource {
    const typename Stored<DT>::T* atlas;
    const VolDev* vol;
    const LevelDev *L, *F;
    BrickAt at;
    bool bad = false;  // a source brick was not resident (its voxels read as slot 0's)
    __device__ __forceinline__ uint32_t word(int x, int y, int z) {
        const int fx = 2 * min(at.x + x, L->D[0] - 1), fy = 2 * min(at.y + y, L->D[1] - 1), fz = 2 * min(at.z + z, L->D[2] - 1);
        const int s = vol->bshift, m = vol->bmask;
        uint32_t cs = __ldg(vol->pt + F->pt_off + (uint32_t)((fx >> s) + F->nb[0] * ((fy >> s) + F->nb[1] * (fz >> s))));
        if (cs == kInvalidSlot) {
            bad = true;
            cs = 0u;
        }
        const bool nx = fx + 1 < F->D[0], ny = fy + 1 < F->D[1], nz = fz + 1 < F->D[2];
        const int lx = fx & m, ly = fy & m, lz = fz & m, B = m + 1;
        uint32_t c[2][4];
        if constexpr (Q) {
            const unsigned long long e = (unsigned long long)cs * vol->slot_entries + (unsigned)((lz * B + ly) * B + lx);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const typename Stored<DT>::T* p = atlas + (e + (q && nz ? (unsigned)(B * B) : 0u)) * 4;
                if constexpr (DT == VOL_U8) {
                    const uchar4 v = *(const uchar4*)p;
                    c[q][0] = v.x, c[q][1] = v.y, c[q][2] = v.z, c[q][3] = v.w;
                } else if constexpr (DT == VOL_F32) {
                    const uint4 v = *(const uint4*)p;
                    c[q][0] = v.x, c[q][1] = v.y, c[q][2] = v.z, c[q][3] = v.w;
                } else {
                    const ushort4 v = *(const ushort4*)p;
                    c[q][0] = v.x, c[q][1] = v.y, c[q][2] = v.z, c[q][3] = v.w;
                }
                // components (x, y), (x+1, y), (x, y+1), (x+1, y+1)
                if (!nx) c[q][1] = c[q][0], c[q][3] = c[q][2];
                if (!ny) c[q][2] = c[q][0], c[q][3] = c[q][1];
            }
        } else {
            const int B1 = B + 1;
            const typename Stored<DT>::T* p = atlas + (unsigned long long)cs * vol->slot_elems + (unsigned)((lz * B1 + ly) * B1 + lx);
#pragma unroll
            for (int q = 0; q < 8; ++q)
                c[q >> 2][q & 3] = to_word<DT>(p[((q & 1) && nx ? 1 : 0) + ((q & 2) && ny ? B1 : 0) + ((q & 4) && nz ? B1 * B1 : 0)]);
        }
        if constexpr (DT == VOL_U8 || DT == VOL_U16) {
            uint32_t sum = 4u;
#pragma unroll
            for (int q = 0; q < 8; ++q) sum += c[q >> 2][q & 3];
            return sum >> 3;
        } else {
            float sum = 0.0f;
#pragma unroll
            for (int q = 0; q < 8; ++q) sum = __fadd_rn(sum, word_value<DT>(c[q >> 2][q & 3]));
            sum = __fmul_rn(sum, 0.125f);
            if constexpr (DT == VOL_F16) return to_word<DT>(__float2half_rn(sum));
            else return __float_as_uint(sum);
        }
    }
};

// the slot itself (its words are in place already: only its ranges are taken)
template <int DT, bool Q>
struct SlotSource {
    const typename Stored<DT>::T* slot;
    int B;
    __device__ __forceinline__ uint32_t word(int x, int y, int z) const {
        const int i = Q ? 4 * ((z * B + min(y, B - 1)) * B + min(x, B - 1)) + (x == B) + 2 * (y == B)
                           : (z * (B + 1) + y) * (B + 1) + x;
        return to_word<DT>(slot[i]);
    }
};

// One CTA fills one slot from its source and takes the slot's value ranges on the way, in one
// pass.  The ranges: of the whole slot (brick plus apron), by which the render loop skips bricks
// that the transfer function maps to zero opacity; and per macro-cell (local voxels [c M, c M + M]
// per axis: every corner a trilinear sample inside the cell reads) the span of TF entries
// [lo, hi] a lookup there can touch: the entries of the coordinates of the cell's smallest and
// largest value, widened by one entry on each side for the last-bit rounding of the interpolation
// (floats may overshoot their corners by an ulp).  A cell holding a NaN, or one whose range is not
// ordered, spans every entry.
//
// Bound: HBM (the source once, the slot once).  A unit of work is one row of macro-cells along x,
// min(B, 32) voxels long, on as many lanes: for each of its M + 1 slices the lanes read the M + 1
// rows coalesced (the next voxel along x comes from the neighbouring lane), write the slice's
// entries, 32 x 16 B at most per store, and keep their columns' minimum and maximum; the M lanes of
// a cell are reduced by shuffles at the end.  The rows and slices that two cells share are read
// again, from L1 or L2.
// WRITE: store the words; MS: log2 M.
// Uploads: 512 threads at 2 CTAs per SM (64 registers); one CTA per SM is slower (512^3 u16 update,
// 32^3 bricks: 1.10 against 1.02 ms), 256-thread CTAs too.  The filter holds 8 words per voxel of a
// slice and takes one CTA per SM: at 64 registers its small levels, where latency counts, take 34
// to 52 us instead of 25 to 40, the large one as long.
// Measured, 512^3 u16 into quad slots (0.27 GB read, 1.07 GB written): 1033 (upload) + 708 (ranges)
// -> 257 us; its first coarser level 627 + 138 -> 125 us; a time step (upload, pyramid, 1280x720
// frame) with a slot list allocated per call 3.30 -> 0.84 ms.
constexpr int kFillThreads = 512;

template <int DT, int MS, bool WRITE, class Source>
__device__ __forceinline__ void fill_slot(Source& src, typename Stored<DT>::T* slot, const VolDev& vol, float2* range,
                                          uint16_t* cells) {
    constexpr int M = 1 << MS;
    const int B = vol.bmask + 1, B1 = B + 1, cb = vol.cbits, CB = 1 << cb;
    const int XS = min(B, 32), xsegs = B / XS;
    const int units = CB * CB * xsegs, nsub = (int)blockDim.x / XS;
    const int lane = threadIdx.x % XS;
    const float inf = __int_as_float(0x7f800000);
    float lo = inf, hi = -inf;
    for (int u0 = 0; u0 < units; u0 += nsub) {
        const int uu = u0 + (int)threadIdx.x / XS, u = min(uu, units - 1);
        const bool mine = uu < units;  // (a lane past the last unit repeats it and writes nothing)
        const int xs = u % xsegs, cy = (u / xsegs) & (CB - 1), cz = u / (xsegs * CB);
        const int x = xs * XS + lane;
        float clo = inf, chi = -inf;
        bool nan = false;
        for (int zz = 0; zz <= M; ++zz) {
            const int z = (cz << MS) + zz, y0 = cy << MS;
            uint32_t v[M + 1], n[M + 1];
#pragma unroll
            for (int y = 0; y <= M; ++y) v[y] = src.word(x, y0 + y, z);
            // the column past the segment: lane y reads row y (every lane row M), for the last lane
            const uint32_t e = src.word(xs * XS + XS, y0 + (lane & (M - 1)), z), e_last = src.word(xs * XS + XS, y0 + M, z);
#pragma unroll
            for (int y = 0; y <= M; ++y) {
                n[y] = __shfl_down_sync(0xFFFFFFFFu, v[y], 1, XS);
                const uint32_t f = y < M ? __shfl_sync(0xFFFFFFFFu, e, y, XS) : e_last;
                if (lane == XS - 1) n[y] = f;
            }
#pragma unroll
            for (int y = 0; y <= M; ++y) {
                const float a = word_value<DT>(v[y]), b = word_value<DT>(n[y]);
                if (DT == VOL_F16 || DT == VOL_F32) nan |= a != a || b != b;
                clo = fminf(clo, fminf(a, b));
                chi = fmaxf(chi, fmaxf(a, b));
            }
            if (WRITE && mine && (zz < M || cz == CB - 1)) {
                if (vol.quad) {
                    typename Stored<DT>::T* p = slot + 4ll * ((z * B + y0) * B + x);
#pragma unroll
                    for (int y = 0; y < M; ++y)
                        store4<DT>(p + 4 * y * B, from_word<DT>(v[y]), from_word<DT>(n[y]), from_word<DT>(v[y + 1]),
                                   from_word<DT>(n[y + 1]));
                } else {
                    typename Stored<DT>::T* p = slot + (z * B1 + y0) * B1 + x;
#pragma unroll
                    for (int y = 0; y <= M; ++y)
                        if (y < M || cy == CB - 1) {
                            p[y * B1] = from_word<DT>(v[y]);
                            if (x == B - 1) p[y * B1 + 1] = from_word<DT>(n[y]);
                        }
                }
            }
        }
        lo = fminf(lo, clo);
        hi = fmaxf(hi, chi);
        if (cells) {
#pragma unroll
            for (int o = 1; o < M; o <<= 1) {
                clo = fminf(clo, __shfl_xor_sync(0xFFFFFFFFu, clo, o));
                chi = fmaxf(chi, __shfl_xor_sync(0xFFFFFFFFu, chi, o));
                if (DT == VOL_F16 || DT == VOL_F32) nan |= __shfl_xor_sync(0xFFFFFFFFu, nan, o) != 0;
            }
            if (mine && (lane & (M - 1)) == 0) {
                uint16_t span = 0xFF00u;  // entries 0 .. 255
                if (!nan && clo <= chi) {
                    const int ilo = max((int)stored_coord<DT>(clo) - 1, 0);
                    const int ihi = min((int)stored_coord<DT>(chi) + 2, 255);
                    span = (uint16_t)(ilo | (ihi << 8));
                }
                cells[(((cz << cb) | cy) << cb) | (x >> MS)] = span;
            }
        }
    }
    // the slot's range over the CTA
    __shared__ float s_lo[kFillThreads / 32], s_hi[kFillThreads / 32];
    for (int o = 16; o; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xFFFFFFFFu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xFFFFFFFFu, hi, o));
    }
    if ((threadIdx.x & 31) == 0) {
        s_lo[threadIdx.x >> 5] = lo;
        s_hi[threadIdx.x >> 5] = hi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)blockDim.x / 32; ++w) {
            lo = fminf(lo, s_lo[w]);
            hi = fmaxf(hi, s_hi[w]);
        }
        *range = make_float2(lo, hi);
    }
    __syncthreads();
}

// The slot written by brick b of a launch: its words, range and cells.
template <int DT>
struct SlotAt {
    typename Stored<DT>::T* slot;
    float2* range;
    uint16_t* cells;
    __device__ __forceinline__ SlotAt(typename Stored<DT>::T* atlas, const VolDev& vol, float2* r, uint16_t* c, uint32_t s)
        : slot(atlas + (unsigned long long)s * vol.slot_elems), range(r + s),
          cells(c ? c + ((unsigned long long)s << (3 * vol.cbits)) : nullptr) {}
};

template <int SRC, int DST, int MS>
__global__ void __launch_bounds__(kFillThreads, 2) k_upload_level(const typename Stored<SRC>::T* __restrict__ src,
                                                               typename Stored<DST>::T* atlas, const __grid_constant__ VolDev vol,
                                                               int level, float2* range, uint16_t* cells,
                                                               const uint32_t* __restrict__ slots, long long nbricks) {
    const LevelDev& L = vol.lv[level];
    for (long long b = blockIdx.x; b < nbricks; b += gridDim.x) {
        const uint32_t s = slots[b];
        if (s == kInvalidSlot) continue;
        const SlotAt<DST> at(atlas, vol, range, cells, s);
        LevelSource<SRC, DST> level{src, brick_at(L, b, vol.bshift), L.D[0] - 1, L.D[1] - 1, L.D[2] - 1};
        fill_slot<DST, MS, true>(level, at.slot, vol, at.range, at.cells);
    }
}

template <int DT, int MS, bool Q>
__global__ void __launch_bounds__(kFillThreads, 1) k_downsample(typename Stored<DT>::T* atlas, const __grid_constant__ VolDev vol,
                                                             int level, float2* range, uint16_t* cells,
                                                             const uint32_t* __restrict__ slots, long long nbricks, unsigned* err) {
    const LevelDev &L = vol.lv[level], &F = vol.lv[level - 1];
    for (long long b = blockIdx.x; b < nbricks; b += gridDim.x) {
        const uint32_t s = slots[b];
        if (s == kInvalidSlot) continue;
        const SlotAt<DT> at(atlas, vol, range, cells, s);
        CoarseSource<DT, Q> coarse{atlas, &vol, &L, &F, brick_at(L, b, vol.bshift)};
        fill_slot<DT, MS, true>(coarse, at.slot, vol, at.range, at.cells);
        if (coarse.bad) atomicAdd(err, 1u);
    }
}

// Copies n bytes with the threads of a CTA; dst 16-byte aligned, src at any byte.  16 bytes of dst
// per thread from the two aligned 16-byte words of src they lie in (host memory is read across the
// chip link: single bytes reached 46 GB/s there); the words that reach outside [src, src + n) are
// read byte by byte.
__device__ __forceinline__ void copy_bytes(void* dst, const void* src, unsigned n) {
    const unsigned sh = (unsigned)(uintptr_t)src & 15u;
    const uint4* a = (const uint4*)((uintptr_t)src - sh);  // word i: src bytes 16 i - sh ...
    const unsigned full = n / 16u;
    const unsigned bits = (sh & 3u) * 8u, w0 = sh >> 2;
#pragma unroll 2
    for (unsigned i = threadIdx.x; i < full; i += blockDim.x) {
        uint4 out;
        if (sh == 0u) {
            out = __ldg(a + i);
        } else if (i > 0u && 16u * (i + 2u) - sh <= n) {
            const uint4 lo = __ldg(a + i), hi = __ldg(a + i + 1);
            const uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
            uint32_t t[5];  // the words w0 .. w0 + 4
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                t[q] = w[q];
                if (w0 == 1u) t[q] = w[q + 1];
                if (w0 == 2u) t[q] = w[q + 2];
                if (w0 == 3u) t[q] = w[q + 3 > 7 ? 7 : q + 3];
            }
            out = make_uint4(__funnelshift_r(t[0], t[1], bits), __funnelshift_r(t[1], t[2], bits),
                             __funnelshift_r(t[2], t[3], bits), __funnelshift_r(t[3], t[4], bits));
        } else {
            uint32_t o[4] = {0u, 0u, 0u, 0u};
#pragma unroll
            for (int q = 0; q < 16; ++q) o[q >> 2] |= (uint32_t)((const uint8_t*)src)[16u * i + q] << (8 * (q & 3));
            out = make_uint4(o[0], o[1], o[2], o[3]);
        }
        ((uint4*)dst)[i] = out;
    }
    for (unsigned i = 16u * full + threadIdx.x; i < n; i += blockDim.x) ((uint8_t*)dst)[i] = ((const uint8_t*)src)[i];
}

// n bricks of (B+1)^3 voxels each (compact, apron included), packed in src (device memory, or the
// mapped host ring: read once, in order), into slots[i]; then the slot's ranges from the words just
// written (in L2).
template <int SRC, int DST, int MS, bool Q>
__global__ void __launch_bounds__(kFillThreads, 2) k_upload_bricks(const typename Stored<SRC>::T* __restrict__ src,
                                                                typename Stored<DST>::T* atlas,
                                                                const __grid_constant__ VolDev vol, float2* range, uint16_t* cells,
                                                                const uint32_t* __restrict__ slots, long long n) {
    const int B = vol.bmask + 1, B1 = B + 1;
    const int nvox = B1 * B1 * B1;
    for (long long b = blockIdx.x; b < n; b += gridDim.x) {
        const uint32_t s = slots[b];
        if (s == kInvalidSlot) continue;
        const SlotAt<DST> at(atlas, vol, range, cells, s);
        const typename Stored<SRC>::T* p = src + b * nvox;
        if constexpr (!Q && SRC == DST) {
            copy_bytes(at.slot, p, nvox * (unsigned)sizeof(*p));
        } else if constexpr (!Q) {
            for (int i = threadIdx.x; i < nvox; i += blockDim.x) at.slot[i] = Convert<SRC, DST>::run(p[i]);
        } else {
            for (int r = threadIdx.x; r < B * B * B1; r += blockDim.x) {
                const int x = r & (B - 1), y = (r >> vol.bshift) & (B - 1), z = r >> (2 * vol.bshift);
                const int i = (z * B1 + y) * B1 + x;
                store4<DST>(at.slot + 4ll * r, Convert<SRC, DST>::run(p[i]), Convert<SRC, DST>::run(p[i + 1]),
                            Convert<SRC, DST>::run(p[i + B1]), Convert<SRC, DST>::run(p[i + B1 + 1]));
            }
        }
        __syncthreads();
        SlotSource<DST, Q> filled{at.slot, B};
        fill_slot<DST, MS, false>(filled, at.slot, vol, at.range, at.cells);
    }
}

// Adjoint of one box-filter level (k_downsample): fine voxel i has the single parent i >> 1 per
// axis, and along an axis of odd size the last fine voxel fills both child places of its
// parent (the filter replaces the missing child by it), so it takes 2 shares there.
__global__ void k_downsample_transpose(const float* __restrict__ coarse, float* __restrict__ fine, int Fx, int Fy,
                                       int Fz) {
    const long long n = (long long)Fx * Fy * Fz;
    const int Cx = (Fx + 1) / 2, Cy = (Fy + 1) / 2;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int x = (int)(i % Fx), y = (int)((i / Fx) % Fy), z = (int)(i / ((long long)Fx * Fy));
        const int m = ((Fx & 1) && x == Fx - 1 ? 2 : 1) * ((Fy & 1) && y == Fy - 1 ? 2 : 1) * ((Fz & 1) && z == Fz - 1 ? 2 : 1);
        const float g = coarse[(x >> 1) + (long long)Cx * ((y >> 1) + (long long)Cy * (z >> 1))];
        if (g != 0.0f) fine[i] += g * (0.125f * (float)m);
    }
}

__global__ void k_pt_update(uint32_t* pt, const uint32_t* idx, const uint32_t* val, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) atomicExch(&pt[idx[i]], val[i]);
}

}  // namespace

// threads of a CTA: one lane per voxel of a unit's row for every unit of the brick, at most kFillThreads
static int fill_threads(const VolDev& vol) {
    const int B = vol.bmask + 1, xs = std::min(B, 32);
    const int lanes = ((1 << (2 * vol.cbits)) * (B / xs)) * xs;
    return std::min(kFillThreads, std::max(32, lanes));
}
static unsigned fill_grid(long long nbricks) { return (unsigned)std::min<long long>(nbricks, 1ll << 30); }

#define VOLRC_PAIRS(X)                                                                                     \
    X(VOL_U8, VOL_U8) X(VOL_U16, VOL_U16) X(VOL_F16, VOL_F16) X(VOL_F32, VOL_F32) X(VOL_U16, VOL_F16)      \
    X(VOL_U8, VOL_F32) X(VOL_U16, VOL_F32)
// the cell edges of the brick sizes 4 (4 voxels), 8 .. 64 (8) and 128 (16)
#define VOLRC_CELL_EDGES(X) X(2) X(3) X(4)
static_assert(kCellShift == 3, "the cell edges listed in VOLRC_CELL_EDGES");

cudaError_t launch_upload_level(int dst, int src_t, const void* src, const VolDev& vol, int level, float2* range,
                                uint16_t* cells, const uint32_t* slots, long long nbricks, cudaStream_t s) {
    if (nbricks <= 0) return cudaSuccess;
#define VOLRC_EDGE(MS)                                                                                             \
    if (vol.cshift == MS) {                                                                                        \
        k_upload_level<S_, D_, MS><<<fill_grid(nbricks), fill_threads(vol), 0, s>>>(                               \
            (const Stored<S_>::T*)src, (Stored<D_>::T*)vol.atlas, vol, level, range, cells, slots, nbricks);       \
        return cudaGetLastError();                                                                                 \
    }
#define VOLRC_UP(S, D)                          \
    if (src_t == S && dst == D) {               \
        constexpr int S_ = S, D_ = D;           \
        VOLRC_CELL_EDGES(VOLRC_EDGE)            \
    }
    VOLRC_PAIRS(VOLRC_UP)
#undef VOLRC_UP
#undef VOLRC_EDGE
    return cudaErrorInvalidValue;
}

cudaError_t launch_upload_bricks(int dst, int src_t, const void* src, const VolDev& vol, float2* range, uint16_t* cells,
                                 const uint32_t* slots, long long n, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
#define VOLRC_EDGE(MS)                                                                                              \
    if (vol.cshift == MS) {                                                                                         \
        const auto fn = vol.quad ? k_upload_bricks<S_, D_, MS, true> : k_upload_bricks<S_, D_, MS, false>;          \
        fn<<<fill_grid(n), kFillThreads, 0, s>>>((const Stored<S_>::T*)src, (Stored<D_>::T*)vol.atlas, vol, range,  \
                                                 cells, slots, n);                                                  \
        return cudaGetLastError();                                                                                  \
    }
#define VOLRC_UP(S, D)                          \
    if (src_t == S && dst == D) {               \
        constexpr int S_ = S, D_ = D;           \
        VOLRC_CELL_EDGES(VOLRC_EDGE)            \
    }
    VOLRC_PAIRS(VOLRC_UP)
#undef VOLRC_UP
#undef VOLRC_EDGE
    return cudaErrorInvalidValue;
}

cudaError_t launch_downsample(int dtype, const VolDev& vol, int level, float2* range, uint16_t* cells,
                              const uint32_t* slots, long long nbricks, unsigned* err, cudaStream_t s) {
    if (nbricks <= 0) return cudaSuccess;
#define VOLRC_EDGE(MS)                                                                                          \
    if (vol.cshift == MS) {                                                                                     \
        const auto fn = vol.quad ? k_downsample<D_, MS, true> : k_downsample<D_, MS, false>;                    \
        fn<<<fill_grid(nbricks), fill_threads(vol), 0, s>>>((Stored<D_>::T*)vol.atlas, vol, level, range, cells, \
                                                            slots, nbricks, err);                               \
        return cudaGetLastError();                                                                              \
    }
#define VOLRC_DOWN(D)                           \
    if (dtype == D) {                           \
        constexpr int D_ = D;                   \
        VOLRC_CELL_EDGES(VOLRC_EDGE)            \
    }
    VOLRC_DOWN(VOL_U8) VOLRC_DOWN(VOL_U16) VOLRC_DOWN(VOL_F16) VOLRC_DOWN(VOL_F32)
#undef VOLRC_DOWN
#undef VOLRC_EDGE
    return cudaErrorInvalidValue;
}

cudaError_t launch_downsample_transpose(const float* coarse, float* fine, const int Dfine[3], cudaStream_t s) {
    const long long n = (long long)Dfine[0] * Dfine[1] * Dfine[2];
    if (n <= 0) return cudaSuccess;
    const long long blocks = std::min<long long>((n + 255) / 256, 65536);
    k_downsample_transpose<<<(unsigned)blocks, 256, 0, s>>>(coarse, fine, Dfine[0], Dfine[1], Dfine[2]);
    return cudaGetLastError();
}

cudaError_t launch_pt_update(uint32_t* pt, const uint32_t* idx, const uint32_t* val, int n, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    k_pt_update<<<(n + 255) / 256, 256, 0, s>>>(pt, idx, val, n);
    return cudaGetLastError();
}

}  // namespace volrc
