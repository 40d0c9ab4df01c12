// Fused correction + sparse matrix-vector product (Sec. 5.2, Sec. 6.4) on the pixel-tiled
// layout.  Every form ends with the same deterministic phase 2; phase 1 comes in three kernels,
// all persistent, one CTA per SM, their stages filled by bulk, tensor (or cp.async) copies that
// mbarriers track, every wait bounded:
//
//   frames_kernel: a work item is a pixel tile (or a piece of a heavy one) for every frame of
//     the launch.  One producer warp copies the item's units and entries (location, weight,
//     per-entry dark) once into a ring of entry buffers and streams the tile's pixels, G frames
//     at a time, into a ring of plane stages; 15 consumer warps take units of eight segments,
//     four lanes a segment and G frames a lane, and write one partial sum per (segment, frame).
//     Batches, the propagated variance of two frames or more, the per-pixel-corrected form.
//   single_kernel: a stage holds an item's units, entries and the planes given (image, dark, flat,
//     solid angle, polarisation) of one frame; 15 consumer warps correct the tile's pixels in
//     shared memory, then reduce the units.  Single frames in both precisions (also without
//     allocation), the many-detector plan, the normalisation sums N, the variance of one frame.
//   phase1_kernel: one item per tile with the planes of one frame, or of fpi frames, and the
//     tile's entries in a ring of stages.  The cp.async copy engine, and what does not fit the
//     other two (FP32 single frames of large tiles go through single_planes_kernel, which
//     writes the corrected frame and its normalisation, and frames_kernel).
//   phase 2: per (row, frame), the row's segment partials summed in a fixed order; then S, N, C
//     and I = S / N.  C = sum w is the layout's (count_layout).
//
// Where a segment is one matrix row's entries inside one tile, long runs cut in pieces of 96
// entries.  The image cast, the dark and flat * solid angle * polarisation are applied inside these
// kernels or in one per-pixel pass (the paper runs separate cast / correction / memset / integrate
// kernels).  FP32 sums are Kahan-compensated (Sec. 5.2.2); FP64 sums are plain.  No atomics touch
// the sums, so results are bit-reproducible run to run, and a frame gives the same bits alone or
// in any batch.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstring>
#include <memory>
#include <new>
#include <vector>

#include "common.cuh"

namespace azint {

namespace {

// phase1_kernel's warps.  With the cp.async engine the staging holds an FP32 frame up: 2167 x 2070
// pixels with four corrections took 120 us with 4 + 16, 114 with 6 + 14, 108 with 8 + 12 and 119 with
// 8 + 16 warps, a batch of 16 frames 437, 402, 374 and 407.
constexpr int kProducers = 8;                               // producer warps per CTA
constexpr int kConsumers = 12;                              // consumer warps per CTA
constexpr int kThreads = 32 * (kProducers + kConsumers);
constexpr uint32_t kFullCount = 32u * kProducers + 1u;       // arrivals completing a stage
constexpr int kMaxPlanes = 12;
constexpr int kMaxStages = 8;

enum Mode { MODE_SINGLE = 0, MODE_NORM = 1, MODE_FRAMES = 2 };

// Everything phase 1 and phase 2 need about one integrator and its inputs.
struct Inst {
    // tiled layout
    const int32_t *row_slot_ptr;
    const uint16_t *ent_loc;
    const void *ent_w;
    int ny, nx, th, tw, srow, ss, ntx, nseg, nrows;
    int64_t npix;
    // inputs
    const char *img;  // first frame of this launch
    int n_frames, fpi, n_groups;
    const float *dark, *flat, *sa, *pol;
    // scratch and outputs
    void *partial;       // [planes][nseg] in the accumulation type
    float *norm;         // [2][nrows] N, C (FP32 batched path)
    void *oI, *oS, *oN, *oC;
    int frame_out0;      // first output frame of this launch
    int64_t item_begin, row_begin;
    int n_items;
    int stage_entries;
    int *status;
    const int32_t *tile_desc, *tile_rec;  // per active tile: descriptor [8] and record
    const float *ent_dark;                // frames pass: dark of each entry's pixel (or NULL)
    const CUtensorMap *maps;              // many-instance launch: this instance's [5][4] maps
    int norm_is_count;  // single-frame phase 2: N is the count too, not the partials' second row
    const void *count;  // [nrows] in the accumulation type: the layout's C
};

struct StageGeom {
    uint32_t plane_words;   // words per plane slot
    uint32_t plane_region;  // bytes of the plane region
    uint32_t ent_cap;       // entry capacity (staged entries)
    uint32_t stage_bytes;   // bytes per stage (multiple of 128)
    uint32_t rec_cap;       // bytes reserved for the tile record
    int ent_dk;             // entries carry a staged per-entry dark (frames pass)
    int nstages;            // pipeline depth
};

// Number of planes staged per item and the base address of plane `pl`: image frames
// first, then the corrections the mode reads (dark for single/frames; flat, solid angle,
// polarisation for single/norm), skipping absent ones.
template <int MODE>
__device__ __forceinline__ int plane_count(const Inst &d, int nimg) {
    int n = nimg;
    if (MODE == MODE_SINGLE && d.dark) ++n;
    if (MODE != MODE_FRAMES) n += (d.flat != nullptr) + (d.sa != nullptr) + (d.pol != nullptr);
    return n;
}

template <int MODE>
__device__ __forceinline__ const char *plane_base(const Inst &d, int f0, int nimg, int pl, int &kind) {
    if (pl < nimg) { kind = 0; return d.img + (size_t)(f0 + pl) * (size_t)d.npix * 4u; }
    int k = pl - nimg;
    if (MODE == MODE_SINGLE && d.dark) { if (k == 0) { kind = 1; return (const char *)d.dark; } --k; }
    if (MODE != MODE_FRAMES) {
        if (d.flat) { if (k == 0) { kind = 2; return (const char *)d.flat; } --k; }
        if (d.sa) { if (k == 0) { kind = 3; return (const char *)d.sa; } --k; }
        if (d.pol) { if (k == 0) { kind = 4; return (const char *)d.pol; } --k; }
    }
    kind = -1;
    return nullptr;
}

__device__ __forceinline__ const Inst &inst_of(const Inst &single, const Inst *multi, int n_inst,
                                               int64_t item) {
    if (!multi) return single;
    int lo = 0, hi = n_inst;  // last instance with item_begin <= item
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (multi[mid].item_begin <= item) lo = mid; else hi = mid;
    }
    return multi[lo];
}

struct TileDesc {
    int t, rec_off, rec_words, e_off, ne, ns;
};

__device__ __forceinline__ TileDesc load_desc(const Inst &d, int64_t local) {
    const int a = (int)(local / d.n_groups);
    const int4 *p = reinterpret_cast<const int4 *>(d.tile_desc) + 2 * (size_t)a;
    const int4 x = __ldg(p), y = __ldg(p + 1);
    return TileDesc{x.x, x.y, x.z, x.w, y.x, y.y};
}

// Descriptors of a CTA's items, 32 at a time: lane l holds the one of item 32 b + l of the CTA, and
// the next 32 are read while these are used.  (Read one or two items ahead, each item waited for
// its descriptor's trip to memory: about 1 us an item where an item has few stages.)
__device__ __forceinline__ TileDesc shfl_desc(const TileDesc &d, int l) {
    return TileDesc{__shfl_sync(0xffffffffu, d.t, l), __shfl_sync(0xffffffffu, d.rec_off, l),
                    __shfl_sync(0xffffffffu, d.rec_words, l), __shfl_sync(0xffffffffu, d.e_off, l),
                    __shfl_sync(0xffffffffu, d.ne, l), __shfl_sync(0xffffffffu, d.ns, l)};
}

// Words between two staged planes: four 128-byte aligned row-class slots and a band of 32
// words that holds zeros (the padding entries of the matrix point there: their weight is 0
// and the value they read is 0, whatever the image holds).  Planes are spread over the
// shared-memory banks by per-plane shifts of 4 * s words that the copies apply.
constexpr uint32_t kZeroBand = 32;
__host__ __device__ __forceinline__ uint32_t plane_stride(int ss) { return 4u * (uint32_t)ss + kZeroBand; }

// Four 2D tensor maps per staged array, one per tile-row class (rows of equal index mod 4,
// 16 * nx bytes apart).  Index: 0 image, 1 dark, 2 flat, 3 solid angle, 4 polarisation.
struct TmaSet {
    CUtensorMap m[5][4];
};

// Stage layout: [header 256 B][tile record][planes][entry locs][entry weights].
// Header ints: 0 ns, 1 group, 2 nimg, 3..6 word offsets of dark, flat, solid angle,
// polarisation in the plane region (-1 = absent), 7 tile, 8 entry offset, 16.. image planes.
constexpr uint32_t kHeaderBytes = 256;

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}

__device__ __forceinline__ void cp_async_arrive(uint64_t *bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// Producer warps: stage work item `local` of instance d.  Warp 0 writes the item header and
// bulk-copies (TMA) the tile record and entries.  Each plane of the tile is staged as four
// row classes (tile rows of equal index mod 4, which are 16 * nx bytes apart in global
// memory): with the TMA engine one 2D tensor copy per class -- a box of srow x (th / 4)
// words into a 128-byte aligned slot -- and with the cp.async engine the same words in
// 16-byte pieces spread over all producer lanes.  For a plane whose base address is beta
// words mod 4 and whose first tile row is global row g0, class k goes to slot
// s = (k - g0) mod 4, and the box starts at column X = c0 - 4 (flag + spread) where
// off_k = (beta + k nx) mod 4, c_s = (nx s) mod 4, phi = (beta + nx g0) mod 4,
// flag = (c_s + phi - off_k) / 4 in {0, 1} and spread = plane mod 4.  Pixel (ly, c0 + lx)
// then sits at the build-time offset plus phi + 4 spread, the per-plane shift the consumers
// add.  Every producer thread makes one arrival per item (deferred until its cp.async copies
// land) and lane 0 of warp 0 one more after publishing the header: kFullCount arrivals.
template <int MODE, class WT, bool TMA>
__device__ void produce(const Inst &d, const TmaSet &tm, int64_t local, const TileDesc &td,
                        unsigned char *stage, const StageGeom &sg, uint64_t *bar, int *ctr,
                        int pwarp) {
    const int lane = threadIdx.x & 31;
    const int group = (int)(local % d.n_groups);
    const int t = td.t;
    const int ti = t / d.ntx, tj = t - ti * d.ntx;
    const int r0 = ti * d.th, c0 = tj * d.tw;
    const int f0 = group * d.fpi;
    const int nimg = MODE == MODE_SINGLE ? 1 : (MODE == MODE_FRAMES ? min(d.fpi, d.n_frames - f0) : 0);
    const int np = plane_count<MODE>(d, nimg);
    const uint32_t pw = plane_stride(d.ss);
    const int nu = d.nx & 3;
    const int rows4 = d.th >> 2;          // rows per class in a tile
    const int boxw = d.srow;              // words per staged row (tw + 20)
    unsigned char *rec_dst = stage + kHeaderBytes;
    uint32_t *planes = reinterpret_cast<uint32_t *>(stage + kHeaderBytes + sg.rec_cap);
    unsigned char *eloc = stage + kHeaderBytes + sg.rec_cap + sg.plane_region;
    unsigned char *ew = eloc + sg.ent_cap * 2u;
    const uint32_t ne = (uint32_t)td.ne;
    const bool stage_e = d.stage_entries != 0;

    // plane geometry: array base, first global row of the tile in that array, rows in it
    auto plane_geo = [&](int pl, const char *&arr, int64_t &g0, int64_t &rows_total, int &kind) {
        if (pl < nimg) {
            kind = 0;
            arr = d.img;
            g0 = (int64_t)(f0 + pl) * d.ny + r0;
            rows_total = (int64_t)d.n_frames * d.ny;
        } else {
            plane_base<MODE>(d, f0, nimg, pl, kind);
            arr = kind == 1 ? (const char *)d.dark : kind == 2 ? (const char *)d.flat
                : kind == 3 ? (const char *)d.sa : (const char *)d.pol;
            g0 = r0;
            rows_total = d.ny;
        }
    };

    if (pwarp == 0) {
        uint32_t mine = 0;
        if (TMA) {
            // lane pl * 4 + k copies class k of plane pl
            for (int job = lane; job < 4 * np; job += 32) {
                const int pl = job >> 2, k = job & 3;
                const char *arr;
                int64_t g0, rows_total;
                int kind;
                plane_geo(pl, arr, g0, rows_total, kind);
                const int phi = (int)(g0 & 3);
                const int sl = (k - phi) & 3;
                if (g0 + sl < rows_total) mine += (uint32_t)(boxw * rows4 * 4);
            }
        }
        const bool dk = MODE == MODE_FRAMES && d.ent_dark != nullptr && stage_e;
        if (lane == 0) {
            mine += (uint32_t)td.rec_words * 4u;
            if (stage_e) mine += ne * 2u + ne * (uint32_t)sizeof(WT);
            if (dk) mine += ne * 4u;
        }
        fence_proxy_async_smem();
        if (mine)
            asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)),
                         "r"(mine)
                         : "memory");
        if (lane == 0) {
            bulk_g2s(rec_dst, d.tile_rec + td.rec_off, (uint32_t)td.rec_words * 4u, bar);
            if (stage_e && ne) {
                bulk_g2s(eloc, d.ent_loc + td.e_off, ne * 2u, bar);
                bulk_g2s(ew, static_cast<const WT *>(d.ent_w) + td.e_off, ne * (uint32_t)sizeof(WT), bar);
            }
            if (dk && ne) bulk_g2s(ew + sg.ent_cap * (uint32_t)sizeof(WT), d.ent_dark + td.e_off, ne * 4u, bar);
        }
        if (TMA) {
            for (int job = lane; job < 4 * np; job += 32) {
                const int pl = job >> 2, k = job & 3;
                const char *arr;
                int64_t g0, rows_total;
                int kind;
                plane_geo(pl, arr, g0, rows_total, kind);
                const int beta = (int)((reinterpret_cast<uintptr_t>(arr) >> 2) & 3u);
                const int phi_row = (int)(g0 & 3);
                const int sl = (k - phi_row) & 3;
                if (g0 + sl >= rows_total) continue;
                const int phi = (beta + nu * phi_row) & 3;
                const int offk = (beta + k * nu) & 3;
                const int cs = (nu * sl) & 3;
                const int flag = (cs + phi - offk) >> 2;
                const int x = c0 - 4 * (flag + (pl & 3));
                uint32_t *dst = planes + (size_t)pl * pw + (size_t)sl * d.ss;
                const int y = (int)((g0 + sl - k) >> 2);
                const CUtensorMap *map = d.maps ? d.maps + 4 * kind + k : &tm.m[kind][k];
                asm volatile(
                    "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
                    " [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_addr(dst)),
                    "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_addr(bar))
                    : "memory");
            }
        }
    }
    if (!TMA) {
        // the same words as the tensor copies: for every (plane, tile row) a run of boxw / 4
        // 16-byte pieces, the first of which holds column c0 - phi - c_s - 4 spread; eight lanes
        // per run.  Tile row ly is row ly / 4 of slot ly mod 4.  Lane pl forms plane pl's
        // geometry once an item.  (Formed for every run, an FP32 frame with four corrections took
        // 134 us in place of 115 on 2048 x 2048 pixels with 48 x 40 tiles, 128 in place of 120 on
        // 2167 x 2070 with 16 x 64.)
        const char *arr = nullptr;
        int64_t first = 0, elems = 0;  // element of the staged word 0 of row 0, elements of the array
        int rows = 0;                  // rows of the tile in the array
        if (lane < np) {
            int64_t g0, rows_total;
            int kind;
            plane_geo(lane, arr, g0, rows_total, kind);
            const int beta = (int)((reinterpret_cast<uintptr_t>(arr) >> 2) & 3u);
            const int phi = (beta + nu * (int)(g0 & 3)) & 3;
            first = g0 * d.nx + c0 - phi - 4 * (lane & 3);
            elems = rows_total * d.nx;
            rows = (int)min((int64_t)d.th, rows_total - g0);
        }
        const int sub = lane >> 3, l8 = lane & 7;
        const int nchunk = boxw >> 2;
        int pl = 0, ly = pwarp * 4 + sub;
        for (int r = pwarp * 4; r < np * d.th; r += 4 * kProducers, ly += 4 * kProducers) {
            while (ly >= d.th) { ly -= d.th; ++pl; }
            const char *a = reinterpret_cast<const char *>(
                __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(arr), pl));
            const int64_t f = __shfl_sync(0xffffffffu, first, pl), n = __shfl_sync(0xffffffffu, elems, pl);
            if (ly >= __shfl_sync(0xffffffffu, rows, pl) || pl >= np) continue;
            uint32_t *dst = planes + (size_t)pl * pw + (size_t)(ly & 3) * d.ss + (size_t)(ly >> 2) * boxw;
            const int64_t e0 = f + (int64_t)ly * d.nx - ((nu * ly) & 3);  // first element of the run
            const char *src = a + 4 * e0;                 // 16-byte aligned by construction
            for (int c = l8; c < nchunk; c += 8) {
                // copy every piece that overlaps the array; a piece is 16-byte aligned, so the
                // words it holds outside the array share a 16-byte granule with one inside it
                const int64_t ec = e0 + 4 * c;
                if (ec + 3 >= 0 && ec < n) cp_async16(dst + 4 * c, src + 16 * c);
            }
        }
        cp_async_arrive(bar);  // deferred arrival when this thread's copies have landed
    } else {
        mbar_arrive(bar);
    }
    if (pwarp == 0) {
        // the zero band of every plane of this item (planes of different instances have
        // different strides, so the bands move from item to item)
        for (int pl = 0; pl < np; ++pl) planes[(size_t)pl * pw + pw - kZeroBand + lane] = 0u;
        __syncwarp();
    }
    if (pwarp == 0) {
        int *h = reinterpret_cast<int *>(stage);
        if (lane == 0) {
            h[0] = td.ns; h[1] = group; h[2] = nimg; h[3] = h[4] = h[5] = h[6] = -1;
            h[7] = t; h[8] = td.e_off;
            *ctr = 0;  // segment claim counter of this stage
        }
        __syncwarp();
        for (int pl = lane; pl < np; pl += 32) {  // a lane per plane
            const char *arr;
            int64_t g0, rows_total;
            int kind;
            plane_geo(pl, arr, g0, rows_total, kind);
            const int beta = (int)((reinterpret_cast<uintptr_t>(arr) >> 2) & 3u);
            const int phi = (beta + nu * (int)(g0 & 3)) & 3;
            const int o = (int)(pl * pw + phi + 4 * (pl & 3));
            if (kind == 0) h[16 + pl] = o; else h[2 + kind] = o;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bar);  // publishes the header and the counter
    }
}

template <int DT>
__device__ __forceinline__ float img_f32(uint32_t w) {
    if (DT == AZ_DTYPE_F32) return __uint_as_float(w);
    if (DT == AZ_DTYPE_U32) return __uint2float_rn(w);
    return __int2float_rn((int)w);
}
template <int DT>
__device__ __forceinline__ double img_f64(uint32_t w) {
    if (DT == AZ_DTYPE_F32) return (double)__uint_as_float(w);
    if (DT == AZ_DTYPE_U32) return (double)w;
    return (double)(int)w;
}

// Accumulators: Kahan (FP32 compensated) or plain double.
template <class A> struct Acc;
template <> struct Acc<float> {
    Kahan k;
    __device__ void zero() { k.s = 0.f; k.nc = 0.f; }
    __device__ void add(float w, float v) { kahan_add(k, w, v); }
    __device__ void merge(const Acc<float> &o) { kahan_merge(k, o.k); }
    __device__ void merge_xor(int m) {
        // lower lane's partial sum on the left: every lane ends with lane 0's value
        const Kahan o = shfl_xor(k, m);
        if ((threadIdx.x & m) != 0) {
            Kahan l = o;
            kahan_merge(l, k);
            k = l;
        } else {
            kahan_merge(k, o);
        }
    }
    // the partner lane's sum merged in, the lower lane's on the left (its value is right on
    // the lower lane of each pair; the upper lane ends with the pair in the other order)
    __device__ void merge_lower_left(int m) {
        const Kahan o = shfl_xor(k, m);
        if ((threadIdx.x & m) == 0) kahan_merge(k, o);
    }
    __device__ float value() const { return kahan_value(k); }
};
template <> struct Acc<double> {
    double s;
    __device__ void zero() { s = 0.0; }
    __device__ void add(double w, double v) { s = __fma_rn(w, v, s); }
    __device__ void merge(const Acc<double> &o) { s += o.s; }
    __device__ void merge_xor(int m) { s += __shfl_xor_sync(0xffffffffu, s, m); }
    __device__ void merge_lower_left(int m) {
        const double o = __shfl_xor_sync(0xffffffffu, s, m);
        if ((threadIdx.x & m) == 0) s = s + o;
    }
    __device__ double value() const { return s; }
};

// What a consumer needs about its instance, loaded once per item into registers.
struct ConsumerParams {
    void *partial;
    const uint16_t *ent_loc;
    const void *ent_w;
    const float *ent_dark;
    int nseg, fpi, stage_entries;
};

__device__ __forceinline__ ConsumerParams consumer_params(const Inst &d) {
    return ConsumerParams{d.partial, d.ent_loc, d.ent_w, d.ent_dark, d.nseg, d.fpi, d.stage_entries};
}

template <class WT> struct W4;
template <> struct W4<float> {
    static __device__ __forceinline__ void load(const float *p, float w[4]) {
        const float4 v = *reinterpret_cast<const float4 *>(p);
        w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
    }
};
template <> struct W4<double> {
    static __device__ __forceinline__ void load(const double *p, double w[4]) {
        const double2 a = *reinterpret_cast<const double2 *>(p);
        const double2 b = *reinterpret_cast<const double2 *>(p + 2);
        w[0] = a.x; w[1] = a.y; w[2] = b.x; w[3] = b.y;
    }
};

// Two FP32 values in one 64-bit register, operated on by the packed f32x2 instructions
// (round to nearest, no flush): each half gives exactly the scalar result.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 f2_pack(float lo, float hi) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void f2_unpack(f32x2 x, float &lo, float &hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(x));
}
__device__ __forceinline__ f32x2 f2_add(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 f2_fma(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// a - b as b (-1) + a: the same single rounding of the same exact value.
__device__ __forceinline__ f32x2 f2_sub(f32x2 a, f32x2 b) {
    return f2_fma(b, 0xbf800000bf800000ull, a);
}
// Two Kahan accumulators stepped together: the same operations as kahan_add on each half.
__device__ __forceinline__ void kahan2_add(f32x2 &s, f32x2 &nc, f32x2 w, f32x2 v) {
    const f32x2 y = f2_fma(w, v, nc);
    const f32x2 t = f2_add(s, y);
    nc = f2_sub(y, f2_sub(t, s));
    s = t;
}
// ... and merged: kahan_merge on each half.
__device__ __forceinline__ void kahan2_merge(f32x2 &as, f32x2 &an, f32x2 bs, f32x2 bn) {
    const f32x2 t = f2_add(as, bs);
    const f32x2 z = f2_sub(t, as);
    const f32x2 e = f2_add(f2_sub(as, f2_sub(t, z)), f2_sub(bs, z));
    an = f2_add(f2_add(an, bn), e);
    as = t;
}

// Frames pass: one lane per (segment, frame).  A warp takes 32 / Q segments at a time from the
// stage's claim counter; the Q lanes of a segment share its entry stream (broadcast reads) and
// lane q sums cast(image) - dark of frame q of the item over all of the segment's entries.
// Segments start on a multiple of 4 entries and hold whole quads (the layout pads them with
// entries of weight 0 that read the plane's zero band).  Entries are read four at a time (one
// 8-byte read of the locations, 16-byte reads of the weights and per-entry darks); entry e
// goes to accumulator e mod 4 and the four are combined as ((a0 + a1) + (a2 + a3)).  Every quantity of every pass is reduced
// by this same sequence of operations, so a flat image with unit corrections gives S == N bit
// for bit, and a frame integrated alone or in a batch gives the same bits.
template <int Q, class AT, class WT, int MODE, int DT, bool SE>
__device__ void consume_serial(const ConsumerParams &cp, const unsigned char *stage,
                               const StageGeom &sg, int *ctr) {
    static_assert(MODE == MODE_FRAMES, "the single and norm passes have their own consumer");
    constexpr int R = 32 / Q;
    const int lane = threadIdx.x & 31;
    const int sub = lane / Q, q = lane % Q;
    const int *h = reinterpret_cast<const int *>(stage);
    const int ns = h[0], group = h[1], nimg = h[2];
    const int oimg = h[16 + q];
    const bool active = q < nimg;
    const int *slots = reinterpret_cast<const int *>(stage + kHeaderBytes) + 4;
    const uint16_t *starts = reinterpret_cast<const uint16_t *>(slots + ns);
    const uint32_t *planes = reinterpret_cast<const uint32_t *>(stage + kHeaderBytes + sg.rec_cap);
    const uint16_t *L;
    const WT *W;
    const float *DK;
    if constexpr (SE) {
        const unsigned char *eb = stage + kHeaderBytes + sg.rec_cap + sg.plane_region;
        L = reinterpret_cast<const uint16_t *>(eb);
        W = reinterpret_cast<const WT *>(eb + sg.ent_cap * 2u);
        DK = reinterpret_cast<const float *>(eb + sg.ent_cap * (2u + (uint32_t)sizeof(WT)));
    } else {
        L = cp.ent_loc + h[8];
        W = static_cast<const WT *>(cp.ent_w) + h[8];
        DK = cp.ent_dark ? cp.ent_dark + h[8] : nullptr;
    }
    const bool has_dk = sg.ent_dk;
    AT *out = static_cast<AT *>(cp.partial) + (size_t)(group * cp.fpi + q) * cp.nseg;
    while (true) {
        int b = 0;
        if (lane == 0) b = atomicAdd(ctr, R);
        b = __shfl_sync(0xffffffffu, b, 0);
        if (b >= ns) break;
        const int sl = b + sub;
        int e0 = 0, e1 = 0, slot = 0;
        if (sl < ns) {
            e0 = starts[sl];
            e1 = starts[sl + 1];
            slot = slots[sl];
        }
        if (!active) e1 = e0;
        Acc<AT> acc[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[j].zero();
        for (int qd = e0; qd < e1; qd += 4) {
            const uint2 l2 = *reinterpret_cast<const uint2 *>(L + qd);
            const int loc[4] = {(int)(l2.x & 0xffffu), (int)(l2.x >> 16), (int)(l2.y & 0xffffu),
                                (int)(l2.y >> 16)};
            WT w[4];
            W4<WT>::load(W + qd, w);
            float dk[4] = {0.f, 0.f, 0.f, 0.f};
            if (has_dk) {
                const float4 v = *reinterpret_cast<const float4 *>(DK + qd);
                dk[0] = v.x; dk[1] = v.y; dk[2] = v.z; dk[3] = v.w;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float v = img_f32<DT>(planes[oimg + loc[j]]);
                if (has_dk) v = __fsub_rn(v, dk[j]);
                acc[j].add((AT)w[j], (AT)v);
            }
        }
        acc[0].merge(acc[1]);
        acc[2].merge(acc[3]);
        acc[0].merge(acc[2]);
        if (sl < ns && active) out[slot] = acc[0].value();
    }
}

// Single-frame and norm modes, four lanes per segment: lane j of a segment keeps accumulator j of
// the sums (the entries e = j mod 4, in order), with per entry x = image - dark and n = ((1 flat)
// solid angle) polarisation, each added with its weight (FP32: compensated, the two sums stepped
// as a packed pair; FP64: fused multiply-adds); the four lanes are merged by shuffles as
// ((a0 + a1) + (a2 + a3)), the order every other reduction of the library uses, so a frame's
// FP32 sums have the bits of the frames kernel's.  A quarter of the chain per lane, every
// lane busy, eight segments per claim.  The norm mode sums n only (X false).  C = sum w is the
// layout's (count_layout), and without flat, solid angle and polarisation so is N.
// (Summing C too, and n unpacked, a 2527 x 2463 frame on the cp.async engine took 150 us in place of
// 142 in FP32 with four corrections, 88 in place of 81 without, and 291 in place of 258 in FP64.)
template <class AT, class WT, int DT, bool SE, bool X>
__device__ void consume_split(const ConsumerParams &cp, const unsigned char *stage, const StageGeom &sg, int *ctr) {
    const int lane = threadIdx.x & 31;
    const int j = lane & 3, sub = lane >> 2;
    const int *h = reinterpret_cast<const int *>(stage);
    const int ns = h[0];
    const int odark = h[3], oflat = h[4], osa = h[5], opol = h[6];
    const int oimg = h[16];
    const bool norm = oflat >= 0 || osa >= 0 || opol >= 0;
    const int *slots = reinterpret_cast<const int *>(stage + kHeaderBytes) + 4;
    const uint16_t *starts = reinterpret_cast<const uint16_t *>(slots + ns);
    const uint32_t *planes = reinterpret_cast<const uint32_t *>(stage + kHeaderBytes + sg.rec_cap);
    const uint16_t *L;
    const WT *W;
    if constexpr (SE) {
        const unsigned char *eb = stage + kHeaderBytes + sg.rec_cap + sg.plane_region;
        L = reinterpret_cast<const uint16_t *>(eb);
        W = reinterpret_cast<const WT *>(eb + sg.ent_cap * 2u);
    } else {
        L = cp.ent_loc + h[8];
        W = static_cast<const WT *>(cp.ent_w) + h[8];
    }
    AT *out = static_cast<AT *>(cp.partial);
    auto image = [&](int loc) -> AT {
        if (sizeof(AT) == 8) {
            AT x = (AT)img_f64<DT>(planes[oimg + loc]);
            if (odark >= 0) x = x - (AT)__uint_as_float(planes[odark + loc]);
            return x;
        }
        float v = img_f32<DT>(planes[oimg + loc]);
        if (odark >= 0) v = __fsub_rn(v, __uint_as_float(planes[odark + loc]));
        return (AT)v;
    };
    auto normal = [&](int loc) -> AT {
        AT n = AT(1);
        if (oflat >= 0) n = n * (AT)__uint_as_float(planes[oflat + loc]);
        if (osa >= 0) n = n * (AT)__uint_as_float(planes[osa + loc]);
        if (opol >= 0) n = n * (AT)__uint_as_float(planes[opol + loc]);
        return n;
    };
    while (true) {
        int b = 0;
        if (lane == 0) b = atomicAdd(ctr, 8);
        b = __shfl_sync(0xffffffffu, b, 0);
        if (b >= ns) break;
        const int sl = b + sub;
        const bool live = sl < ns;
        const int e0 = live ? starts[sl] : 0, e1 = live ? starts[sl + 1] : 0, slot = live ? slots[sl] : 0;
        Acc<AT> a0, a1;  // the first quantity's sum (X: x, else n), and n's
        a0.zero();
        a1.zero();
        if (X && norm) {
            if constexpr (sizeof(AT) == 4) {
                f32x2 s = 0ull, c = 0ull;
                for (int e = e0 + j; e < e1; e += 4) {
                    const int loc = L[e];
                    const float w = W[e];
                    kahan2_add(s, c, f2_pack(w, w), f2_pack(image(loc), normal(loc)));
                }
                f2_unpack(s, a0.k.s, a1.k.s);
                f2_unpack(c, a0.k.nc, a1.k.nc);
            } else {
                for (int e = e0 + j; e < e1; e += 4) {
                    const int loc = L[e];
                    const AT w = (AT)W[e];
                    a0.add(w, image(loc));
                    a1.add(w, normal(loc));
                }
            }
        } else {
            for (int e = e0 + j; e < e1; e += 4) a0.add((AT)W[e], X ? image(L[e]) : normal(L[e]));
        }
        // lanes 0 and 2 form a0 + a1 and a2 + a3 (lower lane on the left); lane 0 adds them
        a0.merge_lower_left(1);
        a0.merge_lower_left(2);
        if (X && norm) { a1.merge_lower_left(1); a1.merge_lower_left(2); }
        if (live && j == 0) {
            out[slot] = a0.value();
            if (X && norm) out[(size_t)cp.nseg + slot] = a1.value();
        }
    }
}

template <class AT, class WT, int MODE, int NIMG, int DT>
__device__ __forceinline__ void consume_dispatch(const ConsumerParams &cp, const unsigned char *stage,
                                                 const StageGeom &sg, int *ctr) {
    if constexpr (MODE != MODE_FRAMES) {
        if (cp.stage_entries) consume_split<AT, WT, DT, true, MODE == MODE_SINGLE>(cp, stage, sg, ctr);
        else consume_split<AT, WT, DT, false, MODE == MODE_SINGLE>(cp, stage, sg, ctr);
    } else {
        if (cp.stage_entries) consume_serial<NIMG, AT, WT, MODE, DT, true>(cp, stage, sg, ctr);
        else consume_serial<NIMG, AT, WT, MODE, DT, false>(cp, stage, sg, ctr);
    }
}

// Warp-specialised persistent kernel.  The first kProducers warps produce: for each work item of
// this CTA (static round robin) they wait until the stage is free (empty barrier), copy the item
// into it and arm the full barrier.  The kConsumers others consume: they wait for the item's
// full barrier, claim and reduce its segments, and release the stage (empty barrier, one
// arrival per consumer warp).  Every wait is bounded; a wait that gives up records
// AZ_ETIMEOUT in the status word, raises the CTA's abort flag and leaves, the producer
// first giving its own copies in flight a bounded grace period.
template <class AT, class WT, int MODE, int NIMG, int DT, bool TMA>
__global__ void __launch_bounds__(kThreads, 1)
phase1_kernel(const __grid_constant__ Inst single, const Inst *__restrict__ multi, int n_inst,
              int64_t n_items, StageGeom sg, const __grid_constant__ TmaSet tm) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    // tensor copies want 128-byte aligned destinations: align explicitly (128 bytes of slack)
    unsigned char *smem = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 127u) & ~static_cast<uintptr_t>(127u));
    const int S = sg.nstages;
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + (size_t)S * sg.stage_bytes);
    uint64_t *empty = full + S;
    int *ctr = reinterpret_cast<int *>(empty + S);
    volatile int *abort_flag = ctr + S;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int *status = single.status ? single.status : multi[0].status;
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full[s], kFullCount);
            mbar_init(&empty[s], kConsumers);
        }
        *abort_flag = 0;
        fence_barrier_init();
    }
    __syncthreads();
    if (warp < kProducers) {
        int k = 0;
        int64_t item = blockIdx.x;
        // the instance of the current and of the next item, searched for again only when an
        // item leaves the range of the last one found
        const Inst *dc = &single, *dn = &single;
        auto find = [&](int64_t it, const Inst *hint) -> const Inst * {
            if (!multi || (it >= hint->item_begin && it < hint->item_begin + hint->n_items)) return hint;
            return &inst_of(single, multi, n_inst, it);
        };
        // One instance: descriptors of the CTA's items 32 at a time, lane l the one of item 32 b + l
        // (as in frames_kernel; read one item ahead, an item waits for the trip to memory).
        // Several: the next item's while this one is staged.
        auto read = [&](int b) {
            const int64_t it = (int64_t)blockIdx.x + (int64_t)(32 * b + lane) * gridDim.x;
            return it < n_items ? load_desc(single, it) : TileDesc{};
        };
        TileDesc td{}, cur{}, nxt{};
        if (!multi) {
            cur = read(0);
            nxt = read(1);
        } else if (item < n_items) {
            dc = dn = &inst_of(single, multi, n_inst, item);
            td = load_desc(*dc, item - dc->item_begin);
        }
        for (; item < n_items; item += gridDim.x, ++k) {
            const int s = k % S, n = k / S;
            TileDesc tn{};
            if (!multi) {
                if (k > 0 && (k & 31) == 0) {
                    cur = nxt;
                    nxt = read((k >> 5) + 1);
                }
                td = shfl_desc(cur, k & 31);
            } else {
                const int64_t next = item + gridDim.x;
                dc = dn;
                if (next < n_items) {
                    dn = find(next, dc);
                    tn = load_desc(*dn, next - dn->item_begin);
                }
            }
            bool ok = true;
            if (n > 0) ok = mbar_wait_bounded(&empty[s], (uint32_t)((n - 1) & 1));
            ok = __all_sync(0xffffffffu, ok);
            if (__any_sync(0xffffffffu, !ok || *abort_flag != 0)) {  // warp-uniform decision
                if (lane == 0) {
                    if (!ok) atomicExch(status, AZ_ETIMEOUT);
                    *abort_flag = 1;
                    for (int j = k - 1; j >= 0 && j >= k - S; --j)  // grace for own copies
                        mbar_wait_bounded(&full[j % S], (uint32_t)((j / S) & 1));
                }
                asm volatile("cp.async.wait_all;" ::: "memory");
                break;
            }
            produce<MODE, WT, TMA>(*dc, tm, item - dc->item_begin, td, smem + (size_t)s * sg.stage_bytes,
                                   sg, &full[s], &ctr[s], warp);
            td = tn;
        }
    } else {
        int k = 0;
        // a CTA's items (every gridDim.x-th) mostly stay in one instance for many rounds:
        // the instance's parameters are looked up again only when the item leaves its range
        ConsumerParams cp = consumer_params(single);
        int64_t cur_begin = 0, cur_end = multi ? 0 : n_items;
        for (int64_t item = blockIdx.x; item < n_items; item += gridDim.x, ++k) {
            const int s = k % S, n = k / S;
            if (item < cur_begin || item >= cur_end) {
                const Inst &d = inst_of(single, multi, n_inst, item);
                cp = consumer_params(d);
                cur_begin = d.item_begin;
                cur_end = d.item_begin + d.n_items;
            }
            bool ok = mbar_wait_bounded(&full[s], (uint32_t)(n & 1));
            ok = __all_sync(0xffffffffu, ok);
            if (__any_sync(0xffffffffu, !ok || *abort_flag != 0)) {  // warp-uniform decision
                if (lane == 0) {
                    if (!ok) atomicExch(status, AZ_ETIMEOUT);
                    *abort_flag = 1;
                }
                break;
            }
            consume_dispatch<AT, WT, MODE, NIMG, DT>(cp, smem + (size_t)s * sg.stage_bytes, sg, &ctr[s]);
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[s]);
        }
    }
}

// ------------------------------------------------------------------------------------
// frames pass with tile-resident entries
// ------------------------------------------------------------------------------------
// The batched frames pass spends most of its bytes on pixels, so a work item is one pixel tile (or a
// piece of a heavy one) for every frame of the launch: the item's units and entries (location,
// weight, dark) are copied once into one of two or more entry buffers and stay there while the
// tile's pixels stream through a ring of plane stages, G frames per stage.  One producer warp
// issues every copy (bulk and tensor TMA); 15 consumer warps reduce.
//
// What bounds it (64 frames of 2527 x 2463 pixels, 9.63 M entries): staging alone runs at the
// copy peak (246 us a launch), with the consumers it takes 343 us; the kernel before this one took
// 468 us.  The consumers are held by shared memory (77% of its throughput; 43% of the wavefronts
// are bank conflicts of the gathers) and by the FP32 pipe, which a packed f32x2 instruction
// occupies for two cycles.  Why this form:
//   - a lane sums one accumulator of one segment for all frames of a stage, so a unit of eight
//     segments reads each entry once for eight frames: 7 words of metadata and 16 gathers per 256
//     products.  One lane per (segment, frame) read 40 bytes of metadata per quad and frame group;
//     four frames per lane measured 7% slower than eight, two 28%.
//   - a box of depth D moves one row class of D frames: four copies per 8-frame stage instead of
//     sixteen, which takes the issue of the copies off the critical path.
//   - consumers take units from one counter across stages and items instead of passing every
//     stage together, so nobody waits for the slowest warp of a stage (11 to 15 consumer warps
//     are within 3%, 19 are 4% slower).
//   - sub.rn.f32x2 takes extra instructions, a multiply-add by -1 does not.
constexpr int kFrConsumers = 15;
constexpr int kFrThreads = 32 * (1 + kFrConsumers);
constexpr int kFrMaxStages = 16;
constexpr int kFrMaxEbufs = 6;
constexpr int kUnitWords = 10;           // a unit in the item's record: first step, steps, 8 slots
constexpr uint32_t kFrUnits = 1u << 19;  // arrivals that complete a stage's release barrier
// What the frames kernel sums per entry: w (img), w (img - dark), or w^2 max(img, 0) (the
// propagated Poisson variance of the signal sum).
enum ValueMode { VM_PLAIN = 0, VM_DARK = 1, VM_VAR = 2 };

// Three-dimensional maps of the frames: [q][c] covers the rows of equal index c mod 4 of the
// frames f = q mod 4, in (x, class row, frame / 4).  Rows of a class are 16 nx bytes apart and
// frames four apart 16 npix bytes, so any width and height meets the 16-byte stride rule, and a
// box of depth D copies one class of a tile's rows from D frames.
struct FrMaps {
    CUtensorMap m[4][4];
};

struct FrArgs {
    int n_frames, n_groups, n_tiles;      // frames in the launch, stages per item, items
    int nq, ld, nd;                       // a stage: nq values of q, D = 2^ld frames of each; nd
                                          // stages cover the frames of one q
    const int32_t *desc, *rec;            // per item: descriptor [8] and its units
    const uint16_t *ent_loc;
    const float *ent_w, *ent_dark;        // ent_dark: NULL without a dark
    float *partial;                       // [n_frames][nseg]
    int nseg, ny, nx, th, tw, ntx;
    int slot, cstride;                    // words: rows of a class, class stride
    int beta, fphase;                     // word phase of frame 0, and npix mod 4 (a frame's step)
    int *status;
    int var;                              // sum w^2 max(img, 0) instead of w img
};

struct FrGeom {
    uint32_t rec_cap;       // bytes for the tile record (multiple of 128)
    uint32_t ent_cap;       // entry capacity (multiple of 8)
    uint32_t ebuf_bytes;    // one entry buffer (multiple of 128)
    int nebufs;             // entry buffers in the ring (2 .. kFrMaxEbufs)
    uint32_t block_bytes;   // plane ring block: fslots planes
    int spb;                // stages per block (fslots / G)
    int nblocks, nstages;   // blocks and plane stages of the ring
    int dk;                 // entries carry a dark
};

__device__ __forceinline__ TileDesc fr_desc(const FrArgs &a, int item) {
    const int4 *p = reinterpret_cast<const int4 *>(a.desc) + 2 * (size_t)item;
    const int4 x = __ldg(p), y = __ldg(p + 1);
    return TileDesc{x.x, x.y, x.z, x.w, y.x, y.y};
}

// One thread: the tile's record, entry locations, weights and darks into entry buffer `eb`.
__device__ __forceinline__ void fr_stage_entries(const FrArgs &a, const FrGeom &fg, const TileDesc &td,
                                                 unsigned char *eb, uint64_t *bar) {
    const uint32_t ne = (uint32_t)td.ne;
    const uint32_t bytes = (uint32_t)td.rec_words * 4u + ne * (fg.dk ? 10u : 6u);
    fence_proxy_async_smem();
    mbar_arrive_expect_tx(bar, bytes);
    bulk_g2s(eb, a.rec + td.rec_off, (uint32_t)td.rec_words * 4u, bar);
    if (ne) {
        unsigned char *el = eb + fg.rec_cap;
        unsigned char *ew = el + fg.ent_cap * 2u;
        bulk_g2s(el, a.ent_loc + td.e_off, ne * 2u, bar);
        bulk_g2s(ew, a.ent_w + td.e_off, ne * 4u, bar);
        if (fg.dk) bulk_g2s(ew + fg.ent_cap * 4u, a.ent_dark + td.e_off, ne * 4u, bar);
    }
}

// The producer warp: stage g of an item into the planes at `dst`.  Stage g holds, for nq values
// of q from q0 on, the D frames q + 4 (D db + d), d < D; lane (qi, c) copies row class c of the D
// frames of q0 + qi with one 3D tensor copy (frames after the last are filled with zeros, and
// never reduced).  Plane i = qi D + d sits i a.slot words into each class's stretch of a.cstride
// words.  Class c's box starts at the 16-byte aligned column that puts pixel (ly, c0 + lx) at
// word c_s + phi + lx of its row for every class, c_s = (nx c) mod 4 (part of the entries'
// locations) and phi the word phase of the frame.
__device__ __forceinline__ void fr_stage_planes(const FrArgs &a, const FrMaps &fm, const TileDesc &td, int g,
                                                uint32_t dst, uint64_t *bar) {
    const int lane = threadIdx.x & 31;
    const int ti = td.t / a.ntx, tj = td.t - ti * a.ntx;
    const int c0 = tj * a.tw;
    const int qg = g / a.nd, db = g - qg * a.nd;
    const int qi = lane >> 2, c = lane & 3, q = qg * a.nq + qi;
    const int d0 = db << a.ld;                       // first frame of q in this stage: q + 4 d0
    const bool on = qi < a.nq && q + 4 * d0 < a.n_frames && c < a.ny;
    const uint32_t box = (uint32_t)(a.slot << a.ld) * 4u;
    const uint32_t n = (uint32_t)__popc(__ballot_sync(0xffffffffu, on));
    fence_proxy_async_smem();
    if (lane == 0) mbar_arrive_expect_tx(bar, n * box);
    __syncwarp();
    if (on) {
        const int phi = (a.beta + q * a.fphase) & 3, cs = ((a.nx & 3) * c) & 3;
        const int x = c0 - ((phi + cs) & 4);
        const uint32_t to = dst + (uint32_t)(c * a.cstride + (qi << a.ld) * a.slot) * 4u;
        asm volatile(
            "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
            " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(to),
            "l"(reinterpret_cast<uint64_t>(&fm.m[q][c])), "r"(x), "r"(ti * (a.th >> 2)), "r"(d0), "r"(smem_addr(bar))
            : "memory");
    }
}

// Load of a 4-byte word of shared memory at a 32-bit shared-window address (the gathers of
// the consumers index the staged planes with 32-bit arithmetic).
__device__ __forceinline__ uint32_t lds_u32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

// One unit of work of a consumer warp: eight segments of the tile for the G frames of a stage.
// Four lanes share a segment: lane j keeps accumulator j, i.e. the entries e = j mod 4 in order,
// for all G frames at once (stepped as packed f32x2 pairs), so that an entry's location, weight
// and dark are read from shared memory once for G frames.  The unit's entries are stored step by
// step, 32 to a step in lane order (a lane whose segment has ended gets weight 0 and the
// segment's last pixel), so these reads touch no bank twice and the loop has no branches.  The
// four accumulators are then merged as ((a0 + a1) + (a2 + a3)) by exchanges that halve the frames
// a lane keeps (a merge gives the same bits in either order: its rounding error is formed
// exactly).  Each value is formed by the operations of consume_serial in the same order, so a
// frame's sums do not depend on the kernel or on the frames it shares a stage with.
// unit: first step, steps, the segments' eight slots (-1: none).
// tab: of the stage's frames, the offset (bytes) of plane i from the stage's first word, and
// the frame's row of the partial sums (-1: past the last frame).
template <int G, int DT, int VM>
__device__ __forceinline__ void fr_unit(const FrArgs &a, const FrGeom &fg, const unsigned char *eb, uint32_t planes,
                                        const int2 *tab, int u) {
    static_assert(G == 1 || G == 2 || G == 4 || G == 8, "frames per stage");
    constexpr int H = G > 1 ? G / 2 : 1;
    const int lane = threadIdx.x & 31;
    const int j = lane & 3;
    const int *unit = reinterpret_cast<const int *>(eb) + kUnitWords * u;
    const int n = unit[1], slot = unit[2 + (lane >> 2)];
    const int e0 = unit[0] * 32 + lane;
    const uint16_t *L = reinterpret_cast<const uint16_t *>(eb + fg.rec_cap) + e0;
    const float *W = reinterpret_cast<const float *>(eb + fg.rec_cap + fg.ent_cap * 2u) + e0;
    const float *D = W + fg.ent_cap;
    uint32_t P[G];
#pragma unroll
    for (int i = 0; i < G; ++i) P[i] = planes + (uint32_t)tab[i].x;
    f32x2 s[H], c[H];
    Kahan k0{0.f, 0.f};
#pragma unroll
    for (int i = 0; i < H; ++i) s[i] = c[i] = 0ull;
#pragma unroll 4
    for (int t = 0; t < n; ++t) {
        const uint32_t o = (uint32_t)L[32 * t] << 2;
        float w = W[32 * t];
        float d = 0.f;
        if (VM == VM_DARK) d = D[32 * t];
        if (VM == VM_VAR) w = __fmul_rn(w, w);
        float v[G];
#pragma unroll
        for (int i = 0; i < G; ++i) v[i] = img_f32<DT>(lds_u32(P[i] + o));
        if (VM == VM_VAR) {
#pragma unroll
            for (int i = 0; i < G; ++i) v[i] = fmaxf(v[i], 0.f);
        }
        if constexpr (G == 1) {
            if (VM == VM_DARK) v[0] = __fsub_rn(v[0], d);
            kahan_add(k0, w, v[0]);
        } else {
            const f32x2 w2 = f2_pack(w, w), d2 = f2_pack(d, d);
#pragma unroll
            for (int i = 0; i < H; ++i) {
                f32x2 x = f2_pack(v[2 * i], v[2 * i + 1]);
                if (VM == VM_DARK) x = f2_sub(x, d2);
                kahan2_add(s[i], c[i], w2, x);
            }
        }
    }
    // lanes j, j ^ 1 form a0 + a1 and a2 + a3, lanes j, j ^ 2 the sum of the two
    auto put = [&](int i, const Kahan &k) {
        const int f = tab[i].y;
        if (slot >= 0 && f >= 0) a.partial[(size_t)f * (size_t)a.nseg + slot] = kahan_value(k);
    };
    if constexpr (G == 1) {
        kahan_merge(k0, shfl_xor(k0, 1));
        kahan_merge(k0, shfl_xor(k0, 2));
        if (j == 0) put(0, k0);
    } else if constexpr (G == 2) {
        Kahan x0, x1;
        f2_unpack(s[0], x0.s, x1.s);
        f2_unpack(c[0], x0.nc, x1.nc);
        Kahan k = (j & 1) ? x1 : x0;
        kahan_merge(k, shfl_xor((j & 1) ? x0 : x1, 1));
        kahan_merge(k, shfl_xor(k, 2));
        if (j < 2) put(j, k);
    } else {
        constexpr int K = H / 2;  // pairs a lane keeps after the first exchange
        f32x2 ks[K], kn[K];
#pragma unroll
        for (int i = 0; i < K; ++i) {
            const f32x2 os = (j & 1) ? s[i] : s[K + i], on = (j & 1) ? c[i] : c[K + i];
            ks[i] = (j & 1) ? s[K + i] : s[i];
            kn[i] = (j & 1) ? c[K + i] : c[i];
            kahan2_merge(ks[i], kn[i], __shfl_xor_sync(0xffffffffu, os, 1), __shfl_xor_sync(0xffffffffu, on, 1));
        }
        Kahan x0, x1;
        if constexpr (G == 4) {
            f2_unpack(ks[0], x0.s, x1.s);
            f2_unpack(kn[0], x0.nc, x1.nc);
            Kahan k = (j & 2) ? x1 : x0;
            kahan_merge(k, shfl_xor((j & 2) ? x0 : x1, 2));
            put(2 * (j & 1) + (j >> 1), k);
        } else {
            f32x2 fs = (j & 2) ? ks[1] : ks[0], fn = (j & 2) ? kn[1] : kn[0];
            const f32x2 os = (j & 2) ? ks[0] : ks[1], on = (j & 2) ? kn[0] : kn[1];
            kahan2_merge(fs, fn, __shfl_xor_sync(0xffffffffu, os, 2), __shfl_xor_sync(0xffffffffu, on, 2));
            f2_unpack(fs, x0.s, x1.s);
            f2_unpack(fn, x0.nc, x1.nc);
            put(4 * (j & 1) + (j & 2), x0);
            put(4 * (j & 1) + (j & 2) + 1, x1);
        }
    }
}

// Bounded grace wait for copies this CTA issued before giving up (every wait is bounded).
__device__ __forceinline__ void fr_drain(uint64_t *bar, uint32_t parity) { (void)mbar_wait_bounded(bar, parity); }

// Consumer warps take units (8 segments of a stage) from one counter of the CTA: item after
// item, stage after stage, longest segments first, so that a warp that finishes early goes on
// with the next stage (or item) that has landed.  A stage is released by its units: the
// producer first makes up the difference to the barrier's fixed count.  The entry buffer of an
// item is free when its last stage is, which the producer learns by waiting for that stage.
template <int G, int DT, int VM>
__global__ void __launch_bounds__(kFrThreads, 1)
frames_kernel(const __grid_constant__ FrArgs a, FrGeom fg, const __grid_constant__ FrMaps fm) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 127u) & ~static_cast<uintptr_t>(127u));
    const int S = fg.nstages;
    const int NE = fg.nebufs;
    unsigned char *ebuf0 = smem;
    unsigned char *ring = smem + (size_t)NE * fg.ebuf_bytes;
    uint64_t *efull = reinterpret_cast<uint64_t *>(ring + (size_t)fg.nblocks * fg.block_bytes);
    uint64_t *pfull = efull + NE;
    uint64_t *pempty = pfull + S;
    int2 *ftab = reinterpret_cast<int2 *>(pempty + S);            // [n_groups][G]
    uint32_t *sbase = reinterpret_cast<uint32_t *>(ftab + a.n_groups * G);  // [S] stages' first word
    int *ctr = reinterpret_cast<int *>(sbase + S);
    volatile int *abort_flag = ctr + 1;
    volatile int *issued = ctr + 2;  // plane stages and items' entries the producer has issued
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < NE; ++i) mbar_init(&efull[i], 1);
        for (int i = 0; i < S; ++i) {
            mbar_init(&pfull[i], 1);
            mbar_init(&pempty[i], kFrUnits);
        }
        *ctr = 0;
        *abort_flag = 0;
        issued[0] = issued[1] = 0;
        fence_barrier_init();
    }
    for (int t = threadIdx.x; t < a.n_groups * G; t += kFrThreads) {
        const int g = t / G, i = t - g * G;
        const int qg = g / a.nd, db = g - qg * a.nd;
        const int q = qg * a.nq + (i >> a.ld), f = q + 4 * ((db << a.ld) + (i & ((1 << a.ld) - 1)));
        ftab[t] = make_int2(4 * (i * a.slot + ((a.beta + q * a.fphase) & 3)), f < a.n_frames ? f : -1);
    }
    // blocks of fslots planes (interleaved by row class), spb stages of G planes in each
    for (int t = threadIdx.x; t < S; t += kFrThreads)
        sbase[t] = smem_addr(ring) + (uint32_t)(t / fg.spb) * fg.block_bytes + (uint32_t)((t % fg.spb) * G * a.slot) * 4u;
    __syncthreads();
    const int step = (int)gridDim.x;
    if (warp == 0) {
        // entries: ke items issued; a buffer is free again when the last stage of the item NE
        // before is, i.e. once `free_items` items are known to be done
        int ke = 0, free_items = NE;
        uint32_t j = 0;  // plane stages issued
        bool stop = false;
        auto read = [&](int b) {
            const int64_t it = (int64_t)blockIdx.x + (int64_t)(32 * b + lane) * step;
            return it < a.n_tiles ? fr_desc(a, (int)it) : TileDesc{};
        };
        TileDesc e_cur = read(0), e_nxt = read(1), p_cur = e_cur, p_nxt = e_nxt;  // entries, planes
        const int items = (a.n_tiles - (int)blockIdx.x + step - 1) / step;
        auto issue_entries = [&]() {
            while (ke < free_items && ke < items) {
                const TileDesc td = shfl_desc(e_cur, ke & 31);
                if (lane == 0)
                    fr_stage_entries(a, fg, td, ebuf0 + (size_t)(ke % NE) * fg.ebuf_bytes, &efull[ke % NE]);
                ++ke;
                if ((ke & 31) == 0) {
                    e_cur = e_nxt;
                    e_nxt = read((ke >> 5) + 1);
                }
                if (lane == 0) {
                    __threadfence_block();
                    issued[1] = ke;
                }
            }
        };
        issue_entries();
        int s = 0;          // stage in the ring, and the parity of the ring's turn
        uint32_t turn = 0;
        int seen_g = 0;  // stages known to be done, within the item free_items - NE
        for (int k = 0; k < items && !stop; ++k) {
            if (k > 0 && (k & 31) == 0) {
                p_cur = p_nxt;
                p_nxt = read((k >> 5) + 1);
            }
            const TileDesc td = shfl_desc(p_cur, k & 31);
            const uint32_t units = (uint32_t)td.ns;
            for (int g = 0; g < a.n_groups; ++g, ++j, s = s + 1 == S ? 0 : s + 1, turn ^= (s == 0)) {
                if (j >= (uint32_t)S) {
                    bool ok = mbar_wait_bounded(&pempty[s], turn ^ 1u);
                    ok = __all_sync(0xffffffffu, ok);
                    if (__any_sync(0xffffffffu, !ok || *abort_flag != 0)) {  // warp-uniform decision
                        stop = true;
                        if (!ok && lane == 0) atomicExch(a.status, AZ_ETIMEOUT);
                        break;
                    }
                    if (++seen_g == a.n_groups) {
                        seen_g = 0;
                        ++free_items;
                        issue_entries();
                    }
                }
                if (lane == 0) mbar_arrive_n(&pempty[s], kFrUnits - units);
                fr_stage_planes(a, fm, td, g, sbase[s], &pfull[s]);
                if (lane == 0) {
                    __threadfence_block();
                    issued[0] = (int)j + 1;
                }
            }
        }
        if (stop && lane == 0) {
            *abort_flag = 1;
            // grace for this CTA's own copies still in flight
            for (uint32_t jj = j > (uint32_t)S ? j - S : 0; jj < j; ++jj) fr_drain(&pfull[jj % S], (jj / S) & 1);
            for (int kk = ke > NE ? ke - NE : 0; kk < ke; ++kk) fr_drain(&efull[kk % NE], (uint32_t)((kk / NE) & 1));
        }
        return;
    }
    // consumers
    auto give_up = [&]() {
        if (lane == 0) { atomicExch(a.status, AZ_ETIMEOUT); *abort_flag = 1; }
        return false;
    };
    // The phase `parity` of `bar`, once the producer has issued more than n of what `count`
    // counts: a unit may lie more than a turn of the ring ahead, where the parity alone would be
    // taken for the turn before.
    auto wait = [&](int which, int &known, int n, uint64_t *bar, uint32_t parity) -> bool {
        if (known <= n) {
            known = __shfl_sync(0xffffffffu, issued[which], 0);
            const long long t0 = clock64();
            while (known <= n) {
                __nanosleep(64);
                const bool late = clock64() - t0 > kWaitLimitCycles;
                if (__any_sync(0xffffffffu, late)) return give_up();
                if (__any_sync(0xffffffffu, *abort_flag != 0)) return false;
                known = __shfl_sync(0xffffffffu, issued[which], 0);
            }
        }
        bool ok = mbar_try_wait(bar, parity);
        if (!__all_sync(0xffffffffu, ok)) {
            ok = mbar_wait_bounded(bar, parity);
            if (!__all_sync(0xffffffffu, ok)) return give_up();
            if (__any_sync(0xffffffffu, *abort_flag != 0)) return false;
        }
        return true;
    };
    int stages_known = 0, entries_known = 0;
    // An item's units per stage are read from its descriptor in global memory, 32 items at a time
    // as above: a warp may pass over an item that the others have finished, whose entry buffer
    // holds another item by then.
    auto unit_counts = [&](int b) -> int {
        const int64_t it = (int64_t)blockIdx.x + (int64_t)(32 * b + lane) * step;
        return it < a.n_tiles ? __ldg(a.desc + 8 * it + 5) : 0;
    };
    int n_cur = unit_counts(0), n_nxt = unit_counts(1);
    int64_t item = blockIdx.x;
    int k = 0;                        // this CTA's item number
    int per = __shfl_sync(0xffffffffu, n_cur, 0);  // units per stage
    int first = 0, units = per * a.n_groups;  // the item's first unit and its units
    float inv = 1.f / (float)per;
    int j0 = 0;                       // its first stage
    int jc = 0, s = 0;                // the last unit's stage: its number, place in the ring and
    uint32_t turn = 0;                // the parity of the ring's turn
    int eb = 0;                       // the item's entry buffer and its parity
    uint32_t eturn = 0;
    bool landed = false;              // its entries have been waited for
    int next = 0;
    if (lane == 0) next = atomicAdd(ctr, 1);
    while (true) {
        const int u = __shfl_sync(0xffffffffu, next, 0);
        while (u >= first + units) {
            j0 += a.n_groups;
            first += units;
            item += step;
            ++k;
            if (++eb == NE) { eb = 0; eturn ^= 1u; }
            landed = false;
            if (item >= a.n_tiles) return;
            if ((k & 31) == 0) {
                n_cur = n_nxt;
                n_nxt = unit_counts((k >> 5) + 1);
            }
            per = __shfl_sync(0xffffffffu, n_cur, k & 31);
            inv = 1.f / (float)per;
            units = per * a.n_groups;

        }
        if (lane == 0) next = atomicAdd(ctr, 1);
        // stage of the item and unit of the stage: u - first and per are far below 2^20, so the
        // product's error cannot reach the half that keeps it off the integers
        const int x = u - first;
        const int g = (int)(((float)x + 0.5f) * inv);
        const int j = j0 + g;
        s += j - jc;
        jc = j;
        while (s >= S) { s -= S; turn ^= 1u; }
        if (!landed && !wait(1, entries_known, k, &efull[eb], eturn)) return;
        landed = true;
        if (!wait(0, stages_known, j, &pfull[s], turn)) return;
        fr_unit<G, DT, VM>(a, fg, ebuf0 + (size_t)eb * fg.ebuf_bytes, sbase[s], ftab + g * G, x - g * per);
        __syncwarp();
        if (lane == 0) mbar_arrive(&pempty[s]);
    }
}

// ------------------------------------------------------------------------------------
// one frame per detector: correction and product in one launch
// ------------------------------------------------------------------------------------
// Items are the tiles of one integrator or of several (the many-detector plan).  A stage of the
// ring holds an item's units and entries and the raw planes of its tile (image and the correction
// arrays given).  The consumer warps first correct the tile's pixels once, in shared memory --
// x = image - dark, n = ((1 flat) solid angle) polarisation -- and then reduce the units over x and
// n as fr_unit does, so a pixel is corrected once for its two to three entries and nothing but
// the inputs is read from memory.  Work is taken from one counter, in the order: pixels of item
// 0, then for every item k the pixels of item k + 1 and the units of item k, so that nobody
// waits for pixels that are still being corrected.  C = sum w is kept per layout.
//
// FP64 (one 2527 x 2463 frame, four corrections): the FP64 pipe, whose instructions take 64 cycles a
// warp, conversions to double included, is busy for 82 us of a launch of 122 (67%; shared memory 25%,
// DRAM 24%): per pixel one subtraction and two products (the conversions are done with integer
// instructions, exactly), per entry two multiply-adds.  A call takes 134 us with tiles of 8 x 152 (140 with 8 x 120); correcting every entry and
// forming C each time took 351 us.
// FP32 (the same frame): 70 us a call (80 with 8 x 120), where a pass that wrote two planes to memory
// (28 us) and the frames kernel over them (40 us) took 78 with tiles of 8 x 224.  Of the 66 us of
// the launch with 8 x 120 the copies alone take 60, the entries and the queue without planes 25:
// five arrays are twenty small copies an item.  16 detectors without corrections: 309 us a call,
// 609 through phase1_kernel.
constexpr int kSgWarps = 15;
constexpr int kSgThreads = 32 * (1 + kSgWarps);
constexpr int kSgMaxStages = 8;
// pixels (with their row's margins) of a correction unit: in FP64 small ones, because a warp's pass
// over 32 pixels takes some 400 cycles of the FP64 pipe (6-Mpixel frame: 32 words 158 us, 64 145,
// 128 149, 384 202), in FP32 larger ones, whose cost is the taking of the unit (192 words 3% slower)
constexpr int kSgConv64 = 64, kSgConv32 = 384;
constexpr uint32_t kSgUnits = 1u << 19;  // arrivals that complete a conversion or release barrier

struct SgInst {
    const int32_t *desc, *rec;
    const uint16_t *loc;
    const void *w;             // float or double
    void *partial;             // [2][nseg]: sums of w x, and of w n
    const CUtensorMap *maps;   // [5][4] in device memory, or NULL: the launch parameter
    int nseg, nx, ny, th4, tw, ntx, slot;
    int present;               // bits: image, dark, flat, solid angle, polarisation
    int beta[5];               // word phase of each array
    int n_items;
    int64_t item_begin;
    int *status;
};

struct SgGeom {
    uint32_t rec_cap, loc_cap, w_cap;  // bytes: units, entry locations, weights (multiples of 128)
    uint32_t plane_bytes;              // one raw plane
    uint32_t xn_off;                   // FP64: corrected pixels
    uint32_t stage_bytes;
    int nstages;
};

__device__ __forceinline__ TileDesc sg_desc(const SgInst &d, int64_t local) {
    const int4 *p = reinterpret_cast<const int4 *>(d.desc) + 2 * local;
    const int4 x = __ldg(p), y = __ldg(p + 1);
    return TileDesc{x.x, x.y, x.z, x.w, y.x, y.y};
}
template <class AT> __device__ __forceinline__ int sg_conv_units(const SgInst &d) {
    constexpr int words = sizeof(AT) == 8 ? kSgConv64 : kSgConv32;
    return (4 * d.slot + words - 1) / words;
}
__device__ __forceinline__ int sg_plane(int present, int k) { return __popc(present & ((1 << k) - 1)); }

// Exact conversions to double by integer instructions.
template <int DT>
__device__ __forceinline__ double to_double(uint32_t b) {
    if (DT == AZ_DTYPE_F32) {
        const uint32_t e = (b >> 23) & 255u;
        if (e - 1u < 254u) return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))), (int)(b << 29));
        if ((b << 1) == 0u) return __hiloint2double((int)b, 0);
        return (double)__uint_as_float(b);  // subnormal, infinite, NaN
    }
    const uint32_t sign = DT == AZ_DTYPE_I32 ? b & 0x80000000u : 0u;
    const uint32_t u = sign ? 0u - b : b;
    if (u == 0u) return 0.0;
    const int lz = __clz((int)u);
    const uint32_t m = u << lz;
    return __hiloint2double((int)(sign | (((uint32_t)(1054 - lz) << 20) + ((m & 0x7fffffffu) >> 11))), (int)(m << 21));
}

template <class AT, int DT, bool X, bool N, bool V>
__device__ __forceinline__ void sg_correct(const SgInst &d, const SgGeom &sg, unsigned char *stage, int part) {
    const int lane = threadIdx.x & 31;
    const int words = 4 * d.slot;
    constexpr int kWords = sizeof(AT) == 8 ? kSgConv64 : kSgConv32;
    const int p0 = part * kWords, p1 = min(words, p0 + kWords);
    unsigned char *planes = stage + sg.rec_cap + sg.loc_cap + sg.w_cap;
    auto plane = [&](int k) {  // the words of array k, or NULL
        return (d.present >> k) & 1 ? reinterpret_cast<uint32_t *>(planes + (size_t)sg_plane(d.present, k) * sg.plane_bytes)
                                    : nullptr;
    };
    uint32_t *img = plane(0);
    const float *dark = reinterpret_cast<const float *>(plane(1));
    float *nrm[3] = {reinterpret_cast<float *>(plane(2)), reinterpret_cast<float *>(plane(3)),
                     reinterpret_cast<float *>(plane(4))};
    if constexpr (sizeof(AT) == 8) {
        // x and n side by side at the entries' locations (the rows' phases taken out)
        double *xn = reinterpret_cast<double *>(stage + sg.xn_off);
        for (int p = p0 + lane; p < p1; p += 32) {
            double x = 0.0, n = 1.0;
            if (X) {
                x = to_double<DT>(img[p + d.beta[0]]);
                if (dark) x = x - to_double<AZ_DTYPE_F32>(__float_as_uint(dark[p + d.beta[1]]));
            }
            if (N) {
                bool first = true;
#pragma unroll
                for (int k = 0; k < 3; ++k)
                    if (nrm[k]) {
                        const double f = to_double<AZ_DTYPE_F32>(__float_as_uint(nrm[k][p + d.beta[2 + k]]));
                        n = first ? f : n * f;  // 1 f is f
                        first = false;
                    }
                reinterpret_cast<double2 *>(xn)[p] = make_double2(x, n);
            } else {
                xn[p] = x;
            }
        }
    } else {
        // in place: x over the image, n over the first of its arrays
        float *x = reinterpret_cast<float *>(img);
        const int sh = dark ? d.beta[1] - d.beta[0] : 0;
        int first = -1;
#pragma unroll
        for (int k = 2; k >= 0; --k)
            if (nrm[k]) first = k;
        int s1 = 0, s2 = 0;  // the other arrays' shifts from the first one's words
        if (N && first >= 0) {
            if (first < 1 && nrm[1]) s1 = d.beta[3] - d.beta[2 + first];
            if (first < 2 && nrm[2]) s2 = d.beta[4] - d.beta[2 + first];
        }
        if (sh == 0 && s1 == 0 && s2 == 0) {  // same phases: four pixels at a time
            for (int p = p0 + 4 * lane; p < p1; p += 128) {
                if (X) {
                    const uint4 u = *reinterpret_cast<const uint4 *>(img + p);
                    float4 v = make_float4(img_f32<DT>(u.x), img_f32<DT>(u.y), img_f32<DT>(u.z), img_f32<DT>(u.w));
                    if (V) v = make_float4(fmaxf(v.x, 0.f), fmaxf(v.y, 0.f), fmaxf(v.z, 0.f), fmaxf(v.w, 0.f));
                    if (dark) {
                        const float4 k = *reinterpret_cast<const float4 *>(dark + p);
                        v = make_float4(__fsub_rn(v.x, k.x), __fsub_rn(v.y, k.y), __fsub_rn(v.z, k.z), __fsub_rn(v.w, k.w));
                    }
                    *reinterpret_cast<float4 *>(x + p) = v;
                }
                if (N && first >= 0) {
                    float4 v = *reinterpret_cast<const float4 *>(nrm[first] + p);
#pragma unroll
                    for (int k = 1; k < 3; ++k)
                        if (k > first && nrm[k]) {
                            const float4 f = *reinterpret_cast<const float4 *>(nrm[k] + p);
                            v = make_float4(__fmul_rn(v.x, f.x), __fmul_rn(v.y, f.y), __fmul_rn(v.z, f.z), __fmul_rn(v.w, f.w));
                        }
                    *reinterpret_cast<float4 *>(nrm[first] + p) = v;
                }
            }
        } else {
            // word p of the first array and word p + shift of the others are one pixel
            for (int p = p0 + lane; p < p1; p += 32) {
                if (X) {
                    float v = img_f32<DT>(img[p]);
                    if (V) v = fmaxf(v, 0.f);
                    if (dark) v = __fsub_rn(v, dark[p + sh]);
                    x[p] = v;
                }
                if (N && first >= 0) {
                    float v = nrm[first][p];
                    if (first < 1 && nrm[1]) v = __fmul_rn(v, nrm[1][p + s1]);
                    if (first < 2 && nrm[2]) v = __fmul_rn(v, nrm[2][p + s2]);
                    nrm[first][p] = v;
                }
            }
        }
    }
}

template <class AT, bool X, bool N, bool V>
__device__ __forceinline__ void sg_unit(const SgInst &d, const SgGeom &sg, const unsigned char *stage, int u) {
    const int lane = threadIdx.x & 31, j = lane & 3;
    const int *unit = reinterpret_cast<const int *>(stage) + kUnitWords * u;
    const int n = unit[1], slot = unit[2 + (lane >> 2)];
    const int e0 = unit[0] * 32 + lane;
    const uint16_t *L = reinterpret_cast<const uint16_t *>(stage + sg.rec_cap) + e0;
    const AT *W = reinterpret_cast<const AT *>(stage + sg.rec_cap + sg.loc_cap) + e0;
    AT *out = static_cast<AT *>(d.partial);
    if constexpr (sizeof(AT) == 8) {
        const double *xn = reinterpret_cast<const double *>(stage + sg.xn_off);
        double S = 0.0, M = 0.0;
#pragma unroll 4
        for (int t = 0; t < n; ++t) {
            const double w = W[32 * t];
            const int o = L[32 * t];
            double2 v;
            if (N) v = reinterpret_cast<const double2 *>(xn)[o];
            else v = make_double2(xn[o], 0.0);
            // past the segment's end (weight -0, all its bits: the upper half alone is also that
            // of negative subnormal weights): the value may be infinite
            if (__double_as_longlong(w) == (long long)(1ull << 63)) v = make_double2(0.0, 0.0);
            if (X) S = __fma_rn(w, v.x, S);
            if (N) M = __fma_rn(w, v.y, M);
        }
        // a0 + a1 and a2 + a3, then their sum (addition commutes)
        S += __shfl_xor_sync(0xffffffffu, S, 1);
        S += __shfl_xor_sync(0xffffffffu, S, 2);
        if (N) {
            M += __shfl_xor_sync(0xffffffffu, M, 1);
            M += __shfl_xor_sync(0xffffffffu, M, 2);
        }
        if (slot >= 0 && j == 0) out[slot] = S;
        if (N && slot >= 0 && j == 1) out[(size_t)d.nseg + slot] = M;
    } else {
        const uint32_t planes = smem_addr(stage + sg.rec_cap + sg.loc_cap + sg.w_cap);
        const bool norm = (d.present & 28) != 0;
        const int kn = (d.present & 4) ? 2 : ((d.present & 8) ? 3 : 4);  // the array n lies over
        const uint32_t px = planes + (uint32_t)d.beta[0] * 4u;
        const uint32_t pn = planes + (uint32_t)sg_plane(d.present, kn) * sg.plane_bytes + (uint32_t)d.beta[kn] * 4u;
        if constexpr (X && N) {
            f32x2 s = 0ull, c = 0ull;
#pragma unroll 4
            for (int t = 0; t < n; ++t) {
                const float w = W[32 * t];
                const uint32_t o = (uint32_t)L[32 * t] << 2;
                const float x = __uint_as_float(lds_u32(px + o));
                const float m = norm ? __uint_as_float(lds_u32(pn + o)) : 1.f;
                kahan2_add(s, c, f2_pack(w, w), f2_pack(x, m));
            }
            Kahan k0, k1;
            f2_unpack(s, k0.s, k1.s);
            f2_unpack(c, k0.nc, k1.nc);
            Kahan k = (j & 1) ? k1 : k0;  // even lanes keep S, odd ones N
            kahan_merge(k, shfl_xor((j & 1) ? k0 : k1, 1));
            kahan_merge(k, shfl_xor(k, 2));
            if (slot >= 0 && j < 2) out[(size_t)j * d.nseg + slot] = kahan_value(k);
        } else {
            const uint32_t pv = X ? px : pn;
            Kahan k{0.f, 0.f};
#pragma unroll 4
            for (int t = 0; t < n; ++t) {
                float w = W[32 * t];
                if (V) w = __fmul_rn(w, w);
                kahan_add(k, w, __uint_as_float(lds_u32(pv + ((uint32_t)L[32 * t] << 2))));
            }
            kahan_merge(k, shfl_xor(k, 1));
            kahan_merge(k, shfl_xor(k, 2));
            if (slot >= 0 && j == 0) out[slot] = kahan_value(k);
        }
    }
}

// X: the signal sums S; N: the normalisation sums (with X: after S); V (FP32, the image alone): the
// propagated variance sum w^2 max(img, 0) in place of S.
template <class AT, int DT, bool X, bool N, bool V = false>
__global__ void __launch_bounds__(kSgThreads, 1)
single_kernel(const __grid_constant__ SgInst one, const SgInst *__restrict__ multi, int n_inst, int n_items,
              SgGeom sg, const __grid_constant__ TmaSet tm) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 127u) & ~static_cast<uintptr_t>(127u));
    const int S = sg.nstages;
    uint64_t *full = reinterpret_cast<uint64_t *>(smem + (size_t)S * sg.stage_bytes + 128);
    uint64_t *conv = full + S, *empty = conv + S;
    int *ctr = reinterpret_cast<int *>(empty + S);
    volatile int *abort_flag = ctr + 1, *issued = ctr + 2;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int *status = one.status;
    if (threadIdx.x == 0) {
        for (int i = 0; i < S; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&conv[i], kSgUnits);
            mbar_init(&empty[i], kSgUnits);
        }
        *ctr = 0;
        *abort_flag = 0;
        *issued = 0;
        fence_barrier_init();
    }
    __syncthreads();
    const int step = (int)gridDim.x;
    const int items = (n_items - (int)blockIdx.x + step - 1) / step;
    // Of this CTA's items 32 b + lane (read 32 at a time, as in frames_kernel): the instance and
    // the descriptor.
    auto item_of = [&](int b) { return (int64_t)blockIdx.x + (int64_t)(32 * b + lane) * step; };
    auto inst_index = [&](int64_t it) {
        int lo = 0, hi = multi ? n_inst : 1;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (multi[mid].item_begin <= it) lo = mid; else hi = mid;
        }
        return lo;
    };
    auto inst = [&](int i) -> const SgInst * { return multi ? multi + i : &one; };
    if (warp == 0) {
        int s = 0, k = 0;
        uint32_t turn = 0;
        auto read = [&](int b, int &i) {
            const int64_t it = item_of(b);
            if (it >= n_items) { i = 0; return TileDesc{}; }
            i = inst_index(it);
            const SgInst *d = inst(i);
            return sg_desc(*d, it - d->item_begin);
        };
        int i_cur = 0, i_nxt = 0;
        TileDesc t_cur = read(0, i_cur), t_nxt = read(1, i_nxt);
        for (; k < items; ++k) {
            if (k > 0 && (k & 31) == 0) {
                t_cur = t_nxt;
                i_cur = i_nxt;
                t_nxt = read((k >> 5) + 1, i_nxt);
            }
            const TileDesc td = shfl_desc(t_cur, k & 31);
            const SgInst *d = inst(__shfl_sync(0xffffffffu, i_cur, k & 31));
            if (k >= S) {
                bool ok = mbar_wait_bounded(&empty[s], turn ^ 1u);
                ok = __all_sync(0xffffffffu, ok);
                if (__any_sync(0xffffffffu, !ok || *abort_flag != 0)) {  // warp-uniform decision
                    if (lane == 0) {
                        if (!ok) atomicExch(status, AZ_ETIMEOUT);
                        *abort_flag = 1;
                        // grace for this CTA's own copies still in flight
                        for (int i = k - S; i < k; ++i) (void)mbar_wait_bounded(&full[i % S], (uint32_t)((i / S) & 1));
                    }
                    return;
                }
            }
            unsigned char *stage = smem + (size_t)s * sg.stage_bytes;
            unsigned char *el = stage + sg.rec_cap, *ew = el + sg.loc_cap, *planes = ew + sg.w_cap;
            const int ti = td.t / d->ntx, tj = td.t - ti * d->ntx;
            // lane 4 a + c copies row class c of array a
            const int a = lane >> 2, c = lane & 3;
            const bool on = a < 5 && ((d->present >> a) & 1) && c < d->ny;
            const uint32_t n = (uint32_t)__popc(__ballot_sync(0xffffffffu, on));
            fence_proxy_async_smem();
            if (lane == 0) {
                mbar_arrive_n(&empty[s], kSgUnits - (uint32_t)td.ns);
                mbar_arrive_n(&conv[s], kSgUnits - (uint32_t)sg_conv_units<AT>(*d));
                mbar_arrive_expect_tx(&full[s], (uint32_t)td.rec_words * 4u + (uint32_t)td.ne * (2u + (uint32_t)sizeof(AT)) +
                                                    n * (uint32_t)d->slot * 4u);
                bulk_g2s(stage, d->rec + td.rec_off, (uint32_t)td.rec_words * 4u, &full[s]);
                bulk_g2s(el, d->loc + td.e_off, (uint32_t)td.ne * 2u, &full[s]);
                bulk_g2s(ew, static_cast<const AT *>(d->w) + td.e_off, (uint32_t)td.ne * (uint32_t)sizeof(AT), &full[s]);
            }
            __syncwarp();
            if (on) {
                const int cs = ((d->nx & 3) * c) & 3;
                const int x = tj * d->tw - ((d->beta[a] + cs) & 4);
                const uint32_t to = smem_addr(planes) + (uint32_t)sg_plane(d->present, a) * sg.plane_bytes +
                                    (uint32_t)(c * d->slot) * 4u;
                const CUtensorMap *map = d->maps ? d->maps + 4 * a + c : &tm.m[a][c];
                asm volatile(
                    "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
                    " [%0], [%1, {%2, %3}], [%4];" ::"r"(to),
                    "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(ti * d->th4), "r"(smem_addr(&full[s]))
                    : "memory");
            }
            __syncwarp();
            if (lane == 0) {
                __threadfence_block();
                *issued = k + 1;
            }
            if (++s == S) { s = 0; turn ^= 1u; }
        }
        return;
    }
    auto give_up = [&]() {
        if (lane == 0) { atomicExch(status, AZ_ETIMEOUT); *abort_flag = 1; }
        return false;
    };
    int known = 0;
    // phase `parity` of bar, once item n has been issued (see frames_kernel)
    auto wait = [&](int n, uint64_t *bar, uint32_t parity) -> bool {
        if (known <= n) {
            known = __shfl_sync(0xffffffffu, *issued, 0);
            const long long t0 = clock64();
            while (known <= n) {
                __nanosleep(64);
                const bool late = clock64() - t0 > kWaitLimitCycles;
                if (__any_sync(0xffffffffu, late)) return give_up();
                if (__any_sync(0xffffffffu, *abort_flag != 0)) return false;
                known = __shfl_sync(0xffffffffu, *issued, 0);
            }
        }
        bool ok = mbar_try_wait(bar, parity);
        if (!__all_sync(0xffffffffu, ok)) {
            ok = mbar_wait_bounded(bar, parity);
            if (!__all_sync(0xffffffffu, ok)) return give_up();
            if (__any_sync(0xffffffffu, *abort_flag != 0)) return false;
        }
        return true;
    };
    auto read = [&](int b, int &i) {
        const int64_t it = item_of(b);
        if (it >= n_items) { i = 0; return 0; }
        i = inst_index(it);
        const SgInst *d = inst(i);
        return __ldg(d->desc + 8 * (it - d->item_begin) + 5);
    };
    int i_cur = 0, i_nxt = 0;
    int n_cur = read(0, i_cur), n_nxt = read(1, i_nxt);
    // block k of the order: correction of item k + 1 (nc units), then the units of item k (ne)
    const SgInst *d1 = inst(__shfl_sync(0xffffffffu, i_cur, 0)), *d0 = d1;  // instances of items k + 1 and k
    int k = -1, s0 = 0, s1 = 0, ne = 0, nc = sg_conv_units<AT>(*d1), first = 0;
    uint32_t t0 = 0, t1 = 0;
    int ne1 = __shfl_sync(0xffffffffu, n_cur, 0);                           // units of item k + 1
    int next = 0;
    if (lane == 0) next = atomicAdd(ctr, 1);
    while (true) {
        const int u = __shfl_sync(0xffffffffu, next, 0);
        while (u >= first + nc + ne) {
            first += nc + ne;
            if (k + 1 >= items) return;
            ++k;
            d0 = d1; s0 = s1; t0 = t1; ne = ne1;
            nc = 0;
            if (++s1 == S) { s1 = 0; t1 ^= 1u; }
            const int m = k + 1;
            if (m < items) {
                if ((m & 31) == 0) {
                    n_cur = n_nxt;
                    i_cur = i_nxt;
                    n_nxt = read((m >> 5) + 1, i_nxt);
                }
                d1 = inst(__shfl_sync(0xffffffffu, i_cur, m & 31));
                nc = sg_conv_units<AT>(*d1);
                ne1 = __shfl_sync(0xffffffffu, n_cur, m & 31);
            }
        }
        if (lane == 0) next = atomicAdd(ctr, 1);
        const int x = u - first;
        if (x < nc) {
            if (!wait(k + 1, &full[s1], t1)) return;
            sg_correct<AT, DT, X, N, V>(*d1, sg, smem + (size_t)s1 * sg.stage_bytes, x);
            __syncwarp();
            if (lane == 0) mbar_arrive(&conv[s1]);
        } else {
            if (!wait(k, &conv[s0], t0)) return;
            sg_unit<AT, X, N, V>(*d0, sg, smem + (size_t)s0 * sg.stage_bytes, x - nc);
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[s0]);
        }
    }
}

// Sum of the weights of every segment, by the operations the other reductions use (four
// accumulators, entry e to accumulator e mod 4, merged as ((a0 + a1) + (a2 + a3))).
template <class AT>
__global__ void count_kernel(const int32_t *__restrict__ start, const int32_t *__restrict__ end,
                             const int32_t *__restrict__ slot, const AT *__restrict__ w, int nseg, AT *__restrict__ partial) {
    const int lane = threadIdx.x & 31, j = lane & 3;
    for (int64_t b = ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5) * 8; b < nseg;
         b += (((int64_t)gridDim.x * blockDim.x) >> 5) * 8) {
        const int64_t sg = b + (lane >> 2);
        const int e0 = sg < nseg ? start[sg] : 0, e1 = sg < nseg ? end[sg] : 0;
        Acc<AT> a;
        a.zero();
        for (int e = e0 + j; e < e1; e += 4) a.add(w[e], AT(1));
        a.merge_lower_left(1);
        a.merge_lower_left(2);
        if (sg < nseg && j == 0) partial[slot[sg]] = a.value();
    }
}

// ------------------------------------------------------------------------------------
// phase 2: per-row sums of the partials in a fixed order
// ------------------------------------------------------------------------------------
template <class AT>
__device__ __forceinline__ AT row_sum(const AT *p, int a, int b) {
    const int lane = threadIdx.x & 31;
    Acc<AT> acc;
    acc.zero();
    for (int s = a + lane; s < b; s += 32) acc.add(AT(1), p[s]);
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) acc.merge_xor(m);
    return acc.value();
}

__device__ __forceinline__ const Inst &inst_of_row(const Inst &single, const Inst *multi,
                                                   int n_inst, int64_t row) {
    if (!multi) return single;
    int lo = 0, hi = n_inst;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (multi[mid].row_begin <= row) lo = mid; else hi = mid;
    }
    return multi[lo];
}

// The value row_sum computes, formed by one thread: the 32 lanes' strided sums (virtual lane l
// sums slots l, l + 32, ...) merged by the same tree, depth first, so that a few sums are live.
template <class AT, int M>
__device__ __forceinline__ Acc<AT> row_tree(const AT *p, int n, int l) {
    Acc<AT> x;
    if constexpr (M == 32) {
        x.zero();
        for (int s = l; s < n; s += 32) x.add(AT(1), p[s]);
    } else {
        x = row_tree<AT, 2 * M>(p, n, l);
        // a merge with an empty lane's {+0, +0} changes no bit
        if (l + M < n) x.merge(row_tree<AT, 2 * M>(p, n, l + M));
    }
    return x;
}

template <class AT>
__device__ __forceinline__ AT row_sum_thread(const AT *p, int a, int b) {
    return row_tree<AT, 1>(p + a, b - a, 0).value();
}

// The frame-independent outputs of a batch, where asked for (a copy launch each cost 2 to 4 us).
__device__ __forceinline__ void put_nc(const Inst &d, int r, float N) {
    if (d.oN) static_cast<float *>(d.oN)[r] = N;
    if (d.oC) static_cast<float *>(d.oC)[r] = static_cast<const float *>(d.count)[r];
}

// Phase 2 for rows of few slots (2D patterns have one or two): a thread per row, which in
// frames mode takes kThreadFrames frames (blockIdx.y) so that the row's slot range and N are read
// once for them and the frames' loads are independent.  Bound by memory traffic: a slot's sum is
// read and four (frames: two) outputs written per row, consecutive threads on consecutive rows
// and slots.  A warp per row left 31 lanes idle on one slot and spent five rounds of shuffles:
// 66.6 us for one frame of a 500 x 360 pattern (180 000 rows, S and N) against 12.8 us here,
// 32.8 against 6.0 us in norm mode; in frames mode a thread per (row, frame), which divided 64-bit
// job numbers and read the row's range for every frame, took 50.3 us for 16 frames against 37.2.
constexpr int kThreadFrames = 4;
constexpr int kThreadRows = 4096;

template <class AT, int MODE>
__global__ void __launch_bounds__(256, 4) phase2_thread_kernel(const __grid_constant__ Inst d, int n_frames) {
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= d.nrows) return;
    const int a = d.row_slot_ptr[r], b = d.row_slot_ptr[r + 1];
    const AT *P = static_cast<const AT *>(d.partial);
    if (MODE == MODE_FRAMES) {
        const float N = d.norm[r];
        const int f0 = blockIdx.y * kThreadFrames;
#pragma unroll
        for (int i = 0; i < kThreadFrames; ++i) {
            const int f = f0 + i;
            if (f >= n_frames) break;
            const float S = (float)row_sum_thread<AT>(P + (size_t)f * d.nseg, a, b);
            const size_t o = (size_t)(d.frame_out0 + f) * d.nrows + r;
            if (d.oS) static_cast<float *>(d.oS)[o] = S;
            if (d.oI) static_cast<float *>(d.oI)[o] = N != 0.f ? __fdiv_rn(S, N) : 0.f;
        }
        if (f0 == 0) put_nc(d, r, N);
    } else if (MODE == MODE_SINGLE) {
        const AT S = row_sum_thread<AT>(P, a, b);
        const AT N = d.norm_is_count ? static_cast<const AT *>(d.count)[r] : row_sum_thread<AT>(P + d.nseg, a, b);
        const AT C = static_cast<const AT *>(d.count)[r];
        if (d.oI) static_cast<AT *>(d.oI)[r] = N != AT(0) ? S / N : AT(0);
        if (d.oS) static_cast<AT *>(d.oS)[r] = S;
        if (d.oN) static_cast<AT *>(d.oN)[r] = N;
        if (d.oC) static_cast<AT *>(d.oC)[r] = C;
    } else {
        const AT N = row_sum_thread<AT>(P, a, b);
        d.norm[r] = (float)N;
        put_nc(d, r, (float)N);
    }
}

template <class AT, int MODE>
__global__ void phase2_kernel(const __grid_constant__ Inst single, const Inst *__restrict__ multi,
                              int n_inst, int64_t n_jobs, int n_frames) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t job = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); job < n_jobs;
         job += nw) {
        if (MODE == MODE_FRAMES) {
            // job = frame * nrows + row (single instance)
            const Inst &d = single;
            const int f = (int)(job / d.nrows), r = (int)(job - (int64_t)f * d.nrows);
            const int a = d.row_slot_ptr[r], b = d.row_slot_ptr[r + 1];
            const AT S = row_sum<AT>(static_cast<const AT *>(d.partial) + (size_t)f * d.nseg, a, b);
            if (lane == 0) {
                const float N = d.norm[r];
                const size_t o = (size_t)(d.frame_out0 + f) * d.nrows + r;
                if (d.oS) static_cast<float *>(d.oS)[o] = (float)S;
                if (d.oI) static_cast<float *>(d.oI)[o] = N != 0.f ? __fdiv_rn((float)S, N) : 0.f;
                if (f == 0) put_nc(d, r, N);
            }
        } else {
            const Inst &d = inst_of_row(single, multi, n_inst, job);
            const int r = (int)(job - d.row_begin);
            const int a = d.row_slot_ptr[r], b = d.row_slot_ptr[r + 1];
            const AT *P = static_cast<const AT *>(d.partial);
            if (MODE == MODE_SINGLE) {
                const AT S = row_sum<AT>(P, a, b);
                const AT N = d.norm_is_count ? static_cast<const AT *>(d.count)[r] : row_sum<AT>(P + d.nseg, a, b);
                const AT C = static_cast<const AT *>(d.count)[r];
                if (lane == 0) {
                    const AT I = N != AT(0) ? S / N : AT(0);
                    if (d.oI) static_cast<AT *>(d.oI)[r] = I;
                    if (d.oS) static_cast<AT *>(d.oS)[r] = S;
                    if (d.oN) static_cast<AT *>(d.oN)[r] = N;
                    if (d.oC) static_cast<AT *>(d.oC)[r] = C;
                }
            } else {
                const AT N = row_sum<AT>(P, a, b);
                if (lane == 0) {
                    d.norm[r] = (float)N;
                    put_nc(d, r, (float)N);
                }
            }
        }
    }
}

// ------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------
int g_num_sms = 0;
int g_max_smem = 0;

// Stage dimensions: plane slots of `plane_words` words, `planes` of them, plus (when the
// entries are staged) room for `ent_cap` entries of (uint16 loc, wbytes weight).
constexpr uint32_t kBarrierBytes = 256 + 128;  // barriers, counters, abort flag; alignment slack

StageGeom stage_geom(uint32_t plane_words, int planes, uint32_t ent_cap, int wbytes, uint32_t rec_words,
                     int ent_dk = 0) {
    StageGeom sg;
    sg.plane_words = plane_words;
    sg.plane_region = (uint32_t)planes * plane_words * 4u;
    sg.ent_cap = ent_cap;
    sg.ent_dk = ent_dk;
    sg.rec_cap = (rec_words * 4u + 127u) & ~127u;  // keeps the plane region 128-byte aligned
    uint32_t bytes = kHeaderBytes + sg.rec_cap + sg.plane_region +
                     ent_cap * (2u + (uint32_t)wbytes + (ent_dk ? 4u : 0u));
    sg.stage_bytes = (bytes + 127u) & ~127u;
    // as many stages as fit (at least two, at most kMaxStages)
    const int avail = max_smem_per_block() - (int)kBarrierBytes;
    sg.nstages = std::min(kMaxStages, std::max(2, avail / (int)sg.stage_bytes));
    return sg;
}

uint32_t smem_for(const StageGeom &sg) { return (uint32_t)sg.nstages * sg.stage_bytes + kBarrierBytes; }

// Stage the entries when the largest tile fits twice next to the planes; otherwise the
// reduction reads the entries from global memory.
StageGeom choose_stage(uint32_t plane_words, int planes, uint32_t max_entries, int wbytes,
                       uint32_t rec_words, int &stage_entries, int ent_dk = 0) {
    StageGeom sg = stage_geom(plane_words, planes, max_entries, wbytes, rec_words, ent_dk);
    if ((int)smem_for(sg) <= max_smem_per_block()) {
        stage_entries = 1;
        return sg;
    }
    stage_entries = 0;
    return stage_geom(plane_words, planes, 0, wbytes, rec_words, ent_dk);
}

Inst make_inst(const az_integrator *h, bool fp64) {
    Inst d{};
    const TiledLayout &L = h->tl;
    d.row_slot_ptr = L.row_slot_ptr.as<int32_t>();
    d.ent_loc = L.ent_loc.as<uint16_t>();
    d.ent_w = fp64 ? (const void *)L.ent_w64.p : (const void *)L.ent_w32.p;
    d.ny = h->ny; d.nx = h->nx; d.th = L.th; d.tw = L.tw; d.srow = L.srow; d.ss = L.ss; d.ntx = L.ntx;
    d.nseg = L.nseg; d.nrows = h->nrows;
    d.npix = (int64_t)h->ny * h->nx;
    d.n_frames = 1; d.fpi = 1; d.n_groups = 1;
    d.partial = h->partial.p;
    d.norm = h->norm.as<float>();
    d.count = fp64 ? (const void *)h->count64.p : (const void *)(h->norm.as<float>() + h->nrows);
    d.status = h->status.as<int>();
    d.n_items = L.n_active;
    d.tile_desc = L.tile_desc.as<int32_t>();
    d.tile_rec = L.tile_rec.as<int32_t>();
    return d;
}

template <class AT, class WT, int MODE, int NIMG, int DT, bool TMA>
int run_phase1(const Inst &single, const Inst *multi, int n_inst, int64_t n_items,
               const StageGeom &sg, const TmaSet &tm, cudaStream_t s, Profiler *prof = nullptr) {
    if (n_items <= 0) return AZ_OK;
    const uint32_t smem = smem_for(sg);
    if ((int)smem > max_smem_per_block())
        return fail(AZ_EUNSUPPORTED, "forward: %u bytes of shared memory needed (%d available)",
                    smem, max_smem_per_block());
    auto kern = phase1_kernel<AT, WT, MODE, NIMG, DT, TMA>;
    AZ_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0;
    AZ_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, smem));
    per_sm = std::max(per_sm, 1);
    const int64_t grid = std::min<int64_t>(n_items, (int64_t)num_sms() * per_sm);
    {
        ProfScope ps(prof, MODE == MODE_FRAMES ? 0 : (MODE == MODE_NORM ? 1 : 2), s);
        kern<<<(unsigned)grid, kThreads, smem, s>>>(single, multi, n_inst, n_items, sg, tm);
    }
    AZ_CUDA(cudaGetLastError());
    return AZ_OK;
}

template <class AT, int MODE>
int run_phase2(const Inst &single, const Inst *multi, int n_inst, int64_t n_jobs, int n_frames,
               cudaStream_t s, Profiler *prof = nullptr) {
    if (n_jobs <= 0) return AZ_OK;
    // Rows of few slots on average: a thread per row, if the rows fill the GPU (4096 rows are 16
    // blocks; below that a warp per row has more loads in flight).  A 2D pattern has 1 to 2 slots
    // per row, a 1D one 100 and more: the line at 8 lies between.
    if (!multi && (int64_t)single.nseg <= 8 * (int64_t)single.nrows && single.nrows >= kThreadRows) {
        const int fy = MODE == MODE_FRAMES ? (n_frames + kThreadFrames - 1) / kThreadFrames : 1;
        ProfScope ps(prof, 3, s);
        phase2_thread_kernel<AT, MODE><<<dim3((unsigned)((single.nrows + 255) / 256), (unsigned)fy), 256, 0, s>>>(single, n_frames);
        AZ_CUDA(cudaGetLastError());
        return AZ_OK;
    }
    const int warps_per_block = 8;
    int64_t blocks = (n_jobs + warps_per_block - 1) / warps_per_block;
    blocks = std::min<int64_t>(blocks, (int64_t)num_sms() * 16);
    {
        ProfScope ps(prof, 3, s);
        phase2_kernel<AT, MODE><<<(unsigned)blocks, warps_per_block * 32, 0, s>>>(single, multi, n_inst,
                                                                               n_jobs, n_frames);
    }
    AZ_CUDA(cudaGetLastError());
    return AZ_OK;
}

template <class AT, class WT, int MODE, int NIMG, int DT>
int run_phase1_eng(int engine, const Inst &single, const Inst *multi, int n_inst, int64_t n_items,
                   const StageGeom &sg, const TmaSet &tm, cudaStream_t s, Profiler *prof) {
    if (engine == AZ_COPY_ASYNC)
        return run_phase1<AT, WT, MODE, NIMG, DT, false>(single, multi, n_inst, n_items, sg, tm, s, prof);
    return run_phase1<AT, WT, MODE, NIMG, DT, true>(single, multi, n_inst, n_items, sg, tm, s, prof);
}

template <class AT, class WT, int MODE, int NIMG>
int run_phase1_dt(int dtype, int engine, const Inst &single, const Inst *multi, int n_inst,
                  int64_t n_items, const StageGeom &sg, const TmaSet &tm, cudaStream_t s,
                  Profiler *prof = nullptr) {
    switch (dtype) {
        case AZ_DTYPE_F32:
            return run_phase1_eng<AT, WT, MODE, NIMG, AZ_DTYPE_F32>(engine, single, multi, n_inst, n_items, sg, tm, s, prof);
        case AZ_DTYPE_U32:
            return run_phase1_eng<AT, WT, MODE, NIMG, AZ_DTYPE_U32>(engine, single, multi, n_inst, n_items, sg, tm, s, prof);
        default:
            return run_phase1_eng<AT, WT, MODE, NIMG, AZ_DTYPE_I32>(engine, single, multi, n_inst, n_items, sg, tm, s, prof);
    }
}

// Dark of each tiled entry's pixel (0 for padding entries), gathered once per batch call.
__global__ void gather_dark_kernel(const int32_t *__restrict__ pix, const float *__restrict__ dark,
                                   int64_t n, float *__restrict__ out) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t p = pix[e];
        out[e] = p >= 0 ? dark[p] : 0.f;
    }
}

// ---- tensor maps for the TMA engine --------------------------------------------------
PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;

int get_encoder() {
    if (g_encode) return AZ_OK;
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000,
                                                     cudaEnableDefault, &q);
    if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn)
        return fail(AZ_EUNSUPPORTED, "cuTensorMapEncodeTiled is not available");
    g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    return AZ_OK;
}

// Four maps over `rows_total` rows of nx 4-byte words starting at `arr`: map k covers rows
// g = 4 y + k (16 * nx bytes apart) from the 16-byte aligned address just before row k, so
// that element (x, y) is column x - off_k of row g, off_k = (beta + k nx) mod 4.  Reads
// outside [0, nx + off_k) x [0, rows of class k) return zeros, so no copy reads past a row or
// the array.
int encode_class_maps(const void *arr, int64_t rows_total, int nx, int box_w, int box_h,
                      CUtensorMap out[4]) {
    AZ_TRY(get_encoder());
    const uintptr_t base = reinterpret_cast<uintptr_t>(arr);
    const int beta = (int)((base >> 2) & 3u), nu = nx & 3;
    for (int k = 0; k < 4; ++k) {
        const int offk = (beta + k * nu) & 3;
        const int64_t rows_k = rows_total > k ? (rows_total - k + 3) / 4 : 0;
        if (rows_k == 0) {
            memset(&out[k], 0, sizeof(CUtensorMap));  // never used: the producer skips the class
            continue;
        }
        void *basek = reinterpret_cast<void *>(base + 4u * (uintptr_t)k * (uintptr_t)nx - 4u * (uintptr_t)offk);
        cuuint64_t dims[2] = {(cuuint64_t)(nx + offk), (cuuint64_t)rows_k};
        cuuint64_t strides[1] = {(cuuint64_t)16 * (cuuint64_t)nx};
        cuuint32_t box[2] = {(cuuint32_t)box_w, (cuuint32_t)box_h};
        cuuint32_t estr[2] = {1, 1};
        CUresult r = g_encode(&out[k], CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, basek, dims, strides, box, estr,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return fail(AZ_ECUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
    }
    return AZ_OK;
}

// The engine a launch really uses: the TMA engine needs boxes of at most 256 words.
int engine_for(const az_integrator *h) {
    if (h->copy_engine == AZ_COPY_TMA && h->tl.srow <= 256) return AZ_COPY_TMA;
    return AZ_COPY_ASYNC;
}

// Maps for the arrays a launch stages (image rows_img rows from img; corrections ny rows).
int make_maps(const az_integrator *h, int engine, const void *img, int64_t rows_img, const float *dark,
              const float *flat, const float *sa, const float *pol, TmaSet &tm) {
    memset(&tm, 0, sizeof(tm));
    if (engine != AZ_COPY_TMA) return AZ_OK;
    const int bw = h->tl.srow, bh = h->tl.th / 4;
    const void *arrs[5] = {img, dark, flat, sa, pol};
    for (int i = 0; i < 5; ++i) {
        if (!arrs[i]) continue;
        AZ_TRY(encode_class_maps(arrs[i], i == 0 ? rows_img : h->ny, h->nx, bw, bh, tm.m[i]));
    }
    return AZ_OK;
}

uint32_t plane_words_of(const az_integrator *h) { return plane_stride(h->tl.ss); }
uint32_t rec_words_of(const az_integrator *h) { return (uint32_t)h->tl.max_rec_words; }

// ---- frames kernel with tile-resident entries -----------------------------------------
// alignment slack; barriers, stage addresses, counters; the stages' frames (up to 64 + 3 * 8)
constexpr uint32_t kFrFixedBytes = 128 + 512 + 8 * 96;

// The frames' maps (FrMaps) over nf frames starting at img: map [q][c] starts at the 16-byte
// aligned address just before row c of frame q, so its element (x, y, m) is column
// x - off of row 4 y + c of frame q + 4 m, off = the word phase of that row.  Reads outside the
// rows of the class or after the last frame return zeros.
int encode_frame_maps(const void *img, int nf, int ny, int nx, int box_w, int box_h, int depth, FrMaps &out) {
    AZ_TRY(get_encoder());
    memset(&out, 0, sizeof(out));
    const uintptr_t base = reinterpret_cast<uintptr_t>(img);
    for (int q = 0; q < 4 && q < nf; ++q)
        for (int c = 0; c < 4 && c < ny; ++c) {
            const uintptr_t row = base + 4u * ((uintptr_t)q * (uintptr_t)ny + (uintptr_t)c) * (uintptr_t)nx;
            const int off = (int)((row >> 2) & 3u);
            cuuint64_t dims[3] = {(cuuint64_t)(nx + off), (cuuint64_t)((ny - c + 3) / 4), (cuuint64_t)((nf - q + 3) / 4)};
            cuuint64_t strides[2] = {(cuuint64_t)16 * (cuuint64_t)nx, (cuuint64_t)16 * (cuuint64_t)nx * (cuuint64_t)ny};
            cuuint32_t box[3] = {(cuuint32_t)box_w, (cuuint32_t)box_h, (cuuint32_t)depth};
            cuuint32_t estr[3] = {1, 1, 1};
            CUresult r = g_encode(&out.m[q][c], CU_TENSOR_MAP_DATA_TYPE_UINT32, 3,
                                  reinterpret_cast<void *>(row - 4u * (uintptr_t)off), dims, strides, box, estr,
                                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
            if (r != CUDA_SUCCESS) return fail(AZ_ECUDA, "cuTensorMapEncodeTiled (frames) failed (%d)", (int)r);
        }
    return AZ_OK;
}

// Sizes for G frames per plane stage; false unless two entry buffers and two stages fit.
bool fr_geom(const az_integrator *h, int G, int dk, int n_groups, FrGeom &fg) {
    const TiledLayout &L = h->tl;
    if (L.fslots < G) return false;
    fg.rec_cap = ((uint32_t)L.f_max_rec * 4u + 127u) & ~127u;
    fg.ent_cap = (uint32_t)L.f_max_entries;
    fg.dk = dk;
    fg.ebuf_bytes = (fg.rec_cap + fg.ent_cap * (dk ? 10u : 6u) + 127u) & ~127u;
    fg.block_bytes = 4u * (uint32_t)L.fslots * (uint32_t)L.fslot_words * 4u;
    fg.spb = L.fslots / G;
    auto need = [&](int e, int blocks) {
        return (int64_t)e * fg.ebuf_bytes + (int64_t)blocks * fg.block_bytes + kFrFixedBytes;
    };
    const int64_t smem = max_smem_per_block();
    // two entry buffers and as many plane stages as fit; when a work item has few stages (the
    // entries dominate its copies), more entry buffers too: both rings grow together, so that as
    // many items are in flight for their planes as for their entries
    fg.nebufs = 2;
    fg.nblocks = 0;
    while ((fg.nblocks + 1) * fg.spb <= std::max(kFrMaxStages, fg.spb) && need(2, fg.nblocks + 1) <= smem) ++fg.nblocks;
    fg.nstages = fg.nblocks * fg.spb;
    if (n_groups <= 2 && fg.nstages >= 2) {
        for (int e = 2; e <= kFrMaxEbufs; ++e) {
            const int ns = std::min(kFrMaxStages, std::max(2, n_groups * e));
            const int blocks = (ns + fg.spb - 1) / fg.spb;
            if (need(e, blocks) > smem) break;
            fg.nebufs = e;
            fg.nblocks = blocks;
            fg.nstages = ns;
        }
    }
    // The producer sees a stage's release when it issues the stage nstages later, and an item's
    // entries follow the release of the item nebufs before: more stages than nebufs items have
    // would leave the last items' entries unissued.
    fg.nstages = std::min(fg.nstages, fg.nebufs * n_groups);
    return fg.nstages >= 2;
}

uint32_t fr_smem(const FrGeom &fg) {
    return (uint32_t)fg.nebufs * fg.ebuf_bytes + (uint32_t)fg.nblocks * fg.block_bytes + kFrFixedBytes;
}

template <int G, int DT, int VM>
int fr_launch(const FrArgs &a, const FrGeom &fg, const FrMaps &fm, cudaStream_t s, Profiler *prof,
              int prof_kind) {
    if (a.n_tiles <= 0) return AZ_OK;
    const uint32_t smem = fr_smem(fg);
    auto kern = frames_kernel<G, DT, VM>;
    AZ_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int grid = std::min(a.n_tiles, num_sms());
    {
        ProfScope ps(prof, prof_kind, s);
        kern<<<grid, kFrThreads, smem, s>>>(a, fg, fm);
    }
    AZ_CUDA(cudaGetLastError());
    return AZ_OK;
}

template <int G>
int fr_launch_dt(int dtype, const FrArgs &a, const FrGeom &fg, const FrMaps &tm, cudaStream_t s,
                 Profiler *prof, int kind) {
    const int vm = a.var ? VM_VAR : (a.ent_dark != nullptr ? VM_DARK : VM_PLAIN);
    switch (dtype) {
        case AZ_DTYPE_F32:
            return vm == VM_DARK ? fr_launch<G, AZ_DTYPE_F32, VM_DARK>(a, fg, tm, s, prof, kind)
                 : vm == VM_VAR  ? fr_launch<G, AZ_DTYPE_F32, VM_VAR>(a, fg, tm, s, prof, kind)
                                 : fr_launch<G, AZ_DTYPE_F32, VM_PLAIN>(a, fg, tm, s, prof, kind);
        case AZ_DTYPE_U32:
            return vm == VM_DARK ? fr_launch<G, AZ_DTYPE_U32, VM_DARK>(a, fg, tm, s, prof, kind)
                 : vm == VM_VAR  ? fr_launch<G, AZ_DTYPE_U32, VM_VAR>(a, fg, tm, s, prof, kind)
                                 : fr_launch<G, AZ_DTYPE_U32, VM_PLAIN>(a, fg, tm, s, prof, kind);
        default:
            return vm == VM_DARK ? fr_launch<G, AZ_DTYPE_I32, VM_DARK>(a, fg, tm, s, prof, kind)
                 : vm == VM_VAR  ? fr_launch<G, AZ_DTYPE_I32, VM_VAR>(a, fg, tm, s, prof, kind)
                                 : fr_launch<G, AZ_DTYPE_I32, VM_PLAIN>(a, fg, tm, s, prof, kind);
    }
}

// How a launch of nf frames is cut into stages (a) and laid out in shared memory (fg): frames
// per stage as tuned (8 by default, 4 below that), no more than the launch has; a stage covers nq
// of the four frame classes q and D frames of each, chosen for the fewest stages and then for the
// deepest copies.  False when the TMA engine or the shared memory it needs is not available.
bool fr_plan(const az_integrator *h, int nf, int dk, FrArgs &a, FrGeom &fg, int &G) {
    if (engine_for(h) != AZ_COPY_TMA || h->tl.fslots < 1) return false;
    G = h->frames_per_pass >= 8 ? 8 : 4;
    while (G > 1 && G / 2 >= nf) G >>= 1;
    for (; G >= 1; G >>= 1) {
        a.n_groups = 0;
        for (int ld = 0; (1 << ld) <= G; ++ld) {
            const int nq = G >> ld;
            if (nq > 4 || (nq > 1 && nq / 2 >= nf)) continue;
            const int nd = ((nf + 3) / 4 + (1 << ld) - 1) >> ld;
            const int groups = ((std::min(nf, 4) + nq - 1) / nq) * nd;
            if (a.n_groups == 0 || groups <= a.n_groups) {
                a.n_groups = groups; a.nq = nq; a.ld = ld; a.nd = nd;
            }
        }
        if (a.n_groups > 0 && fr_geom(h, G, dk, a.n_groups, fg)) return true;
    }
    return false;
}

// Frames kernel over `nf` frames starting at `img` (nf <= the partial buffer's frames): per-
// segment partials [nf][nseg] in h->partial.  ent_dark and ent_weights (NULL: the matrix's) are in
// the order of the layout's f_pix.  Returns AZ_EUNSUPPORTED (without error text) when fr_plan
// finds no form.
int frames_v3(az_integrator *h, const void *img, int nf, int dtype, const float *ent_dark,
              int prof_kind, cudaStream_t s, bool var = false, const float *ent_weights = nullptr) {
    FrGeom fg;
    FrArgs a{};
    int G = 0;
    if (!fr_plan(h, nf, ent_dark != nullptr, a, fg, G)) return AZ_EUNSUPPORTED;
    const TiledLayout &L = h->tl;
    a.n_frames = nf; a.n_tiles = L.n_active;
    a.desc = L.f_desc.as<int32_t>(); a.rec = L.f_rec.as<int32_t>();
    a.ent_loc = L.f_loc.as<uint16_t>();
    a.ent_w = ent_weights ? ent_weights : L.f_w32.as<float>();
    a.ent_dark = ent_dark;
    a.var = var ? 1 : 0;
    a.partial = h->partial.as<float>();
    a.nseg = L.nseg; a.ny = h->ny; a.nx = h->nx; a.th = L.th; a.tw = L.tw; a.ntx = L.ntx;
    a.slot = L.fslot_words; a.cstride = L.fslots * L.fslot_words;
    a.beta = (int)((reinterpret_cast<uintptr_t>(img) >> 2) & 3u);
    a.fphase = (int)(((int64_t)h->ny * h->nx) & 3);
    a.status = h->status.as<int>();
    FrMaps fm;
    AZ_TRY(encode_frame_maps(img, nf, h->ny, h->nx, L.srow_f, L.th / 4, 1 << a.ld, fm));
    switch (G) {
        case 1: return fr_launch_dt<1>(dtype, a, fg, fm, s, &h->prof, prof_kind);
        case 2: return fr_launch_dt<2>(dtype, a, fg, fm, s, &h->prof, prof_kind);
        case 4: return fr_launch_dt<4>(dtype, a, fg, fm, s, &h->prof, prof_kind);
        default: return fr_launch_dt<8>(dtype, a, fg, fm, s, &h->prof, prof_kind);
    }
}

// ---- single-frame kernel ----------------------------------------------------------------
constexpr uint32_t kSgFixedBytes = 128 + 128 + 256;  // alignment, margin after the last stage, barriers

// Adds integrator h to the sizes a stage needs.
struct SgNeed {
    uint32_t rec = 0, ent = 0, plane = 0;
    int planes = 0;
    void add(const az_integrator *h, int present) {
        const TiledLayout &L = h->tl;
        rec = std::max(rec, ((uint32_t)L.f_max_rec * 4u + 127u) & ~127u);
        ent = std::max(ent, (uint32_t)L.f_max_entries);
        plane = std::max(plane, 16u * (uint32_t)L.fslot_words);
        planes = std::max(planes, __builtin_popcount((unsigned)present));
    }
};

// False unless two stages fit.
bool sg_geom(const SgNeed &n, bool fp64, bool norm, SgGeom &g) {
    g.rec_cap = n.rec;
    g.loc_cap = (n.ent * 2u + 127u) & ~127u;
    g.w_cap = n.ent * (fp64 ? 8u : 4u);
    g.plane_bytes = n.plane;
    g.xn_off = g.rec_cap + g.loc_cap + g.w_cap + (uint32_t)n.planes * n.plane + 128u;  // margin: phases
    g.stage_bytes = g.xn_off + (fp64 ? n.plane * (norm ? 4u : 2u) : 0u);
    const int64_t avail = (int64_t)max_smem_per_block() - kSgFixedBytes;
    g.nstages = (int)std::min<int64_t>(kSgMaxStages, avail / std::max<uint32_t>(g.stage_bytes, 1u));
    return g.nstages >= 2;
}

SgInst sg_inst(const az_integrator *h, bool fp64, const void *const arrs[5]) {
    const TiledLayout &L = h->tl;
    SgInst d{};
    d.desc = L.f_desc.as<int32_t>(); d.rec = L.f_rec.as<int32_t>();
    d.loc = L.f_loc1.as<uint16_t>();
    d.w = fp64 ? (const void *)L.f_w64.p : (const void *)L.f_w32.p;
    d.partial = h->partial.p;
    d.nseg = L.nseg; d.nx = h->nx; d.ny = h->ny; d.th4 = L.th / 4; d.tw = L.tw; d.ntx = L.ntx; d.slot = L.fslot_words;
    for (int k = 0; k < 5; ++k)
        if (arrs[k]) {
            d.present |= 1 << k;
            d.beta[k] = (int)((reinterpret_cast<uintptr_t>(arrs[k]) >> 2) & 3u);
        }
    d.n_items = L.n_active;
    d.status = h->status.as<int>();
    return d;
}

// Maps of the arrays' row classes in the frames kernel's row pitch.
int sg_maps(const az_integrator *h, const void *const arrs[5], TmaSet &tm) {
    memset(&tm, 0, sizeof(tm));
    for (int k = 0; k < 5; ++k)
        if (arrs[k]) AZ_TRY(encode_class_maps(arrs[k], h->ny, h->nx, h->tl.srow_f, h->tl.th / 4, tm.m[k]));
    return AZ_OK;
}

template <class AT, int DT, bool X, bool N, bool V = false>
int sg_launch(const SgInst &one, const SgInst *multi, int n_inst, int n_items, const SgGeom &sg, const TmaSet &tm,
              cudaStream_t s, Profiler *prof, int kind) {
    if (n_items <= 0) return AZ_OK;
    const uint32_t smem = (uint32_t)sg.nstages * sg.stage_bytes + kSgFixedBytes;
    auto kern = single_kernel<AT, DT, X, N, V>;
    AZ_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    ProfScope ps(prof, kind, s);
    kern<<<std::min(n_items, num_sms()), kSgThreads, smem, s>>>(one, multi, n_inst, n_items, sg, tm);
    AZ_CUDA(cudaGetLastError());
    return AZ_OK;
}

template <class AT>
int sg_launch_dt(int dtype, bool norm, const SgInst &one, const SgInst *multi, int n_inst, int n_items,
                 const SgGeom &sg, const TmaSet &tm, cudaStream_t s, Profiler *prof) {
    switch (dtype) {
        case AZ_DTYPE_F32:
            return norm ? sg_launch<AT, AZ_DTYPE_F32, true, true>(one, multi, n_inst, n_items, sg, tm, s, prof, 2)
                        : sg_launch<AT, AZ_DTYPE_F32, true, false>(one, multi, n_inst, n_items, sg, tm, s, prof, 2);
        case AZ_DTYPE_U32:
            return norm ? sg_launch<AT, AZ_DTYPE_U32, true, true>(one, multi, n_inst, n_items, sg, tm, s, prof, 2)
                        : sg_launch<AT, AZ_DTYPE_U32, true, false>(one, multi, n_inst, n_items, sg, tm, s, prof, 2);
        default:
            return norm ? sg_launch<AT, AZ_DTYPE_I32, true, true>(one, multi, n_inst, n_items, sg, tm, s, prof, 2)
                        : sg_launch<AT, AZ_DTYPE_I32, true, false>(one, multi, n_inst, n_items, sg, tm, s, prof, 2);
    }
}

// flat * solid angle * polarisation per pixel, multiplied in that order from 1 (absent = 1):
// the value the norm reduction multiplies by each weight.
__global__ void norm_pixels_kernel(const float *__restrict__ flat, const float *__restrict__ sa,
                                   const float *__restrict__ pol, int64_t n, float *__restrict__ out) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n;
         p += (int64_t)gridDim.x * blockDim.x) {
        float v = 1.f;
        if (flat) v = __fmul_rn(v, flat[p]);
        if (sa) v = __fmul_rn(v, sa[p]);
        if (pol) v = __fmul_rn(v, pol[p]);
        out[p] = v;
    }
}

// Weight of each entry divided by its pixel's flat * solid angle * polarisation (0 for
// padding entries): the weights of the per-pixel-corrected form; and, with a dark, its pixel's dark.
// (In two passes, each reading the entries' pixels, a call with one 2527 x 2463 frame took 137 us.)
__global__ void gather_wnorm_kernel(const int32_t *__restrict__ pix, const float *__restrict__ w,
                                    const float *__restrict__ npx, const float *__restrict__ dark, int64_t n,
                                    float *__restrict__ out, float *__restrict__ out_dark) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int32_t p = pix[e];
        out[e] = p >= 0 ? __fdiv_rn(w[e], npx[p]) : 0.f;
        if (dark) out_dark[e] = p >= 0 ? dark[p] : 0.f;
    }
}

// One frame's two planes for the frames kernel: [cast(img) - dark] and, with corrections,
// [((1 * flat) * solid angle) * polarisation] -- the values the batched path forms per entry
// (dark) and in its norm pass, with the same roundings.
template <int DT>
__global__ void single_planes_kernel(const void *__restrict__ img, const float *__restrict__ dark,
                                     const float *__restrict__ flat, const float *__restrict__ sa,
                                     const float *__restrict__ pol, int64_t n, int with_norm,
                                     float *__restrict__ out) {
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n;
         p += (int64_t)gridDim.x * blockDim.x) {
        float v = img_f32<DT>(static_cast<const uint32_t *>(img)[p]);
        if (dark) v = __fsub_rn(v, dark[p]);
        out[p] = v;
        if (with_norm) {
            float m = 1.f;
            if (flat) m = __fmul_rn(m, flat[p]);
            if (sa) m = __fmul_rn(m, sa[p]);
            if (pol) m = __fmul_rn(m, pol[p]);
            out[n + p] = m;
        }
    }
}

}  // namespace

int num_sms() {
    if (!g_num_sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev);
        if (g_num_sms <= 0) g_num_sms = 1;
    }
    return g_num_sms;
}

int max_smem_per_block() {
    if (!g_max_smem) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&g_max_smem, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        if (g_max_smem <= 0) g_max_smem = 48 * 1024;
    }
    return g_max_smem;
}

bool wide_tiles_fit(const az_integrator *h) {
    FrGeom fg;
    SgNeed need;
    need.add(h, 31);
    SgGeom sg;
    return fr_geom(h, 8, 1, kMaxFramesPerLaunch / 8, fg) && fg.nstages >= 4 && sg_geom(need, true, true, sg) && sg.nstages >= 3;
}

// C = sum w per row of the current layout, in both precisions (it does not depend on the
// inputs): formed when the layout is built.
int count_layout(az_integrator *h, cudaStream_t s) {
    const TiledLayout &L = h->tl;
    const int32_t *start = L.seg_ent_ptr.as<int32_t>();
    const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>(((int64_t)L.nseg + 63) / 64, (int64_t)num_sms() * 16));
    for (int p = 0; p < 2; ++p) {
        Inst d = make_inst(h, p == 1);
        if (p == 0) {
            count_kernel<float><<<g, 256, 0, s>>>(start, start + L.nseg, L.seg_slot.as<int32_t>(), L.ent_w32.as<float>(),
                                                  L.nseg, h->partial.as<float>());
            AZ_CUDA(cudaGetLastError());
            d.oS = h->norm.as<float>() + h->nrows;
            d.norm_is_count = 1;  // (S only)
            AZ_TRY((run_phase2<float, MODE_SINGLE>(d, nullptr, 1, h->nrows, 1, s)));
        } else {
            count_kernel<double><<<g, 256, 0, s>>>(start, start + L.nseg, L.seg_slot.as<int32_t>(), L.ent_w64.as<double>(),
                                                   L.nseg, h->partial.as<double>());
            AZ_CUDA(cudaGetLastError());
            d.oS = h->count64.p;
            d.norm_is_count = 1;
            AZ_TRY((run_phase2<double, MODE_SINGLE>(d, nullptr, 1, h->nrows, 1, s)));
        }
    }
    return AZ_OK;
}

// One frame through single_kernel; AZ_EUNSUPPORTED (without error text) where it does not fit.
template <class AT>
int forward_one(const az_integrator *h, const void *const arrs[5], int dtype, void *oI, void *oS, void *oN, void *oC,
                void *partial, Profiler *prof, cudaStream_t s) {
    constexpr bool fp64 = sizeof(AT) == 8;
    if (engine_for(h) != AZ_COPY_TMA || h->tl.fslots < 1) return AZ_EUNSUPPORTED;
    SgInst one = sg_inst(h, fp64, arrs);
    one.partial = partial;
    const bool norm = (one.present & 28) != 0;
    SgNeed need;
    need.add(h, one.present);
    SgGeom sg;
    if (!sg_geom(need, fp64, norm, sg)) return AZ_EUNSUPPORTED;
    TmaSet tm;
    AZ_TRY(sg_maps(h, arrs, tm));
    AZ_TRY((sg_launch_dt<AT>(dtype, norm, one, nullptr, 1, one.n_items, sg, tm, s, prof)));
    Inst d = make_inst(h, fp64);
    d.partial = partial;
    d.oI = oI; d.oS = oS; d.oN = oN; d.oC = oC;
    d.norm_is_count = !norm;
    return run_phase2<AT, MODE_SINGLE>(d, nullptr, 1, h->nrows, 1, s, prof);
}

// One FP32 frame with tiles whose six planes and entries do not fit twice: the corrected frame
// and its normalisation written to memory, then the frames kernel over the two.
int forward_planes(az_integrator *h, const void *image, int dtype, const float *dark, const float *flat,
                   const float *sa, const float *pol, void *oI, void *oS, void *oN, void *oC, cudaStream_t s) {
    const bool corr = flat || sa || pol;
    FrArgs fa{};
    FrGeom fg;
    int G = 0;
    if (!fr_plan(h, corr ? 2 : 1, 0, fa, fg, G)) return AZ_EUNSUPPORTED;
    const int64_t npix = (int64_t)h->ny * h->nx;
    if (h->one_planes.bytes < 2 * sizeof(float) * (size_t)npix)
        AZ_TRY(h->one_planes.alloc(2 * sizeof(float) * (size_t)npix));
    float *planes = h->one_planes.as<float>();
    {
        ProfScope ps(&h->prof, 4, s);
        const unsigned g = (unsigned)std::min<int64_t>((npix + 255) / 256, (int64_t)num_sms() * 8);
        const int wn = corr ? 1 : 0;
        switch (dtype) {
            case AZ_DTYPE_F32: single_planes_kernel<AZ_DTYPE_F32><<<g, 256, 0, s>>>(image, dark, flat, sa, pol, npix, wn, planes); break;
            case AZ_DTYPE_U32: single_planes_kernel<AZ_DTYPE_U32><<<g, 256, 0, s>>>(image, dark, flat, sa, pol, npix, wn, planes); break;
            default: single_planes_kernel<AZ_DTYPE_I32><<<g, 256, 0, s>>>(image, dark, flat, sa, pol, npix, wn, planes); break;
        }
        AZ_CUDA(cudaGetLastError());
    }
    const int rc = frames_v3(h, planes, corr ? 2 : 1, AZ_DTYPE_F32, nullptr, 2, s);
    if (rc != AZ_OK) return rc;
    Inst d = make_inst(h, false);
    d.oI = oI; d.oS = oS; d.oN = oN; d.oC = oC;
    d.norm_is_count = !corr;
    return run_phase2<float, MODE_SINGLE>(d, nullptr, 1, h->nrows, 1, s, &h->prof);
}

// One frame through phase1_kernel (tiles or engines the kernels above do not take).
int forward_general(const az_integrator *h, const void *const arrs[5], int dtype, int precision, void *oI, void *oS,
                    void *oN, void *oC, void *partial, Profiler *prof, cudaStream_t s) {
    const bool fp64 = precision == AZ_PREC_FP64;
    const float *const c[4] = {static_cast<const float *>(arrs[1]), static_cast<const float *>(arrs[2]),
                               static_cast<const float *>(arrs[3]), static_cast<const float *>(arrs[4])};
    Inst d = make_inst(h, fp64);
    d.partial = partial;
    d.img = static_cast<const char *>(arrs[0]);
    d.dark = c[0]; d.flat = c[1]; d.sa = c[2]; d.pol = c[3];
    d.oI = oI; d.oS = oS; d.oN = oN; d.oC = oC;
    d.norm_is_count = !(c[1] || c[2] || c[3]);
    const int planes = 1 + (c[0] != nullptr) + (c[1] != nullptr) + (c[2] != nullptr) + (c[3] != nullptr);
    StageGeom sg = choose_stage(plane_words_of(h), planes, (uint32_t)h->tl.max_tile_entries,
                                fp64 ? 8 : 4, rec_words_of(h), d.stage_entries);
    const int eng = engine_for(h);
    TmaSet tm;
    AZ_TRY(make_maps(h, eng, arrs[0], h->ny, c[0], c[1], c[2], c[3], tm));
    if (fp64) {
        AZ_TRY((run_phase1_dt<double, double, MODE_SINGLE, 1>(dtype, eng, d, nullptr, 1, d.n_items, sg, tm, s, prof)));
        return run_phase2<double, MODE_SINGLE>(d, nullptr, 1, h->nrows, 1, s, prof);
    }
    AZ_TRY((run_phase1_dt<float, float, MODE_SINGLE, 1>(dtype, eng, d, nullptr, 1, d.n_items, sg, tm, s, prof)));
    return run_phase2<float, MODE_SINGLE>(d, nullptr, 1, h->nrows, 1, s, prof);
}

int forward_single(const az_integrator *h, const void *image, int dtype, const float *dark,
                   const float *flat, const float *sa, const float *pol, int precision, void *oI,
                   void *oS, void *oN, void *oC, cudaStream_t s) {
    const bool fp64 = precision == AZ_PREC_FP64;
    const void *const arrs[5] = {image, dark, flat, sa, pol};
    Profiler *prof = &h->prof;
    const int rc = fp64 ? forward_one<double>(h, arrs, dtype, oI, oS, oN, oC, h->partial.p, prof, s)
                        : forward_one<float>(h, arrs, dtype, oI, oS, oN, oC, h->partial.p, prof, s);
    if (rc != AZ_EUNSUPPORTED) return rc;
    if (!fp64) {
        const int rp = forward_planes(const_cast<az_integrator *>(h), image, dtype, dark, flat, sa, pol, oI, oS, oN, oC, s);
        if (rp != AZ_EUNSUPPORTED) return rp;
    }
    return forward_general(h, arrs, dtype, precision, oI, oS, oN, oC, h->partial.p, prof, s);
}

// Loads, without launching them, the kernels forward_single_into can launch (both
// precisions, every image type, both copy engines, and phase 2).  Under the CUDA runtime's
// lazy loading a kernel's code is otherwise loaded, and may take device memory, at its first
// launch.
template <class K> int preload_kernel(K k) {
    cudaFuncAttributes fa;
    AZ_CUDA(cudaFuncGetAttributes(&fa, k));
    return AZ_OK;
}
template <class AT, int DT> int preload_single_dt() {
    AZ_TRY((preload_kernel(single_kernel<AT, DT, true, true>)));
    AZ_TRY((preload_kernel(single_kernel<AT, DT, true, false>)));
    AZ_TRY(preload_kernel(phase1_kernel<AT, AT, MODE_SINGLE, 1, DT, true>));
    return preload_kernel(phase1_kernel<AT, AT, MODE_SINGLE, 1, DT, false>);
}
int preload_single_pass() {
    AZ_TRY((preload_single_dt<double, AZ_DTYPE_F32>()));
    AZ_TRY((preload_single_dt<double, AZ_DTYPE_U32>()));
    AZ_TRY((preload_single_dt<double, AZ_DTYPE_I32>()));
    AZ_TRY((preload_single_dt<float, AZ_DTYPE_F32>()));
    AZ_TRY((preload_single_dt<float, AZ_DTYPE_U32>()));
    AZ_TRY((preload_single_dt<float, AZ_DTYPE_I32>()));
    AZ_TRY(preload_kernel(phase2_kernel<double, MODE_SINGLE>));
    AZ_TRY(preload_kernel(phase2_kernel<float, MODE_SINGLE>));
    AZ_TRY((preload_kernel(phase2_thread_kernel<double, MODE_SINGLE>)));
    return preload_kernel(phase2_thread_kernel<float, MODE_SINGLE>);
}

// One frame with the per-segment partial sums in a buffer the caller supplies (at least
// 3 * nseg values of the accumulation type) instead of the integrator's own; no profiling and no
// allocation.  (phase1_kernel, which took every such call before, needed 151 us for a 2527 x 2463
// FP32 frame with four corrections on 8 x 120 tiles and 94 on 8 x 224; this takes 80 and 62, and
// 70 on the default 8 x 152.)
int forward_single_into(const az_integrator *h, const void *image, int dtype, const float *dark,
                        const float *flat, const float *sa, const float *pol, int precision,
                        void *oI, void *oS, void *oN, void *oC, void *partial, cudaStream_t s) {
    const void *const arrs[5] = {image, dark, flat, sa, pol};
    const int rc = precision == AZ_PREC_FP64 ? forward_one<double>(h, arrs, dtype, oI, oS, oN, oC, partial, nullptr, s)
                                             : forward_one<float>(h, arrs, dtype, oI, oS, oN, oC, partial, nullptr, s);
    if (rc != AZ_EUNSUPPORTED) return rc;
    return forward_general(h, arrs, dtype, precision, oI, oS, oN, oC, partial, nullptr, s);
}

int batch_norm(az_integrator *h, const float *flat, const float *sa, const float *pol, float *oN,
               float *oC, cudaStream_t s) {
    const int nrows = h->nrows;
    float *Cdev = h->norm.as<float>() + nrows;
    if (!flat && !sa && !pol) {  // N = C
        if (oC) AZ_CUDA(cudaMemcpyAsync(oC, Cdev, sizeof(float) * nrows, cudaMemcpyDeviceToDevice, s));
        AZ_CUDA(cudaMemcpyAsync(h->norm.as<float>(), Cdev, sizeof(float) * nrows, cudaMemcpyDeviceToDevice, s));
        if (oN) AZ_CUDA(cudaMemcpyAsync(oN, Cdev, sizeof(float) * nrows, cudaMemcpyDeviceToDevice, s));
        return AZ_OK;
    }
    Inst d = make_inst(h, false);
    d.flat = flat; d.sa = sa; d.pol = pol;
    d.oN = oN; d.oC = oC;
    if (engine_for(h) == AZ_COPY_TMA && h->tl.fslots >= 1) {
        // flat * solid angle * polarisation formed per pixel in the tiles of single_kernel: each
        // weight meets the same value as in the norm mode below, through the same accumulation.
        // (2167 x 2070 pixels, one array: 34 us; a pass that wrote it to memory and the frames
        // kernel over it took 39 us with the former layout, 51 us with this one.)
        const void *const arrs[5] = {nullptr, nullptr, flat, sa, pol};
        const SgInst one = sg_inst(h, false, arrs);
        SgNeed need;
        need.add(h, one.present);
        SgGeom g;
        if (sg_geom(need, false, true, g)) {
            TmaSet tm;
            AZ_TRY(sg_maps(h, arrs, tm));
            AZ_TRY((sg_launch<float, AZ_DTYPE_F32, false, true>(one, nullptr, 1, one.n_items, g, tm, s, &h->prof, 1)));
            return run_phase2<float, MODE_NORM>(d, nullptr, 1, h->nrows, 1, s, &h->prof);
        }
        // larger tiles: that plane in memory, one frame of the frames kernel
        FrArgs fa{};
        FrGeom fg;
        int G = 0;
        if (fr_plan(h, 1, 0, fa, fg, G)) {
            const int64_t npix = (int64_t)h->ny * h->nx;
            if (h->tl.norm_frames.bytes < sizeof(float) * (size_t)npix)
                AZ_TRY(h->tl.norm_frames.alloc(sizeof(float) * (size_t)npix));
            {
                ProfScope ps(&h->prof, 4, s);
                const int64_t blocks = std::min<int64_t>((npix + 255) / 256, (int64_t)num_sms() * 8);
                norm_pixels_kernel<<<(unsigned)blocks, 256, 0, s>>>(flat, sa, pol, npix, h->tl.norm_frames.as<float>());
                AZ_CUDA(cudaGetLastError());
            }
            const int rc = frames_v3(h, h->tl.norm_frames.p, 1, AZ_DTYPE_F32, nullptr, 1, s);
            if (rc != AZ_OK) return rc;
            return run_phase2<float, MODE_NORM>(d, nullptr, 1, h->nrows, 1, s, &h->prof);
        }
    }
    const int planes = (flat != nullptr) + (sa != nullptr) + (pol != nullptr);
    StageGeom sg = choose_stage(plane_words_of(h), planes, (uint32_t)h->tl.max_tile_entries, 4,
                                rec_words_of(h), d.stage_entries);
    const int eng = engine_for(h);
    TmaSet tm;
    AZ_TRY(make_maps(h, eng, nullptr, 0, nullptr, flat, sa, pol, tm));
    AZ_TRY((run_phase1_eng<float, float, MODE_NORM, 1, AZ_DTYPE_F32>(eng, d, nullptr, 1, d.n_items, sg, tm, s, &h->prof)));
    AZ_TRY((run_phase2<float, MODE_NORM>(d, nullptr, 1, h->nrows, 1, s, &h->prof)));
    return AZ_OK;
}

// The dark of every entry: in the order of the frames kernel's entries (f) or of the general
// kernel's.
int gather_darks(az_integrator *h, const float *dark, bool f, DevBuf &out, cudaStream_t s) {
    TiledLayout &L = h->tl;
    const int64_t n = f ? L.f_entries : L.padded_nnz;
    if (out.bytes < sizeof(float) * (size_t)n) AZ_TRY(out.alloc(sizeof(float) * (size_t)n));
    const int64_t blocks = std::min<int64_t>((n + 255) / 256, (int64_t)num_sms() * 8);
    ProfScope ps(&h->prof, 4, s);
    gather_dark_kernel<<<(unsigned)std::max<int64_t>(blocks, 1), 256, 0, s>>>(
        (f ? L.f_pix : L.ent_pix).as<int32_t>(), dark, n, out.as<float>());
    AZ_CUDA(cudaGetLastError());
    return AZ_OK;
}

int batch_frames(az_integrator *h, const void *frames, int n, int dtype, const float *dark,
                 float *oI, float *oS, int frame_out0, cudaStream_t s, bool bound_dark, const float *norm,
                 float *oN, float *oC) {
    // the dark of every entry, in entry order, so that the frames pass reads it with the
    // weights instead of staging a dark plane with every group of frames (bound_dark: gathered
    // once by az_set_corrections)
    const int ent_dk = dark != nullptr || bound_dark;
    const int64_t cap = (int64_t)(h->partial_bytes / (sizeof(float) * (size_t)std::max(h->tl.nseg, 1)));
    const int chunk = (int)std::max<int64_t>(1, std::min<int64_t>(cap, kMaxFramesPerLaunch));
    {
        // tile-resident entries (frames_kernel), up to kMaxFramesPerLaunch frames per launch
        FrArgs fa{};
        FrGeom fgeo;
        int G = 0;
        if (n > 0 && fr_plan(h, std::min(chunk, n), ent_dk, fa, fgeo, G)) {
            if (dark && !bound_dark) AZ_TRY(gather_darks(h, dark, true, h->tl.ent_dark, s));
            const float *ent_dark = !ent_dk ? nullptr : (bound_dark ? h->bound_dark[1] : h->tl.ent_dark).as<float>();
            for (int f0 = 0; f0 < n; f0 += chunk) {
                const int nf = std::min(chunk, n - f0);
                Inst d = make_inst(h, false);
                d.img = static_cast<const char *>(frames) + (size_t)f0 * (size_t)d.npix * 4u;
                const int rc = frames_v3(h, d.img, nf, dtype, ent_dark, 0, s);
                if (rc == AZ_EUNSUPPORTED)
                    return fail(AZ_EUNSUPPORTED, "batch of %d frames: the tiles do not fit in shared memory", nf);
                AZ_TRY(rc);
                if (norm) d.norm = const_cast<float *>(norm);
                d.n_frames = nf;
                d.oI = oI; d.oS = oS; d.frame_out0 = frame_out0 + f0;
                if (f0 == 0) { d.oN = oN; d.oC = oC; }
                AZ_TRY((run_phase2<float, MODE_FRAMES>(d, nullptr, 1, (int64_t)nf * h->nrows, nf, s, &h->prof)));
            }
            return AZ_OK;
        }
    }
    if (dark && !bound_dark) AZ_TRY(gather_darks(h, dark, false, h->tl.ent_dark, s));
    const float *ent_dark = (bound_dark ? h->bound_dark[0] : h->tl.ent_dark).as<float>();
    // frames per pass as tuned, halved while two stages of that many frame planes do not fit,
    // or while the tile's entries would not fit beside them (down to 4 frames per pass)
    int fpi = h->frames_per_pass;
    while (fpi > 1) {
        int se = 0;
        const StageGeom g = choose_stage(plane_words_of(h), fpi, (uint32_t)h->tl.max_tile_entries, 4,
                                         rec_words_of(h), se, ent_dk);
        if ((int)smem_for(g) <= max_smem_per_block() && (se || fpi <= 4)) break;
        fpi >>= 1;
    }
    const int chunk_max = (int)std::max<int64_t>(fpi, (cap / fpi) * fpi);
    const int planes = fpi;
    int stage_e = 0;
    StageGeom sg = choose_stage(plane_words_of(h), planes, (uint32_t)h->tl.max_tile_entries, 4,
                                rec_words_of(h), stage_e, ent_dk);
    const int eng = engine_for(h);
    for (int f0 = 0; f0 < n; f0 += chunk_max) {
        const int nf = std::min(chunk_max, n - f0);
        Inst d = make_inst(h, false);
        d.img = static_cast<const char *>(frames) + (size_t)f0 * (size_t)d.npix * 4u;
        d.n_frames = nf; d.fpi = fpi; d.n_groups = (nf + fpi - 1) / fpi;
        d.dark = dark;
        d.ent_dark = ent_dk ? ent_dark : nullptr;
        if (norm) d.norm = const_cast<float *>(norm);
        d.oI = oI; d.oS = oS; d.frame_out0 = frame_out0 + f0;
        if (f0 == 0) { d.oN = oN; d.oC = oC; }
        d.stage_entries = stage_e;
        d.n_items = h->tl.n_active * d.n_groups;
        TmaSet tm;
        AZ_TRY(make_maps(h, eng, d.img, (int64_t)nf * h->ny, nullptr, nullptr, nullptr, nullptr, tm));
        switch (fpi) {
            case 1: AZ_TRY((run_phase1_dt<float, float, MODE_FRAMES, 1>(dtype, eng, d, nullptr, 1, d.n_items, sg, tm, s, &h->prof))); break;
            case 2: AZ_TRY((run_phase1_dt<float, float, MODE_FRAMES, 2>(dtype, eng, d, nullptr, 1, d.n_items, sg, tm, s, &h->prof))); break;
            case 4: AZ_TRY((run_phase1_dt<float, float, MODE_FRAMES, 4>(dtype, eng, d, nullptr, 1, d.n_items, sg, tm, s, &h->prof))); break;
            case 8: AZ_TRY((run_phase1_dt<float, float, MODE_FRAMES, 8>(dtype, eng, d, nullptr, 1, d.n_items, sg, tm, s, &h->prof))); break;
            case 16: AZ_TRY((run_phase1_dt<float, float, MODE_FRAMES, 16>(dtype, eng, d, nullptr, 1, d.n_items, sg, tm, s, &h->prof))); break;
            default: AZ_TRY((run_phase1_dt<float, float, MODE_FRAMES, 32>(dtype, eng, d, nullptr, 1, d.n_items, sg, tm, s, &h->prof))); break;
        }
        AZ_TRY((run_phase2<float, MODE_FRAMES>(d, nullptr, 1, (int64_t)nf * h->nrows, nf, s, &h->prof)));
    }
    return AZ_OK;
}

// The paper's per-pixel-corrected form for n frames: U = sum (w / (flat Omega P)) (img - dark)
// and I = U / C, C = sum w (kept per layout).  Through the frames kernel with the weights
// divided by each pixel's normalisation once per call.
int batch_pixelnorm(az_integrator *h, const void *frames, int n, int dtype, const float *dark,
                    const float *flat, const float *sa, const float *pol, float *oI, float *oU,
                    float *oC, cudaStream_t s) {
    if (engine_for(h) != AZ_COPY_TMA || h->tl.fslots < 1 || h->partial_bytes < 2 * sizeof(float) * (size_t)h->tl.nseg)
        return fail(AZ_EUNSUPPORTED, "az_integrate_batch_pixelnorm: needs the tensor-copy engine (tiles up to 236 pixels wide)");
    TiledLayout &L = h->tl;
    const int64_t npix = (int64_t)h->ny * h->nx;
    const int nrows = h->nrows;
    // C of the current layout
    const float *Cdev = h->norm.as<float>() + nrows;
    if (n == 0) {
        if (oC) AZ_CUDA(cudaMemcpyAsync(oC, Cdev, sizeof(float) * nrows, cudaMemcpyDeviceToDevice, s));
        return AZ_OK;
    }
    // per-pixel normalisation, per-entry corrected weights and darks
    const int64_t pblocks = std::min<int64_t>((npix + 255) / 256, (int64_t)num_sms() * 8);
    const int64_t eblocks = std::max<int64_t>(1, std::min<int64_t>((L.f_entries + 255) / 256, (int64_t)num_sms() * 8));
    if (L.norm_frames.bytes < sizeof(float) * (size_t)npix) AZ_TRY(L.norm_frames.alloc(sizeof(float) * (size_t)npix));
    if (L.ent_wnorm.bytes < sizeof(float) * (size_t)L.f_entries)
        AZ_TRY(L.ent_wnorm.alloc(sizeof(float) * (size_t)L.f_entries));
    if (dark && L.ent_dark.bytes < sizeof(float) * (size_t)L.f_entries)
        AZ_TRY(L.ent_dark.alloc(sizeof(float) * (size_t)L.f_entries));
    const float *ent_dk = dark ? L.ent_dark.as<float>() : nullptr;
    {
        ProfScope ps(&h->prof, 4, s);
        norm_pixels_kernel<<<(unsigned)pblocks, 256, 0, s>>>(flat, sa, pol, npix, L.norm_frames.as<float>());
        gather_wnorm_kernel<<<(unsigned)eblocks, 256, 0, s>>>(L.f_pix.as<int32_t>(), L.f_w32.as<float>(),
                                                              L.norm_frames.as<float>(), dark, L.f_entries,
                                                              L.ent_wnorm.as<float>(), L.ent_dark.as<float>());
        AZ_CUDA(cudaGetLastError());
    }
    const int64_t cap = (int64_t)(h->partial_bytes / (sizeof(float) * (size_t)std::max(L.nseg, 1)));
    const int chunk = (int)std::max<int64_t>(1, std::min<int64_t>(cap, kMaxFramesPerLaunch));
    for (int f0 = 0; f0 < n; f0 += chunk) {
        const int nf = std::min(chunk, n - f0);
        Inst d = make_inst(h, false);
        d.img = static_cast<const char *>(frames) + (size_t)f0 * (size_t)d.npix * 4u;
        const int rc = frames_v3(h, d.img, nf, dtype, ent_dk, 0, s, false, L.ent_wnorm.as<float>());
        if (rc == AZ_EUNSUPPORTED)
            return fail(AZ_EUNSUPPORTED, "az_integrate_batch_pixelnorm: the tiles do not fit in shared memory");
        AZ_TRY(rc);
        d.n_frames = nf;
        d.norm = const_cast<float *>(Cdev);  // I = U / C
        d.oI = oI; d.oS = oU; d.frame_out0 = f0;
        if (f0 == 0) d.oC = oC;
        AZ_TRY((run_phase2<float, MODE_FRAMES>(d, nullptr, 1, (int64_t)nf * nrows, nf, s, &h->prof)));
    }
    return AZ_OK;
}

// One frame's variance sums through single_kernel; AZ_EUNSUPPORTED (without error text) where its
// stages do not fit.
int variance_one(const az_integrator *h, const void *img, int dtype, cudaStream_t s) {
    if (engine_for(h) != AZ_COPY_TMA || h->tl.fslots < 1) return AZ_EUNSUPPORTED;
    const void *const arrs[5] = {img, nullptr, nullptr, nullptr, nullptr};
    const SgInst one = sg_inst(h, false, arrs);
    SgNeed need;
    need.add(h, one.present);
    SgGeom sg;
    if (!sg_geom(need, false, false, sg)) return AZ_EUNSUPPORTED;
    TmaSet tm;
    AZ_TRY(sg_maps(h, arrs, tm));
    switch (dtype) {
        case AZ_DTYPE_F32: return sg_launch<float, AZ_DTYPE_F32, true, false, true>(one, nullptr, 1, one.n_items, sg, tm, s, &h->prof, 0);
        case AZ_DTYPE_U32: return sg_launch<float, AZ_DTYPE_U32, true, false, true>(one, nullptr, 1, one.n_items, sg, tm, s, &h->prof, 0);
        default: return sg_launch<float, AZ_DTYPE_I32, true, false, true>(one, nullptr, 1, one.n_items, sg, tm, s, &h->prof, 0);
    }
}

// Propagated variance of the signal sums, V = sum w^2 max(img, 0), for n frames through the
// frames kernel (chunks of up to kMaxFramesPerLaunch frames), written to oV [n][nrows].
int batch_variance(az_integrator *h, const void *frames, int n, int dtype, float *oV, cudaStream_t s) {
    if (engine_for(h) != AZ_COPY_TMA)
        return fail(AZ_EUNSUPPORTED, "az_integrate_variance: needs the tensor-copy engine (tiles up to 236 pixels wide)");
    const int64_t cap = (int64_t)(h->partial_bytes / (sizeof(float) * (size_t)std::max(h->tl.nseg, 1)));
    const int chunk = (int)std::max<int64_t>(1, std::min<int64_t>(cap, kMaxFramesPerLaunch));
    for (int f0 = 0; f0 < n; f0 += chunk) {
        const int nf = std::min(chunk, n - f0);
        Inst d = make_inst(h, false);
        d.img = static_cast<const char *>(frames) + (size_t)f0 * (size_t)d.npix * 4u;
        int rc = nf == 1 ? variance_one(h, d.img, dtype, s) : AZ_EUNSUPPORTED;
        if (rc == AZ_EUNSUPPORTED) rc = frames_v3(h, d.img, nf, dtype, nullptr, 0, s, true);
        if (rc == AZ_EUNSUPPORTED)
            return fail(AZ_EUNSUPPORTED, "az_integrate_variance: the tiles do not fit in shared memory");
        AZ_TRY(rc);
        d.n_frames = nf;
        d.oI = nullptr; d.oS = oV; d.frame_out0 = f0;
        AZ_TRY((run_phase2<float, MODE_FRAMES>(d, nullptr, 1, (int64_t)nf * h->nrows, nf, s, &h->prof)));
    }
    return AZ_OK;
}

int forward_batch(az_integrator *h, const void *frames, int n, int dtype, const float *dark,
                  const float *flat, const float *sa, const float *pol, float *oI, float *oS,
                  float *oN, float *oC, cudaStream_t s) {
    if (n == 0) return batch_norm(h, flat, sa, pol, oN, oC, s);
    const bool corr = flat || sa || pol;
    if (corr) AZ_TRY(batch_norm(h, flat, sa, pol, nullptr, nullptr, s));
    const float *norm = corr ? nullptr : h->norm.as<float>() + h->nrows;  // N = C
    return batch_frames(h, frames, n, dtype, dark, oI, oS, 0, s, false, norm, oN, oC);
}

// Whether a batch with darks goes through the frames kernel.  (If one frame fits, any number does:
// fr_plan comes down to the same stages.)
bool takes_frames_kernel(const az_integrator *h) {
    FrArgs a{};
    FrGeom fg;
    int G = 0;
    return fr_plan(h, 1, 1, a, fg, G);
}

__global__ void scatter_dark_kernel(const int32_t *__restrict__ pix, const float *__restrict__ ent, int64_t n,
                                    float *__restrict__ dark) {
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x)
        if (pix[e] >= 0) dark[pix[e]] = ent[e];  // (equal values for the entries of a pixel)
}

// The caller's dark is not at hand any more: its pixels from the entries of one order, then the
// entries of the other.  No stream is given: the device is waited for before and after.
int convert_bound_darks(az_integrator *h) {
    const bool f = takes_frames_kernel(h);
    if (!h->corr_bound || !h->corr_dark || h->bound_dark_ok[f]) return AZ_OK;
    const cudaStream_t s = nullptr;
    AZ_CUDA(cudaDeviceSynchronize());
    ScratchScope scope;
    TmpBuf plane;
    AZ_TRY(plane.alloc(sizeof(float) * (size_t)h->ny * (size_t)h->nx));
    const int64_t n = f ? h->tl.padded_nnz : h->tl.f_entries;
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)num_sms() * 8));
    scatter_dark_kernel<<<(unsigned)blocks, 256, 0, s>>>((f ? h->tl.ent_pix : h->tl.f_pix).as<int32_t>(),
                                                         h->bound_dark[!f].as<float>(), n, plane.as<float>());
    AZ_CUDA(cudaGetLastError());
    AZ_TRY(gather_darks(h, plane.as<float>(), f, h->bound_dark[f], s));
    AZ_CUDA(cudaStreamSynchronize(s));
    h->bound_dark_ok[f] = true;
    return AZ_OK;
}

// az_set_corrections: the frame-independent work of a batch formed once -- each entry's dark
// (gathered from `dark`) and N, C per row -- into buffers of their own, which later calls of
// az_integrate_batch do not touch.  The caller's arrays are not read again.
int bind_corrections(az_integrator *h, const float *dark, const float *flat, const float *sa,
                     const float *pol, cudaStream_t s) {
    h->corr_bound = false;
    h->corr_dark = dark != nullptr;
    h->bound_dark_ok[0] = h->bound_dark_ok[1] = false;
    if (dark) {
        const bool f = takes_frames_kernel(h);
        AZ_TRY(gather_darks(h, dark, f, h->bound_dark[f], s));
        h->bound_dark_ok[f] = true;
    }
    if (h->bound_norm.bytes < 2 * sizeof(float) * (size_t)h->nrows)
        AZ_TRY(h->bound_norm.alloc(2 * sizeof(float) * (size_t)h->nrows));
    float *bN = h->bound_norm.as<float>();
    AZ_TRY(batch_norm(h, flat, sa, pol, bN, bN + h->nrows, s));
    h->corr_bound = true;
    return AZ_OK;
}

// Frames through the bound corrections: the frames pass with the bound per-entry darks and
// phase 2 with the bound N.  oN, oC (may be NULL) receive copies of the bound N and C.
int forward_batch_bound(az_integrator *h, const void *frames, int n, int dtype, float *oI, float *oS,
                        float *oN, float *oC, cudaStream_t s) {
    if (!h->corr_bound)
        return fail(AZ_EINVAL, "az_integrate_batch_bound: no corrections are bound (az_set_corrections), "
                               "or the tiled layout changed since they were");
    const float *bN = h->bound_norm.as<float>();
    const size_t rb = sizeof(float) * (size_t)h->nrows;
    if (n == 0) {
        if (oN) AZ_CUDA(cudaMemcpyAsync(oN, bN, rb, cudaMemcpyDeviceToDevice, s));
        if (oC) AZ_CUDA(cudaMemcpyAsync(oC, bN + h->nrows, rb, cudaMemcpyDeviceToDevice, s));
        return AZ_OK;
    }
    return batch_frames(h, frames, n, dtype, nullptr, oI, oS, 0, s, h->corr_dark, bN, oN, oC);
}

// ------------------------------------------------------------------------------------
// heterogeneous instances in one persistent launch
// ------------------------------------------------------------------------------------
struct MultiPlan {
    std::vector<Inst> host;
    DevBuf dev;
    DevBuf maps;  // TMA engine: n TmaSets, one per instance, read by the producers
    int n = 0;
    int dtype = 0, engine = 0;
    int64_t n_items = 0, n_rows = 0;
    StageGeom sg{};
    bool single = false, norm = false;  // through single_kernel; with normalisation sums
    SgGeom sgeo{};
    SgInst first{};
    DevBuf sg_dev;       // SgInst [n]
    std::vector<std::pair<const az_integrator *, int64_t>> layouts;  // integrators and their layouts
    // partial sums of an integrator's second and further instances (the first has its own)
    std::vector<std::unique_ptr<DevBuf>> partials;
    cudaGraphExec_t exec = nullptr;
    cudaGraph_t graph = nullptr;
};

int multi_create(az_integrator *const *hs, int n, const void *const *images, int dtype,
                 const float *const *darks, const float *const *flats, const float *const *sas,
                 const float *const *pols, float *const *oI, float *const *oS, float *const *oN,
                 float *const *oC, void **out) {
    MultiPlan *P = new (std::nothrow) MultiPlan;
    if (!P) return fail(AZ_ENOMEM, "az_multi_create: out of host memory");
    P->n = n;
    P->dtype = dtype;
    int64_t items = 0, rows = 0;
    uint32_t pw = 0, ecap = 0, rw = 0;
    // The TMA engine when every instance can use it: each instance's tensor maps then live in
    // device memory (a launch parameter holds one set only) and the producers read them there.
    P->engine = AZ_COPY_TMA;
    for (int k = 0; k < n; ++k)
        if (engine_for(hs[k]) != AZ_COPY_TMA) P->engine = AZ_COPY_ASYNC;
    // ... through single_kernel, if two stages of the largest instance fit, else phase1_kernel
    P->single = P->engine == AZ_COPY_TMA;
    SgNeed need;
    std::vector<SgInst> sgi;
    for (int k = 0; k < n && P->single; ++k) {
        if (hs[k]->tl.fslots < 1) P->single = false;
        const void *const arrs[5] = {images[k], darks ? darks[k] : nullptr, flats ? flats[k] : nullptr,
                                     sas ? sas[k] : nullptr, pols ? pols[k] : nullptr};
        SgInst d = sg_inst(hs[k], false, arrs);
        need.add(hs[k], d.present);
        P->norm = P->norm || (d.present & 28);
        d.item_begin = sgi.empty() ? 0 : sgi.back().item_begin + sgi.back().n_items;
        sgi.push_back(d);
    }
    if (P->single) P->single = sg_geom(need, false, P->norm, P->sgeo);
    std::vector<TmaSet> maps;
    if (P->engine == AZ_COPY_TMA) {
        maps.resize((size_t)n);
        int rc = P->maps.alloc(sizeof(TmaSet) * (size_t)n);
        for (int k = 0; k < n && rc == AZ_OK; ++k)
        {
            const void *const arrs[5] = {images[k], darks ? darks[k] : nullptr, flats ? flats[k] : nullptr,
                                         sas ? sas[k] : nullptr, pols ? pols[k] : nullptr};
            rc = P->single ? sg_maps(hs[k], arrs, maps[(size_t)k])
                           : make_maps(hs[k], AZ_COPY_TMA, images[k], hs[k]->ny, darks ? darks[k] : nullptr,
                                       flats ? flats[k] : nullptr, sas ? sas[k] : nullptr, pols ? pols[k] : nullptr,
                                       maps[(size_t)k]);
            if (P->single) sgi[(size_t)k].maps = &P->maps.as<TmaSet>()[k].m[0][0];
        }
        if (rc == AZ_OK) {
            cudaError_t e = cudaMemcpy(P->maps.p, maps.data(), sizeof(TmaSet) * (size_t)n, cudaMemcpyHostToDevice);
            if (e != cudaSuccess) rc = fail(AZ_ECUDA, "az_multi_create: %s", cudaGetErrorString(e));
        }
        if (rc != AZ_OK) {
            delete P;
            return rc;
        }
    }
    int planes = 0;
    for (int k = 0; k < n; ++k) {
        const az_integrator *h = hs[k];
        Inst d = make_inst(h, false);
        d.img = static_cast<const char *>(images[k]);
        d.dark = darks ? darks[k] : nullptr;
        d.flat = flats ? flats[k] : nullptr;
        d.sa = sas ? sas[k] : nullptr;
        d.pol = pols ? pols[k] : nullptr;
        d.oI = oI ? oI[k] : nullptr;
        d.oS = oS ? oS[k] : nullptr;
        d.oN = oN ? oN[k] : nullptr;
        d.oC = oC ? oC[k] : nullptr;
        if (P->engine == AZ_COPY_TMA) d.maps = &P->maps.as<TmaSet>()[k].m[0][0];
        d.norm_is_count = P->single ? !P->norm : !(d.flat || d.sa || d.pol);
        d.item_begin = items;
        d.row_begin = rows;
        items += d.n_items;
        rows += h->nrows;
        pw = std::max(pw, plane_words_of(h));
        ecap = std::max(ecap, (uint32_t)h->tl.max_tile_entries);
        rw = std::max(rw, rec_words_of(h));
        planes = std::max(planes, 1 + (d.dark != nullptr) + (d.flat != nullptr) + (d.sa != nullptr) +
                                      (d.pol != nullptr));
        P->host.push_back(d);
    }
    int stage_e = 0;
    P->sg = choose_stage(pw, planes, ecap, 4, rw, stage_e);
    for (auto &d : P->host) d.stage_entries = stage_e;
    for (int k = 0; k < n; ++k) P->layouts.emplace_back(hs[k], hs[k]->layout_no);
    P->n_items = items;
    P->n_rows = rows;
    for (int k = 0; k < n; ++k) {
        if (std::find(hs, hs + k, hs[k]) == hs + k) continue;
        P->partials.emplace_back(new DevBuf);
        const int rp = P->partials.back()->alloc(3 * sizeof(float) * (size_t)std::max(hs[k]->tl.nseg, 1));
        if (rp != AZ_OK) {
            delete P;
            return rp;
        }
        P->host[(size_t)k].partial = P->partials.back()->p;
        if (P->single) sgi[(size_t)k].partial = P->partials.back()->p;
    }
    int rc = P->dev.alloc(sizeof(Inst) * (size_t)n);
    if (rc == AZ_OK) {
        cudaError_t e = cudaMemcpy(P->dev.p, P->host.data(), sizeof(Inst) * (size_t)n, cudaMemcpyHostToDevice);
        if (e != cudaSuccess) rc = fail(AZ_ECUDA, "az_multi_create: %s", cudaGetErrorString(e));
    }
    if (rc == AZ_OK && P->single) {
        P->first = sgi[0];
        rc = P->sg_dev.alloc(sizeof(SgInst) * (size_t)n);
        if (rc == AZ_OK) {
            cudaError_t e = cudaMemcpy(P->sg_dev.p, sgi.data(), sizeof(SgInst) * (size_t)n, cudaMemcpyHostToDevice);
            if (e != cudaSuccess) rc = fail(AZ_ECUDA, "az_multi_create: %s", cudaGetErrorString(e));
        }
    }
    if (rc != AZ_OK) {
        delete P;
        return rc;
    }
    *out = P;
    return AZ_OK;
}

int multi_enqueue(void *plan, cudaStream_t s) {
    MultiPlan *P = static_cast<MultiPlan *>(plan);
    const Inst *dev = P->dev.as<Inst>();
    static TmaSet no_maps;  // zero: the producers read each instance's maps from Inst::maps
    if (P->single)
        AZ_TRY((sg_launch_dt<float>(P->dtype, P->norm, P->first, P->sg_dev.as<SgInst>(), P->n, (int)P->n_items, P->sgeo,
                                    no_maps, s, nullptr)));
    else
        AZ_TRY((run_phase1_dt<float, float, MODE_SINGLE, 1>(P->dtype, P->engine, P->host[0], dev, P->n, P->n_items, P->sg, no_maps, s)));
    AZ_TRY((run_phase2<float, MODE_SINGLE>(P->host[0], dev, P->n, P->n_rows, 1, s)));
    return AZ_OK;
}

int multi_launch(void *plan, int use_graph, cudaStream_t s) {
    MultiPlan *P = static_cast<MultiPlan *>(plan);
    for (size_t k = 0; k < P->layouts.size(); ++k)
        if (P->layouts[k].first->layout_no != P->layouts[k].second)
            return fail(AZ_EINVAL, "az_multi_launch: integrator %d got other tiles (az_set_tuning, az_autotune) since "
                                   "the plan was made: make a new plan", (int)k);
    if (!use_graph) return multi_enqueue(plan, s);
    if (!P->exec) {
        // Run once eagerly (this call's results; it also configures the kernels), then
        // capture the two launches on a private stream: the caller's stream may be the
        // legacy default stream, which cannot be captured.
        AZ_TRY(multi_enqueue(plan, s));
        cudaStream_t cs = nullptr;
        AZ_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
        cudaError_t e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeRelaxed);
        int rc = e == cudaSuccess ? multi_enqueue(plan, cs)
                                  : fail(AZ_ECUDA, "graph capture: %s", cudaGetErrorString(e));
        cudaGraph_t g = nullptr;
        if (e == cudaSuccess) {
            e = cudaStreamEndCapture(cs, &g);
            if (e != cudaSuccess && rc == AZ_OK) rc = fail(AZ_ECUDA, "graph capture: %s", cudaGetErrorString(e));
        }
        cudaStreamDestroy(cs);
        if (rc != AZ_OK) {
            if (g) cudaGraphDestroy(g);
            return rc;
        }
        P->graph = g;
        AZ_CUDA(cudaGraphInstantiate(&P->exec, g, 0));
        return AZ_OK;
    }
    AZ_CUDA(cudaGraphLaunch(P->exec, s));
    return AZ_OK;
}

void multi_destroy(void *plan) {
    MultiPlan *P = static_cast<MultiPlan *>(plan);
    if (!P) return;
    if (P->exec) cudaGraphExecDestroy(P->exec);
    if (P->graph) cudaGraphDestroy(P->graph);
    delete P;
}

}  // namespace azint
