// C ABI of the library: argument validation, handle lifetime, error strings, build
// orchestration, the end-to-end host-buffer path and the tuner.  The device work is done by
// the kernels in geometry.cu, csr_build.cu, integrate.cu, lut.cu and backward.cu (the
// allocation-free entry point and the wait self-test have their own files); the only kernel
// here fills the tuner's synthetic frames.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>

#include "common.cuh"

namespace azint {

namespace {
thread_local char g_err[512] = "";

bool aligned4(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 3u) == 0; }

__global__ void fill_frames_kernel(uint32_t *out, int64_t n, uint32_t seed) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n;
         k += (int64_t)gridDim.x * blockDim.x) {
        uint32_t x = (uint32_t)k * 2654435761u ^ seed;
        x ^= x >> 16;
        x *= 2246822519u;
        x ^= x >> 13;
        out[k] = x & 1023u;
    }
}

int alloc_scratch(az_integrator *h, cudaStream_t s) {
    const size_t nseg = (size_t)std::max(h->tl.nseg, 1);
    const size_t single = 3 * nseg * sizeof(double);
    const size_t frames = (size_t)kMaxFramesPerLaunch * nseg * sizeof(float);
    h->partial_bytes = std::max(single, frames);
    AZ_TRY(alloc_parts(h->slab_scratch, {{&h->partial, h->partial_bytes},
                                         {&h->norm, sizeof(float) * 2 * (size_t)h->nrows},
                                         {&h->count64, sizeof(double) * (size_t)h->nrows},
                                         {&h->adj, sizeof(double) * 2 * (size_t)h->nrows}}));
    return count_layout(h, s);
}

// The layout of th x tw tiles with the scratch that goes with it.
int set_tiles(az_integrator *h, int th, int tw, cudaStream_t s) {
    AZ_TRY(build_tiled_layout(h, th, tw, s));  // (clears layout_ok once it changes anything)
    AZ_TRY(alloc_scratch(h, s));
    h->layout_ok = true;
    return AZ_OK;
}

// After a failed set_tiles: back to the tiles there were.  The error text stays the failure's; if
// these do not fit any more either, the integrator stays without a layout.
void restore_tiles(az_integrator *h, int th, int tw, cudaStream_t s) {
    if (h->layout_ok) return;
    char text[sizeof(g_err)];
    memcpy(text, g_err, sizeof(text));
    cudaStreamSynchronize(s);
    (void)set_tiles(h, th, tw, s);
    memcpy(g_err, text, sizeof(text));
}

// Default tiles.
void default_tile(const az_integrator *h, int &th, int &tw) {
    // az_autotune refines them per matrix.  1D: 8 x 120, or 16 x 64 from 2.1 entries
    // per pixel on -- taller tiles make fewer, longer segments, which pays where the entries set
    // the time, wider rows make fewer pieces of a copy, which pays where the pixels do.  Frames
    // kernel, 8 x 120 against 16 x 64: 683 and 777 us (128 frames of 2527 x 2463 pixels, 1.7
    // entries per pixel), 273 and 244 us (37 frames of 2167 x 2070, 2.6), 45 and 40 us (24 variances
    // of 1043 x 981, 2.8).
    // 2D: 48 x 40 (500 x 360 bins of 2048 x 2048 pixels, 16 frames and one:
    // 91 and 29 us; 32 x 64, where only four frames fit a stage: 109 and 28 us; 24 x 56: 80 and 37).
    // Denser matrices get smaller tiles, so that the stages of the FP64 single-frame kernel (14
    // bytes an entry) still fit and no tile is cut: 962 x 972 pixels with 7.1 entries per pixel,
    // 16 x 40 against 16 x 64: FP64 frame 80 and 260 us, 16 frames 134 and 173 us; with 4.0 entries
    // 48 and 59, 92 and 89 us.
    const double density = (double)h->nnz / (double)std::max(h->n_unmasked, 1);
    th = 8; tw = 24;
    if (density < 20.0) { th = 16; tw = 24; }
    if (density < 10.0) { th = 16; tw = 40; }
    if (density < 5.0) { th = 16; tw = 64; }
    if (h->npt_azim == 0 && density < 2.1) { th = 8; tw = 120; }
    if (h->npt_azim > 0 && density < 2.4) { th = 48; tw = 40; }
}

// Whether 8 x 152 tiles may take the place of the default 8 x 120 (1D, below 1.75 entries per pixel,
// large detectors): a launch of few frames spends about 1.5 us an item, and has a fifth fewer of
// them.  2527 x 2463, full split: one to four frames against bound corrections 73 to 94 us on 8 x
// 120, 64 to 82 here, twenty 205 and 179, 64 380 and 383; an FP64 frame 144 and 139.  Nine matrices of
// 2.9 to 6.2 Mpixel with 1.0 to 1.89 entries per pixel: 8 to 20% for up to 20 frames, 1 to 10% for
// 48.  But the rings are sized for the heaviest tile: where four stages of the frames kernel or
// three of the FP64 single-frame kernel no longer fit, the narrow tiles are faster (2880 x 2880,
// bounding boxes, 1.55: 32 frames 321 and 511 us, an FP64 frame 134 and 185; 2540 x 1800, 1.90: an
// FP64 frame 119 and 173), which wide_tiles_fit says once they are built.  With fewer than twelve
// tiles per SM (1043 x 981) the two are equal within 5%.
int try_wide_tiles(az_integrator *h, cudaStream_t s, bool *kept) {
    *kept = false;
    const int64_t tiles = (int64_t)((h->ny + 7) / 8) * ((h->nx + 151) / 152);
    if (h->npt_azim > 0 || (double)h->nnz >= 1.75 * (double)std::max(h->n_unmasked, 1) || tiles < 12 * (int64_t)num_sms())
        return AZ_OK;
    // the heaviest tile's entries, 10 bytes each and a tenth of padding, twice beside four blocks of
    // planes: if that is too much, the layout is not built to find out
    int64_t most = 0;
    AZ_TRY(heaviest_tile(h, 8, 152, s, &most));
    if (2 * 11 * most + 4 * 16 * 8 * 320 > max_smem_per_block()) return AZ_OK;
    AZ_TRY(build_tiled_layout(h, 8, 152, s));
    *kept = wide_tiles_fit(h);
    return AZ_OK;
}

int finish_build(az_integrator *h, cudaStream_t s) {
    int th = 0, tw = 0;
    default_tile(h, th, tw);
    bool wide = false;
    if (try_wide_tiles(h, s, &wide) != AZ_OK) clear_error();
    if (wide) tw = 152;
    else if (build_tiled_layout(h, th, tw, s) != AZ_OK) {  // a denser matrix: smaller tiles
        clear_error();
        th = 8;
        tw = 64;
        AZ_TRY(build_tiled_layout(h, th, tw, s));
    }
    // The allocation-free entry point takes integrators whose FP64 partial sums fit its fixed
    // array, or whose FP32 ones do (twice the segments).  A matrix past either limit gets larger
    // tiles if they bring it below -- and if there is the memory for that: else its own stay.
    const int64_t most = (int64_t)AZ_NOALLOC_SCRATCH_BYTES / (3 * (int64_t)sizeof(double));
    if (h->tl.nseg > most) {
        const std::vector<std::pair<int, int>> larger =
            h->npt_azim > 0 ? std::vector<std::pair<int, int>>{{32, 64}}
                            : std::vector<std::pair<int, int>>{{16, 64}, {8, 224}};
        const int64_t nseg = h->tl.nseg;
        for (const auto &t : larger) {
            int64_t runs = 0;
            if (count_runs(h, t.first, t.second, s, &runs) != AZ_OK) break;
            if (runs <= most || (nseg > 2 * most && runs <= 2 * most)) {
                if (build_tiled_layout(h, t.first, t.second, s) != AZ_OK) AZ_TRY(build_tiled_layout(h, th, tw, s));
                break;
            }
        }
        clear_error();
    }
    h->frames_per_pass = 8;
    h->rows_per_warp = 32 / h->frames_per_pass;
    AZ_TRY(alloc_scratch(h, s));
    h->layout_ok = true;
    AZ_TRY(h->status.alloc(sizeof(int)));
    AZ_CUDA(cudaMemsetAsync(h->status.p, 0, sizeof(int), s));
    AZ_CUDA(cudaStreamSynchronize(s));
    // the allocation-free entry point's fixed array and kernels, loaded at set-up
    return noalloc_setup();
}

int check_build_args(int ny, int nx, int npt_rad, int npt_azim, int unit, int split) {
    if (ny < 1 || nx < 1) return fail(AZ_ESHAPE, "csr_build: ny, nx must be >= 1 (got %d, %d)", ny, nx);
    if ((int64_t)ny * nx >= INT32_MAX) return fail(AZ_ESHAPE, "csr_build: more than 2^31 - 1 pixels");
    if (npt_rad < 1) return fail(AZ_EINVAL, "csr_build: npt_rad must be >= 1");
    if (npt_azim < 0) return fail(AZ_EINVAL, "csr_build: npt_azim must be >= 0");
    if ((int64_t)npt_rad * std::max(npt_azim, 1) >= (1ll << 30))
        return fail(AZ_EINVAL, "csr_build: too many bins");
    if (unit < AZ_UNIT_2TH_DEG || unit > AZ_UNIT_R_MM) return fail(AZ_EINVAL, "csr_build: bad unit %d", unit);
    if (split < AZ_SPLIT_NONE || split > AZ_SPLIT_FULL) return fail(AZ_EINVAL, "csr_build: bad split %d", split);
    return AZ_OK;
}

int build_common(int ny, int nx, const double *rad, const double *chi, int npt_rad, int npt_azim,
                 int unit, int split, const uint8_t *mask, cudaStream_t s, az_integrator **out) {
    az_integrator *h = new (std::nothrow) az_integrator;
    if (!h) return fail(AZ_ENOMEM, "csr_build: out of host memory");
    cudaGetDevice(&h->device);
    int rc = build_integrator(ny, nx, rad, chi, npt_rad, npt_azim, unit, split, mask, s, h);
    if (rc == AZ_OK) rc = finish_build(h, s);
    if (rc != AZ_OK) {
        cudaStreamSynchronize(s);
        delete h;
        return rc;
    }
    *out = h;
    return AZ_OK;
}

}  // namespace

int check_layout(const az_integrator *h, const char *who) {
    if (h->layout_ok) return AZ_OK;
    return fail(AZ_EINVAL, "%s: the integrator has no tiled layout since a failed az_set_tuning or az_autotune: "
                           "call az_set_tuning again", who);
}

int check_forward(const az_integrator *h, const void *image, int dtype, const float *dark,
                  const float *flat, const float *sa, const float *pol, const char *who) {
    if (!h) return fail(AZ_EINVAL, "%s: NULL integrator", who);
    if (!image) return fail(AZ_EINVAL, "%s: NULL image", who);
    if (dtype < AZ_DTYPE_F32 || dtype > AZ_DTYPE_I32) return fail(AZ_EINVAL, "%s: bad image dtype %d", who, dtype);
    const void *ptrs[5] = {image, dark, flat, sa, pol};
    for (const void *p : ptrs)
        if (p && !aligned4(p)) return fail(AZ_EINVAL, "%s: arrays must be 4-byte aligned", who);
    return AZ_OK;
}

int fail(int code, const char *fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
    return code;
}

void clear_error() { g_err[0] = 0; }

int multi_create(az_integrator *const *hs, int n, const void *const *images, int dtype,
                 const float *const *darks, const float *const *flats, const float *const *sas,
                 const float *const *pols, float *const *oI, float *const *oS, float *const *oN,
                 float *const *oC, void **out);
int multi_launch(void *plan, int use_graph, cudaStream_t s);
void multi_destroy(void *plan);

}  // namespace azint

using namespace azint;

struct az_multi {
    void *plan = nullptr;
};

extern "C" const char *az_last_error(void) { return g_err; }

extern "C" int az_csr_build(const az_geometry *geom, int ny, int nx, int npt_rad, int npt_azim,
                            int unit, int split, const uint8_t *mask_dev, az_stream_t stream,
                            az_integrator **out) {
    clear_error();
    if (!geom || !out) return fail(AZ_EINVAL, "az_csr_build: NULL argument");
    *out = nullptr;
    AZ_TRY(check_build_args(ny, nx, npt_rad, npt_azim, unit, split));
    cudaStream_t s = (cudaStream_t)stream;
    const bool corners = split != AZ_SPLIT_NONE;
    const bool need_chi = npt_azim > 0 || split == AZ_SPLIT_FULL;
    const int64_t npos = corners ? (int64_t)(ny + 1) * (nx + 1) : (int64_t)ny * nx;
    // scratch of the whole build; at first positions, bin coordinates, counts and their sums
    ScratchScope scope;
    ScratchScope::reserve((size_t)npos * 8 * (need_chi ? 3 : 2) + (size_t)ny * nx * 16 + ((size_t)2 << 20));
    TmpBuf rad, chi;
    AZ_TRY(rad.alloc(sizeof(double) * npos));
    if (need_chi) AZ_TRY(chi.alloc(sizeof(double) * npos));
    AZ_TRY(launch_positions(geom->g, ny, nx, unit, corners ? AZ_WHERE_CORNERS : AZ_WHERE_CENTRES,
                            rad.as<double>(), need_chi ? chi.as<double>() : nullptr, s));
    const int rc = build_common(ny, nx, rad.as<double>(), need_chi ? chi.as<double>() : nullptr,
                                npt_rad, npt_azim, unit, split, mask_dev, s, out);
    cudaStreamSynchronize(s);
    return rc;
}

extern "C" int az_csr_build_from_positions(int ny, int nx, const double *rad_dev,
                                           const double *chi_dev, int npt_rad, int npt_azim,
                                           int split, const uint8_t *mask_dev,
                                           az_stream_t stream, az_integrator **out) {
    clear_error();
    if (!rad_dev || !out) return fail(AZ_EINVAL, "az_csr_build_from_positions: NULL argument");
    *out = nullptr;
    AZ_TRY(check_build_args(ny, nx, npt_rad, npt_azim, AZ_UNIT_2TH_DEG, split));
    if ((npt_azim > 0 || split == AZ_SPLIT_FULL) && !chi_dev)
        return fail(AZ_EINVAL, "az_csr_build_from_positions: chi positions are required");
    return build_common(ny, nx, rad_dev, (npt_azim > 0 || split == AZ_SPLIT_FULL) ? chi_dev : nullptr,
                        npt_rad, npt_azim, -1, split, mask_dev, (cudaStream_t)stream, out);
}

extern "C" int az_csr_import(int ny, int nx, int npt_rad, int npt_azim, int unit, int split,
                             const int32_t *indptr_host, const int32_t *indices_host,
                             const double *data_host, double lo, double hi, az_stream_t stream,
                             az_integrator **out) {
    clear_error();
    const char *who = "az_csr_import";
    if (!out || !indptr_host) return fail(AZ_EINVAL, "%s: NULL argument", who);
    *out = nullptr;
    AZ_TRY(check_build_args(ny, nx, npt_rad, npt_azim, unit, split));
    if (!(std::isfinite(lo) && std::isfinite(hi) && lo < hi))
        return fail(AZ_EINVAL, "%s: the radial range [%g, %g] must be finite with lo < hi", who, lo, hi);
    // the whole matrix is checked on the host before any device work
    const int nrows = npt_azim > 0 ? npt_rad * npt_azim : npt_rad;
    const int64_t npix = (int64_t)ny * nx;
    if (indptr_host[0] != 0) return fail(AZ_EINVAL, "%s: indptr[0] must be 0", who);
    for (int r = 0; r < nrows; ++r)
        if (indptr_host[r + 1] < indptr_host[r])
            return fail(AZ_EINVAL, "%s: indptr decreases at row %d", who, r);
    const int64_t nnz = indptr_host[nrows];
    if (nnz == 0) return fail(AZ_ERANGE, "%s: the matrix has no entries", who);
    if (!indices_host || !data_host) return fail(AZ_EINVAL, "%s: NULL indices or data", who);
    for (int r = 0; r < nrows; ++r)
        for (int32_t k = indptr_host[r]; k < indptr_host[r + 1]; ++k) {
            const int32_t p = indices_host[k];
            if (p < 0 || p >= npix)
                return fail(AZ_EINVAL, "%s: entry %d of row %d has pixel %d outside [0, %lld)", who, (int)k, r,
                            (int)p, (long long)npix);
            if (k > indptr_host[r] && p <= indices_host[k - 1])
                return fail(AZ_EINVAL, "%s: the pixels of row %d are not strictly ascending", who, r);
            if (!std::isfinite(data_host[k]))
                return fail(AZ_EINVAL, "%s: entry %d has a non-finite weight", who, (int)k);
        }
    cudaStream_t s = (cudaStream_t)stream;
    az_integrator *h = new (std::nothrow) az_integrator;
    if (!h) return fail(AZ_ENOMEM, "%s: out of host memory", who);
    cudaGetDevice(&h->device);
    h->ny = ny; h->nx = nx; h->npt_rad = npt_rad; h->npt_azim = npt_azim; h->nrows = nrows;
    h->unit = unit; h->split = split; h->nnz = nnz;
    h->lo = lo; h->hi = hi; h->delta = (hi - lo) / npt_rad;
    int rc = import_csr(h, indptr_host, indices_host, data_host, s);
    if (rc == AZ_OK) rc = finish_build(h, s);
    if (rc != AZ_OK) {
        cudaStreamSynchronize(s);
        delete h;
        return rc;
    }
    *out = h;
    return AZ_OK;
}

extern "C" int az_integrator_info(const az_integrator *h, az_info *out) {
    clear_error();
    if (!h || !out) return fail(AZ_EINVAL, "az_integrator_info: NULL argument");
    memset(out, 0, sizeof(*out));
    out->ny = h->ny; out->nx = h->nx; out->npt_rad = h->npt_rad; out->npt_azim = h->npt_azim;
    out->nrows = h->nrows; out->unit = h->unit; out->split = h->split;
    out->n_unmasked = h->n_unmasked; out->nnz = h->nnz;
    out->lo = h->lo; out->hi = h->hi; out->delta = h->delta;
    out->tile_h = h->tl.th; out->tile_w = h->tl.tw;
    out->rows_per_warp = h->rows_per_warp; out->frames_per_pass = h->frames_per_pass;
    out->n_tiles = h->tl.ntiles; out->n_segments = h->tl.nseg;
    out->copy_engine = h->copy_engine;
    out->n_items = h->tl.n_active;
    out->layout = h->layout;
    out->lut_width = h->lut_width;
    const DevBuf *bufs[] = {&h->csr_ptr, &h->csr_idx, &h->csr_w64, &h->csc_ptr, &h->csc_row,
                            &h->csc_w64, &h->csc_w32, &h->tl.tile_seg_ptr, &h->tl.tile_ent_ptr,
                            &h->tl.active_tiles, &h->tl.seg_ent_ptr, &h->tl.seg_slot,
                            &h->tl.row_slot_ptr, &h->tl.ent_loc, &h->tl.f_desc, &h->tl.f_rec, &h->tl.f_loc, &h->tl.f_w32, &h->tl.f_pix, &h->tl.f_loc1, &h->tl.f_w64, &h->count64, &h->tl.ent_w32, &h->tl.ent_w64,
                            &h->partial, &h->norm, &h->adj, &h->status, &h->host_stage,
                            &h->tl.tile_desc, &h->tl.tile_rec, &h->tl.ent_pix, &h->tl.ent_dark,
                            &h->tl.norm_frames, &h->tl.ent_wnorm, &h->lut32, &h->lut64,
                            &h->lut_vals, &h->lut_part, &h->one_planes, &h->bound_dark[0], &h->bound_dark[1],
                            &h->bound_norm};
    int64_t tot = 0;
    for (const DevBuf *b : bufs) tot += (int64_t)b->bytes;
    out->device_bytes = tot;
    return AZ_OK;
}

extern "C" int az_csr_export(const az_integrator *h, int32_t *indptr_host, int32_t *indices_host,
                             double *data_host) {
    clear_error();
    if (!h) return fail(AZ_EINVAL, "az_csr_export: NULL integrator");
    if (indptr_host)
        AZ_CUDA(cudaMemcpy(indptr_host, h->csr_ptr.p, sizeof(int32_t) * (h->nrows + 1), cudaMemcpyDeviceToHost));
    if (indices_host)
        AZ_CUDA(cudaMemcpy(indices_host, h->csr_idx.p, sizeof(int32_t) * h->nnz, cudaMemcpyDeviceToHost));
    if (data_host)
        AZ_CUDA(cudaMemcpy(data_host, h->csr_w64.p, sizeof(double) * h->nnz, cudaMemcpyDeviceToHost));
    return AZ_OK;
}

extern "C" int az_radial_axis(const az_integrator *h, double *out_host) {
    clear_error();
    if (!h || !out_host) return fail(AZ_EINVAL, "az_radial_axis: NULL argument");
    for (int k = 0; k < h->npt_rad; ++k) out_host[k] = h->lo + ((double)k + 0.5) * h->delta;
    return AZ_OK;
}

extern "C" int az_integrator_status(az_integrator *h) {
    clear_error();
    if (!h) return fail(AZ_EINVAL, "az_integrator_status: NULL integrator");
    AZ_CUDA(cudaStreamSynchronize(h->last_stream));
    int st = 0;
    AZ_CUDA(cudaMemcpy(&st, h->status.p, sizeof(int), cudaMemcpyDeviceToHost));
    AZ_CUDA(cudaMemset(h->status.p, 0, sizeof(int)));
    if (st != AZ_OK) return fail(st, "a bounded device-side wait gave up");
    return AZ_OK;
}

extern "C" void az_integrator_destroy(az_integrator *h) {
    if (!h) return;
    cudaDeviceSynchronize();
    if (h->copy_stream) cudaStreamDestroy(h->copy_stream);
    for (cudaEvent_t e : h->copy_events)
        if (e) cudaEventDestroy(e);
    delete h;
}

static int integrate_common(const az_integrator *h, const void *image, int dtype, const float *dark,
                            const float *flat, const float *sa, const float *pol, int precision,
                            void *oI, void *oS, void *oN, void *oC, az_stream_t stream, bool two_d,
                            const char *who) {
    clear_error();
    AZ_TRY(check_forward(h, image, dtype, dark, flat, sa, pol, who));
    if (precision != AZ_PREC_FP64 && precision != AZ_PREC_FP32_COMP)
        return fail(AZ_EINVAL, "%s: bad precision %d", who, precision);
    if (two_d && h->npt_azim == 0) return fail(AZ_ESHAPE, "%s: integrator is 1D", who);
    if (!two_d && h->npt_azim != 0) return fail(AZ_ESHAPE, "%s: integrator is 2D", who);
    const_cast<az_integrator *>(h)->last_stream = (cudaStream_t)stream;
    if (h->layout == AZ_LAYOUT_LUT)
        return lut_forward(h, image, dtype, dark, flat, sa, pol, precision, oI, oS, oN, oC, (cudaStream_t)stream);
    AZ_TRY(check_layout(h, who));
    return forward_single(h, image, dtype, dark, flat, sa, pol, precision, oI, oS, oN, oC,
                          (cudaStream_t)stream);
}

extern "C" int az_integrate1d(const az_integrator *h, const void *image_dev, int image_dtype,
                              const float *dark, const float *flat, const float *solid_angle,
                              const float *polarization, int precision, void *out_I,
                              void *out_sum_signal, void *out_sum_norm, void *out_count,
                              az_stream_t stream) {
    return integrate_common(h, image_dev, image_dtype, dark, flat, solid_angle, polarization,
                            precision, out_I, out_sum_signal, out_sum_norm, out_count, stream,
                            false, "az_integrate1d");
}

extern "C" int az_integrate2d(const az_integrator *h, const void *image_dev, int image_dtype,
                              const float *dark, const float *flat, const float *solid_angle,
                              const float *polarization, int precision, void *out_I,
                              void *out_sum_signal, void *out_sum_norm, void *out_count,
                              az_stream_t stream) {
    return integrate_common(h, image_dev, image_dtype, dark, flat, solid_angle, polarization,
                            precision, out_I, out_sum_signal, out_sum_norm, out_count, stream,
                            true, "az_integrate2d");
}

extern "C" int az_integrate_batch(az_integrator *h, const void *frames_dev, int n_frames,
                                  int image_dtype, const float *dark, const float *flat,
                                  const float *solid_angle, const float *polarization,
                                  float *out_I, float *out_sum_signal, float *out_sum_norm,
                                  float *out_count, az_stream_t stream) {
    clear_error();
    if (n_frames < 0) return fail(AZ_ESHAPE, "az_integrate_batch: n_frames < 0");
    // with no frames only N and C are formed: the frames pointer may be NULL
    static const uint32_t no_frames = 0;
    AZ_TRY(check_forward(h, n_frames == 0 ? &no_frames : frames_dev, image_dtype, dark, flat,
                         solid_angle, polarization, "az_integrate_batch"));
    AZ_TRY(check_layout(h, "az_integrate_batch"));
    h->last_stream = (cudaStream_t)stream;
    if (n_frames == 0 && !out_sum_norm && !out_count) return AZ_OK;
    return forward_batch(h, frames_dev, n_frames, image_dtype, dark, flat, solid_angle,
                         polarization, out_I, out_sum_signal, out_sum_norm, out_count,
                         (cudaStream_t)stream);
}

extern "C" int az_set_corrections(az_integrator *h, const float *dark, const float *flat,
                                  const float *solid_angle, const float *polarization,
                                  az_stream_t stream) {
    clear_error();
    static const uint32_t no_frames = 0;
    AZ_TRY(check_forward(h, &no_frames, AZ_DTYPE_F32, dark, flat, solid_angle, polarization,
                         "az_set_corrections"));
    AZ_TRY(check_layout(h, "az_set_corrections"));
    h->last_stream = (cudaStream_t)stream;
    return bind_corrections(h, dark, flat, solid_angle, polarization, (cudaStream_t)stream);
}

extern "C" int az_integrate_batch_bound(az_integrator *h, const void *frames_dev, int n_frames,
                                        int image_dtype, float *out_I, float *out_sum_signal,
                                        float *out_sum_norm, float *out_count, az_stream_t stream) {
    clear_error();
    if (n_frames < 0) return fail(AZ_ESHAPE, "az_integrate_batch_bound: n_frames < 0");
    static const uint32_t no_frames = 0;
    AZ_TRY(check_forward(h, n_frames == 0 ? &no_frames : frames_dev, image_dtype, nullptr, nullptr,
                         nullptr, nullptr, "az_integrate_batch_bound"));
    AZ_TRY(check_layout(h, "az_integrate_batch_bound"));
    h->last_stream = (cudaStream_t)stream;
    return forward_batch_bound(h, frames_dev, n_frames, image_dtype, out_I, out_sum_signal, out_sum_norm,
                               out_count, (cudaStream_t)stream);
}

extern "C" int az_integrate_batch_pixelnorm(az_integrator *h, const void *frames_dev, int n_frames,
                                            int image_dtype, const float *dark, const float *flat,
                                            const float *solid_angle, const float *polarization,
                                            float *out_I, float *out_sum_corrected, float *out_count,
                                            az_stream_t stream) {
    clear_error();
    if (n_frames < 0) return fail(AZ_ESHAPE, "az_integrate_batch_pixelnorm: n_frames < 0");
    static const uint32_t no_frames = 0;
    AZ_TRY(check_forward(h, n_frames == 0 ? &no_frames : frames_dev, image_dtype, dark, flat,
                         solid_angle, polarization, "az_integrate_batch_pixelnorm"));
    AZ_TRY(check_layout(h, "az_integrate_batch_pixelnorm"));
    h->last_stream = (cudaStream_t)stream;
    return batch_pixelnorm(h, frames_dev, n_frames, image_dtype, dark, flat, solid_angle, polarization,
                           out_I, out_sum_corrected, out_count, (cudaStream_t)stream);
}

extern "C" int az_integrate_variance(az_integrator *h, const void *frames_dev, int n_frames,
                                     int image_dtype, float *out_sum_variance, az_stream_t stream) {
    clear_error();
    if (n_frames < 0) return fail(AZ_ESHAPE, "az_integrate_variance: n_frames < 0");
    if (n_frames == 0) return AZ_OK;
    AZ_TRY(check_forward(h, frames_dev, image_dtype, nullptr, nullptr, nullptr, nullptr,
                         "az_integrate_variance"));
    if (!out_sum_variance) return fail(AZ_EINVAL, "az_integrate_variance: NULL output");
    AZ_TRY(check_layout(h, "az_integrate_variance"));
    h->last_stream = (cudaStream_t)stream;
    return batch_variance(h, frames_dev, n_frames, image_dtype, out_sum_variance, (cudaStream_t)stream);
}

extern "C" int az_integrate_batch_host(az_integrator *h, const void *frames_host, int n_frames,
                                       int image_dtype, const float *dark, const float *flat,
                                       const float *solid_angle, const float *polarization,
                                       float *out_I_host, float *out_sum_signal_host,
                                       az_stream_t stream) {
    clear_error();
    AZ_TRY(check_forward(h, frames_host, image_dtype, dark, flat, solid_angle, polarization,
                         "az_integrate_batch_host"));
    if (n_frames < 0) return fail(AZ_ESHAPE, "az_integrate_batch_host: n_frames < 0");
    if (n_frames == 0) return AZ_OK;
    AZ_TRY(check_layout(h, "az_integrate_batch_host"));
    cudaStream_t s = (cudaStream_t)stream;
    const size_t fbytes = (size_t)h->ny * h->nx * 4u;
    const size_t obytes = (size_t)h->nrows * sizeof(float);
    const int chunk = std::max(1, std::min(16, n_frames));
    // two device buffers of `chunk` frames and their outputs
    const size_t per = chunk * (fbytes + 2 * obytes);
    if (h->host_stage.bytes < 2 * per) AZ_TRY(h->host_stage.alloc(2 * per));
    char *base = h->host_stage.as<char>();
    char *fr[2] = {base, base + per};
    float *oi[2], *os[2];
    for (int b = 0; b < 2; ++b) {
        oi[b] = reinterpret_cast<float *>(fr[b] + chunk * fbytes);
        os[b] = oi[b] + (size_t)chunk * h->nrows;
    }
    int rc = AZ_OK;
    auto ck = [&](cudaError_t e) {
        if (e != cudaSuccess && rc == AZ_OK) rc = fail(AZ_ECUDA, "az_integrate_batch_host: %s", cudaGetErrorString(e));
    };
    // the upload stream and its events live with the integrator (created once)
    if (!h->copy_stream) ck(cudaStreamCreateWithFlags(&h->copy_stream, cudaStreamNonBlocking));
    for (cudaEvent_t &e : h->copy_events)
        if (!e) ck(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    if (rc != AZ_OK) return rc;
    cudaStream_t cp = h->copy_stream;
    cudaEvent_t start = h->copy_events[0];
    cudaEvent_t up[2] = {h->copy_events[1], h->copy_events[2]};
    cudaEvent_t done[2] = {h->copy_events[3], h->copy_events[4]};
    if (rc == AZ_OK) {
        ck(cudaEventRecord(start, s));
        ck(cudaStreamWaitEvent(cp, start, 0));
        rc = batch_norm(h, flat, solid_angle, polarization, nullptr, nullptr, s);
    }
    const int nchunks = (n_frames + chunk - 1) / chunk;
    // upload chunk 0 (and 1) ahead, then: compute k on `s` while `cp` uploads k+1
    auto upload = [&](int k) {
        const int b = k & 1, f0 = k * chunk, nf = std::min(chunk, n_frames - f0);
        ck(cudaMemcpyAsync(fr[b], static_cast<const char *>(frames_host) + (size_t)f0 * fbytes,
                           (size_t)nf * fbytes, cudaMemcpyHostToDevice, cp));
        ck(cudaEventRecord(up[b], cp));
    };
    if (rc == AZ_OK) upload(0);
    for (int k = 0; k < nchunks && rc == AZ_OK; ++k) {
        const int b = k & 1, f0 = k * chunk, nf = std::min(chunk, n_frames - f0);
        if (k + 1 < nchunks) {
            if (k >= 1) ck(cudaStreamWaitEvent(cp, done[(k + 1) & 1], 0));  // buffer free again
            upload(k + 1);
        }
        ck(cudaStreamWaitEvent(s, up[b], 0));
        if (rc == AZ_OK) rc = batch_frames(h, fr[b], nf, image_dtype, dark, oi[b], os[b], 0, s);
        if (out_I_host)
            ck(cudaMemcpyAsync(out_I_host + (size_t)f0 * h->nrows, oi[b], (size_t)nf * obytes,
                               cudaMemcpyDeviceToHost, s));
        if (out_sum_signal_host)
            ck(cudaMemcpyAsync(out_sum_signal_host + (size_t)f0 * h->nrows, os[b], (size_t)nf * obytes,
                               cudaMemcpyDeviceToHost, s));
        ck(cudaEventRecord(done[b], s));
    }
    ck(cudaStreamSynchronize(s));
    ck(cudaStreamSynchronize(cp));
    h->last_stream = s;
    return rc;
}

extern "C" int az_integrate_backward(const az_integrator *h, const void *grad_I, const void *I,
                                     const void *sum_norm, const float *solid_angle,
                                     const float *polarization, int precision,
                                     void *out_grad_image, void *out_grad_flat,
                                     az_stream_t stream) {
    clear_error();
    if (!h || !grad_I || !I || !sum_norm) return fail(AZ_EINVAL, "az_integrate_backward: NULL argument");
    if (precision != AZ_PREC_FP64 && precision != AZ_PREC_FP32_COMP)
        return fail(AZ_EINVAL, "az_integrate_backward: bad precision %d", precision);
    if (!out_grad_image && !out_grad_flat) return AZ_OK;
    AZ_TRY(check_layout(h, "az_integrate_backward"));  // (its scratch)
    const_cast<az_integrator *>(h)->last_stream = (cudaStream_t)stream;
    return backward(h, grad_I, I, sum_norm, solid_angle, polarization, precision, out_grad_image,
                    out_grad_flat, (cudaStream_t)stream);
}

extern "C" int az_multi_create(az_integrator *const *handles, int n, const void *const *images,
                               int image_dtype, const float *const *darks,
                               const float *const *flats, const float *const *solid_angles,
                               const float *const *polarizations, float *const *out_I,
                               float *const *out_sum_signal, float *const *out_sum_norm,
                               float *const *out_count, az_multi **out) {
    clear_error();
    if (!handles || !images || !out || n < 1) return fail(AZ_EINVAL, "az_multi_create: bad arguments");
    *out = nullptr;
    if (image_dtype < AZ_DTYPE_F32 || image_dtype > AZ_DTYPE_I32)
        return fail(AZ_EINVAL, "az_multi_create: bad image dtype %d", image_dtype);
    for (int k = 0; k < n; ++k) {
        if (!handles[k] || !images[k]) return fail(AZ_EINVAL, "az_multi_create: NULL handle or image %d", k);
        AZ_TRY(check_forward(handles[k], images[k], image_dtype, darks ? darks[k] : nullptr,
                             flats ? flats[k] : nullptr, solid_angles ? solid_angles[k] : nullptr,
                             polarizations ? polarizations[k] : nullptr, "az_multi_create"));
        AZ_TRY(check_layout(handles[k], "az_multi_create"));
    }
    az_multi *m = new (std::nothrow) az_multi;
    if (!m) return fail(AZ_ENOMEM, "az_multi_create: out of host memory");
    int rc = multi_create(handles, n, images, image_dtype, darks, flats, solid_angles, polarizations,
                          out_I, out_sum_signal, out_sum_norm, out_count, &m->plan);
    if (rc != AZ_OK) {
        delete m;
        return rc;
    }
    *out = m;
    return AZ_OK;
}

extern "C" int az_multi_launch(az_multi *plan, int use_graph, az_stream_t stream) {
    clear_error();
    if (!plan || !plan->plan) return fail(AZ_EINVAL, "az_multi_launch: NULL plan");
    return multi_launch(plan->plan, use_graph, (cudaStream_t)stream);
}

extern "C" void az_multi_destroy(az_multi *plan) {
    if (!plan) return;
    cudaDeviceSynchronize();
    multi_destroy(plan->plan);
    delete plan;
}

extern "C" int az_profile_enable(az_integrator *h, int enable) {
    clear_error();
    if (!h) return fail(AZ_EINVAL, "az_profile_enable: NULL integrator");
    h->prof.on = enable != 0;
    return AZ_OK;
}

extern "C" int az_profile_read(az_integrator *h, az_profile *out) {
    clear_error();
    if (!h || !out) return fail(AZ_EINVAL, "az_profile_read: NULL argument");
    memset(out, 0, sizeof(*out));
    int rc = AZ_OK;
    for (auto &r : h->prof.recs) {
        float ms = 0.f;
        cudaError_t e = cudaEventSynchronize(r.b);
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, r.a, r.b);
        if (e != cudaSuccess && rc == AZ_OK) rc = fail(AZ_ECUDA, "az_profile_read: %s", cudaGetErrorString(e));
        if (r.kind >= 0 && r.kind < AZ_PROF_KINDS) {
            out->launches[r.kind] += 1;
            out->total_ms[r.kind] += ms;
        }
        h->prof.pool.push_back(r.a);
        h->prof.pool.push_back(r.b);
    }
    h->prof.recs.clear();
    return rc;
}

extern "C" int az_set_copy_engine(az_integrator *h, int engine) {
    clear_error();
    if (!h) return fail(AZ_EINVAL, "az_set_copy_engine: NULL integrator");
    if (engine != AZ_COPY_TMA && engine != AZ_COPY_ASYNC)
        return fail(AZ_EINVAL, "az_set_copy_engine: bad engine %d", engine);
    const int before = h->copy_engine;
    h->copy_engine = engine;
    const int rc = convert_bound_darks(h);
    if (rc != AZ_OK) h->copy_engine = before;
    return rc;
}

extern "C" int az_set_tuning(az_integrator *h, int tile_h, int tile_w, int rows_per_warp,
                             int frames_per_pass) {
    clear_error();
    if (!h) return fail(AZ_EINVAL, "az_set_tuning: NULL integrator");
    if (tile_h < 0 || tile_w < 0 || (tile_w % 4) != 0)
        return fail(AZ_EINVAL, "az_set_tuning: tile_w must be a multiple of 4");
    auto pow2_upto32 = [](int v) { return v == 1 || v == 2 || v == 4 || v == 8 || v == 16 || v == 32; };
    if (rows_per_warp && !pow2_upto32(rows_per_warp))
        return fail(AZ_EINVAL, "az_set_tuning: rows_per_warp must be 1, 2, 4, 8, 16 or 32");
    if (frames_per_pass && !pow2_upto32(frames_per_pass))
        return fail(AZ_EINVAL, "az_set_tuning: frames_per_pass must be 1, 2, 4, 8, 16 or 32");
    if (rows_per_warp && frames_per_pass && rows_per_warp * frames_per_pass != 32)
        return fail(AZ_EINVAL, "az_set_tuning: rows_per_warp * frames_per_pass must be 32");
    const int th = tile_h ? tile_h : h->tl.th, tw = tile_w ? tile_w : h->tl.tw;
    if (th != h->tl.th || tw != h->tl.tw || !h->layout_ok) {
        if ((int64_t)th * (tw + 8) > 65535 || th < 1 || tw < 4)
            return fail(AZ_EINVAL, "az_set_tuning: tile %dx%d out of range", th, tw);
        const int th0 = h->tl.th, tw0 = h->tl.tw;
        cudaDeviceSynchronize();
        const int rc = set_tiles(h, th, tw, nullptr);
        if (rc != AZ_OK) {
            restore_tiles(h, th0, tw0, nullptr);
            cudaDeviceSynchronize();
            return rc;
        }
        AZ_CUDA(cudaDeviceSynchronize());
    }
    if (rows_per_warp) h->frames_per_pass = 32 / rows_per_warp;
    if (frames_per_pass) h->frames_per_pass = frames_per_pass;
    h->rows_per_warp = 32 / h->frames_per_pass;
    return AZ_OK;
}

// One FP32 frame through the tiled form and through the look-up table; the faster becomes
// the single-frame layout.  The table is built for the trial if missing and small enough
// (at most four times the bytes of the matrix's entries), and freed again if it loses.
static int tune_layout(az_integrator *h, const void *frame, const float *dark, cudaStream_t s) {
    const bool had_table = h->lut32.p != nullptr;
    if (!had_table) {
        int64_t wmax = 0;
        {
            std::vector<int32_t> ptr((size_t)h->nrows + 1);
            AZ_CUDA(cudaMemcpy(ptr.data(), h->csr_ptr.p, sizeof(int32_t) * ptr.size(), cudaMemcpyDeviceToHost));
            for (int b = 0; b < h->nrows; ++b) wmax = std::max<int64_t>(wmax, ptr[b + 1] - ptr[b]);
        }
        if (wmax * h->nrows > 4 * std::max<int64_t>(h->nnz, 1)) return AZ_OK;  // the tiled form stays
        if (lut_build(h, AZ_PREC_FP32_COMP, s) != AZ_OK) {
            clear_error();
            return AZ_OK;
        }
    }
    DevBuf out;
    AZ_TRY(out.alloc(sizeof(float) * 4 * (size_t)h->nrows));
    float *o = out.as<float>();
    const int rows = h->nrows;
    cudaEvent_t e0, e1;
    AZ_CUDA(cudaEventCreate(&e0));
    AZ_CUDA(cudaEventCreate(&e1));
    double t[2] = {1e30, 1e30};
    for (int lay = 0; lay < 2; ++lay) {
        h->layout = lay;
        for (int rep = 0; rep < 4; ++rep) {
            cudaEventRecord(e0, s);
            int rc;
            if (lay == AZ_LAYOUT_LUT) {
                rc = lut_forward(h, frame, AZ_DTYPE_U32, dark, nullptr, nullptr, nullptr, AZ_PREC_FP32_COMP, o,
                                 o + rows, o + 2 * rows, o + 3 * rows, s);
            } else {
                // what az_integrate1d/2d run in FP32 with the tiled form
                rc = forward_single(h, frame, AZ_DTYPE_U32, dark, nullptr, nullptr, nullptr, AZ_PREC_FP32_COMP, o,
                                    o + rows, o + 2 * rows, o + 3 * rows, s);
            }
            cudaEventRecord(e1, s);
            cudaEventSynchronize(e1);
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            if (rc != AZ_OK) {
                clear_error();
                break;
            }
            if (rep > 0) t[lay] = std::min<double>(t[lay], ms);
        }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    h->layout = t[AZ_LAYOUT_LUT] < t[AZ_LAYOUT_TILED] ? AZ_LAYOUT_LUT : AZ_LAYOUT_TILED;
    if (h->layout == AZ_LAYOUT_TILED && !had_table) {
        h->lut32.release();
        if (!h->lut64.p) {
            h->lut_vals.release();
            h->lut_part.release();
            h->lut_width = 0;
        }
    }
    return AZ_OK;
}

// The tiles az_autotune times: the integrator's own first, the default of its matrix, and others:
// small ones where the entries are many (16 x 40 with 7.1 entries per pixel: a batch of 16 frames 121
// us, 16 x 64 173; an FP64 frame 77 and 260).
static std::vector<std::pair<int, int>> trial_tiles(const az_integrator *h) {
    std::vector<std::pair<int, int>> out{{h->tl.th, h->tl.tw}};
    int th = 0, tw = 0;
    default_tile(h, th, tw);
    out.emplace_back(th, tw);
    for (const auto &t : {std::pair<int, int>{8, 120}, {16, 64}, {16, 96}, {16, 56}, {32, 64}}) out.push_back(t);
    if ((double)h->nnz < 4.0 * (double)std::max(h->n_unmasked, 1))
        for (const auto &t : {std::pair<int, int>{8, 224}, {8, 152}, {48, 40}, {24, 56}}) out.push_back(t);
    else
        for (const auto &t : {std::pair<int, int>{8, 64}, {16, 40}, {16, 24}, {8, 24}}) out.push_back(t);
    for (size_t k = 0; k < out.size(); ++k)
        out.erase(std::remove(out.begin() + k + 1, out.end(), out[k]), out.end());
    return out;
}

extern "C" int az_autotune_tiles(const az_integrator *h, int32_t *tiles, int capacity, int *n_tiles) {
    clear_error();
    if (!h || !n_tiles || capacity < 0 || (capacity > 0 && !tiles)) return fail(AZ_EINVAL, "az_autotune_tiles: bad argument");
    const auto t = trial_tiles(h);
    *n_tiles = (int)t.size();
    for (int k = 0; k < std::min(capacity, *n_tiles); ++k) {
        tiles[2 * k] = t[(size_t)k].first;
        tiles[2 * k + 1] = t[(size_t)k].second;
    }
    return AZ_OK;
}

extern "C" int az_autotune(az_integrator *h, int n_trial_frames, az_stream_t stream,
                           double *best_ms) {
    clear_error();
    if (!h) return fail(AZ_EINVAL, "az_autotune: NULL integrator");
    if (n_trial_frames < 1) return fail(AZ_EINVAL, "az_autotune: n_trial_frames must be >= 1");
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t npix = (int64_t)h->ny * h->nx;
    DevBuf frames, outI, outS, dark;
    AZ_TRY(frames.alloc(sizeof(uint32_t) * npix * n_trial_frames));
    AZ_TRY(outI.alloc(sizeof(float) * (size_t)h->nrows * n_trial_frames));
    AZ_TRY(outS.alloc(sizeof(float) * (size_t)h->nrows * n_trial_frames));
    AZ_TRY(dark.alloc(sizeof(float) * npix));
    AZ_CUDA(cudaMemsetAsync(dark.p, 0, sizeof(float) * npix, s));
    fill_frames_kernel<<<num_sms() * 8, 256, 0, s>>>(frames.as<uint32_t>(), npix * n_trial_frames, 12345u);
    AZ_CUDA(cudaGetLastError());
    const int th0 = h->tl.th, tw0 = h->tl.tw, fpp0 = h->frames_per_pass, engine0 = h->copy_engine;
    cudaEvent_t e0, e1;
    AZ_CUDA(cudaEventCreate(&e0));
    AZ_CUDA(cudaEventCreate(&e1));
    const auto tiles = trial_tiles(h);
    const int fpps[] = {4, 8, 16};
    const int engines[] = {AZ_COPY_TMA, AZ_COPY_ASYNC};
    double best = 1e30;
    int bt = -1, bf = h->frames_per_pass, be = h->copy_engine;
    for (int ti = 0; ti < (int)tiles.size(); ++ti) {
        if (set_tiles(h, tiles[(size_t)ti].first, tiles[(size_t)ti].second, s) != AZ_OK ||
            batch_norm(h, nullptr, nullptr, nullptr, nullptr, nullptr, s) != AZ_OK) {
            clear_error();
            continue;
        }
        for (int eg : engines)
            for (int f : fpps) {
                if (eg == AZ_COPY_TMA && f > 8) continue;  // the frames kernel takes eight at most
                h->frames_per_pass = f;
                h->copy_engine = eg;
                float best_t = 1e30f;
                bool ok = true;
                for (int rep = 0; rep < 3 && ok; ++rep) {
                    cudaEventRecord(e0, s);
                    ok = batch_frames(h, frames.p, n_trial_frames, AZ_DTYPE_U32, dark.as<float>(),
                                      outI.as<float>(), outS.as<float>(), 0, s) == AZ_OK;
                    cudaEventRecord(e1, s);
                    cudaEventSynchronize(e1);
                    float ms = 0.f;
                    cudaEventElapsedTime(&ms, e0, e1);
                    if (rep > 0) best_t = std::min(best_t, ms);
                }
                clear_error();
                if (ok && best_t < best) {
                    best = best_t;
                    bt = ti; bf = f; be = eg;
                }
            }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    const int rc = bt < 0 ? fail(AZ_EUNSUPPORTED, "az_autotune: no configuration ran")
                          : set_tiles(h, tiles[(size_t)bt].first, tiles[(size_t)bt].second, s);
    if (rc != AZ_OK) {  // as it was
        h->frames_per_pass = fpp0;
        h->copy_engine = engine0;
        if (h->tl.th != th0 || h->tl.tw != tw0) h->layout_ok = false;
        restore_tiles(h, th0, tw0, s);
        cudaStreamSynchronize(s);
        return rc;
    }
    h->frames_per_pass = bf;
    h->rows_per_warp = 32 / bf;
    h->copy_engine = be;
    AZ_TRY(tune_layout(h, frames.p, dark.as<float>(), s));
    AZ_CUDA(cudaStreamSynchronize(s));
    if (best_ms) *best_ms = best / n_trial_frames;
    return AZ_OK;
}
