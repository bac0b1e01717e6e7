// Plane phase: dispatch to the per-type kernels (tc_fft_f64.cu, tc_fft_f32.cu,
// tc_fft_df.cu; templates and the description of the transforms in
// tc_fft_impl.cuh; fixed point: tc_fx_*.cu) and the transform-length table.
#include "tc_internal.h"

void tc_plane_kernel_f64(const TcDev& d, int which, cudaStream_t s, int tile0, int ntiles);
void tc_plane_kernel_f32(const TcDev& d, int which, cudaStream_t s, int tile0, int ntiles);
void tc_plane_kernel_df(const TcDev& d, int which, cudaStream_t s, int tile0, int ntiles);
void tc_plane_kernel_batch_f64(const TcDev& d0, const TcDev* ds, const int2* ymap, int nplanes, int which, cudaStream_t s);
void tc_plane_kernel_batch_f32(const TcDev& d0, const TcDev* ds, const int2* ymap, int nplanes, int which, cudaStream_t s);
void tc_plane_kernel_batch_df(const TcDev& d0, const TcDev* ds, const int2* ymap, int nplanes, int which, cudaStream_t s);
cudaError_t tc_plane_attributes_f64();
cudaError_t tc_plane_attributes_f32();
cudaError_t tc_plane_attributes_df();
cudaError_t tc_rows_phys_attributes();
#define FX_GROUP(TAG)                                                                                                   \
    bool tc_fx_z_##TAG(const TcDev&, const TcDev*, const int2*, int, int, cudaStream_t, int, int);                      \
    bool tc_fx_rows_##TAG(const TcDev&, const TcDev*, const int2*, int, cudaStream_t);                                  \
    bool tc_fx_phys_##TAG(const TcDev&, int4, cudaStream_t);                                                            \
    bool tc_fx_order_##TAG(int, int4&);                                                                                 \
    bool tc_fx_attributes_##TAG(int, int, cudaError_t&);                                                                \
    void tc_fx_phys_attributes_##TAG(cudaError_t&);
FX_GROUP(a) FX_GROUP(b) FX_GROUP(c) FX_GROUP(d)
#undef FX_GROUP

void tc_fx_plane_kernel(const TcDev& d, const TcDev* ds, const int2* ymap, int nplanes, int which, cudaStream_t s,
                        int col0, int ncols) {
    if (which == 1) {
        (void)(tc_fx_rows_a(d, ds, ymap, nplanes, s) || tc_fx_rows_b(d, ds, ymap, nplanes, s) ||
               tc_fx_rows_c(d, ds, ymap, nplanes, s) || tc_fx_rows_d(d, ds, ymap, nplanes, s));
    } else {
        (void)(tc_fx_z_a(d, ds, ymap, nplanes, which, s, col0, ncols) || tc_fx_z_b(d, ds, ymap, nplanes, which, s, col0, ncols) ||
               tc_fx_z_c(d, ds, ymap, nplanes, which, s, col0, ncols) || tc_fx_z_d(d, ds, ymap, nplanes, which, s, col0, ncols));
    }
}

bool tc_fx_to_physical(const TcDev& d, const double2* field, cudaStream_t s) {
    if (!d.phx) return false;
    TcDev dd = d;
    dd.u = const_cast<double2*>(field);                 // read only
    dd.Mtx = dd.Mt;
    dd.Mzx = dd.Mz;
    int4 zr = make_int4(1, 1, 1, 1);
    (void)(tc_fx_order_a(d.Mz, zr) || tc_fx_order_b(d.Mz, zr) || tc_fx_order_c(d.Mz, zr) || tc_fx_order_d(d.Mz, zr));
    tc_fx_plane_kernel(dd, nullptr, nullptr, d.Nr, 3, s, 0, d.Nh);
    (void)(tc_fx_phys_a(dd, zr, s) || tc_fx_phys_b(dd, zr, s) || tc_fx_phys_c(dd, zr, s) || tc_fx_phys_d(dd, zr, s));
    return true;
}

cudaError_t tc_fx_attributes(int Mtx, int Mzx) {
    cudaError_t e = cudaSuccess;
    tc_fx_attributes_a(Mtx, Mzx, e);
    tc_fx_attributes_b(Mtx, Mzx, e);
    tc_fx_attributes_c(Mtx, Mzx, e);
    tc_fx_attributes_d(Mtx, Mzx, e);
    return e;
}

cudaError_t tc_fx_physical_attributes() {
    cudaError_t e = cudaSuccess;
    tc_fx_phys_attributes_a(e);
    tc_fx_phys_attributes_b(e);
    tc_fx_phys_attributes_c(e);
    tc_fx_phys_attributes_d(e);
    return e;
}

bool tc_fft_fixed_length(int M) {
    for (int m : {12, 18, 24, 36, 48, 72, 96, 144, 192, 288, 384, 576, 768, 1152, 1536})
        if (M == m) return true;
    return false;
}

void tc_launch_plane_kernel_tiles(const TcDev& d, int which, cudaStream_t s, int tile0, int ntiles) {
    if (d.fx) tc_fx_plane_kernel(d, nullptr, nullptr, d.Nr, which, s, tile0 * d.ztile, ntiles * d.ztile);
    else if (d.prec == 1) tc_plane_kernel_f32(d, which, s, tile0, ntiles);
    else if (d.prec == 2) tc_plane_kernel_df(d, which, s, tile0, ntiles);
    else tc_plane_kernel_f64(d, which, s, tile0, ntiles);
}

void tc_launch_plane_kernel_batch(const TcDev& d0, const TcDev* ds, const int2* ymap, int nplanes, int which,
                                  cudaStream_t s) {
    if (d0.fx) tc_fx_plane_kernel(d0, ds, ymap, nplanes, which, s, 0, d0.Nh);
    else if (d0.prec == 1) tc_plane_kernel_batch_f32(d0, ds, ymap, nplanes, which, s);
    else if (d0.prec == 2) tc_plane_kernel_batch_df(d0, ds, ymap, nplanes, which, s);
    else tc_plane_kernel_batch_f64(d0, ds, ymap, nplanes, which, s);
}

void tc_launch_plane_kernel(const TcDev& d, int which, cudaStream_t s) {
    tc_launch_plane_kernel_tiles(d, which, s, 0, d.Nh / d.ztile);
}

void tc_launch_plane_phase(const TcDev& d, cudaStream_t s) {
    for (int w = 0; w < 3; ++w) tc_launch_plane_kernel(d, w, s);
}

// Shared-memory opt-in of the FFT kernels (called once per device, before any
// stream capture).
cudaError_t tc_set_kernel_attributes() {
    cudaError_t e = cudaSuccess;
    for (cudaError_t r : {tc_plane_attributes_f64(), tc_plane_attributes_f32(), tc_plane_attributes_df(),
                          tc_rows_phys_attributes()})
        if (r != cudaSuccess) e = r;
    return e;
}
