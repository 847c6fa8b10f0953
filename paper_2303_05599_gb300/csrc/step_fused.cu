// Single-event launch of the field step: the FP32 strip kernel
// (strip_body.cuh) or the FP64 tile kernel (fused_body.cuh), both writing the
// site E, B of t_n beside the fields of step n + 1.
#include "small_body.cuh"
#include "strip_body.cuh"

namespace gl {

template <typename R, int TX, int TY>
__global__ void __launch_bounds__(TX * TY) fused_step_kernel(Fields<R> in, Fields<R> out,
                                                             typename Prec<R>::V* site, StepR<R> a) {
    fused_tile<R, TX, TY>(in, out, site, a, blockIdx.x);
}

template <typename R, int TX, int TY>
static void launch_t(void* in, void* out, void* site, int N, int64_t n, double dt, cudaStream_t st) {
    using T = Tile<R, TX, TY>;
    // the dynamic shared-memory limit is a per-device function attribute
    static bool attr[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr[dev]) {
        cudaFuncSetAttribute(fused_step_kernel<R, TX, TY>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)T::bytes);
        attr[dev] = true;
    }
    const int64_t Vn = (int64_t)N * N;
    StepArgs a = step_args(N, (N + TX - 1) / TX, n, dt, 0);
    const int tiles_y = (N + TY - 1) / TY;
    fused_step_kernel<R, TX, TY><<<a.tiles_x * tiles_y, TX * TY, T::bytes, st>>>(
        carve_fields<R>(in, Vn), carve_fields<R>(out, Vn), (typename Prec<R>::V*)site, step_r<R>(a));
}

// FP32: blocks of up to WPB warps take as many consecutive segments of the
// event's strips per item and run them in step; `items` items strided over the
// grid
template <int WPB, int MINB>
__global__ void __launch_bounds__(WPB * 32, MINB) strip_step_kernel(Fields<float> in, Fields<float> out, float4* site,
                                                                     int N, StripStep a, int items, int seg) {
    extern __shared__ __align__(16) unsigned char strip_smem[];
    StripWarpSmem* S = (StripWarpSmem*)strip_smem;
    const int wib = threadIdx.x >> 5;
    const int64_t nseg = strip_segments(N, seg);
    for (int it = blockIdx.x; it < items; it += gridDim.x) {
        const int64_t j = (int64_t)it * (blockDim.x >> 5) + wib;
        strip_run_segment(S[wib], in, out, site, N, j < nseg ? j : nseg - 1, j < nseg, a, seg);
    }
}

static int sm_count() {
    static int sms[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) dev = 0;
    if (!sms[dev]) cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev);
    return sms[dev] > 0 ? sms[dev] : 1;
}

// warps a block and warps an SM of FP32 launch shape `tile`
static void strip_shape(int tile, int* wpb, int* warps_sm) {
    *wpb = tile == 1 ? 12 : 8;
    *warps_sm = tile == 1 ? 12 : tile == 2 ? 8 : 16;
}

template <int WPB, int MINB>
static void launch_strip(void* in, void* out, void* site, int N, int64_t n, double dt, int every, int seg,
                         cudaStream_t st) {
    // the dynamic shared-memory limit is a per-device function attribute
    static bool attr[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev >= 0 && dev < 64 && !attr[dev]) {
        cudaFuncSetAttribute(strip_step_kernel<WPB, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             WPB * (int)sizeof(StripWarpSmem));
        attr[dev] = true;
    }
    const int64_t Vn = (int64_t)N * N;
    const StripPlan p = strip_plan(&N, 1, WPB, WPB * MINB, sm_count(), seg);
    const int items = (int)((strip_segments(N, p.seg) + p.wpb - 1) / p.wpb);
    int grid = sm_count() * (WPB * MINB / p.wpb);
    if (grid > items) grid = items;
    strip_step_kernel<WPB, MINB><<<grid, p.wpb * 32, p.wpb * sizeof(StripWarpSmem), st>>>(
        carve_fields<float>(in, Vn), carve_fields<float>(out, Vn), (float4*)site, N, strip_step(n, dt, every), items,
        p.seg);
}

__global__ void __launch_bounds__(SmallTile::NT) small_step_kernel(Fields<double> in, Fields<double> out, double2* site,
                                                                  StepR<double> a) {
    small_tile(in, out, site, a, blockIdx.x);
}

void launch_fused_step(int prec, void* in, void* out, void* site, int N, int64_t n, double dt, int reunit_every,
                       int tile, int seg, cudaStream_t st) {
    if (prec == 0) {
        // FP64: 4x4 tiles of four warps for small lattices, else 16x8 (103 KB of
        // shared memory) or 32x2
        if (small64(tiles64(N), sm_count())) {
            const int64_t Vn = (int64_t)N * N;
            const int nt = small_tiles_x(N);
            small_step_kernel<<<nt * nt, SmallTile::NT, sizeof(SmallTile), st>>>(
                carve_fields<double>(in, Vn), carve_fields<double>(out, Vn), (double2*)site,
                step_r<double>(step_args(N, nt, n, dt, 0)));
        } else if (tile == 2) launch_t<double, 32, 2>(in, out, site, N, n, dt, st);
        else launch_t<double, TILE64_X, TILE64_Y>(in, out, site, N, n, dt, st);
    } else if (tile == 1) {
        launch_strip<12, 1>(in, out, site, N, n, dt, reunit_every, seg, st);
    } else if (tile == 2) {
        launch_strip<8, 1>(in, out, site, N, n, dt, reunit_every, seg, st);
    } else {
        launch_strip<8, 2>(in, out, site, N, n, dt, reunit_every, seg, st);
    }
}

int strip_model_seg(int N, int tile) {
    int wpb, warps_sm;
    strip_shape(tile, &wpb, &warps_sm);
    return strip_plan(&N, 1, wpb, warps_sm, sm_count(), 0).seg;
}

// Launch shape of an event that has not been tuned.  Lattices that leave the
// SMs with one or two warps a scheduler take the 8-warp shape (203 registers a
// thread), larger ones the 12-warp shape, which needs three to pay: 256^2 19.6
// against 20.3 us, 300^2 24.7 against 24.5 us, 1024^2 153 against 139 us (trial
// launches, the best segment length of each shape).
int strip_default_tile(int N) { return (int64_t)N * N <= (int64_t)sm_count() * 8 * 32 * 4 ? 2 : 1; }

}  // namespace gl
