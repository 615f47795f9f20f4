// fftfx.cu -- host side of the fixed-point passes (fftfx.cuh): which plans take
// them, their launches, and their tables.
#include "fftfx.cuh"
#include "sg_launch.cuh"

namespace sg {

static const FxKernels* fx_kernels(int n)
{
    static const FxKernels table[] = {fx_kernels_lg6(), fx_kernels_lg7(),  fx_kernels_lg8(), fx_kernels_lg9(),
                                      fx_kernels_lg10(), fx_kernels_lg11(), fx_kernels_lg12()};
    const int lg = sg_ilog2(n);
    return lg >= FX_MIN_LG && lg <= FX_MAX_LG ? &table[lg - FX_MIN_LG] : nullptr;
}

// the maps of wa, wb, wc for row blocks of R rows, or null
static const CUtensorMap* fx_maps(const PlanView& p, int R)
{
    if (!p.maps) return nullptr;
    for (int k = 0; k < 2; k++)
        if (p.maps[k].R == R) return p.maps[k].m;
    return nullptr;
}

bool fx_rows_ok(const PlanView& p)
{
    const FxKernels* k = p.twx ? fx_kernels(p.nphi) : nullptr;
    return k && p.nu % k->rows == 0 && fx_maps(p, k->rows);
}
bool fx_cols_len(const PlanView& p) { return p.twx && fx_kernels(2 * p.nu); }
bool fx_cols_ok(const PlanView& p) { return p.kfr && p.kfp && fx_cols_len(p); }

cudaError_t launch_fx_r2c(const PlanView& p, const double* x0, const double* x1, cudaStream_t st)
{
    const FxKernels& k = *fx_kernels(p.nphi);
    const int b = x1 ? 1 : 0, units = b ? p.nu : p.nu / 2, per = b ? k.rows : k.r2c_slots;
    const CUtensorMap* m = fx_maps(p, k.rows);
    cudaError_t e = set_smem(k.r2c[b], k.r2c_smem[b]);
    if (e != cudaSuccess) return e;
    return launch_pdl(k.r2c[b], (units + per - 1) / per, k.r2c_threads[b], k.r2c_smem[b], st, x0, x1,
                      b ? p.wpost : p.wpre, p.wdf, (double2*)p.wa, p.nu, (const fxw*)p.twx, p.err, m[0], m[2]);
}

cudaError_t launch_fx_cols(const PlanView& p, bool adjoint, cudaStream_t st)
{
    const FxKernels& k = *fx_kernels(2 * p.nu);
    const int half = p.nphi / 2, grid = (half + k.cols_slots - 1) / k.cols_slots;
    const double2 *A = (const double2*)p.wa, *C = (const double2*)p.wc;
    cudaError_t e;
    if (adjoint) {
        if ((e = set_smem(k.bwd_cols, k.cols_smem)) != cudaSuccess) return e;
        return launch_pdl(k.bwd_cols, grid, k.cols_threads, k.cols_smem, st, A, C, (const fx2*)p.kfr,
                          (const fx2*)p.kfp, (double2*)p.wb, half, (const fxw*)p.twx, p.err);
    }
    if ((e = set_smem(k.fwd_cols, k.cols_smem)) != cudaSuccess) return e;
    return launch_pdl(k.fwd_cols, grid, k.cols_threads, k.cols_smem, st, A, (const fx2*)p.kfr, (const fx2*)p.kfp,
                      (double2*)p.wb, (double2*)p.wc, half, (const fxw*)p.twx, p.err);
}

cudaError_t launch_fx_c2r(const PlanView& p, double* y0, double* y1, cudaStream_t st)
{
    const FxKernels& k = *fx_kernels(p.nphi);
    const int b = y1 ? 0 : 1;
    const CUtensorMap* m = fx_maps(p, k.rows);
    cudaError_t e = set_smem(k.c2r[b], k.c2r_smem[b]);
    if (e != cudaSuccess) return e;
    return launch_pdl(k.c2r[b], p.nu / k.rows, k.c2r_threads[b], k.c2r_smem[b], st, b ? p.wpre : p.wpost, p.wdf, y0,
                      y1, p.nu, (const fxw*)p.twx, p.err, m[1], m[2]);
}

size_t fx_twiddle_bytes() { return (size_t)(FX_SMAX - FX_SMIN + 1) * fx_tw_entries() * sizeof(fxw); }
const void* fx_twiddles()
{
    static const std::vector<fxw> table = fx_twiddle_table();  // made once, thread-safe
    return table.data();
}

// one block per mode's row: its exponent, then its entries (fx_spec_entry)
__device__ __forceinline__ double2 fx_spec_value(const double2* p) { return *p; }
__device__ __forceinline__ double2 fx_spec_value(const dfloat2* p)
{
    return double2{df_to_double(p->x), df_to_double(p->y)};
}
template <typename V>
__global__ void __launch_bounds__(256) k_fx_spectra(const V* __restrict__ kr, const V* __restrict__ kp,
                                                    fx2* __restrict__ fr, fx2* __restrict__ fp, int nu)
{
    __shared__ unsigned top;
    const size_t at = (size_t)blockIdx.x * (nu + 2);
    const V* in = (blockIdx.y ? kp : kr) + at;
    fx2* out = (blockIdx.y ? fp : fr) + at;
    if (threadIdx.x == 0) top = 0;
    __syncthreads();
    unsigned h = 0;
    for (int i = threadIdx.x; i <= nu; i += blockDim.x) {
        const double2 k = fx_spec_value(in + i);
        h = max(h, max(fx_abshi(k.x), fx_abshi(k.y)));
    }
    atomicMax(&top, h);
    __syncthreads();
    const int F = fx_field(top);
    for (int i = threadIdx.x; i <= nu; i += blockDim.x) {
        const double2 k = fx_spec_value(in + i);
        out[i] = fx_spec_entry(k.x, k.y, F);
    }
    // the row's exponent; a table with an infinity or NaN marks its mode bad
    if (threadIdx.x == 0) out[nu + 1] = fx2{top >= 0x7ff00000u ? FX_BAD : fx_spec_exp(F), 0};
}

cudaError_t launch_fx_spectra(const PlanView& p, bool df, cudaStream_t st)
{
    const dim3 grid(p.nphi / 2 + 1, 2);
    if (df)
        k_fx_spectra<<<grid, 256, 0, st>>>((const dfloat2*)p.kr, (const dfloat2*)p.kp, (fx2*)p.kfr, (fx2*)p.kfp, p.nu);
    else
        k_fx_spectra<<<grid, 256, 0, st>>>((const double2*)p.kr, (const double2*)p.kp, (fx2*)p.kfr, (fx2*)p.kfp, p.nu);
    return cudaGetLastError();
}

}  // namespace sg
