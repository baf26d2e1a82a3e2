// sde_tally.cu -- the small kernels around the transport: spot preparation, the tally's sum and
// the dose conversion.  They are apart from the transport kernel because that file is compiled
// with subnormal numbers flushed to zero and these treat every input exactly.
#include <math.h>

#include "sde_internal.cuh"
#include "sde_transport.h"

namespace sde {

// Sum of the tally (the deposited energy of the balance), added to *out.
__global__ void k_sum_u64(const unsigned long long* __restrict__ v, size_t n, unsigned long long* out) {
    unsigned long long acc = 0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        acc += v[i];
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
    if ((threadIdx.x & 31) == 0 && acc) atomicAdd(out, acc);
}

// Spot records -> device form and the inclusive prefix of history counts;
// sets the work-queue cursor to the first history id of the run.  One block.
__global__ void __launch_bounds__(1024) k_prep_spots(const sde_spot* raw, int n, SpotDev* out,
                                                     unsigned long long* prefix,
                                                     unsigned long long* counters, unsigned int* err,
                                                     double ox, double oy, double oz, double ihx, double ihy,
                                                     double ihz, double e_min, double e_lim,
                                                     unsigned long long h_begin) {
    __shared__ unsigned long long scan[1024];
    unsigned long long carry = 0;
    for (int base = 0; base < n; base += blockDim.x) {
        int i = base + threadIdx.x;
        unsigned long long nh = 0;
        if (i < n) {
            sde_spot s = raw[i];
            double un = s.ux * s.ux + s.uy * s.uy + s.uz * s.uz;
            bool ok = s.E_MeV > e_min && s.E_MeV + 5.0 * s.sigma_E_MeV <= e_lim && s.sigma_E_MeV >= 0.0 &&
                      s.sigma_xy_mm >= 0.0 && s.sigma_xy_mm < 1e4 && s.sigma_angle_rad >= 0.0 &&
                      s.sigma_angle_rad < 1.0 && un > 0.0 && isfinite(un) && isfinite(s.x_mm) &&
                      isfinite(s.y_mm) && isfinite(s.z_mm);
            SpotDev d = {};
            if (ok) {
                nh = s.n_hist;
                double inv = rsqrt(un);
                double x = s.ux * inv, y = s.uy * inv, z = s.uz * inv;
                double sg = copysign(1.0, z);
                double a = -1.0 / (sg + z), b = x * y * a;
                d.E = (float)s.E_MeV;
                d.sE = (float)s.sigma_E_MeV;
                d.sxy = (float)s.sigma_xy_mm;
                d.sang = (float)s.sigma_angle_rad;
                const double sx = s.sigma_xy_mm * ihx, sy = s.sigma_xy_mm * ihy, sz = s.sigma_xy_mm * ihz;
                d.px = (float)((s.x_mm - ox) * ihx);
                d.py = (float)((s.y_mm - oy) * ihy);
                d.pz = (float)((s.z_mm - oz) * ihz);
                d.ux = (float)x;
                d.uy = (float)y;
                d.uz = (float)z;
                d.e1x = (float)((1.0 + sg * x * x * a) * sx);
                d.e1y = (float)(sg * b * sy);
                d.e1z = (float)(-sg * x * sz);
                d.e2x = (float)(b * sx);
                d.e2y = (float)((sg + y * y * a) * sy);
                d.e2z = (float)(-y * sz);
            } else {
                atomicOr(err, kErrBadSpot);
            }
            out[i] = d;
        }
        scan[threadIdx.x] = nh;
        __syncthreads();
        for (int off = 1; off < (int)blockDim.x; off <<= 1) {
            unsigned long long add = threadIdx.x >= (unsigned)off ? scan[threadIdx.x - off] : 0ull;
            __syncthreads();
            scan[threadIdx.x] += add;
            __syncthreads();
        }
        if (i < n) prefix[i + 1] = carry + scan[threadIdx.x];
        carry += scan[blockDim.x - 1];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        prefix[0] = 0;
        counters[kCntCursor] = h_begin;
    }
}

// Dose to medium (Sec. 2.2.2): tally units -> J over voxel mass (kg).  The FP64 unit of
// this GPU is narrow and a double division is a long sequence on it, so 1/mass is the
// FP32 reciprocal refined by one Newton step in FP64 (relative error ~1e-14).  Even so it is
// FP64 operations that bound a dense dose, and most voxels of most doses hold nothing: those
// are written as zeros without reading their density.  Four voxels a thread are in flight.
template <typename T>
__global__ void __launch_bounds__(256) k_convert(const unsigned long long* __restrict__ edep,
                                                 const float* __restrict__ rho, size_t nv, double unit_J,
                                                 double vol_kg_per_rho, T* __restrict__ dose) {
    constexpr int kAhead = 4;
    const size_t step = (size_t)gridDim.x * blockDim.x;
    for (size_t v0 = blockIdx.x * (size_t)blockDim.x + threadIdx.x; v0 < nv; v0 += kAhead * step) {
        unsigned long long e[kAhead];
        float r[kAhead];
#pragma unroll
        for (int i = 0; i < kAhead; ++i) e[i] = v0 + i * step < nv ? edep[v0 + i * step] : 0ull;
#pragma unroll
        for (int i = 0; i < kAhead; ++i) r[i] = e[i] ? rho[v0 + i * step] : 0.f;
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
            if (v0 + i * step >= nv) break;
            double out = 0.0;
            if (r[i] > 0.f) {
                const double mass = (double)r[i] * vol_kg_per_rho;
                double y = (double)__frcp_rn(__double2float_rn(mass));
                y = fma(y, fma(-mass, y, 1.0), y);
                out = (double)e[i] * unit_J * y;
            }
            dose[v0 + i * step] = (T)out;
        }
    }
}

// ---------------------------------------------------------------- launchers
cudaError_t launch_prep(const sde_spot* raw, int n, SpotDev* out, unsigned long long* prefix,
                        unsigned long long* counters, unsigned int* err, const double o[3], const double h[3],
                        double e_min, double e_lim, cudaStream_t st, unsigned long long h_begin) {
    k_prep_spots<<<1, 1024, 0, st>>>(raw, n, out, prefix, counters, err, o[0], o[1], o[2], 1.0 / h[0], 1.0 / h[1],
                                     1.0 / h[2], e_min, e_lim, h_begin);
    return cudaGetLastError();
}

cudaError_t launch_sum_u64(const unsigned long long* v, size_t n, unsigned long long* out, int num_sms,
                           cudaStream_t st) {
    k_sum_u64<<<num_sms * 4, 256, 0, st>>>(v, n, out);
    return cudaGetLastError();
}

cudaError_t launch_convert(const unsigned long long* edep, const float* rho, size_t nv, double unit_J,
                           double vol_kg_per_rho, double* dose, int num_sms, cudaStream_t st) {
    int blocks = num_sms * 8;
    k_convert<double><<<blocks, 256, 0, st>>>(edep, rho, nv, unit_J, vol_kg_per_rho, dose);
    return cudaGetLastError();
}

cudaError_t launch_convert_f32(const unsigned long long* edep, const float* rho, size_t nv, double unit_J,
                               double vol_kg_per_rho, float* dose, int num_sms, cudaStream_t st) {
    int blocks = num_sms * 8;
    k_convert<float><<<blocks, 256, 0, st>>>(edep, rho, nv, unit_J, vol_kg_per_rho, dose);
    return cudaGetLastError();
}

}  // namespace sde
