// Ray directions (Eq. txty, Eq. raypos), the finalize pass (maps in rayid order),
// the source-redshift moments (Eqs. Isources, Isources1) and the shear maps.
#include "rr_internal.h"

namespace rr {
namespace {

// Zeros in the accumulators and the counter of ray rid.
__device__ __forceinline__ void clear_ray(const RayState& st, long long rid)
{
    const float2 z = make_float2(0.f, 0.f);
    st.kacc[rid] = z;
    st.bacc[rid] = z;
    if (st.kmom) {
        st.kmom[rid] = z;
        st.bmom[rid] = z;
    }
    if (st.g1acc) {
        st.g1acc[rid] = z;
        st.g2acc[rid] = z;
    }
    st.nseg[rid] = 0;
}

// Rows [row0, row0 + nrows) of an nx x ny bundle; rid counts from row row0. The
// ray's accumulators and the state's words are zeroed on the way.
//
// Bound by the FP64 pipe (sincos, a square root and two divisions a ray, on a
// GPU whose FP64 rate is 1/64 of its FP32 rate), not by the 56 bytes a ray
// writes. The angle grid of Eq. (txty) is antisymmetric, theta(n - 1 - i) =
// -theta(i) exactly, and theta_x, theta_y enter theta only squared: one thread
// computes |theta|, its sine and cosine and the two quotients once and writes
// the four rays (+-theta_x, +-theta_y), whose components differ in sign only
// (bit for bit what each ray's own evaluation gives). A thread's first ray is
// (ix, iy) in the lower quarter of the whole bundle; of its rows only those in
// the band are written. (kx, ky: fov / (2 (n - 1)), divided on the host.)
// 2048^2 rays: 679 us with one evaluation a ray, 143 us now (1024^2: 171 -> 39).
__global__ void init_state_kernel(int nx, int ny, int row0, int nrows, double kx, double ky, const RayState st)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *st.err = 0;
        *st.words = Words{0, 0, 0};
    }
    const int hx = (nx + 1) / 2, hy = (ny + 1) / 2;
    const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= (long long)hx * hy) return;
    const int ix = (int)(q % hx), iy = (int)(q / hx);
    const int mx = nx - 1 - ix, my = ny - 1 - iy;
    const bool lower = iy >= row0 && iy < row0 + nrows, upper = my != iy && my >= row0 && my < row0 + nrows;
    if (!lower && !upper) return;
    // Eq. (txty) with 0-based pixel indices, as (2i - (N-1)) U / (2(N-1)): the
    // central pixel of an odd row is at exactly 0; a single ray per side sits at 0
    const double tx = nx > 1 ? (double)(2 * ix - (nx - 1)) * kx : 0.0;
    const double ty = ny > 1 ? (double)(2 * iy - (ny - 1)) * ky : 0.0;
    const double th = sqrt(tx * tx + ty * ty);
    double n0 = 0.0, n1 = 0.0, n2 = 1.0;
    if (th > 0.0) {
        // (sin th cos ph, sin th sin ph, cos th) with cos ph = tx/th, sin ph = ty/th
        double s, c;
        sincos(th, &s, &c);
        n0 = s * (tx / th);
        n1 = s * (ty / th);
        n2 = c;
    }
    const float h0 = (float)n0, h1 = (float)n1, h2 = (float)n2;
    const float l0 = (float)(n0 - (double)h0), l1 = (float)(n1 - (double)h1), l2 = (float)(n2 - (double)h2);
    auto put = [&](int x, int y, bool fx, bool fy) {
        const long long rid = (long long)(y - row0) * nx + x;
        // (0 - v, not -v: a zero component stays +0, as in the ray's own evaluation)
        if (st.dir) {
            st.dir[3 * rid] = fx ? 0.0 - n0 : n0;
            st.dir[3 * rid + 1] = fy ? 0.0 - n1 : n1;
            st.dir[3 * rid + 2] = n2;
        }
        st.dirh[rid] = make_float4(fx ? 0.f - h0 : h0, fy ? 0.f - h1 : h1, h2, 0.f);
        st.dirl[rid] = make_float4(fx ? 0.f - l0 : l0, fy ? 0.f - l1 : l1, l2, 0.f);
        clear_ray(st, rid);
    };
    if (lower) {
        put(ix, iy, false, false);
        if (mx != ix) put(mx, iy, true, false);
    }
    if (upper) {
        put(ix, my, false, true);
        if (mx != ix) put(mx, my, true, true);
    }
}

__device__ __forceinline__ double ff(float2 v) { return (double)v.x + (double)v.y; }

// Maps from the accumulators; for the moments form (kmom, bmom not null)
// kappa = A - B / chi_s per channel (Eq. Isources); for Method A (add_born)
// kappa = the gradient and surface terms plus the density term (Eq. kappa2).
// The block that finishes last publishes the segment total and hands it and
// the error word to the host: no memset before and no copies after the kernel,
// which took longer than the kernel on a small bundle.
// Bound by HBM (36 bytes a ray): two rays a thread in 16-byte accesses where the
// maps are 16-byte aligned (PAIR), one fence a block.
template <bool PAIR>
__global__ void finalize_kernel(int nrays, const RayState st, double* out_kappa, double* out_kborn, HostWords* host,
                                double inv_chi_s, int add_born)
{
    __shared__ unsigned long long block_sum;
    if (threadIdx.x == 0) block_sum = 0;
    __syncthreads();
    auto kappa = [&](float2 k, float2 b, long long i) {
        return st.kmom ? ff(k) - ff(st.kmom[i]) * inv_chi_s : (add_born ? ff(k) + ff(b) : ff(k));
    };
    auto born = [&](float2 b, long long i) { return st.bmom ? ff(b) - ff(st.bmom[i]) * inv_chi_s : ff(b); };
    unsigned long long wide = 0;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const long long first = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if constexpr (PAIR) {
        for (long long i = first; i < nrays / 2; i += stride) {
            const float4 k = reinterpret_cast<const float4*>(st.kacc)[i], b = reinterpret_cast<const float4*>(st.bacc)[i];
            const uint2 n = reinterpret_cast<const uint2*>(st.nseg)[i];
            const float2 k0 = make_float2(k.x, k.y), k1 = make_float2(k.z, k.w);
            const float2 b0 = make_float2(b.x, b.y), b1 = make_float2(b.z, b.w);
            if (out_kappa)
                reinterpret_cast<double2*>(out_kappa)[i] = make_double2(kappa(k0, b0, 2 * i), kappa(k1, b1, 2 * i + 1));
            if (out_kborn)
                reinterpret_cast<double2*>(out_kborn)[i] = make_double2(born(b0, 2 * i), born(b1, 2 * i + 1));
            wide += (unsigned long long)n.x + n.y;
        }
    }
    for (long long i = PAIR ? (nrays & ~1LL) + first : first; i < nrays; i += stride) {
        const float2 k = st.kacc[i], b = st.bacc[i];
        if (out_kappa) out_kappa[i] = kappa(k, b, i);
        if (out_kborn) out_kborn[i] = born(b, i);
        wide += st.nseg[i];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) wide += __shfl_down_sync(0xffffffffu, wide, o);
    if ((threadIdx.x & 31) == 0 && wide) atomicAdd(&block_sum, wide);
    __syncthreads();
    if (threadIdx.x != 0) return;
    atomicAdd(&st.words->sum, block_sum);
    __threadfence();
    if (atomicAdd(&st.words->done, 1u) == gridDim.x - 1) {
        const unsigned long long t = atomicExch(&st.words->sum, 0ull);
        st.words->total = t;
        st.words->done = 0;
        if (host) {
            host->total = t;
            host->err = atomicOr(st.err, 0u);
        }
    }
}

// Zeros in one state (blockIdx.y: the part), in a loop over its rays.
__device__ __forceinline__ void clear_state(const RayState& st, long long n)
{
    if (blockIdx.y == 0 && threadIdx.x == 0) *st.err = 0;
    for (long long i = (long long)blockIdx.y * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.y * blockDim.x)
        clear_ray(st, i);
}

__global__ void clear_state_kernel(const ClearItem item) { clear_state(item.st, item.nrays); }

// blockIdx.x: the state
__global__ void clear_states_kernel(const ClearItem* __restrict__ items)
{
    const ClearItem item = items[blockIdx.x];
    clear_state(item.st, item.nrays);
}

__global__ void collect_words_kernel(const ClearItem* __restrict__ items, int n, HostWords* out)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        out[i].total = items[i].st.words->total;
        out[i].err = *items[i].st.err;
    }
}

// The four moments (A_kappa, B_kappa, A_born, B_born) as FP64 rows.
__global__ void moments_kernel(int nrays, const float2* __restrict__ kacc, const float2* __restrict__ kmom,
                               const float2* __restrict__ bacc, const float2* __restrict__ bmom, double* out)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nrays) return;
    out[i] = ff(kacc[i]);
    out[nrays + i] = ff(kmom[i]);
    out[2LL * nrays + i] = ff(bacc[i]);
    out[3LL * nrays + i] = ff(bmom[i]);
}

// The shear maps from their float-float accumulators.
__global__ void shear_out_kernel(int nrays, const float2* __restrict__ g1acc, const float2* __restrict__ g2acc,
                                 double* gamma1, double* gamma2)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nrays) return;
    gamma1[i] = ff(g1acc[i]);
    gamma2[i] = ff(g2acc[i]);
}

// kappa for sources at chi_k from the moments at the end and at chi_k
// (Eqs. Isources, Isources1): A(chi_k) = A_end - A_k, B(chi_k) = B_end - B_k.
__global__ void source_kappa_kernel(const double* __restrict__ m_end, const double* __restrict__ m_k,
                                    long long nrays, double inv_chi_k, double* kappa, double* kborn)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nrays) return;
    double a = m_end[i], b = m_end[nrays + i], ab = m_end[2 * nrays + i], bb = m_end[3 * nrays + i];
    if (m_k) {
        a -= m_k[i];
        b -= m_k[nrays + i];
        ab -= m_k[2 * nrays + i];
        bb -= m_k[3 * nrays + i];
    }
    kappa[i] = a - b * inv_chi_k;
    if (kborn) kborn[i] = ab - bb * inv_chi_k;
}

}  // namespace

cudaError_t launch_moments(int nrays, const float2* kacc, const float2* kmom, const float2* bacc, const float2* bmom,
                           double* out, cudaStream_t s)
{
    const int nt = 256;
    moments_kernel<<<(unsigned)(((long long)nrays + nt - 1) / nt), nt, 0, s>>>(nrays, kacc, kmom, bacc, bmom, out);
    return cudaGetLastError();
}

cudaError_t launch_shear_out(int nrays, const float2* g1acc, const float2* g2acc, double* gamma1, double* gamma2,
                             cudaStream_t s)
{
    const int nt = 256;
    shear_out_kernel<<<(unsigned)(((long long)nrays + nt - 1) / nt), nt, 0, s>>>(nrays, g1acc, g2acc, gamma1, gamma2);
    return cudaGetLastError();
}

cudaError_t launch_source_kappa(const double* m_end, const double* m_k, long long nrays, double chi_k, double* kappa,
                                double* kborn, cudaStream_t s)
{
    const int nt = 256;
    source_kappa_kernel<<<(unsigned)((nrays + nt - 1) / nt), nt, 0, s>>>(m_end, m_k, nrays, 1.0 / chi_k, kappa, kborn);
    return cudaGetLastError();
}

cudaError_t launch_init_state(const rr_bundle_desc& b, const RayState& st, cudaStream_t s, int row0, int nrows)
{
    if (nrows < 0) nrows = b.ny;
    const long long quarter = (long long)((b.nx + 1) / 2) * ((b.ny + 1) / 2);
    const double kx = b.nx > 1 ? b.fov_x / (2.0 * (b.nx - 1)) : 0.0, ky = b.ny > 1 ? b.fov_y / (2.0 * (b.ny - 1)) : 0.0;
    const int nt = 256;
    init_state_kernel<<<(unsigned)((quarter + nt - 1) / nt), nt, 0, s>>>(b.nx, b.ny, row0, nrows, kx, ky, st);
    return cudaGetLastError();
}

cudaError_t launch_clear_states(const ClearItem* items, int n, cudaStream_t s)
{
    clear_states_kernel<<<dim3((unsigned)n, 64), 256, 0, s>>>(items);
    return cudaGetLastError();
}

cudaError_t launch_clear_state(const ClearItem& item, cudaStream_t s)
{
    const long long parts = (item.nrays + 255) / 256;
    clear_state_kernel<<<dim3(1, (unsigned)(parts < 1216 ? parts : 1216)), 256, 0, s>>>(item);
    return cudaGetLastError();
}

cudaError_t launch_collect_words(const ClearItem* items, int n, HostWords* out, cudaStream_t s)
{
    collect_words_kernel<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(items, n, out);
    return cudaGetLastError();
}

cudaError_t launch_finalize(int nrays, const RayState& st, double* out_kappa, double* out_kborn, HostWords* host,
                            cudaStream_t s, double chi_s, bool add_born)
{
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int nt = 256;
    const bool pair = (reinterpret_cast<uintptr_t>(out_kappa) & 15u) == 0 &&
                      (reinterpret_cast<uintptr_t>(out_kborn) & 15u) == 0 && nrays > 1;
    long long blocks = ((long long)nrays / (pair ? 2 : 1) + nt - 1) / nt;
    const long long cap = (long long)(sms > 0 ? sms : 1) * 8;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    const double ics = (st.kmom && chi_s > 0) ? 1.0 / chi_s : 0.0;
    if (pair)
        finalize_kernel<true><<<(unsigned)blocks, nt, 0, s>>>(nrays, st, out_kappa, out_kborn, host, ics, add_born ? 1 : 0);
    else
        finalize_kernel<false><<<(unsigned)blocks, nt, 0, s>>>(nrays, st, out_kappa, out_kborn, host, ics, add_born ? 1 : 0);
    return cudaGetLastError();
}

}  // namespace rr
