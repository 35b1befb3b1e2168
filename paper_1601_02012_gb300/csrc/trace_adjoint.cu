// Adjoint of the cell-by-cell integration (the transpose of rr_trace_step).
//
// kappa and Born kappa are linear in the records, so the gradient of a loss
// with respect to the records is the transpose of the forward map: the walk
// of a logged step is replayed (geometry only) and every segment's weights
// dI/dq of its 8 corners (or its centre) are scattered back, scaled by the
// per-ray dL/dkappa and dL/dkappa_born.
#include "walk.cuh"

namespace rr {
namespace {

// Transpose of line_cubic: given the weights J_N of the cubic's coefficients
// e_{N-1} in the segment integral, the weight of each corner value q[m].
__device__ __forceinline__ void line_cubic_adjoint(const float J[4], float u0, float u1, float u2, float v0,
                                                   float v1, float v2, float W[8])
{
    const float E0 = J[0] * u2 + J[1] * v2;
    const float E1 = J[1] * u2 + J[2] * v2;
    const float E2 = J[2] * u2 + J[3] * v2;
    const float M0[2] = {J[0] - E0, E0};
    const float M1[2] = {J[1] - E1, E1};
    const float M2[2] = {J[2] - E2, E2};
#pragma unroll
    for (int kk = 0; kk < 2; ++kk) {
        const float C = fmaf(M0[kk], u1, M1[kk] * v1);
        const float D = fmaf(M1[kk], u1, M2[kk] * v1);
        const float A0 = M0[kk] - C, A1 = C;
        const float B0 = M1[kk] - D, B1 = D;
        // x-step for the pairs jk = 2 kk (j = 0) and 2 kk + 1 (j = 1)
        const float d0 = fmaf(A0, u0, B0 * v0);
        const float d1 = fmaf(A1, u0, B1 * v0);
        W[4 * kk + 0] = A0 - d0;
        W[4 * kk + 1] = d0;
        W[4 * kk + 2] = A1 - d1;
        W[4 * kk + 3] = d1;
    }
}

// Warps per block of the adjoint launch (the default ray tile), and the floats
// of one row of a warp's staging area: 32 lanes and a pad, so that the 16-byte
// reads of eight different rows fall into different banks.
constexpr int kAdjWarps = 4;
constexpr int kRow = 36;

// The warp's G matrix: G_c of lane k, the factor of channel c in lane k's
// contributions (gk w_c for the six tidal channels, gb for delta), is constant
// along its ray. Lane l keeps the row c = l & 7 for all 32 lanes k, in registers
// for the whole walk.
__device__ __forceinline__ void load_factors(const float G[7], float* __restrict__ sm, float4 row[8])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int c = 0; c < 7; ++c) sm[c * kRow + lane] = G[c];
    sm[7 * kRow + lane] = 0.f;
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 8; ++i) row[i] = *reinterpret_cast<const float4*>(sm + (lane & 7) * kRow + 4 * i);
    __syncwarp();
}

// The contributions of a ray whose derivative is infinite or NaN, one by one:
// in the product they would reach every point the warp flushes (0 x NaN).
template <class PT>
__device__ __noinline__ void add_alone(double* __restrict__ grad, float4 n, float gk, float gb, int nr, PT P0, PT Da,
                                       PT Db, float F0, float F1, float F2, float F3)
{
    const float w[6] = {n.y * n.y + n.z * n.z, n.x * n.x + n.z * n.z, n.x * n.x + n.y * n.y,
                        -2.f * n.x * n.y,      -2.f * n.x * n.z,      -2.f * n.y * n.z};
    for (int r = 0; r < nr; ++r) {
        const float f = r == 0 ? F0 : (r == 1 ? F1 : (r == 2 ? F2 : F3));
        if (f == 0.f) continue;
        double* p = grad + 8 * (size_t)(P0 + ((r & 1) ? Da : 0) + ((r & 2) ? Db : 0));
        for (int c = 0; c < 6; ++c)
            if (gk != 0.f) atomicAdd(p + c, (double)(gk * f * w[c]));
        if (gb != 0.f) atomicAdd(p + 6, (double)(gb * f));
    }
}

// Adds F[r] G_c to channel c of the gradient records of the points P0 + {0, Da,
// Db, Da + Db} (r = 0 .. 3: the corners of the face a crossing leaves; NR = 1:
// P0 alone, the cell of the NGP form), for every lane with `part` set; all
// lanes of the warp take part in the call.
//
// The records hold 8 FP64 sums, one per channel {Hxx, Hyy, Hzz, Hxy, Hxz, Hyz,
// delta, 0} (64 B), where thousands of contributions of both signs meet.
// Neighbouring rays are far closer together than a cell, so the lanes mostly
// flush the same face. Per round the lanes on the face of the first lane not
// done yet are summed: sum_k F_r[k] G_c[k] over them is a 4 x 32 by 32 x 8
// product, lane l computing the entry (l >> 3, l & 7) from the F rows in shared
// memory (4 stores, 8 broadcast 16-byte reads) and its own G row in registers,
// and adding it with one FP64 reduction. One round serves three quarters of the
// crossings, two most others (a warp that straddles a cell plane). Storing every
// lane's 28 products and summing columns, as an earlier form did, moved five
// times the shared-memory data.
template <int NR, class PT>
__device__ __forceinline__ void flush_points(double* __restrict__ grad, PT P0, PT Da, PT Db, const float* F, bool part,
                                             const float4 row[8], float* __restrict__ sm)
{
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int mr = lane >> 3, mc = lane & 7;
    unsigned todo = __ballot_sync(FULL, part);
    while (todo) {
        const int lead = __ffs(todo) - 1;
        const PT k0 = __shfl_sync(FULL, P0, lead);
        const PT ka = NR == 4 ? __shfl_sync(FULL, Da, lead) : 0, kb = NR == 4 ? __shfl_sync(FULL, Db, lead) : 0;
        const bool in = (todo >> lane & 1) && P0 == k0 && (NR == 1 || (Da == ka && Db == kb));
        todo &= ~__ballot_sync(FULL, in);
        __syncwarp();
#pragma unroll
        for (int r = 0; r < NR; ++r) sm[r * kRow + lane] = in ? F[r] : 0.f;
        __syncwarp();
        if (NR == 4 || mr == 0) {
            float2 x = make_float2(0.f, 0.f), y = make_float2(0.f, 0.f);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const float4 f = *reinterpret_cast<const float4*>(sm + mr * kRow + 4 * i);
                x = __ffma2_rn(make_float2(f.x, f.y), make_float2(row[i].x, row[i].y), x);
                y = __ffma2_rn(make_float2(f.z, f.w), make_float2(row[i].z, row[i].w), y);
            }
            const float v = (x.x + y.x) + (x.y + y.y);
            const PT key = k0 + ((mr & 1) ? ka : 0) + ((mr & 2) ? kb : 0);
            if (mc < 7 && v != 0.f) atomicAdd(grad + 8 * (size_t)key + mc, (double)v);
        }
    }
}

// Adjoint of one sub-step (B.first + blockIdx.x % pieces) of one step: replays the walk and, for
// every point the ray's segments read (the 8 vertices of each cell, or its
// centre), accumulates dI/dq of the segment integrals (the transpose of the
// forward map) while the point stays in the ray's current cell; a point is
// flushed into the gradient records once per residency.
//
// The sub-steps are independent (each starts from its own float-float point and
// the records take sums), so each is a thread of its own: a small bundle fills
// the GPU by shorter ones. The lanes of a warp stay together to the warp's last
// crossing, those that are done adding nothing: every flush is one of a whole
// warp. Consecutive blocks are the sub-steps of one ray tile: the first sub-steps
// of all rays add to the few points around the observer, and run together
// (sub-step slowest) they queued for those points' L2 lines, for a time that
// depended on where the records lay in memory (3.25 to 3.63 ms; now 3.00 ms).
// Bound by issue slots and the shared-memory round trip of the flush (FP64 and L2
// atomics below 21 %); 4 blocks per SM, 5 are 4 % slower. One step of 256 cells,
// 1024^2 rays: backward 5.39 -> 3.00 ms; two steps of 32 cells, 96^2 rays: 287 ->
// 58 us.
template <int INTERP, class R, bool PER, class PT>
__global__ void __launch_bounds__(32 * kAdjWarps, (INTERP == RR_TRILINEAR && sizeof(R) == 4) ? 4 : 1)
    trace_adjoint_kernel(const TraceArgs A, const AdjArgs B, const TileCfg tc)
{
    constexpr bool F64 = sizeof(R) == 8;
    constexpr bool TRI = INTERP == RR_TRILINEAR;
    constexpr unsigned FULL = 0xffffffffu;
    __shared__ __align__(16) float stage[kAdjWarps * 8 * kRow];
    float* sm = stage + (threadIdx.x >> 5) * 8 * kRow;
    int ix, iy;
    const int pieces = gridDim.x / B.tiles_x;
    tile_ray(tc, blockIdx.x / pieces, blockIdx.y, ix, iy);
    const bool ray = ix < A.nx && iy < A.ny;
    const long long rid = ray ? (long long)iy * A.nx + ix : 0;
    const float gk = ray && B.dkappa ? (float)(B.dkappa[rid] * B.kscale) : 0.f;
    const float gb = ray && B.dkborn ? (float)(B.dkborn[rid] * B.bscale) : 0.f;
    bool alive = ray && (gk != 0.f || gb != 0.f);
    RayRange rg;
    if (alive && !ray_range<PER>(A, rid, rg)) alive = false;
    const int j = B.first + blockIdx.x % pieces;
    int nsub = 1;
    float dsub = 0.f;
    if (!F64 && alive) {
        nsub = PER ? A.nsub : max(1, (int)ceilf(rg.Lf / A.sub_len));
        dsub = PER ? A.dsub : rg.Lf / (float)nsub;
    }
    if (j >= nsub) alive = false;
    if (!__any_sync(FULL, alive)) return;
    const bool odd = alive && !(isfinite(gk) && isfinite(gb));   // adds on its own (add_alone)
    const bool any_odd = __any_sync(FULL, odd);
    const int nn[3] = {A.n0, A.n1, A.n2};
    const R chis = (R)A.chi_s;
    const R ichis = F64 ? (R)(1.0 / A.chi_s) : (R)A.inv_chi_s_f;
    const R eps_rel = F64 ? (R)1.4551915228366852e-11 : (R)4.76837158203125e-07;
    const PT st[3] = {(PT)A.n1 * (PT)A.n2, (PT)A.n2, 1};
    Walk<R> W;
    // point index of the cell's entry corner (vertex vlo on every axis) and the
    // index step from vlo to vhi per axis (periodic wrap included), modulo 2^32
    // for grids of at most 2^32 points and modulo 2^64 for larger ones (PT); NGP:
    // the cell's index
    PT P0 = 0, D[3] = {0, 0, 0};
    if (alive) {
        float bh, bl, Lj, D0j;
        sub_step(rg, j, nsub, dsub, bh, bl, Lj, D0j);
        walk_setup<R>(A, rid, bh, bl, Lj, D0j, rg.hi, rg.lo, W);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            P0 += (PT)(TRI ? W.vlo[a] : W.c[a]) * st[a];
            D[a] = (PT)(W.vhi[a] - W.vlo[a]) * st[a];
        }
    }
    float4 row[8];
    {
        const bool sum = alive && !odd;
        const float G[7] = {sum ? gk * W.w[0] : 0.f, sum ? gk * W.w[1] : 0.f, sum ? gk * W.w[2] : 0.f,
                            sum ? gk * W.w[3] : 0.f, sum ? gk * W.w[4] : 0.f, sum ? gk * W.w[5] : 0.f,
                            sum ? gb : 0.f};
        load_factors(G, sm, row);
    }
    const bool work = alive;
    // a face (or cell) of this ray into the records, with the warp
    auto flush = [&](PT P, PT Da, PT Db, const float* F, bool part) {
        constexpr int NR = TRI ? 4 : 1;
        flush_points<NR, PT>(B.grad, P, Da, Db, F, part && !odd, row, sm);
        if (any_odd && odd && part)
            add_alone<PT>(B.grad, A.dirh[rid], B.dkappa ? (float)(B.dkappa[rid] * B.kscale) : 0.f,
                      B.dkborn ? (float)(B.dkborn[rid] * B.bscale) : 0.f, NR, P, Da, Db, F[0], F[TRI ? 1 : 0],
                      F[TRI ? 2 : 0], F[TRI ? 3 : 0]);
        __syncwarp();
    };
    const R L = W.L, chiA0 = W.chiA0, D0 = W.D0;
    const R eps_end = L * eps_rel;
    float S[TRI ? 8 : 1] = {0.f};
    R sig = 0;
    R T[3] = {W.T0[0], W.T0[1], W.T0[2]};
    R kf[3] = {(R)0, (R)0, (R)0};   // crossings so far
    int left = alive ? W.max_iter : 0;
    bool overflow = false;
    while (true) {
        bool e1 = false, e2 = false, cross = false;
        if (alive) {
            const bool p1 = T[1] < T[0];
            const R t01 = p1 ? T[1] : T[0];
            e2 = T[2] < t01;
            e1 = !e2 && p1;
            R tend = e2 ? T[2] : t01;
            cross = tend < L - eps_end;
            if (!cross) tend = L;
            const R t = tend - sig;
            if (t > tend * eps_rel) {
                R u[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) u[a] = fmin(fmax(fma(sig - T[a], W.v[a], W.cu[a]), (R)0), (R)1);
                const R chiA = chiA0 - sig;
                const R G0 = (D0 + sig) * chiA * ichis;
                const R G1 = (2 * chiA - chis) * ichis;
                const R G2 = -ichis;
                const R t2 = t * t;
                const R J1 = t * (G0 + t * (G1 * (R)0.5 + t * G2 * (R)(1.0 / 3.0)));
                if constexpr (TRI) {
                    const float J[4] = {(float)J1,
                                        (float)(t2 * (G0 * (R)0.5 + t * (G1 * (R)(1.0 / 3.0) + t * G2 * (R)0.25))),
                                        (float)(t2 * t * (G0 * (R)(1.0 / 3.0) + t * (G1 * (R)0.25 + t * G2 * (R)0.2))),
                                        (float)(t2 * t2 * (G0 * (R)0.25 + t * (G1 * (R)0.2 + t * G2 * (R)(1.0 / 6.0))))};
                    float Wm[8];
                    line_cubic_adjoint(J, (float)u[0], (float)u[1], (float)u[2], (float)W.v[0], (float)W.v[1],
                                       (float)W.v[2], Wm);
#pragma unroll
                    for (int m = 0; m < 8; ++m) S[m] += Wm[m];
                } else {
                    S[0] += (float)J1;
                }
            }
            sig = tend;
        }
        if (!__any_sync(FULL, cross)) break;
        const bool e0 = !e1 && !e2;
        if constexpr (TRI) {
            // the 4 corners on the entry face along e leave the ray's cell:
            // corner m of the cell has bit a set when it lies on vhi along
            // axis a; r = 0..3 runs over the face's corners, the first of
            // the two other axes (a < b) as bit 0
            const float F[4] = {S[0], e0 ? S[2] : S[1], e2 ? S[2] : S[4], e0 ? S[6] : (e1 ? S[5] : S[3])};
            flush(P0, e0 ? D[1] : D[0], e2 ? D[1] : D[2], F, cross);
            // the exit face's sums become the entry face's
            if (cross) {
                const float s1 = S[1], s2 = S[2], s3 = S[3], s4 = S[4], s5 = S[5], s6 = S[6], s7 = S[7];
                S[0] = e0 ? s1 : (e1 ? s2 : s4);
                S[1] = e0 ? 0.f : (e1 ? s3 : s5);
                S[2] = e0 ? s3 : (e1 ? 0.f : s6);
                S[3] = e2 ? s7 : 0.f;
                S[4] = e0 ? s5 : (e1 ? s6 : 0.f);
                S[5] = e1 ? s7 : 0.f;
                S[6] = e0 ? s7 : 0.f;
                S[7] = 0.f;
            }
        } else {
            flush(P0, 0, 0, S, cross);
            if (cross) S[0] = 0.f;
        }
        alive = cross;
        if (cross) {
#pragma unroll
            for (int a = 0; a < 3; ++a)
                if (a == 0 ? e0 : (a == 1 ? e1 : e2)) {
                    if (!TRI || !PER) {
                        const int ncell = W.c[a] + W.sgn[a], nc = wrap_once(ncell, nn[a]);
                        // the ray leaves the box (no wrap): what is pending is flushed below
                        if (!PER && !A.periodic && (ncell < 0 || ncell >= nn[a])) alive = false;
                        if constexpr (!TRI) P0 += (PT)(nc - W.c[a]) * st[a];
                        W.c[a] = nc;
                    }
                    if constexpr (TRI) {
                        const int nvhi = wrap_once(W.vhi[a] + W.sgn[a], nn[a]);
                        P0 += D[a];
                        D[a] = (PT)(nvhi - W.vhi[a]) * st[a];
                        W.vhi[a] = nvhi;
                    }
                    kf[a] += (R)1;
                    T[a] = fma(kf[a], W.td[a], W.T0[a]);
                }
            if (--left < 0) {
                overflow = true;
                alive = false;
            }
        }
    }
    // flush everything still pending
    if constexpr (TRI) {
        const float lo[4] = {S[0], S[1], S[2], S[3]}, hi[4] = {S[4], S[5], S[6], S[7]};
        flush(P0, D[0], D[1], lo, work);
        flush(P0 + D[2], D[0], D[1], hi, work);
    } else {
        flush(P0, 0, 0, S, work);
    }
    if (overflow) atomicOr(A.err, kErrStepLimit);
}

using AdjKernel = void (*)(const TraceArgs, const AdjArgs, const TileCfg);

template <int INTERP, class R>
AdjKernel adj_kernel(const TraceArgs& a)
{
    // (64-bit point indices: one kernel for periodic and bounded grids)
    if ((long long)a.n0 * a.n1 * a.n2 > (1LL << 32)) return trace_adjoint_kernel<INTERP, R, false, unsigned long long>;
    return a.periodic ? trace_adjoint_kernel<INTERP, R, true, uint32_t> : trace_adjoint_kernel<INTERP, R, false, uint32_t>;
}

}  // namespace

cudaError_t launch_trace_adjoint(const TraceArgs& args, const AdjArgs& b, int interp, bool fp64_dda, cudaStream_t s)
{
    const TileCfg t{};
    dim3 grid = tile_grid(t, args.nx, args.ny);
    const int nt = 32 * t.bwx * t.bwy;
    if (nt > 32 * kAdjWarps) return cudaErrorInvalidConfiguration;   // the staging area holds kAdjWarps warps
    TraceArgs a = args;
    if (!fp64_dda) {
        // sub-steps of the forward walk's length (32 cells) where these give
        // every SM sub-partition 8 warps; shorter ones, of 4 cells at least, for
        // smaller bundles, which a few serial walks leave mostly idle
        const long long warps = (long long)grid.x * grid.y * kAdjWarps;
        int dev = 0, sms = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        const long long want = (sms > 0 ? sms : 1) * 4LL * 8;
        const float longest = a.sub_len, shortest = longest * (4.f / 32.f);
        float len = longest;
        if (warps * a.nsub < want) {
            const float pieces = (float)((want + warps - 1) / warps);
            len = fminf(longest, fmaxf(shortest, a.Lf / pieces));
        }
        a.sub_len = len;
        a.nsub = (int)fmaxf(1.f, fminf(ceilf(a.Lf / len), 1e9f));
        a.dsub = a.Lf / (float)a.nsub;
    }
    AdjKernel k;
    if (interp == RR_TRILINEAR) k = fp64_dda ? adj_kernel<RR_TRILINEAR, double>(a) : adj_kernel<RR_TRILINEAR, float>(a);
    else k = fp64_dda ? adj_kernel<RR_NGP, double>(a) : adj_kernel<RR_NGP, float>(a);
    const int pieces = fp64_dda ? 1 : a.nsub;
    AdjArgs g = b;
    g.tiles_x = (int)grid.x;
    const int most = 0x7fffffff / g.tiles_x;   // sub-steps in a launch (grid.x < 2^31)
    for (int done = 0, n; done < pieces; done += n) {
        n = pieces - done < most ? pieces - done : most;
        g.first = done;
        grid.x = (unsigned)(g.tiles_x * n);
        k<<<grid, nt, 0, s>>>(a, g, t);
    }
    return cudaGetLastError();
}

}  // namespace rr
