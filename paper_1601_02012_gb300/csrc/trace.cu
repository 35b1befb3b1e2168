// Cell-by-cell line-of-sight integration over one step (Secs. 2.5-2.6, 3.2).
//
// One thread owns one ray; a warp owns an 8 x 4 tile of neighbouring pixels,
// so that its rays sit in the same or adjacent cells at every chi and the
// record gathers of a warp mostly hit the same 128-byte lines (served by L1).
//
// Per ray and step:
//  * Setup: the start point obs + chi_a n (Eq. raypos) and its cell. In the
//    FP32 form this is float-float arithmetic (chi_a, n, obs and 1/h carried
//    as pairs of floats, ~2^-46 relative), because GB300 issues FP64 at a
//    small fraction of the FP32 rate; the plain form uses FP64. The distances
//    from the start point to the cell's two faces on each axis are both
//    obtained with full relative precision.
//  * The walk runs in cell-local "mirrored" coordinates u_a in [0, 1] that
//    grow along the motion (-n). The path to the k-th face crossing on axis a
//    is T0_a + k td_a (one rounding, no drift); the nearest crossing picks the
//    exit face (the exit-plane rule of Sec. 2.5.1, Eq. disttocross), ties go
//    to the lowest axis. The step ends when the path reaches chi_a - chi_b.
//  * Trilinear mode keeps the projected values of the cell's 8 vertices in
//    registers; crossing a face keeps the 4 shared vertices and gathers the 4
//    new ones (2 x 16-byte loads each), issued before the current segment's
//    arithmetic.
//  * Along the segment, chi = chi_A - s for s in [0, t]; the trilinear field
//    restricted to the line is a cubic in s (the d_N of Appendix B, written
//    about the entry point) and the lensing kernel is the quadratic
//    g(chi_A - s); the segment integral (Eq. Iclensing) is the exact
//    sum_N e_N J_N with J_N = int_0^t g(chi_A - s) s^(N-1) ds.
//  * Sums over the segments of a step are compensated FP32 (Kahan); the step
//    total times the step's scale is added to the ray's float-float
//    accumulator (~48 bits).
#include <type_traits>

#include "walk.cuh"

namespace rr {
namespace {

// Crossing face e of the mirrored cell: the 4 corners on the exit side become
// the entry side and the 4 new corner values p come in on the exit side, slot
// by slot as selects on e (e0: e = 0, e1: e = 1): the rays of a warp rarely
// cross the same face at the same iteration, and branches would diverge (2 %
// slower on the production pass).
__device__ __forceinline__ void shift_corners(float2 q[8], const float2 p[4], bool e0, bool e1)
{
    const bool e2 = !e0 && !e1;
    float2 n[8];
    n[0] = e2 ? q[4] : (e1 ? q[2] : q[1]);
    n[1] = e2 ? q[5] : (e1 ? q[3] : p[0]);
    n[2] = e2 ? q[6] : (e1 ? p[0] : q[3]);
    n[3] = e2 ? q[7] : p[1];
    n[4] = e2 ? p[0] : (e1 ? q[6] : q[5]);
    n[5] = e2 ? p[1] : (e1 ? q[7] : p[2]);
    n[6] = e0 ? q[7] : p[2];
    n[7] = p[3];
#pragma unroll
    for (int i = 0; i < 8; ++i) q[i] = n[i];
}

// a shared-memory read that the compiler neither hoists nor merges
__device__ __forceinline__ float4 lds_again(unsigned a)
{
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
    return v;
}

// (gamma1, gamma2) of N records. The twelve weights are read again for each
// crossing (three 16-byte reads) instead of holding registers through the
// segment's arithmetic, where they spilled (228 -> 116 bytes; 256^3, 1024^2 rays,
// 20 steps: 4.36 -> 4.21 ms).
template <int N>
__device__ __forceinline__ void shear_pairs(unsigned sw, const Rec* r, float2* g)
{
    const float4 a = lds_again(sw), b = lds_again(sw + 16 * NT_MAX), c = lds_again(sw + 32 * NT_MAX);
    const float w1[6] = {a.x, a.y, a.z, a.w, b.x, b.y}, w2[6] = {b.z, b.w, c.x, c.y, c.z, c.w};
#pragma unroll
    for (int i = 0; i < N; ++i) g[i] = make_float2(project(w1, r[i]), project(w2, r[i]));
}

// What the sub-steps of one ray's step accumulate and hand on.
template <class R>
struct PieceState {
    // per-step sums of (kappa, Born kappa): packed Kahan pairs (FP32) or FP64
    Acc2 s2;
    Acc2 s2m;   // moments form: the B moments; shear form: (gamma1, gamma2)
    Acc<R> sk, sb;
    // Method A: n . grad Phi and g at the start and at the end of the interval
    float qa = 0.f, ga = 0.f, qb = 0.f, gb = 0.f;
    uint32_t cnt = 0;
    int pc0 = -1, pc1 = -1, pc2 = -1;   // cell where the previous sub-step ended
    bool overflow = false;
};

// The form's own per-ray constants.
struct RayWeights {
    unsigned sw;          // shear form: the Q weights of gamma1, gamma2 in shared memory
    float4 nd;            // Method A: the direction, for n . grad Phi
};

template <int FORM>
__device__ __forceinline__ void ray_weights(const TraceArgs& A, long long rid, RayWeights& V)
{
    if constexpr (FORM == kFormShear) {
        __shared__ float4 sw[3 * NT_MAX];
        float w1[6], w2[6];
        shear_weights(A.dirh[rid], w1, w2);
        sw[threadIdx.x] = make_float4(w1[0], w1[1], w1[2], w1[3]);
        sw[NT_MAX + threadIdx.x] = make_float4(w1[4], w1[5], w2[0], w2[1]);
        sw[2 * NT_MAX + threadIdx.x] = make_float4(w2[2], w2[3], w2[4], w2[5]);
        V.sw = (unsigned)__cvta_generic_to_shared(sw + threadIdx.x);
    }
    if constexpr (FORM == kFormMethodA) V.nd = A.dirh[rid];
}

// The FP32 walk's slivers, in units of the path: 4 ulp (see walk_piece).
constexpr float kSliver = 4.76837158203125e-07f;

// One ray over one step. INTERP: RR_NGP or RR_TRILINEAR. R: float
// (compensated FP32 walk) or double (plain FP64 walk). FORM (FP32 only):
// kFormKahan (default), kFormPlain (uncompensated FP32 sums within and across
// steps, for comparison), kFormMoments (the moments A = int chi Q and
// B = int chi^2 Q of Eq. Isources instead of kappa: the kernel g becomes chi
// and chi^2, i.e. (G0, G1, G2) = (chi_A, -1, 0) and (chi_A^2, -2 chi_A, 1)) or
// kFormShear (kappa and Born kappa, and the shear pair (gamma1, gamma2) of Eqs.
// gamma1, gamma2 from a second projection of the same records, carried as a
// second packed pair through the same segments) or kFormMethodA (Method A,
// Eq. kappa2, on gradient records {grad Phi, delta}: the first channel
// integrates n . grad Phi with the kernel dg/dchi and adds the step's surface
// terms -g n.grad Phi at the start and +g n.grad Phi at the end of the traced
// interval (Eq. 2nterm); the second is the Born term as in the other forms) or
// kFormGeneric (two scalar fields from float2 records, each with its own
// quadratic kernel K(chi): the generic integrals of Eqs. Ic, Icfinal).
// ADDR: how the trilinear walk addresses its records.
//  kAddrIndex:  vertex indices per axis, with periodic wrap (any grid).
//  kAddrPlanes: the 64-bit record offsets of the mirrored cell's two vertex
//               planes per axis (entry and exit side), with wrap, so that a
//               record's offset is two additions: the FP64 walk's. (In FP32,
//               one step through 8 periods of 24^3: 1014 us, by indices 960.)
//  kAddrAuto:   kAddrFlat for the sub-steps whose own cells and vertex planes
//               lie inside the grid without a wrap (counted exactly as the walk
//               will cross them, so a ray that ends on the box face z = 0 still
//               qualifies), up to the first that does not; the ray's rest out
//               of line, its outside sub-steps by kAddrIndex. Whole-grid records
//               of steps the host cannot clear: steps that reach the observer
//               on the box face, bounded boxes, batches. Grids of fewer than
//               2^31 points. (One step of 1024^2 rays through 256 cells down to
//               z = 0: 3.13 ms by vertex planes, 2.35 ms; a batch of 16 cones
//               12.30 ms by vertex indices, 9.20 ms. With both loops in one
//               function, or a call inside the sub-steps' loop, the rare path's
//               registers spill into the common one: 2.45 to 2.68 ms.)
//  kAddrFlat:   no wrap: a 32-bit point index B of the mirrored cell's entry
//               corner and a constant signed stride d_a per axis (the next
//               vertex plane along the motion), so the 8 corners are B plus
//               sums of the d_a and a crossing of face e is B += d_e. Valid
//               when no ray of the step comes within a cell of the periodic
//               seam and the grid has fewer than 2^31 points: the host checks
//               the step's footprint box; each sub-step checks its own cell
//               range first and, outside it, flags kErrRange and reads nothing.
template <int INTERP, class R, int FORM, int ADDR>
__device__ __forceinline__ void walk_piece(const TraceArgs& A, const float4* rec, Walk<R>& W, const RayWeights& V,
                                           int j, bool resume, PieceState<R>& S)
{
    using OT = unsigned long long;
    constexpr bool PLANES = ADDR == kAddrPlanes;
    constexpr bool F64 = sizeof(R) == 8;
    constexpr bool SH = !F64 && FORM == kFormShear;
    constexpr bool MA = !F64 && FORM == kFormMethodA;
    constexpr bool GEN = !F64 && FORM == kFormGeneric;
    // one record per point: 2 float4 of the tidal tensor, 1 gradient float4
    // (Method A) or a float2 scalar pair (generic form)
    using PR = typename std::conditional<MA, float4, typename std::conditional<GEN, float2, Rec>::type>::type;
    const int nn[3] = {A.n0, A.n1, A.n2};
    const long long sx = (long long)A.n1 * A.n2, sy = A.n2;
    const R chis = (R)A.chi_s;
    const R ichis = F64 ? (R)(1.0 / A.chi_s) : (R)A.inv_chi_s_f;
    int* c = W.c;
    const int* sgn = W.sgn;
    int* k = W.k;
    // offsets of the entry-side (plo) and exit-side (phi) vertex planes per
    // axis (PLANES), or the vertex indices themselves
    const OT st[3] = {(OT)A.n1 * (OT)A.n2, (OT)A.n2, (OT)1};
    OT plo[3], phi[3];
    int* vlo = W.vlo;
    int* vhi = W.vhi;
    if constexpr (PLANES) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            plo[a] = (OT)vlo[a] * st[a];
            phi[a] = (OT)vhi[a] * st[a];
        }
    }
    const R* T0 = W.T0;
    const R* td = W.td;
    const R* v = W.v;
    const R* cu = W.cu;
    const float* w = W.w;
    const R L = W.L, chiA0 = W.chiA0, D0 = W.D0;
    // Crossings closer together than the walk resolves are one crossing: a
    // crossing within eps_rel * L of the step's end, and a segment shorter
    // than eps_rel * (its end), are rounding slivers at an edge or corner the
    // ray passes through; they are neither integrated nor counted. FP32: 4 ulp
    // of the path. FP64: 2^-36, above the error the FP64 start point carries
    // into a crossing distance (ulp(|p|) / |n_a|) for rays 1e-4 rad off an axis.
    const R eps_rel = F64 ? (R)1.4551915228366852e-11 : (R)kSliver;
    const R eps_end = L * eps_rel;
    const int max_iter = W.max_iter;
    auto fetch = [&](long long i) -> PR {
        if constexpr (MA) return load_grad_rec(rec, i);
        else if constexpr (GEN) return __ldg(reinterpret_cast<const float2*>(rec) + i);
        else return load_rec(rec, i);
    };
    // (the channel pair the walk integrates) of a record
    auto pair = [&](const PR& r) -> float2 {
        if constexpr (MA) return radial_pair(V.nd, r);
        else if constexpr (GEN) return r;
        else return make_float2(project(w, r), r.b.z);
    };
    int iter = 0;

    // Field cache: (projected kappa value, delta) at the 8 mirrored corners
    // (trilinear) or at the cell centre (NGP); the shear form also keeps
    // (gamma1, gamma2) values there.
    float2 q2[8];
    float2 g2[SH ? 8 : 1];
    if (INTERP == RR_TRILINEAR) {
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            long long o;
            if constexpr (PLANES) {
                o = (long long)(((m & 1) ? phi[0] : plo[0]) + ((m & 2) ? phi[1] : plo[1]) +
                                ((m & 4) ? phi[2] : plo[2]));
            } else {
                const int gx = (m & 1) ? vhi[0] : vlo[0];
                const int gy = (m & 2) ? vhi[1] : vlo[1];
                const int gz = (m & 4) ? vhi[2] : vlo[2];
                o = gx * sx + gy * sy + gz;
            }
            const PR r = fetch(o);
            q2[m] = pair(r);
            if constexpr (SH) shear_pairs<1>(V.sw, &r, &g2[m]);
        }
    } else {
        const PR r = fetch(c[0] * sx + c[1] * sy + c[2]);
        q2[0] = pair(r);
        if constexpr (SH) shear_pairs<1>(V.sw, &r, &g2[0]);
    }

    // (a resumed first segment is not a new one; it is integrated below unless
    // the walk starts on its exit face)
    if (resume && T0[0] > (R)0 && T0[1] > (R)0 && T0[2] > (R)0) --S.cnt;
    R sig = 0;                       // path from the sub-step start to the segment entry
    R T[3] = {T0[0], T0[1], T0[2]};  // path to the next face crossing per axis
    while (true) {
        // exit plane: the nearest face crossing (lowest axis on ties)
        R tend = T[0];
        int e = 0;
        if (T[1] < tend) { tend = T[1]; e = 1; }
        if (T[2] < tend) { tend = T[2]; e = 2; }
        const bool last = !(tend < L - eps_end);
        if (last) tend = L;
        const R t = tend - sig;
        // mirrored entry point of this segment
        R u[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            u[a] = fmin(fmax(fma(sig - T[a], v[a], cu[a]), (R)0), (R)1);
        }

        // Prefetch the next cell's new records before this segment's arithmetic.
        // (register arrays are indexed only through unrolled loops, never by e)
        int ncell = 0, ne = 1;
        OT nph = 0;     // offset of the vertex plane beyond the exit face (PLANES)
        int nvhi = 0;   // its vertex index (otherwise)
        PR nr[4];
        if (!last) {
#pragma unroll
            for (int a = 0; a < 3; ++a)
                if (a == e) {
                    ncell = c[a] + sgn[a];
                    ne = nn[a];
                    // the exit-side plane one vertex further along the motion, with wrap
                    if constexpr (PLANES) {
                        const OT span = st[a] * (OT)nn[a];
                        if (sgn[a] > 0) nph = phi[a] + st[a] == span ? (OT)0 : phi[a] + st[a];
                        else nph = phi[a] == 0 ? span - st[a] : phi[a] - st[a];
                    } else {
                        nvhi = wrap_once(vhi[a] + sgn[a], nn[a]);
                    }
                }
            if (INTERP == RR_TRILINEAR) {
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const int pb = r & 1, qb2 = r >> 1;
                    if constexpr (PLANES) {
                        const OT ox = e == 0 ? nph : (pb ? phi[0] : plo[0]);
                        const OT oy = e == 1 ? nph : (e == 0 ? (pb ? phi[1] : plo[1]) : (qb2 ? phi[1] : plo[1]));
                        const OT oz = e == 2 ? nph : (qb2 ? phi[2] : plo[2]);
                        nr[r] = fetch((long long)(ox + oy + oz));
                    } else {
                        const int gx = e == 0 ? nvhi : (pb ? vhi[0] : vlo[0]);
                        const int gy = e == 1 ? nvhi : (e == 0 ? (pb ? vhi[1] : vlo[1]) : (qb2 ? vhi[1] : vlo[1]));
                        const int gz = e == 2 ? nvhi : (qb2 ? vhi[2] : vlo[2]);
                        nr[r] = fetch(gx * sx + gy * sy + gz);
                    }
                }
            } else {
                const int cx = e == 0 ? wrap_once(ncell, nn[0]) : c[0];
                const int cy = e == 1 ? wrap_once(ncell, nn[1]) : c[1];
                const int cz = e == 2 ? wrap_once(ncell, nn[2]) : c[2];
                nr[0] = fetch(cx * sx + cy * sy + cz);
            }
        }
        if constexpr (MA) {
            // the surface terms of Eq. (2nterm): n . grad Phi and g at the start
            // of the traced interval (the first segment's entry) and at its end
            // (the exit of the segment that ends the interval: the last one,
            // or, without wrap, the one leaving the box)
            if (j == 0 && iter == 0) {
                S.qa = INTERP == RR_TRILINEAR ? trilinear_x(q2, u[0], u[1], u[2]) : q2[0].x;
                S.ga = D0 * chiA0 * ichis;
            }
            if (last || (!A.periodic && (ncell < 0 || ncell >= ne))) {
                if (INTERP == RR_TRILINEAR) {
                    float ue[3];
#pragma unroll
                    for (int a = 0; a < 3; ++a) ue[a] = fminf(fmaxf(fmaf(t, v[a], u[a]), 0.f), 1.f);
                    S.qb = trilinear_x(q2, ue[0], ue[1], ue[2]);
                } else {
                    S.qb = q2[0].x;
                }
                float G0, G1, G2;
                kernel_coeffs(t, sig, chiA0, D0, chis, ichis, G0, G1, G2);
                S.gb = fmaf(t, fmaf(t, G2, G1), G0);
            }
        }

        if (t > tend * eps_rel) {
            if constexpr (!F64 && FORM == kFormMoments) {
                const float chiA = chiA0 - sig;
                if (INTERP == RR_TRILINEAR) {
                    float2 e2[4];
                    line_cubic2(q2, bc2(u[0]), bc2(u[1]), bc2(u[2]), bc2(v[0]), bc2(v[1]), bc2(v[2]), e2);
                    S.s2.add(dot_kernel(e2, t, chiA, -1.f, 0.f));
                    S.s2m.add(dot_kernel(e2, t, chiA * chiA, -2.f * chiA, 1.f));
                } else {
                    S.s2.add(segment_ngp(q2[0], t, chiA, -1.f, 0.f));
                    S.s2m.add(segment_ngp(q2[0], t, chiA * chiA, -2.f * chiA, 1.f));
                }
            } else if constexpr (GEN) {
                // each channel's kernel about the entry point: K(chi_A - s) =
                // K(chi_A) - K'(chi_A) s + k2 s^2
                const float chiA = chiA0 - sig;
                const float2 G0 = make_float2(fmaf(chiA, fmaf(chiA, A.kq[2], A.kq[1]), A.kq[0]),
                                              fmaf(chiA, fmaf(chiA, A.kq[5], A.kq[4]), A.kq[3]));
                const float2 G1 = make_float2(-fmaf(2.f * A.kq[2], chiA, A.kq[1]), -fmaf(2.f * A.kq[5], chiA, A.kq[4]));
                const float2 G2 = make_float2(A.kq[2], A.kq[5]);
                if (INTERP == RR_TRILINEAR) {
                    float2 e2[4];
                    line_cubic2(q2, bc2(u[0]), bc2(u[1]), bc2(u[2]), bc2(v[0]), bc2(v[1]), bc2(v[2]), e2);
                    S.s2.add(dot_kernel_pair(e2, t, G0, G1, G2));
                } else {
                    const float2 tt = bc2(t);
                    const float2 J1 = __fmul2_rn(tt, __ffma2_rn(tt, __ffma2_rn(tt, __fmul2_rn(G2, bc2(1.f / 3.f)),
                                                                              __fmul2_rn(G1, bc2(0.5f))), G0));
                    S.s2.add(__fmul2_rn(q2[0], J1));
                }
            } else if constexpr (MA) {
                float G0, G1, G2;
                kernel_coeffs(t, sig, chiA0, D0, chis, ichis, G0, G1, G2);
                S.s2.add(INTERP == RR_TRILINEAR
                           ? segment_trilinear_a(q2, u[0], u[1], u[2], v[0], v[1], v[2], t, G0, G1, G2)
                           : segment_ngp_a(q2[0], t, G0, G1, G2));
            } else if constexpr (!F64) {
                float G0, G1, G2;
                kernel_coeffs(t, sig, chiA0, D0, chis, ichis, G0, G1, G2);
                const float2 x = INTERP == RR_TRILINEAR
                                     ? segment_trilinear(q2, u[0], u[1], u[2], v[0], v[1], v[2], t, G0, G1, G2)
                                     : segment_ngp(q2[0], t, G0, G1, G2);
                if constexpr (FORM == kFormPlain) S.s2.s = __fadd2_rn(S.s2.s, x);
                else S.s2.add(x);
                if constexpr (SH)
                    S.s2m.add(INTERP == RR_TRILINEAR
                                ? segment_trilinear(g2, u[0], u[1], u[2], v[0], v[1], v[2], t, G0, G1, G2)
                                : segment_ngp(g2[0], t, G0, G1, G2));
            } else {
                // lensing kernel g(chi_A - s) = G0 + G1 s + G2 s^2 about the entry
                // point; J_N and the sums rounded as written (the single-launch and
                // the batch kernels must give the same values)
                const double chiA = chiA0 - sig;
                const double G0 = (D0 + sig) * chiA * ichis;
                const double G1 = __dmul_rn(__fma_rn(2.0, chiA, -(double)chis), ichis);
                const double G2 = -ichis;
                const double t2 = __dmul_rn(t, t);
                const double tn[4] = {t, t2, __dmul_rn(t2, t), __dmul_rn(t2, t2)};
                const double ca[4] = {1.0, 0.5, 1.0 / 3.0, 0.25};
                const double cb[4] = {0.5, 1.0 / 3.0, 0.25, 0.2};
                const double cc[4] = {1.0 / 3.0, 0.25, 0.2, 1.0 / 6.0};
                double J[4];
#pragma unroll
                for (int n = 0; n < 4; ++n)
                    J[n] = __dmul_rn(tn[n], __fma_rn(t, __fma_rn(t, __dmul_rn(G2, cc[n]), __dmul_rn(G1, cb[n])),
                                                   __dmul_rn(G0, ca[n])));
                if (INTERP == RR_TRILINEAR) {
                    float2 e2[4];
                    line_cubic2(q2, bc2((float)u[0]), bc2((float)u[1]), bc2((float)u[2]), bc2((float)v[0]),
                                bc2((float)v[1]), bc2((float)v[2]), e2);
                    double xk = __dmul_rn((double)e2[0].x, J[0]), xb = __dmul_rn((double)e2[0].y, J[0]);
#pragma unroll
                    for (int n = 1; n < 4; ++n) {
                        xk = __fma_rn((double)e2[n].x, J[n], xk);
                        xb = __fma_rn((double)e2[n].y, J[n], xb);
                    }
                    S.sk.add((R)xk);
                    S.sb.add((R)xb);
                } else {
                    S.sk.add((R)__dmul_rn((double)q2[0].x, J[0]));
                    S.sb.add((R)__dmul_rn((double)q2[0].y, J[0]));
                }
            }
            ++S.cnt;
        }
        sig = tend;
        if (last) break;

        // cross the exit face e
        if (!A.periodic && (ncell < 0 || ncell >= ne)) break;
#pragma unroll
        for (int a = 0; a < 3; ++a)
            if (a == e) {
                c[a] = wrap_once(ncell, nn[a]);
                if constexpr (PLANES) {
                    plo[a] = phi[a];
                    phi[a] = nph;
                } else {
                    vlo[a] = vhi[a];
                    vhi[a] = nvhi;
                }
                k[a] += 1;
                if constexpr (F64) T[a] = fma((R)k[a], td[a], T0[a]);
                else T[a] = fmaf(i2f_exact(k[a]), td[a], T0[a]);
            }
        if (INTERP == RR_TRILINEAR) {
            float2 p2[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) p2[r] = pair(nr[r]);
            shift_corners(q2, p2, e == 0, e == 1);
            if constexpr (SH) {
#pragma unroll
                for (int r = 0; r < 4; ++r) shear_pairs<1>(V.sw, &nr[r], &p2[r]);
                shift_corners(g2, p2, e == 0, e == 1);
            }
        } else {
            q2[0] = pair(nr[0]);
            if constexpr (SH) shear_pairs<1>(V.sw, &nr[0], &g2[0]);
        }
        if (++iter > max_iter) {
            S.overflow = true;
            break;
        }
    }
    S.pc0 = c[0]; S.pc1 = c[1]; S.pc2 = c[2];
}

// The contribution of one segment of the FP32 walk (path sig .. tend of the
// sub-step, corner pairs q and, for the shear, g; NGP: the cell's own pair) to
// the step's sums;
// slivers are skipped. SELECT: by selecting the old sums afterwards instead of
// branching around the arithmetic (three control instructions a segment):
// default form 21.52 -> 21.23 ms per production pass; the shear form, with twice
// the sums, and the kernels without registers to spare keep the branch.
template <int INTERP, int FORM, bool SELECT>
__device__ __forceinline__ void add_segment(const TraceArgs& A, const Walk<float>& W, const float2* q,
                                            const float2* g, const float T[3], float sig, float tend,
                                            PieceState<float>& S)
{
    constexpr bool TRI = INTERP == RR_TRILINEAR;
    const float t = tend - sig;
    // mirrored entry point of this segment
    float u[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) u[a] = TRI ? __saturatef(fmaf(sig - T[a], W.v[a], W.cu[a])) : 0.f;
    const bool live = t > tend * kSliver;
    if (!SELECT && !live) return;
    const PieceState<float> S0 = S;
    const float chis = A.chi_sf, ichis = A.inv_chi_s_f;
    float2 e[4];
    if constexpr (TRI)
        line_cubic2(q, bc2(u[0]), bc2(u[1]), bc2(u[2]), bc2(W.v[0]), bc2(W.v[1]), bc2(W.v[2]), e);
    const float chiA = W.chiA0 - sig;
    if constexpr (FORM == kFormMoments) {
        S.s2.add(TRI ? dot_kernel(e, t, chiA, -1.f, 0.f) : segment_ngp(q[0], t, chiA, -1.f, 0.f));
        S.s2m.add(TRI ? dot_kernel(e, t, chiA * chiA, -2.f * chiA, 1.f)
                      : segment_ngp(q[0], t, chiA * chiA, -2.f * chiA, 1.f));
    } else if constexpr (FORM == kFormGeneric) {
        // each channel's kernel about the entry point: K(chi_A - s) = K(chi_A) -
        // K'(chi_A) s + k2 s^2
        const float2 G0 = make_float2(fmaf(chiA, fmaf(chiA, A.kq[2], A.kq[1]), A.kq[0]),
                                      fmaf(chiA, fmaf(chiA, A.kq[5], A.kq[4]), A.kq[3]));
        const float2 G1 = make_float2(-fmaf(2.f * A.kq[2], chiA, A.kq[1]), -fmaf(2.f * A.kq[5], chiA, A.kq[4]));
        const float2 G2 = make_float2(A.kq[2], A.kq[5]), tt = bc2(t);
        if constexpr (TRI) S.s2.add(dot_kernel_pair(e, t, G0, G1, G2));
        else
            S.s2.add(__fmul2_rn(q[0], __fmul2_rn(tt, __ffma2_rn(tt, __ffma2_rn(tt, __fmul2_rn(G2, bc2(1.f / 3.f)),
                                                                              __fmul2_rn(G1, bc2(0.5f))), G0))));
    } else {
        float G0, G1, G2;
        kernel_coeffs(t, sig, W.chiA0, W.D0, chis, ichis, G0, G1, G2);
        float2 x;
        if constexpr (TRI) x = FORM == kFormMethodA ? dot_kernel_a(e, t, G0, G1, G2) : dot_kernel(e, t, G0, G1, G2);
        else x = FORM == kFormMethodA ? segment_ngp_a(q[0], t, G0, G1, G2) : segment_ngp(q[0], t, G0, G1, G2);
        if constexpr (FORM == kFormPlain) S.s2.s = __fadd2_rn(S.s2.s, x);
        else S.s2.add(x);
        if constexpr (FORM == kFormShear)
            S.s2m.add(TRI ? segment_trilinear(g, u[0], u[1], u[2], W.v[0], W.v[1], W.v[2], t, G0, G1, G2)
                          : segment_ngp(g[0], t, G0, G1, G2));
    }
    ++S.cnt;
    if (SELECT && !live) S = S0;
}

// walk_piece with flat addressing (FP32): the same segments with the same
// arithmetic. The loop holds crossings only; the segment that ends the
// sub-step follows it, once for the whole warp, without the loads, the
// projections and the corner shift that a crossing needs, and one test ends the
// loop on the last segment and on the cap alike. Bound by issue slots and the
// FP32 pipes (FMA 60 % and ALU 42 % busy at 72 % issue, 7.0 warp instructions a
// segment); production pass, trace kernels 22.62 -> 21.52 ms without the last
// segment in the loop, 20.83 ms with one test, 20.33 ms with the ray's constants
// hoisted (kHoist), 19.72 ms with the new corners projected before the crossing's
// bookkeeping, 19.40 ms with the crossings of all axes evaluated anew and the
// shift's selects ordered by the z face, the commonest (one step of 256 cells
// 2.24 -> 2.13 ms, batch 8.91 -> 8.36 ms), and 18.70 ms (batch 8.14 ms) with
// ray_consts' test for rates whose inverse overflows, on which the loop compiles
// to 8 % fewer instructions.
// (B, D0, fd, SEAM: flat_start's; more: another sub-step follows; WIDE: a record in one 32-byte load)
template <int INTERP, int FORM, bool SELECT, bool SEAM, bool WIDE = true>
__device__ __forceinline__ void walk_flat(const TraceArgs& A, const float4* rec, const Walk<float>& W, const RayWeights& V, bool first,
                                          bool more, bool resume, int B, const int D0[3], const int fd[3],
                                          PieceState<float>& S)
{
    constexpr bool TRI = INTERP == RR_TRILINEAR;
    constexpr bool SH = FORM == kFormShear;
    constexpr bool MA = FORM == kFormMethodA;
    constexpr bool GEN = FORM == kFormGeneric;
    using PR = typename std::conditional<MA, float4, typename std::conditional<GEN, float2, Rec>::type>::type;
    auto fetch = [&](int i) -> PR {
        if constexpr (MA) return load_grad_rec(rec, (unsigned)i);
        else if constexpr (GEN) return __ldg(reinterpret_cast<const float2*>(rec) + (unsigned)i);
        else if constexpr (WIDE) return load_rec32(rec, (unsigned)i);
        else return load_rec(rec, (unsigned)i);
    };
    auto pair = [&](const PR& r) -> float2 {
        if constexpr (MA) return radial_pair(V.nd, r);
        else if constexpr (GEN) return r;
        else return make_float2(project(W.w, r), r.b.z);
    };
    constexpr int NQ = TRI ? 8 : 1;   // corners, or the cell (B: its index)
    float2 q[NQ], g[SH ? NQ : 1];
#pragma unroll
    for (int m = 0; m < NQ; ++m) {
        const PR r = fetch(B + ((m & 1) ? D0[0] : 0) + ((m & 2) ? D0[1] : 0) + ((m & 4) ? D0[2] : 0));
        q[m] = pair(r);
        if constexpr (SH) shear_pairs<1>(V.sw, &r, &g[m]);
    }
    float sig = 0.f;                          // path from the sub-step start to the segment entry
    float T[3] = {W.T0[0], W.T0[1], W.T0[2]};   // path to the next face crossing per axis
    float kf[3] = {0.f, 0.f, 0.f};            // crossings so far
    int D[3] = {D0[0], D0[1], D0[2]};         // entry to exit side of the cell (fd but for SEAM)
    const float lim = W.L - W.L * kSliver;
    int left = W.max_iter + 1;
    // (a resumed first segment is not a new one; it is integrated unless the
    // walk starts on its exit face)
    if (resume && T[0] > 0.f && T[1] > 0.f && T[2] > 0.f) --S.cnt;
    if constexpr (MA) {
        // the surface term of Eq. (2nterm) at the start of the traced interval
        if (first) {
            float u[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) u[a] = __saturatef(fmaf(sig - T[a], W.v[a], W.cu[a]));
            if constexpr (TRI) S.qa = trilinear_x(q, u[0], u[1], u[2]);
            else S.qa = q[0].x;
            S.ga = W.D0 * W.chiA0 * A.inv_chi_s_f;
        }
    }
    while (true) {
        // exit plane: the nearest face crossing (lowest axis on ties)
        const bool p1 = T[1] < T[0];
        const float t01 = fminf(T[1], T[0]);
        const bool e2 = T[2] < t01;
        const float tend = fminf(T[2], t01);
        if (!(tend < lim) | (left == 0)) break;
        --left;
        const bool e0 = !e2 && !p1, e1 = !e2 && p1;
        // the new exit-side corners, loaded ahead of this segment's arithmetic:
        // the plane beyond the exit side along e, plus 0, d_A, d_B, d_A + d_B over
        // the other two axes A < B
        const int fde = e2 ? fd[2] : (p1 ? fd[1] : fd[0]);
        const int de = SEAM ? (e2 ? D[2] : (p1 ? D[1] : D[0])) : fde;
        const int P = B + de + fde;
        const int dA = e0 ? D[1] : D[0];
        const int dB = e2 ? D[1] : D[2];
        PR r[TRI ? 4 : 1];
        if constexpr (TRI) {
            r[0] = fetch(P);
            r[1] = fetch(P + dA);
            r[2] = fetch(P + dB);
            r[3] = fetch(P + dA + dB);
        } else {
            r[0] = fetch(B + de);   // the next cell
        }
        add_segment<INTERP, FORM, SELECT>(A, W, q, g, T, sig, tend, S);
        if constexpr (TRI) {
            float2 p[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) p[i] = pair(r[i]);
            shift_corners(q, p, e0, e1);
            if constexpr (SH) {
                shear_pairs<4>(V.sw, r, p);
                shift_corners(g, p, e0, e1);
            }
        } else {
            q[0] = pair(r[0]);
            if constexpr (SH) shear_pairs<1>(V.sw, &r[0], &g[0]);
        }
        // cross the exit face
        sig = tend;
        B += de;
        if constexpr (SEAM) {
            if (e0) D[0] = fd[0];
            if (e1) D[1] = fd[1];
            if (e2) D[2] = fd[2];
        }
        // (every axis' next crossing evaluated again, the same but for axis e: no
        // predicates, no chain through the exit axis)
        kf[0] += e0 ? 1.f : 0.f;
        kf[1] += e1 ? 1.f : 0.f;
        kf[2] += e2 ? 1.f : 0.f;
        T[0] = fmaf(kf[0], W.td[0], W.T0[0]);
        T[1] = fmaf(kf[1], W.td[1], W.T0[1]);
        T[2] = fmaf(kf[2], W.td[2], W.T0[2]);
    }
    // (no crossing left: the cap ended the walk, or it ended on its last allowed one)
    if (left == 0 && fminf(fminf(T[0], T[1]), T[2]) < lim) {
        S.overflow = true;
        return;
    }
    add_segment<INTERP, FORM, SELECT>(A, W, q, g, T, sig, W.L, S);
    if constexpr (MA) {
        // the surface term at the end of the interval (the last sub-step's stays)
        const float t = W.L - sig;
        float u[3];
#pragma unroll
        for (int a = 0; a < 3; ++a)
            u[a] = __saturatef(fmaf(t, W.v[a], __saturatef(fmaf(sig - T[a], W.v[a], W.cu[a]))));
        if constexpr (TRI) S.qb = trilinear_x(q, u[0], u[1], u[2]);
        else S.qb = q[0].x;
        float G0, G1, G2;
        kernel_coeffs(t, sig, W.chiA0, W.D0, A.chi_sf, A.inv_chi_s_f, G0, G1, G2);
        S.gb = fmaf(t, fmaf(t, G2, G1), G0);
    }
    if (more) {
        // the cell the walk ended in (a box-local walk may have passed the seam, once)
        S.pc0 = wrap_once(W.c[0] + W.sgn[0] * f2i_exact(kf[0]), A.n0);
        S.pc1 = wrap_once(W.c[1] + W.sgn[1] * f2i_exact(kf[1]), A.n1);
        S.pc2 = wrap_once(W.c[2] + W.sgn[2] * f2i_exact(kf[2]), A.n2);
    }
}

// The flat walk's start: the point index B of the sub-step's entry corner, the
// index step D per axis to the first cell's exit side and fd from plane to plane
// along the motion; whether every vertex plane the sub-step can read lies inside
// the records' box. SEAM (the whole grid's records): crossings are counted as
// the walk will make them, not two more than the path allows, and the entry side
// of the first cell may be the periodic image of plane 0 (a ray that comes in
// through the far face): D is then not fd. NGP: cells for vertices (B the cell's
// index, D = fd).
template <int INTERP, bool SEAM>
__device__ __forceinline__ bool flat_start(const TraceArgs& A, const Walk<float>& W, int& B, int D[3], int fd[3])
{
    const int nn[3] = {A.n0, A.n1, A.n2};
    bool inside = true;
    B = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        // box-local vertex and cell coordinates (the records' box starts at fo,
        // periodically)
        const int sa = a == 0 ? A.fs0 : (a == 1 ? A.fs1 : 1);
        int vl = (INTERP == RR_TRILINEAR ? W.vlo[a] : W.c[a]) - A.fo[a];
        if (vl < 0) vl += nn[a];
        int cl = W.c[a] - A.fo[a];
        if (cl < 0) cl += nn[a];
        B += vl * sa;
        fd[a] = W.sgn[a] * sa;
        D[a] = SEAM && INTERP == RR_TRILINEAR ? (W.vhi[a] - W.vlo[a]) * sa : fd[a];
        // crossings this sub-step can make on axis a; cells c .. c + sgn K,
        // vertex planes one further
        int K = 0;
        if (W.T0[a] < W.L) {
            const float x = (W.L - W.T0[a]) * W.v[a];
            if (x < 4194304.f) K = f2i_exact(x) + 2;
            else inside = false;
            if constexpr (SEAM) {
                // the walk crosses face k (k = 0, 1, ...) on this axis while
                // T_k = T0 + k td < L - eps_end, and T_k never decreases with k:
                // drop the margin that the walk's own test rules out
                const float lim = W.L - W.L * kSliver;
#pragma unroll
                for (int r = 0; r < 3; ++r)
                    if (K > 0 && !(fmaf((float)(K - 1), W.td[a], W.T0[a]) < lim)) --K;
            }
        }
        constexpr int up = INTERP == RR_TRILINEAR ? 1 : 0;
        const int lo = W.sgn[a] > 0 ? cl : cl - K, hi = W.sgn[a] > 0 ? cl + K + up : (SEAM ? cl : cl + 1);
        if (lo < 0 || hi > A.fe[a] - 1) inside = false;
    }
    return inside;
}

// A sub-step that resumes inside the previous one's last cell does not start a
// new cell segment.
template <class R>
__device__ __forceinline__ bool resumes(const Walk<R>& W, const PieceState<R>& S, int j)
{
    return j > 0 && W.c[0] == S.pc0 && W.c[1] == S.pc1 && W.c[2] == S.pc2;
}

// The sub-steps j .. nsub - 1 of a ray from the first that does not lie inside
// the grid, out of line (kAddrAuto): those inside by flat offsets, the others by
// wrapped vertex indices. It sets the walk up from the ray's interval alone and
// the caller has left its loop, so that the common path keeps no register for it.
template <int INTERP, int FORM>
__device__ __noinline__ void finish_ray(const TraceArgs& A, const float4* rec, long long rid, float ch, float cl,
                                        float Lf, float D0f, int j, int nsub, float dsub, PieceState<float>& state)
{
    const RayRange rg{ch, cl, Lf, D0f, 0.0, 0.0};
    PieceState<float> S = state;
    RayWeights V;
    ray_weights<FORM>(A, rid, V);
    for (; j < nsub && !S.overflow; ++j) {
        float bh, bl, Lj, D0j;
        sub_step(rg, j, nsub, dsub, bh, bl, Lj, D0j);
        Walk<float> W;
        walk_setup<float>(A, rid, bh, bl, Lj, D0j, 0.0, 0.0, W);
        int B, D[3], fd[3];
        const bool inside = flat_start<INTERP, true>(A, W, B, D, fd), resume = resumes(W, S, j);
        if (inside) walk_flat<INTERP, FORM, false, INTERP == RR_TRILINEAR, false>(A, rec, W, V, j == 0, j + 1 < nsub, resume, B, D, fd, S);
        else walk_piece<INTERP, float, FORM, kAddrIndex>(A, rec, W, V, j, resume, S);
    }
    state = S;
}

// Whether a multi-step kernel sets a ray's constants up once, outside its loop
// over the steps, and takes the sub-steps' division from the host. Production
// pass, trace kernels: default form 20.83 -> 20.33 ms; 256^3, 1024^2 rays, 20
// steps: shear 4.46 -> 4.37, moments 2.90 -> 2.82, Method A (with selects for
// slivers) 2.52 -> 2.41 ms; the kernels that choose their addressing spill.
template <int ADDR>
constexpr bool kHoist = ADDR == kAddrFlat;

// PER: periodic bundles only. REGACC: one of several steps of a launch; acc and
// W0 (the ray's constants) live across them. BATCH: in the persistent kernel. A0: the kernel's own arguments (A,
// but for the step's fields in a multi-step kernel), whose address finish_ray
// takes.
template <int INTERP, class R, int FORM, int ADDR, bool PER, bool REGACC = false, bool BATCH = false>
__device__ __forceinline__ void trace_ray(const TraceArgs& A, const TraceArgs& A0, int ix, int iy, RayAcc* acc = nullptr,
                                          const Walk<R>* W0 = nullptr)
{
    static_assert(!REGACC || (FORM != kFormPlain && sizeof(R) == 4), "register accumulators: FP32 compensated forms");
    constexpr bool AUTO = ADDR == kAddrAuto;
    constexpr bool FLAT = ADDR == kAddrFlat || AUTO;
    static_assert(!FLAT || sizeof(R) == 4, "flat addressing: FP32 walk");
    constexpr bool F64 = sizeof(R) == 8;
    constexpr bool SH = !F64 && FORM == kFormShear;
    constexpr bool MA = !F64 && FORM == kFormMethodA;
    const long long rid = (long long)iy * A.nx + ix;
    RayRange rg;
    if (!ray_range<PER>(A, rid, rg)) return;
    if (!REGACC || !acc->loaded) {
        prefetch_l2(A.kacc + rid);
        prefetch_l2(A.bacc + rid);
        prefetch_l2(A.nseg + rid);
        if constexpr (SH) {
            prefetch_l2(A.g1acc + rid);
            prefetch_l2(A.g2acc + rid);
        }
    }
    // FP32: sub-steps of at most sub_len, so that the path variable stays small
    constexpr bool HOIST = REGACC && kHoist<ADDR>;
    const int nsub = F64 ? 1 : (HOIST ? A.nsub : max(1, (int)ceilf(rg.Lf / A.sub_len)));
    const float dsub = HOIST ? A.dsub : rg.Lf / (float)nsub;

    RayWeights V;
    ray_weights<FORM>(A, rid, V);
    Walk<R> W;
    if constexpr (HOIST) W = *W0;
    PieceState<R> S;
    int rest = -1;   // AUTO: the first sub-step that does not lie inside
    for (int j = 0; j < nsub && !S.overflow; ++j) {
    float bh, bl, Lj, D0j;
    sub_step(rg, j, nsub, dsub, bh, bl, Lj, D0j);
    walk_setup<R, false, !HOIST>(A, rid, bh, bl, Lj, D0j, rg.hi, rg.lo, W);
    if constexpr (FLAT) {
        int B, D[3], fd[3];
        if (!flat_start<INTERP, AUTO>(A, W, B, D, fd)) {
            if constexpr (AUTO) rest = j;
            else atomicOr(A.err, kErrRange);
            break;
        }
        // (see add_segment; kernels that hold more, and the NGP walk at 64
        // registers, branch)
        constexpr bool SELECT = INTERP == RR_TRILINEAR && !BATCH && !(AUTO && REGACC) &&
                                FORM != kFormShear;
        walk_flat<INTERP, FORM, SELECT, AUTO && INTERP == RR_TRILINEAR>(A, A.rec, W, V, j == 0, j + 1 < nsub, resumes(W, S, j), B, D, fd, S);
    } else {
        walk_piece<INTERP, R, FORM, ADDR>(A, A.rec, W, V, j, resumes(W, S, j), S);
    }
    }
    if constexpr (AUTO) {
        if (rest >= 0) {
            PieceState<R> Q = S;
            finish_ray<INTERP, FORM>(A0, A.rec, rid, rg.ch, rg.cl, rg.Lf, rg.D0f, rest, nsub, dsub, Q);
            S = Q;
        }
    }

    if constexpr (MA) {
        S.s2.add(make_float2(-S.ga * S.qa, 0.f));
        S.s2.add(make_float2(S.gb * S.qb, 0.f));
    }
    if constexpr (!F64) {
        S.sk.s = S.s2.s.x; S.sk.c = S.s2.c.x;
        S.sb.s = S.s2.s.y; S.sb.c = S.s2.c.y;
    }
    if (S.overflow) atomicOr(A.err, kErrStepLimit);
    if (!S.sk.finite() || !S.sb.finite()) atomicOr(A.err, kErrNonFinite);
    if constexpr (REGACC) {
        // the first step of the launch: the ray's state from memory
        if (!acc->loaded) {
            acc->k = A.kacc[rid];
            acc->b = A.bacc[rid];
            acc->n = A.nseg[rid];
            if constexpr (SH) {
                acc->x1 = A.g1acc[rid];
                acc->x2 = A.g2acc[rid];
            }
            if constexpr (FORM == kFormMoments) {
                acc->x1 = A.kmom[rid];
                acc->x2 = A.bmom[rid];
            }
            acc->loaded = true;
        }
    }
    if constexpr (SH) {
        float gh, gl;
        if (!S.s2m.finite()) atomicOr(A.err, kErrNonFinite);
        two_sum(S.s2m.s.x, -S.s2m.c.x, gh, gl);
        if constexpr (REGACC) acc->x1 = ff_mul_add(acc->x1, gh, gl, A.sch, A.scl);
        else A.g1acc[rid] = ff_mul_add(A.g1acc[rid], gh, gl, A.sch, A.scl);
        two_sum(S.s2m.s.y, -S.s2m.c.y, gh, gl);
        if constexpr (REGACC) acc->x2 = ff_mul_add(acc->x2, gh, gl, A.sch, A.scl);
        else A.g2acc[rid] = ff_mul_add(A.g2acc[rid], gh, gl, A.sch, A.scl);
    }
    if constexpr (FORM == kFormMoments) {
        float mh, ml;
        if (!S.s2m.finite()) atomicOr(A.err, kErrNonFinite);
        two_sum(S.s2m.s.x, -S.s2m.c.x, mh, ml);
        if constexpr (REGACC) acc->x1 = ff_mul_add(acc->x1, mh, ml, A.sch, A.scl);
        else A.kmom[rid] = ff_mul_add(A.kmom[rid], mh, ml, A.sch, A.scl);
        two_sum(S.s2m.s.y, -S.s2m.c.y, mh, ml);
        if constexpr (REGACC) acc->x2 = ff_mul_add(acc->x2, mh, ml, A.bsh, A.bsl);
        else A.bmom[rid] = ff_mul_add(A.bmom[rid], mh, ml, A.bsh, A.bsl);
    }
    if constexpr (FORM == kFormPlain) {
        // plain FP32 across steps too: the high word only
        A.kacc[rid] = make_float2(fmaf(S.sk.s, A.sch, A.kacc[rid].x), 0.f);
        A.bacc[rid] = make_float2(fmaf(S.sb.s, A.bsh, A.bacc[rid].x), 0.f);
        A.nseg[rid] += S.cnt;
        return;
    }
    float kh, kl, bh, bl;
    S.sk.pair(kh, kl);
    S.sb.pair(bh, bl);
    if constexpr (REGACC) {
        acc->k = ff_mul_add(acc->k, kh, kl, A.sch, A.scl);
        acc->b = ff_mul_add(acc->b, bh, bl, A.bsh, A.bsl);
        acc->n += S.cnt;
        return;
    }
    A.kacc[rid] = ff_mul_add(A.kacc[rid], kh, kl, A.sch, A.scl);
    A.bacc[rid] = ff_mul_add(A.bacc[rid], bh, bl, A.bsh, A.bsl);
    A.nseg[rid] += S.cnt;
}


// Blocks of NT_MAX threads per SM: the NGP walk's default sums need few
// registers outside their rare path (256^3, 1024^2 rays, 20 steps: 1199 us with 2
// blocks, 1072 with 3, 1012 with 4, at 64 registers); the trilinear ones spill
// into their loop with more than 2.
template <int INTERP, class R, int FORM>
constexpr int kBlocks = INTERP == RR_NGP && sizeof(R) == 4 && (FORM == kFormKahan || FORM == kFormPlain) ? 4 : 2;

template <int INTERP, class R, int FORM, int ADDR, bool PER>
__global__ void __launch_bounds__(NT_MAX, kBlocks<INTERP, R, FORM>) trace_kernel(const __grid_constant__ TraceArgs A, const TileCfg t)
{
    prefetch_ahead(A, t);
    int ix, iy;
    tile_ray(t, blockIdx.x, blockIdx.y, ix, iy);
    if (ix < A.nx && iy < A.ny) trace_ray<INTERP, R, FORM, ADDR, PER>(A, A, ix, iy);
}

// Consecutive steps of one bundle in one launch (the default FP32 form): each
// thread walks its ray through the steps in order, every step reading its own
// records with its own interval and scales, the ray's accumulators kept in
// registers in between. Per step the arithmetic is that of trace_kernel, so
// the result equals one trace_kernel launch per step bit for bit; what goes
// is the per-launch and per-step traffic of the ray state (directions,
// accumulators) and all launches but one.
template <int INTERP, int ADDR, int FORM, bool PER>
__global__ void __launch_bounds__(NT_MAX, kBlocks<INTERP, float, FORM>)
    trace_steps_kernel(const __grid_constant__ TraceArgs A, const __grid_constant__ StepBlock S, const TileCfg t)
{
    prefetch_ahead(A, t);
    int ix, iy;
    tile_ray(t, blockIdx.x, blockIdx.y, ix, iy);
    if (ix >= A.nx || iy >= A.ny) return;
    RayAcc acc;
    acc.loaded = false;
    Walk<float> W0;
    if constexpr (kHoist<ADDR>) ray_consts<float>(A, (long long)iy * A.nx + ix, W0);
    for (int g = 0; g < S.n; ++g) {
        const StepArgs& st = S.s[g];
        TraceArgs As = A;
        As.rec = st.rec;
        As.chi_a = st.chi_a; As.chi_b = st.chi_b;
        As.cah = st.cah; As.cal = st.cal;
        As.Lf = st.Lf; As.D0f = st.D0f;
        As.nsub = st.nsub; As.dsub = st.dsub;
        As.sch = st.sch; As.scl = st.scl;
        As.bsh = st.bsh; As.bsl = st.bsl;
        As.fo[0] = st.fo[0]; As.fo[1] = st.fo[1]; As.fo[2] = st.fo[2];
        As.fe[0] = st.fe[0]; As.fe[1] = st.fe[1]; As.fe[2] = st.fe[2];
        As.fs0 = st.fs0; As.fs1 = st.fs1;
        trace_ray<INTERP, float, FORM, ADDR, PER, true>(As, A, ix, iy, &acc, &W0);
    }
    if (acc.loaded) {
        const long long rid = (long long)iy * A.nx + ix;
        A.kacc[rid] = acc.k;
        A.bacc[rid] = acc.b;
        A.nseg[rid] = acc.n;
        if constexpr (FORM == kFormShear) {
            A.g1acc[rid] = acc.x1;
            A.g2acc[rid] = acc.x2;
        }
        if constexpr (FORM == kFormMoments) {
            A.kmom[rid] = acc.x1;
            A.bmom[rid] = acc.x2;
        }
    }
}

// Persistent work queue over the ray tiles of many bundles (lightcones): each
// block takes `chunk` consecutive tiles from a global counter (monotonic, no
// waiting), finds the bundle by binary search in the tile offsets, stages that
// bundle's arguments in shared memory and traces the tile.
template <int INTERP, class R, int ADDR, bool PER>
__global__ void __launch_bounds__(NT_MAX, kBlocks<INTERP, R, kFormKahan>) trace_batch_kernel(const BatchArgs B)
{
    __shared__ TraceArgs sA;
    __shared__ int s_item, s_cone;
    const int total = B.tile_start[B.ncones];
    while (true) {
        if (threadIdx.x == 0) s_item = atomicAdd(B.counter, B.chunk);
        __syncthreads();
        const int item0 = s_item;
        __syncthreads();
        if (item0 >= total) break;
        for (int c = 0; c < B.chunk; ++c) {
            const int item = item0 + c;
            if (item >= total) break;
            if (threadIdx.x == 0) {
                int lo = 0, hi = B.ncones - 1;   // last cone with tile_start <= item
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (B.tile_start[mid] <= item) lo = mid;
                    else hi = mid - 1;
                }
                s_cone = lo;
            }
            __syncthreads();
            const int cone = s_cone;
            {
                const int* src = reinterpret_cast<const int*>(B.cones + cone);
                int* dst = reinterpret_cast<int*>(&sA);
                for (int i = threadIdx.x; i < (int)(sizeof(TraceArgs) / sizeof(int)); i += blockDim.x)
                    dst[i] = __ldg(src + i);
            }
            __syncthreads();
            const int local = item - B.tile_start[cone];
            const int ntx = B.tiles_x[cone];
            int ix, iy;
            tile_ray(B.tile, local % ntx, local / ntx, ix, iy);
            if (ix < sA.nx && iy < sA.ny) trace_ray<INTERP, R, kFormKahan, ADDR, PER, false, true>(sA, sA, ix, iy);
            __syncthreads();
        }
    }
}

}  // namespace

dim3 tile_grid(const TileCfg& t, int nx, int ny)
{
    const int bx = t.wx * t.bwx, by = (32 / t.wx) * t.bwy;
    return dim3((unsigned)((nx + bx - 1) / bx), (unsigned)((ny + by - 1) / by));
}

bool tile_ok(const TileCfg& t)
{
    return (t.wx == 1 || t.wx == 2 || t.wx == 4 || t.wx == 8 || t.wx == 16 || t.wx == 32) && t.bwx >= 1 &&
           t.bwy >= 1 && t.bwx * t.bwy * 32 <= NT_MAX;
}

namespace {

template <int INTERP, class R, int FORM, int ADDR>
cudaError_t launch_addr(const TraceArgs& a, const dim3& grid, int nt, cudaStream_t s, const TileCfg& t)
{
    if (a.periodic) trace_kernel<INTERP, R, FORM, ADDR, true><<<grid, nt, 0, s>>>(a, t);
    else trace_kernel<INTERP, R, FORM, ADDR, false><<<grid, nt, 0, s>>>(a, t);
    return cudaGetLastError();
}

template <int INTERP, class R, int FORM>
cudaError_t launch_one(const TraceArgs& a, const dim3& grid, int nt, cudaStream_t s, const TileCfg& t,
                       bool wrapped = false)
{
    if constexpr (sizeof(R) == 4) {
        // fewer than 2^31 points
        if (a.fe[0] > 0 && !(wrapped && INTERP == RR_TRILINEAR))
            return launch_addr<INTERP, R, FORM, kAddrAuto>(a, grid, nt, s, t);
    }
    return launch_addr<INTERP, R, FORM, FORM == kFormKahan && INTERP == RR_TRILINEAR && sizeof(R) == 8 ? kAddrPlanes : kAddrIndex>(
        a, grid, nt, s, t);
}

template <int FORM>
cudaError_t launch_form(const TraceArgs& a, int interp, const dim3& grid, int nt, cudaStream_t s, const TileCfg& t,
                        bool wrapped)
{
    return interp == RR_TRILINEAR ? launch_one<RR_TRILINEAR, float, FORM>(a, grid, nt, s, t, wrapped)
                                  : launch_one<RR_NGP, float, FORM>(a, grid, nt, s, t);
}

}  // namespace

cudaError_t launch_trace(const TraceArgs& a, int interp, bool fp64_dda, cudaStream_t s, const TileCfg& t,
                         int form, bool flat, bool wrapped)
{
    if (!tile_ok(t)) return cudaErrorInvalidValue;
    const dim3 grid = tile_grid(t, a.nx, a.ny);
    const int nt = 32 * t.bwx * t.bwy;
    if (flat && !fp64_dda && interp == RR_TRILINEAR && a.periodic) {
        switch (form) {
        case kFormPlain: trace_kernel<RR_TRILINEAR, float, kFormPlain, kAddrFlat, true><<<grid, nt, 0, s>>>(a, t); break;
        case kFormMoments: trace_kernel<RR_TRILINEAR, float, kFormMoments, kAddrFlat, true><<<grid, nt, 0, s>>>(a, t); break;
        case kFormGeneric: trace_kernel<RR_TRILINEAR, float, kFormGeneric, kAddrFlat, true><<<grid, nt, 0, s>>>(a, t); break;
        case kFormMethodA: trace_kernel<RR_TRILINEAR, float, kFormMethodA, kAddrFlat, true><<<grid, nt, 0, s>>>(a, t); break;
        case kFormShear: trace_kernel<RR_TRILINEAR, float, kFormShear, kAddrFlat, true><<<grid, nt, 0, s>>>(a, t); break;
        default: trace_kernel<RR_TRILINEAR, float, kFormKahan, kAddrFlat, true><<<grid, nt, 0, s>>>(a, t); break;
        }
        return cudaGetLastError();
    }
    if (fp64_dda)
        return interp == RR_TRILINEAR ? launch_one<RR_TRILINEAR, double, kFormKahan>(a, grid, nt, s, t)
                                      : launch_one<RR_NGP, double, kFormKahan>(a, grid, nt, s, t);
    switch (form) {
    case kFormPlain: return launch_form<kFormPlain>(a, interp, grid, nt, s, t, wrapped);
    case kFormMoments: return launch_form<kFormMoments>(a, interp, grid, nt, s, t, wrapped);
    case kFormGeneric: return launch_form<kFormGeneric>(a, interp, grid, nt, s, t, wrapped);
    case kFormMethodA: return launch_form<kFormMethodA>(a, interp, grid, nt, s, t, wrapped);
    // (the shear form's 128-register cap of two resident blocks spills a few
    // bytes; 168 registers without spills measured 2 % slower)
    case kFormShear: return launch_form<kFormShear>(a, interp, grid, nt, s, t, wrapped);
    default: return launch_form<kFormKahan>(a, interp, grid, nt, s, t, wrapped);
    }
}

template <int FORM>
static cudaError_t launch_steps_form(const TraceArgs& a, const StepBlock& b, int interp, bool flat, dim3 grid, int nt,
                              const TileCfg& t, cudaStream_t s)
{
    // trilinear (grids of fewer than 2^31 points): steps that all take the flat
    // addressing (periodic), or choose it per sub-step, as NGP steps do
    if (interp == RR_TRILINEAR) {
        if (flat && a.periodic) trace_steps_kernel<RR_TRILINEAR, kAddrFlat, FORM, true><<<grid, nt, 0, s>>>(a, b, t);
        else if (a.periodic) trace_steps_kernel<RR_TRILINEAR, kAddrAuto, FORM, true><<<grid, nt, 0, s>>>(a, b, t);
        else trace_steps_kernel<RR_TRILINEAR, kAddrAuto, FORM, false><<<grid, nt, 0, s>>>(a, b, t);
    } else {
        if (a.fe[0] <= 0) trace_steps_kernel<RR_NGP, kAddrIndex, FORM, false><<<grid, nt, 0, s>>>(a, b, t);
        else if (a.periodic) trace_steps_kernel<RR_NGP, kAddrAuto, FORM, true><<<grid, nt, 0, s>>>(a, b, t);
        else trace_steps_kernel<RR_NGP, kAddrAuto, FORM, false><<<grid, nt, 0, s>>>(a, b, t);
    }
    return cudaGetLastError();
}

cudaError_t launch_trace_steps(const TraceArgs& a, const StepBlock& b, int interp, bool flat, cudaStream_t s,
                               int form)
{
    const TileCfg t{};
    if (b.n < 1 || b.n > kMaxStepBlock) return cudaErrorInvalidValue;
    const dim3 grid = tile_grid(t, a.nx, a.ny);
    const int nt = 32 * t.bwx * t.bwy;
    switch (form) {
    case kFormKahan: return launch_steps_form<kFormKahan>(a, b, interp, flat, grid, nt, t, s);
    case kFormShear: return launch_steps_form<kFormShear>(a, b, interp, flat, grid, nt, t, s);
    case kFormMoments: return launch_steps_form<kFormMoments>(a, b, interp, flat, grid, nt, t, s);
    case kFormMethodA: return launch_steps_form<kFormMethodA>(a, b, interp, flat, grid, nt, t, s);
    case kFormGeneric: return launch_steps_form<kFormGeneric>(a, b, interp, flat, grid, nt, t, s);
    default: return cudaErrorInvalidValue;
    }
}

namespace {

using BatchKernel = void (*)(const BatchArgs);

// small: every bundle's grid has fewer than 2^31 points; periodic: every bundle is
template <bool PER>
BatchKernel batch_kernel_of(int interp, bool fp64_dda, bool small)
{
    if (interp == RR_TRILINEAR) {
        if (fp64_dda) return trace_batch_kernel<RR_TRILINEAR, double, kAddrIndex, PER>;
        return small ? trace_batch_kernel<RR_TRILINEAR, float, kAddrAuto, PER>
                     : trace_batch_kernel<RR_TRILINEAR, float, kAddrIndex, PER>;
    }
    if (fp64_dda) return trace_batch_kernel<RR_NGP, double, kAddrIndex, PER>;
    return small ? trace_batch_kernel<RR_NGP, float, kAddrAuto, PER> : trace_batch_kernel<RR_NGP, float, kAddrIndex, PER>;
}

BatchKernel batch_kernel(int interp, bool fp64_dda, bool small, bool periodic)
{
    return periodic ? batch_kernel_of<true>(interp, fp64_dda, small) : batch_kernel_of<false>(interp, fp64_dda, small);
}

}  // namespace

cudaError_t launch_trace_batch(const BatchArgs& b, int interp, bool fp64_dda, int blocks, cudaStream_t s, bool small,
                               bool periodic)
{
    if (!tile_ok(b.tile) || b.chunk < 1 || blocks < 1) return cudaErrorInvalidValue;
    const int nt = 32 * b.tile.bwx * b.tile.bwy;
    batch_kernel(interp, fp64_dda, small, periodic)<<<blocks, nt, 0, s>>>(b);
    return cudaGetLastError();
}

int batch_blocks_per_sm(int interp, bool fp64_dda, bool periodic, const TileCfg& t)
{
    const int nt = 32 * t.bwx * t.bwy;
    int n = 0;
    const cudaError_t e =
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, batch_kernel(interp, fp64_dda, true, periodic), nt, 0);
    return (e == cudaSuccess && n > 0) ? n : 1;
}
}  // namespace rr
