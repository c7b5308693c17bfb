// Immersed-boundary kernels: MLS interpolation at markers and hydrodynamic
// probes (Sec. 2.2, Eqs. uLag, l2norm, intKernel; Sec. 2.3, Eqs. hydroForP,
// hydroForNu), membrane forces + Verlet update + spreading (Sec. 2.3,
// Eqs. strainFor, bendFor, volFor, newtonSoft, verletPos, verletVel;
// Sec. 2.2, Eq. bodyforce) and the rigid-body Newton-Euler update
// (Eqs. linearVelRig, angularVelRig).
//
// Per step and body: k_moments streams the populations once for every node
// of the body's support region (predictor density and velocity), k_mls
// fits at every marker and probe from those node moments, and one
// structure kernel updates the markers and spreads the IB force.
#include "lbib_device.cuh"
#include "lbib_kernels.h"
#include "sweep_cell.cuh"

namespace lbib {

constexpr int kStructThreads = 128;  // threads per block of the structure kernels (16 markers)
constexpr double kAlpha = 0.3;    // Eq. (intKernel)
constexpr double kRw = 1.3;       // support size r_w (Sec. 2.2)
constexpr double kProbe = 1.2;    // probe length (Sec. 2.3)
constexpr int kBoxLo = 3, kBoxHi = 4;  // node margins that cover marker and probe supports

__device__ __forceinline__ float rcp(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double rcp(double x) { return 1.0 / x; }

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// ---------------------------------------------------------------------------
// Predictor moments on the support region: for every node of the box,
// pull the 19 populations (f_i(x) = f*_i(x - e_i)) and store
// rho - 1 and u* = (sum f e + g_ext/2)/rho.  Grid-stride over the box
// recorded on the device by the previous step's update.
// ---------------------------------------------------------------------------
// Support-region moments, node-interleaved: mom[4 node + q] holds rho - 1
// and the predictor velocity u*_x, u*_y, u*_z of node `node`, so that the
// MLS gather of one support node is a single 16-byte (FP32) or two
// 16-byte (FP64) loads.
__device__ __forceinline__ void mom_store(float *m, int node, float a, float b, float c, float d) {
    reinterpret_cast<float4 *>(m)[node] = make_float4(a, b, c, d);
}
__device__ __forceinline__ void mom_store(double *m, int node, double a, double b, double c, double d) {
    reinterpret_cast<double2 *>(m)[2 * node] = make_double2(a, b);
    reinterpret_cast<double2 *>(m)[2 * node + 1] = make_double2(c, d);
}
template <bool kCG>
__device__ __forceinline__ void mom_load(const float *m, int node, float *v) {
    const float4 q = ld_ro<kCG>(reinterpret_cast<const float4 *>(m) + node);
    v[0] = q.x;
    v[1] = q.y;
    v[2] = q.z;
    v[3] = q.w;
}
template <bool kCG>
__device__ __forceinline__ void mom_load(const double *m, int node, double *v) {
    const double2 a = ld_ro<kCG>(reinterpret_cast<const double2 *>(m) + 2 * node);
    const double2 b = ld_ro<kCG>(reinterpret_cast<const double2 *>(m) + 2 * node + 1);
    v[0] = a.x;
    v[1] = a.y;
    v[2] = b.x;
    v[3] = b.y;
}

template <typename S, typename R, bool kCG = false>
__device__ __forceinline__ void moments_body(const S *__restrict__ fin, const Lattice &L, const int *__restrict__ box,
                                             int *__restrict__ box_next, R *__restrict__ mom,
                                             uint32_t *__restrict__ step_inc, const int vb, const int nvb) {
    // the step counter and the support box are read and written by other
    // kernels of the step (or other work items of a persistent launch):
    // L2 accesses, coherent across SMs
    if (step_inc && vb == 0 && threadIdx.x == 0) atomicAdd(step_inc, 1u);  // read by the later kernels of the step
    const int n[3] = {L.nx, L.ny, L.nz};
    int lo[3], ext[3];
    for (int a = 0; a < 3; ++a) {
        long long l = __ldcg(box + a), h = __ldcg(box + 3 + a);
        if (L.bc[a] == kWall) {
            l = l < 0 ? 0 : l;
            h = h > n[a] - 1 ? n[a] - 1 : h;
        } else if (h - l + 1 > n[a]) {
            l = 0;
            h = n[a] - 1;
        }
        lo[a] = (int)l;
        ext[a] = h < l ? 0 : (int)(h - l + 1);
    }
    if (vb == 0 && threadIdx.x < 6) box_next[threadIdx.x] = threadIdx.x < 3 ? 0x7fffffff : (int)0x80000000;
    const int total = ext[0] * ext[1] * ext[2];
    const int nxy = L.nx * L.ny;
    const long long st = L.stride;
    for (int k = vb * blockDim.x + threadIdx.x; k < total; k += nvb * blockDim.x) {
        int c[3] = {lo[0] + k % ext[0], lo[1] + (k / ext[0]) % ext[1], lo[2] + k / (ext[0] * ext[1])};
        int cm[3], cp[3];
        for (int a = 0; a < 3; ++a) {
            if (L.bc[a] == kPeriodic) c[a] = wrap_periodic(c[a], n[a]);
            int vm = c[a] - 1, vp = c[a] + 1;
            if (vm < 0) vm = L.bc[a] == kPeriodic ? n[a] - 1 : 0;
            if (vp >= n[a]) vp = L.bc[a] == kPeriodic ? 0 : n[a] - 1;
            cm[a] = vm;
            cp[a] = vp;
        }
        R drho = R(0), jx = R(0), jy = R(0), jz = R(0);
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const int sx = ex(i) > 0 ? cm[0] : ex(i) < 0 ? cp[0] : c[0];
            const int sy = ey(i) > 0 ? cm[1] : ey(i) < 0 ? cp[1] : c[1];
            const int sz = ez(i) > 0 ? cm[2] : ez(i) < 0 ? cp[2] : c[2];
            const R gi = Pop<S, R>::from(ld_ro<kCG>(fin + (long long)i * st + (sx + L.nx * sy + nxy * sz)));
            drho += gi;
            if (ex(i) > 0) jx += gi;
            if (ex(i) < 0) jx -= gi;
            if (ey(i) > 0) jy += gi;
            if (ey(i) < 0) jy -= gi;
            if (ez(i) > 0) jz += gi;
            if (ez(i) < 0) jz -= gi;
        }
        const int node = c[0] + L.nx * c[1] + nxy * c[2];
        const R rho = R(1) + drho;
        mom_store(mom, node, drho, (jx + R(0.5) * pick<R>(L.gext_d[0], L.gext_f[0])) / rho,
                  (jy + R(0.5) * pick<R>(L.gext_d[1], L.gext_f[1])) / rho,
                  (jz + R(0.5) * pick<R>(L.gext_d[2], L.gext_f[2])) / rho);
    }
}

template <typename S, typename R>
__global__ void __launch_bounds__(kNodeThreads) k_moments(const S *__restrict__ fin, Lattice L, const int *__restrict__ box,
                                                 int *__restrict__ box_next, R *__restrict__ mom,
                                                 uint32_t *__restrict__ step_inc) {
    chain_release();  // the MLS kernel may be scheduled beside this one
    moments_body<S, R>(fin, L, box, box_next, mom, step_inc, blockIdx.x, gridDim.x);
}

constexpr int kRec = 16;  // R values of a marker's transfer record (BodyView::phi)

// 1/d in FP64 from the FP32 reciprocal refined by two Newton steps
// (relative error ~1e-7 -> ~1e-14 -> below the double rounding).  d must lie
// in the FP32 normal range, or the seed is infinite or zero: callers bound it.
__device__ __forceinline__ double recip64(double d) {
    double r = (double)__frcp_rn((float)d);
    r = fma(r, fma(-d, r, 1.0), r);
    r = fma(r, fma(-d, r, 1.0), r);
    return r;
}

// Inverse of a symmetric positive definite 4x4 matrix given by its upper
// triangle (00,01,02,03,11,12,13,22,23,33), as the adjugate over the
// determinant, both from the 2x2 minors of the top and bottom row pairs
// (a shallow dependency chain: FP64 latency, not throughput, limits this
// per-point solve).  Returns false unless kMinDet < determinant < kMaxDet:
// the bounds keep the FP32 seed of recip64 finite and normal.  An MLS moment
// matrix has entries of at most 27 * 1.5^2 (weights <= 1, offsets <= 1.5),
// so det < 4e7 always, and the centre node with the three nearer face
// neighbours (all within 1.22 of the point: weights >= 5e-5, unit offsets)
// keep det above ~1e-16; a determinant outside the bounds marks a singular
// support.
constexpr double kMinDet = 1e-30, kMaxDet = 1e30;
__device__ __forceinline__ bool spd_inverse4(const double *a, double *inv) {
    const double m00 = a[0], m01 = a[1], m02 = a[2], m03 = a[3];
    const double m11 = a[4], m12 = a[5], m13 = a[6], m22 = a[7], m23 = a[8], m33 = a[9];
    // rows 0,1 and rows 2,3 (symmetric: m10 = m01, ...)
    const double s0 = m00 * m11 - m01 * m01;
    const double s1 = m00 * m12 - m02 * m01;
    const double s2 = m00 * m13 - m03 * m01;
    const double s3 = m01 * m12 - m02 * m11;
    const double s4 = m01 * m13 - m03 * m11;
    const double s5 = m02 * m13 - m03 * m12;
    const double c5 = m22 * m33 - m23 * m23;
    const double c4 = m12 * m33 - m13 * m23;
    const double c3 = m12 * m23 - m13 * m22;
    const double c2 = m02 * m33 - m03 * m23;
    const double c1 = m02 * m23 - m03 * m22;
    const double c0 = m02 * m13 - m03 * m12;
    const double det = s0 * c5 - s1 * c4 + s2 * c3 + s3 * c2 - s4 * c1 + s5 * c0;
    if (!(det > kMinDet && det < kMaxDet)) return false;
    const double id = recip64(det);
    // rows of the adjugate (the matrix is symmetric, so is its inverse)
    inv[0] = (m11 * c5 - m12 * c4 + m13 * c3) * id;
    inv[1] = (-m01 * c5 + m02 * c4 - m03 * c3) * id;
    inv[2] = (m13 * s5 - m23 * s4 + m33 * s3) * id;
    inv[3] = (-m12 * s5 + m22 * s4 - m23 * s3) * id;
    inv[5] = (m00 * c5 - m02 * c2 + m03 * c1) * id;
    inv[6] = (-m03 * s5 + m23 * s2 - m33 * s1) * id;
    inv[7] = (m02 * s5 - m22 * s2 + m23 * s1) * id;
    inv[10] = (m03 * s4 - m13 * s2 + m33 * s0) * id;
    inv[11] = (-m02 * s4 + m12 * s2 - m23 * s0) * id;
    inv[15] = (m02 * s3 - m12 * s1 + m22 * s0) * id;
    inv[4] = inv[1];
    inv[8] = inv[2];
    inv[9] = inv[6];
    inv[12] = inv[3];
    inv[13] = inv[7];
    inv[14] = inv[11];
    return true;
}

// The same in FP32 by the root-free Cholesky factors A = L D L^T (L unit
// lower triangular, M = L^-1): A^-1 = M^T D^-1 M.  Backward stable, so for
// moment sums that are themselves FP32 it is as accurate as an FP64 inverse
// of the same sums (both leave errors of the order of the sums' own rounding
// in the fits), at FP32 issue rates.  Returns false unless every pivot is
// positive and finite (a singular support).
__device__ __forceinline__ bool spd_inverse4(const float *a, float *inv) {
    const float d0 = a[0], r0 = rcp(d0);
    const float l10 = a[1] * r0, l20 = a[2] * r0, l30 = a[3] * r0;
    const float d1 = a[4] - l10 * a[1], r1 = rcp(d1);
    const float t21 = a[5] - l10 * a[2], t31 = a[6] - l10 * a[3];
    const float l21 = t21 * r1, l31 = t31 * r1;
    const float d2 = a[7] - l20 * a[2] - l21 * t21, r2 = rcp(d2);
    const float t32 = a[8] - l20 * a[3] - l21 * t31;
    const float l32 = t32 * r2;
    const float d3 = a[9] - l30 * a[3] - l31 * t31 - l32 * t32, r3 = rcp(d3);
    // M = L^-1
    const float m10 = -l10, m21 = -l21, m32 = -l32;
    const float m20 = l21 * l10 - l20;
    const float m31 = l32 * l21 - l31;
    const float m30 = -l30 - l31 * m10 - l32 * m20;
    const float q10 = m10 * r1, q20 = m20 * r2, q21 = m21 * r2, q30 = m30 * r3, q31 = m31 * r3, q32 = m32 * r3;
    inv[0] = r0 + m10 * q10 + m20 * q20 + m30 * q30;
    inv[1] = q10 + m20 * q21 + m30 * q31;
    inv[2] = q20 + m30 * q32;
    inv[3] = q30;
    inv[5] = r1 + m21 * q21 + m31 * q31;
    inv[6] = q21 + m31 * q32;
    inv[7] = q31;
    inv[10] = r2 + m32 * q32;
    inv[11] = q32;
    inv[15] = r3;
    inv[4] = inv[1];
    inv[8] = inv[2];
    inv[9] = inv[6];
    inv[12] = inv[3];
    inv[13] = inv[7];
    inv[14] = inv[11];
    return d0 > 0.f && d0 < 1e30f && d1 > 0.f && d2 > 0.f && d3 > 0.f;
}

// Squared distance with the products and sums rounded one by one in the
// order (x^2 + y^2) + z^2, as a plain sum of squares is.
__device__ __forceinline__ double dist2_exact(double a, double b, double c) {
    return __dadd_rn(__dadd_rn(__dmul_rn(a, a), __dmul_rn(b, b)), __dmul_rn(c, c));
}

// The FP64 decision r_k <= 1 for the support nodes in `near` (bit i + 3 j +
// 9 k: offsets i - 1, j - 1, k - 1 from the point's base node).
__device__ __noinline__ unsigned support_exact(unsigned near, double fx, double fy, double fz, double cut) {
    unsigned in = 0u;
    while (near) {
        const int q = __ffs((int)near) - 1;
        near &= near - 1u;
        const double e0 = (double)(q % 3 - 1) - fx, e1 = (double)((q / 3) % 3 - 1) - fy, e2 = (double)(q / 9 - 1) - fz;
        if (dist2_exact(e0, e1, e2) <= cut) in |= 1u << q;
    }
    return in;
}

// One axis of the support weight W = exp(-(r/alpha)^2) of Eq. (intKernel),
// which is a product over the axes: w[i] = exp(-(d[i]/(r_w alpha))^2) at the
// offsets d[i] = i - 1 - f.  (Each from its own exponential: opposite offsets
// then have equal weights, and the sums of a mirrored support mirror exactly.)
template <typename R>
__device__ __forceinline__ void axis_weights(R f, R *d, R *w) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        d[i] = R(i - 1) - f;
        const R t = d[i] * R(1.0 / (kRw * kAlpha));
        w[i] = exp(-(t * t));
    }
}

// A node coordinate's image on the lattice; on walled axes bases are clamped
// so that the support lies inside.
__device__ __forceinline__ int support_coord(const Lattice &L, int a, int c) {
    const int n = a == 0 ? L.nx : a == 1 ? L.ny : L.nz;
    if (L.bc[a] != kPeriodic) return c;
    if (c < 0)
        c += n;
    else if (c >= n)
        c -= n;
    return wrap_periodic(c, n);
}

// Coordinate of the node nearest to x (any that is on the lattice, for a run
// that has diverged).
__device__ __forceinline__ int near_coord(const Lattice &L, int a, double x) {
    const int n = a == 0 ? L.nx : a == 1 ? L.ny : L.nz, c = __double2int_rn(x);
    return L.bc[a] == kPeriodic ? support_coord(L, a, c) : min(max(c, 0), n - 1);
}

// Transfer record of marker p: row 0 of A^-1 (4), the offset X - base (3) and
// the three axes' weights (9), from which every support node's transfer
// weight phi_k = W_k (A^-1 p_k)_0 follows; base node and the bits of the
// nodes with r_k <= 1 in node[4 p ..].
__device__ __forceinline__ void store_record(float *rec, const float *v) {
#pragma unroll
    for (int q = 0; q < kRec / 4; ++q)
        reinterpret_cast<float4 *>(rec)[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
}
__device__ __forceinline__ void store_record(double *rec, const double *v) {
#pragma unroll
    for (int q = 0; q < kRec / 2; ++q) reinterpret_cast<double2 *>(rec)[q] = make_double2(v[2 * q], v[2 * q + 1]);
}

// Sums a body takes over its MLS points: the enclosed volume times 6, or a
// rigid body's force and moment.
__device__ __forceinline__ int body_sums(const BodyView &B) { return B.rigid ? 6 : 1; }

// Momentum exchange: triangle t's share of minus the IB force of the
// previous step (sum_l A_l F_l) and of its moment about x_c (arm: X_c - x_c).
template <typename R>
__device__ __forceinline__ void exchange_force(const BodyView &B, int t, R area, const R *arm, R *f) {
    if (B.centroid) {
        for (int c = 0; c < 3; ++c) f[c] = -area * R(B.Flc[3 * t + c]);
        f[3] = arm[1] * f[2] - arm[2] * f[1];
        f[4] = arm[2] * f[0] - arm[0] * f[2];
        f[5] = arm[0] * f[1] - arm[1] * f[0];
        return;
    }
    // each corner carries a third of the triangle's area
    const R c = -area / R(3);
    const R *Xr = (const R *)B.Xrel;
    R xc[3];
    for (int a = 0; a < 3; ++a) xc[a] = R(__ldcg(B.rstate + RigidState::XC + a) - B.origin[a]);
    for (int q = 0; q < 3; ++q) {
        const int v = B.tri[3 * t + q];
        const R Fv[3] = {c * R(B.Fl[3 * v]), c * R(B.Fl[3 * v + 1]), c * R(B.Fl[3 * v + 2])};
        const R r[3] = {Xr[3 * v] - xc[0], Xr[3 * v + 1] - xc[1], Xr[3 * v + 2] - xc[2]};
        for (int a = 0; a < 3; ++a) f[a] += Fv[a];
        f[3] += r[1] * Fv[2] - r[2] * Fv[1];
        f[4] += r[2] * Fv[0] - r[0] * Fv[2];
        f[5] += r[0] * Fv[1] - r[1] * Fv[0];
    }
}

// MLS at markers and probes, one thread per point.  Points 0..nm-1 are the
// markers (the vertices, or the triangle centroids); point nm + 2t + side is
// the probe of triangle t on the outer (side 0) or inner (side 1) face.  With p_k = (1, x_k - X) the fit of a
// field f is a = A^-1 b_f, A = sum_k W_k p_k p_k^T, b_f = sum_k W_k p_k f_k
// (Eq. l2norm), i.e. f(X) = a_0 and grad f = (a_1, a_2, a_3).
//  positions: the point (probes: triangle geometry), the nearest node base =
//           floor(X + 1/2) and the exact offset X - base.
//           Nothing here reads the moments: with kChain it runs while the
//           moments kernel ends, and so reads the positions at the L2
//           (chain_release's comment);
//  sums:    W is a product over the axes but for its cut-off r_k <= 1 (a bit
//           per node, decided exactly as in FP64), so the ten sums of A and
//           the sixteen of b (fields less those of the centre node) are formed
//           axis by axis: x within each row of three nodes, then y, then z
//           (about 800 operations a point; 1250 when formed node by node);
//  solve:   inverse of A (FP64 adjugate in the FP64 path, FP32 L D L^T in
//           the FP32 one); markers get U = (A^-1 b_u)_0 + u_c (Eq. uLag),
//           probes the pressure c_s^2 rho and the traction
//           rho nu (grad u + grad u^T) . n from the fits (membranes keep
//           them per triangle, rigid bodies sum the forces and moments).
//           A rigid body's two probes of a triangle are rounded and summed
//           apart, so both take their pressure less that of the node nearest
//           to the triangle's first corner: an offset of the density leaves
//           before the first rounding (density 1.1, sphere of radius 4 to 8,
//           error of the FP32 angular impulse against FP64: 10 to 21e-9 with
//           the full pressures, 3 to 14e-9 as differences per triangle,
//           3 to 14e-9 so).  Its density is fetched with the moments for all
//           points, without a branch: 48^3 FP32 sphere 18.67 us a step (18.26
//           with the full pressures, 18.98 with a branch), 64^3 capsule 19.1 to
//           19.2 (19.02, 19.3).
template <typename R, bool kCG = false, bool kChain = false>
__device__ __forceinline__ void mls_body(const R *mom, const Lattice &L, const BodyView &B, int *err,
                                         const int vb) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nm = B.nm, npts = nm + 2 * B.nt;
    const int slot = vb * blockDim.x + threadIdx.x;
    const int n[3] = {L.nx, L.ny, L.nz};
    const int p = slot < npts ? (B.perm ? B.perm[slot] : slot) : -1;

    // ---------------- positions ----------------
    double vol = 0.0, frac[3] = {0.0, 0.0, 0.0};
    R nrm[3] = {R(0), R(0), R(0)}, arm[3] = {R(0), R(0), R(0)}, area = R(0);  // probes: normal, X_c - x_c, area
    int base[3] = {2, 2, 2}, ref = 0;  // ref: the node whose density a rigid body's probe refers to
    if (p >= 0) {
        double P[3];
        if (p < nm && B.centroid) {
            const int *tv = B.tri + 3 * p;
            for (int a = 0; a < 3; ++a)
                P[a] = (__ldcg(B.X + 3 * tv[0] + a) + __ldcg(B.X + 3 * tv[1] + a) + __ldcg(B.X + 3 * tv[2] + a)) / 3.0;
        } else if (p < nm) {
            for (int a = 0; a < 3; ++a) P[a] = __ldcg(B.X + 3 * p + a);
        } else {
            // probe X_c +- 1.2 n, with X_c = x_0 + (e1 + e2)/3 and the
            // triangle's edges and normal from origin-relative positions
            const int t = (p - nm) >> 1, side = (p - nm) & 1;
            const int tv[3] = {B.tri[3 * t], B.tri[3 * t + 1], B.tri[3 * t + 2]};
            const R *Xr = (const R *)B.Xrel;
            R r0[3], e1[3], e2[3];
            for (int a = 0; a < 3; ++a) {
                P[a] = __ldcg(B.X + 3 * tv[0] + a);
                r0[a] = __ldcg(Xr + 3 * tv[0] + a);
                e1[a] = __ldcg(Xr + 3 * tv[1] + a) - r0[a];
                e2[a] = __ldcg(Xr + 3 * tv[2] + a) - r0[a];
            }
            const R N[3] = {e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2],
                            e1[0] * e2[1] - e1[1] * e2[0]};
            const R nn = sqrt(N[0] * N[0] + N[1] * N[1] + N[2] * N[2]);
            const R inn = R(1) / nn, sg = side ? R(-kProbe) : R(kProbe);
            R *tg = (R *)B.tri_geo + 8 * t;
            area = R(0.5) * nn;
            if (B.rigid)
                ref = near_coord(L, 0, P[0]) + L.nx * (near_coord(L, 1, P[1]) + L.ny * near_coord(L, 2, P[2]));
            for (int a = 0; a < 3; ++a) {
                nrm[a] = N[a] * inn;
                const R c3 = (e1[a] + e2[a]) / R(3);
                P[a] += (double)(c3 + sg * nrm[a]);
                arm[a] = r0[a] + c3;
                if (side == 0) {
                    tg[a] = nrm[a];
                    tg[4 + a] = arm[a];
                }
            }
            if (side == 0) {
                tg[3] = area;
                if (!B.rigid)
                    vol = (double)r0[0] * (double)N[0] + (double)r0[1] * (double)N[1] + (double)r0[2] * (double)N[2];
            }
            if (B.rigid)
                for (int a = 0; a < 3; ++a) arm[a] -= R(__ldcg(B.rstate + RigidState::XC + a) - B.origin[a]);
        }
        bool bad = false, diverged = false;
        for (int a = 0; a < 3; ++a) {
            if (!(fabs(P[a]) < kMaxMarkerCoord)) {  // non-finite or runaway: flag, keep indices sane
                diverged = true;
                P[a] = 0.0;
            }
            int b = __double2int_rd(P[a] + 0.5);  // floor(X + 1/2)
            if (L.bc[a] == kWall && (b - 1 < 1 || b + 1 > n[a] - 2)) {
                bad = true;
                b = b < 2 ? 2 : (b > n[a] - 3 ? n[a] - 3 : b);
            }
            base[a] = b;
            frac[a] = P[a] - (double)b;
        }
        if (diverged)
            atomicCAS(err, 0, kErrDiverged);
        else if (bad)
            atomicCAS(err, 0, kErrBodyWall);
    }
    // weights and the support's nodes (r_k <= 1, Eq. intKernel): FP32 squared
    // distances, and the FP64 ones of nodes whose decision FP32 rounding
    // (below 1e-6 here) could flip
    R d[3][3], w[3][3];
    unsigned in = 0u, near = 0u;
    {
        float sq[3][3];
        for (int a = 0; a < 3; ++a) {
            axis_weights(R(frac[a]), d[a], w[a]);
            const float f = float(frac[a]);
#pragma unroll
            for (int i = 0; i < 3; ++i) sq[a][i] = (float(i - 1) - f) * (float(i - 1) - f);
        }
#pragma unroll
        for (int q = 0; q < 27; ++q) {
            const float t = sq[0][q % 3] + (sq[1][(q / 3) % 3] + sq[2][q / 9]) - L.dist2_cut_f;
            if (t <= 0.f) in |= 1u << q;
            if (fabsf(t) <= 1e-5f) near |= 1u << q;
        }
        if (near) in = (in & ~near) | support_exact(near, frac[0], frac[1], frac[2], L.dist2_cut);
    }
    if constexpr (kChain) chain_wait();  // (kCG: no read-only loads behind it)
    R f6[6] = {R(0), R(0), R(0), R(0), R(0), R(0)};  // rigid: the point's share of the force and moment
    if (p >= 0) {
    // ---------------- sums ----------------
    int ox[3], oy[3], oz[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        ox[i] = support_coord(L, 0, base[0] + i - 1);
        oy[i] = L.nx * support_coord(L, 1, base[1] + i - 1);
        oz[i] = L.nx * L.ny * support_coord(L, 2, base[2] + i - 1);
    }
    // fit f - f_c, f_c the moments of the centre node (always in the
    // support): the same fit, since MLS reproduces constants, but the sums
    // and the solve then carry the field's variation over the support rather
    // than its size, which the gradients at the probes (small differences of
    // the fitted values) need
    R fc[4];
    mom_load<kCG>(mom, ox[1] + oy[1] + oz[1], fc);
    const R fr = ld_ro<kCG>(mom + 4 * (size_t)(p >= nm && B.rigid ? ref : ox[1] + oy[1] + oz[1]));
    // A: 00, 01, 02, 03, 11, 12, 13, 22, 23, 33; b[c]: 1, x, y, z
    R A[10], b[4][4];
#pragma unroll
    for (int q = 0; q < 10; ++q) A[q] = R(0);
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int q = 0; q < 4; ++q) b[c][q] = R(0);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        R T[6], Tf[4][3];  // sums over the plane: 1, x, y, xx, xy, yy; fields: 1, x, y
#pragma unroll
        for (int q = 0; q < 6; ++q) T[q] = R(0);
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int q = 0; q < 3; ++q) Tf[c][q] = R(0);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            R S0 = R(0), S1 = R(0), S2 = R(0), F0[4], F1[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) F0[c] = F1[c] = R(0);
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                R v[4];
                mom_load<kCG>(mom, ox[i] + oy[j] + oz[k], v);
                const R a0 = (in >> (i + 3 * j + 9 * k)) & 1u ? w[0][i] : R(0), a1 = a0 * d[0][i];
                S0 += a0;
                S1 += a1;
                S2 += a1 * d[0][i];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const R f = v[c] - fc[c];
                    F0[c] += a0 * f;
                    F1[c] += a1 * f;
                }
            }
            const R w1 = w[1][j], w1d = w1 * d[1][j];
            T[0] += w1 * S0;
            T[1] += w1 * S1;
            T[2] += w1d * S0;
            T[3] += w1 * S2;
            T[4] += w1d * S1;
            T[5] += (w1d * d[1][j]) * S0;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                Tf[c][0] += w1 * F0[c];
                Tf[c][1] += w1 * F1[c];
                Tf[c][2] += w1d * F0[c];
            }
        }
        const R w2 = w[2][k], w2d = w2 * d[2][k];
        A[0] += w2 * T[0];
        A[1] += w2 * T[1];
        A[2] += w2 * T[2];
        A[3] += w2d * T[0];
        A[4] += w2 * T[3];
        A[5] += w2 * T[4];
        A[6] += w2d * T[1];
        A[7] += w2 * T[5];
        A[8] += w2d * T[2];
        A[9] += (w2d * d[2][k]) * T[0];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            b[c][0] += w2 * Tf[c][0];
            b[c][1] += w2 * Tf[c][1];
            b[c][2] += w2 * Tf[c][2];
            b[c][3] += w2d * Tf[c][0];
        }
    }

    // ---------------- solve ----------------
    R Ai[16];
    if (!spd_inverse4(A, Ai)) atomicCAS(err, 0, -1);
    if (p < nm) {
        double *Uo = B.centroid ? B.Uc : B.U;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const R *bu = b[1 + c];
            Uo[3 * p + c] = (double)(fc[1 + c] + (Ai[3] * bu[3] + Ai[2] * bu[2] + Ai[1] * bu[1] + Ai[0] * bu[0]));
        }
        R rec[kRec];
#pragma unroll
        for (int q = 0; q < 4; ++q) rec[q] = Ai[q];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            rec[4 + a] = R(frac[a]);
#pragma unroll
            for (int i = 0; i < 3; ++i) rec[7 + 3 * a + i] = w[a][i];
        }
        store_record((R *)B.phi + (size_t)kRec * p, rec);
        reinterpret_cast<int4 *>(B.node)[p] = make_int4(base[0], base[1], base[2], (int)in);
    } else {
        // fits: c_f[i] = sum_m Ai[i][m] b_f[m], plus the centre value for
        // the value (i = 0)
        const R c0 = Ai[0] * b[0][0] + Ai[1] * b[0][1] + Ai[2] * b[0][2] + Ai[3] * b[0][3];
        R gr[3][3];
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const R *bu = b[1 + c], *row = Ai + 4 * (a + 1);
                gr[c][a] = row[0] * bu[0] + row[1] * bu[1] + row[2] * bu[2] + row[3] * bu[3];
            }
        const int t = (p - nm) >> 1, side = (p - nm) & 1;
        const R rn = (R(1) + (c0 + fc[0])) * pick<R>(L.nu_d, L.nu_f);
        const R pr0 = (c0 + (B.rigid ? fc[0] - fr : fc[0])) / R(3);  // p - c_s^2 rho0 (rigid: less that of node ref)
        R tr[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            R acc = R(0);
#pragma unroll
            for (int a = 0; a < 3; ++a) acc += (gr[c][a] + gr[a][c]) * nrm[a];
            tr[c] = rn * acc;
        }
        if (!B.rigid) {
            R *pr = (R *)B.probe + 8 * t + 4 * side;
            pr[0] = pr0;
            for (int c = 0; c < 3; ++c) pr[1 + c] = tr[c];
        } else if (!B.rigid_force) {
            // the probe's side of the stress jump (Eqs. hydroForP, hydroForNu):
            // +-(-p n + tau . n) A and its moment about x_c
            const R sA = side ? -area : area;
            for (int c = 0; c < 3; ++c) f6[c] = (tr[c] - pr0 * nrm[c]) * sA;
            f6[3] = arm[1] * f6[2] - arm[2] * f6[1];
            f6[4] = arm[2] * f6[0] - arm[0] * f6[2];
            f6[5] = arm[0] * f6[1] - arm[1] * f6[0];
        } else if (side == 0) {
            exchange_force<R>(B, t, area, arm, f6);
        }
    }
    }
    // the block's partial sums, in a fixed order: enclosed volume (membranes)
    // or force and moment (rigid bodies)
    __shared__ double red[6][8];
    const int nw = blockDim.x >> 5;
    if (B.rigid) {
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            const R sum = warp_sum(f6[q]);
            if (lane == 0) red[q][warp] = (double)sum;
        }
    } else {
        vol = warp_sum(vol);
        if (lane == 0) red[0][warp] = vol;
    }
    __syncthreads();
    if ((int)threadIdx.x < body_sums(B)) {
        double acc = 0.0;
        for (int k = 0; k < nw; ++k) acc += red[threadIdx.x][k];
        B.part[body_sums(B) * vb + threadIdx.x] = acc;
    }
}

// The same with four lanes per point, for few points (mls_quads): lane a < 3
// forms the point's component and the weights of axis a, and lane q takes
// field q (rho - 1, u_x, u_y, u_z), with the sums of A split by the power of x
// over lanes 0 to 2.  A point's chain of operations is about a third of
// mls_body's (FP64: 385 instead of 1080 warp instructions, each holding its
// SM quarter for 64 cycles), over four times the warps.
constexpr int kQuadThreads = 128;  // 32 points a block
// x / 3, rounded as the division (whose FP64 form takes a dozen operations)
template <typename R>
__device__ __forceinline__ R third(R x) {
    const R q = x * R(1.0 / 3.0);
    return fma(fma(R(-3), q, x), R(1.0 / 3.0), q);
}
template <typename R>
__device__ __forceinline__ void mls_quad_body(const R *mom, const Lattice &L, const BodyView &B, int *err,
                                              const int vb) {
    const unsigned kFull = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, q = lane & 3, qb = lane & ~3;
    auto from = [&](auto v, int src) { return __shfl_sync(kFull, v, qb | src); };  // lane src of the point
    const int a = q < 3 ? q : 0, a1 = (a + 1) % 3, a2 = (a + 2) % 3;
    const int nm = B.nm, npts = nm + 2 * B.nt;
    const int slot = vb * (kQuadThreads / 4) + (threadIdx.x >> 2);
    const int p = slot < npts ? (B.perm ? B.perm[slot] : slot) : -1;
    const bool probe = p >= nm;
    const int t = probe ? (p - nm) >> 1 : 0, side = (p - nm) & 1;

    // ---------------- positions: component a ----------------
    double P = 0.0;
    int rc = 0;  // rigid: coordinate of the node whose density the probe refers to
    R r0 = R(0), e1 = R(0), e2 = R(0);
    if (probe) {
        const int *tv = B.tri + 3 * t;
        const int i0 = tv[0], i1 = tv[1], i2 = tv[2];
        const R *Xr = (const R *)B.Xrel;
        P = __ldcg(B.X + 3 * i0 + a);
        if (B.rigid) rc = near_coord(L, a, P);
        r0 = __ldcg(Xr + 3 * i0 + a);
        e1 = __ldcg(Xr + 3 * i1 + a) - r0;
        e2 = __ldcg(Xr + 3 * i2 + a) - r0;
    } else if (p >= 0 && B.centroid) {
        const int *tv = B.tri + 3 * p;
        P = (__ldcg(B.X + 3 * tv[0] + a) + __ldcg(B.X + 3 * tv[1] + a) + __ldcg(B.X + 3 * tv[2] + a)) / 3.0;
    } else if (p >= 0) {
        P = __ldcg(B.X + 3 * p + a);
    }
    const R e1b = from(e1, a1), e1c = from(e1, a2), e2b = from(e2, a1), e2c = from(e2, a2);
    const R N = e1b * e2c - e1c * e2b;
    const R N0 = from(N, 0), N1 = from(N, 1), N2 = from(N, 2);
    const R nn = sqrt(N0 * N0 + N1 * N1 + N2 * N2), area = R(0.5) * nn;
    R nrm = R(0), arm = R(0);
    if (probe) {
        nrm = N * (R(1) / nn);
        const R c3 = third(e1 + e2);
        P += (double)(c3 + (side ? R(-kProbe) : R(kProbe)) * nrm);
        arm = r0 + c3;
        if (side == 0) {
            R *tg = (R *)B.tri_geo + 8 * t;
            if (q < 3) {
                tg[a] = nrm;
                tg[4 + a] = arm;
            } else {
                tg[3] = area;
            }
        }
        if (B.rigid) arm -= R(__ldcg(B.rstate + RigidState::XC + a) - B.origin[a]);
    }
    double vol = 0.0;  // on lane 0
    if (!B.rigid) {
        const double v = (double)r0 * (double)N;
        vol = from(v, 0) + from(v, 1) + from(v, 2);
        if (q != 0 || !probe || side != 0) vol = 0.0;
    }
    const int n = a == 0 ? L.nx : a == 1 ? L.ny : L.nz;
    bool diverged = false, bad = false;
    if (!(fabs(P) < kMaxMarkerCoord)) {  // non-finite or runaway: flag, keep indices sane
        diverged = p >= 0;
        P = 0.0;
    }
    int base = __double2int_rd(P + 0.5);  // floor(X + 1/2)
    if (L.bc[a] == kWall && (base - 1 < 1 || base + 1 > n - 2)) {
        bad = p >= 0;
        base = base < 2 ? 2 : (base > n - 3 ? n - 3 : base);
    }
    const double frac = P - (double)base;
    const unsigned mdiv = __ballot_sync(kFull, diverged) >> qb & 7u, mbad = __ballot_sync(kFull, bad) >> qb & 7u;
    if (q == 0 && mdiv)
        atomicCAS(err, 0, kErrDiverged);
    else if (q == 0 && mbad)
        atomicCAS(err, 0, kErrBodyWall);

    // ---------------- weights, support and nodes ----------------
    const R fR = R(frac), f0 = from(fR, 0), f1 = from(fR, 1), f2 = from(fR, 2);
    const double g0 = from(frac, 0), g1 = from(frac, 1), g2 = from(frac, 2);
    unsigned in = 0u, near = 0u;
    {
        const float fx = float(f0), fy = float(f1), fz = float(f2);
        float sx[3], sy[3], sz[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            sx[i] = (float(i - 1) - fx) * (float(i - 1) - fx);
            sy[i] = (float(i - 1) - fy) * (float(i - 1) - fy);
            sz[i] = (float(i - 1) - fz) * (float(i - 1) - fz);
        }
#pragma unroll
        for (int k = 0; k < 27; ++k) {
            const float s = sx[k % 3] + (sy[(k / 3) % 3] + sz[k / 9]) - L.dist2_cut_f;
            if (s <= 0.f) in |= 1u << k;
            if (fabsf(s) <= 1e-5f) near |= 1u << k;
        }
        if (near) in = (in & ~near) | support_exact(near, g0, g1, g2, L.dist2_cut);
    }
    R wx[3], wxd[3], wxp[3], wy[3], wyd[3], wydd[3], wz[3], wzd[3], wzdd[3];
    {
        R d[3], w[3];
        axis_weights(fR, d, w);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const R wd = w[i] * d[i], wdd = wd * d[i];
            wx[i] = from(w[i], 0);
            wxd[i] = from(wd, 0);
            const R xdd = from(wdd, 0);
            wxp[i] = q == 0 ? wx[i] : q == 1 ? wxd[i] : xdd;
            wy[i] = from(w[i], 1);
            wyd[i] = from(wd, 1);
            wydd[i] = from(wdd, 1);
            wz[i] = from(w[i], 2);
            wzd[i] = from(wd, 2);
            wzdd[i] = from(wdd, 2);
        }
    }
    int ox[3], oy[3], oz[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const int o = (a == 0 ? 1 : a == 1 ? L.nx : L.nx * L.ny) * support_coord(L, a, base + i - 1);
        ox[i] = from(o, 0);
        oy[i] = from(o, 1);
        oz[i] = from(o, 2);
    }
    const int centre = ox[1] + oy[1] + oz[1];
    const int ref = B.rigid ? from(rc, 0) + L.nx * (from(rc, 1) + L.ny * from(rc, 2)) : centre;
    chain_wait();

    // ---------------- sums: field q, and A by the power of x ----------------
    const R *mq = mom + q;
    const R fc = ld_ca(mq + 4 * (size_t)centre), fr = ld_ca(mom + 4 * (size_t)ref);
    R b[4] = {R(0), R(0), R(0), R(0)};
    R C00 = R(0), C10 = R(0), C20 = R(0), C01 = R(0), C11 = R(0), C02 = R(0);  // y and z powers
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        R T0 = R(0), T1 = R(0), T2 = R(0), U0 = R(0), U1 = R(0), U2 = R(0);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            R F0 = R(0), F1 = R(0), S = R(0);
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const R f = ld_ca(mq + 4 * (size_t)(ox[i] + oy[j] + oz[k])) - fc;
                const bool on = (in >> (i + 3 * j + 9 * k)) & 1u;
                F0 += (on ? wx[i] : R(0)) * f;
                F1 += (on ? wxd[i] : R(0)) * f;
                S += on ? wxp[i] : R(0);
            }
            T0 += wy[j] * F0;
            T1 += wy[j] * F1;
            T2 += wyd[j] * F0;
            U0 += wy[j] * S;
            U1 += wyd[j] * S;
            U2 += wydd[j] * S;
        }
        b[0] += wz[k] * T0;
        b[1] += wz[k] * T1;
        b[2] += wz[k] * T2;
        b[3] += wzd[k] * T0;
        C00 += wz[k] * U0;
        C10 += wz[k] * U1;
        C20 += wz[k] * U2;
        C01 += wzd[k] * U0;
        C11 += wzd[k] * U1;
        C02 += wzdd[k] * U0;
    }
    const R A[10] = {from(C00, 0), from(C00, 1), from(C10, 0), from(C01, 0), from(C00, 2),
                     from(C10, 1), from(C01, 1), from(C20, 0), from(C11, 0), from(C02, 0)};

    // ---------------- solve ----------------
    R Ai[16];
    if (!spd_inverse4(A, Ai) && p >= 0) atomicCAS(err, 0, -1);
    const R fit = Ai[3] * b[3] + Ai[2] * b[2] + Ai[1] * b[1] + Ai[0] * b[0], val = fc + fit;
    const int b0 = from(base, 0), b1 = from(base, 1), b2 = from(base, 2);
    const R x0 = wx[0], x1 = wx[1], x2 = wx[2], y0 = wy[0], y1 = wy[1], y2 = wy[2], z0 = wz[0], z1 = wz[1], z2 = wz[2];
    if (p >= 0 && !probe) {
        double *Uo = B.centroid ? B.Uc : B.U;
        if (q > 0) Uo[3 * p + q - 1] = (double)val;
        // the transfer record, four values a lane
        R *rec = (R *)B.phi + (size_t)kRec * p + 4 * q;
        rec[0] = q == 0 ? Ai[0] : q == 1 ? f0 : q == 2 ? x1 : y2;
        rec[1] = q == 0 ? Ai[1] : q == 1 ? f1 : q == 2 ? x2 : z0;
        rec[2] = q == 0 ? Ai[2] : q == 1 ? f2 : q == 2 ? y0 : z1;
        rec[3] = q == 0 ? Ai[3] : q == 1 ? x0 : q == 2 ? y1 : z2;
        if (q == 0) reinterpret_cast<int4 *>(B.node)[p] = make_int4(b0, b1, b2, (int)in);
    }
    // probes: lane q > 0 has the gradient of velocity component q - 1
    R g[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const R *row = Ai + 4 * (c + 1);
        g[c] = row[0] * b[0] + row[1] * b[1] + row[2] * b[2] + row[3] * b[3];
    }
    const R cr = from(val, 0), n0 = from(nrm, 0), n1 = from(nrm, 1), n2 = from(nrm, 2);
    R acc = g[0] * n0 + g[1] * n1 + g[2] * n2;  // row of the gradient, and below its column
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const R col = from(g[c], 1) * n0 + from(g[c], 2) * n1 + from(g[c], 3) * n2;
        if (q == c + 1) acc += col;
    }
    // p - c_s^2 rho0 (rigid: less that of node ref)
    const R tr = (R(1) + cr) * pick<R>(L.nu_d, L.nu_f) * acc, pr0 = third(from(B.rigid ? (fc - fr) + fit : val, 0));
    if (probe && !B.rigid) ((R *)B.probe + 8 * t + 4 * side)[q] = q == 0 ? pr0 : tr;
    __shared__ double red[6][kQuadThreads / 32];
    if (B.rigid) {
        // the probe's side of the stress jump, or the momentum exchange:
        // component q - 1 of force and moment on lane q > 0
        const R ar[3] = {from(arm, 0), from(arm, 1), from(arm, 2)};
        R F = R(0), M = R(0);
        if (B.rigid_force) {
            R f6[6] = {R(0), R(0), R(0), R(0), R(0), R(0)};
            if (probe && side == 0 && q == 0) exchange_force<R>(B, t, area, ar, f6);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const R Fc = from(f6[c], 0), Mc = from(f6[3 + c], 0);
                if (q == c + 1) {
                    F = Fc;
                    M = Mc;
                }
            }
        } else {
            const R nq = q == 1 ? n0 : q == 2 ? n1 : n2;
            if (probe && q > 0) F = (tr - pr0 * nq) * (side ? -area : area);
            const R F0 = from(F, 1), F1 = from(F, 2), F2 = from(F, 3);
            if (q == 1) M = ar[1] * F2 - ar[2] * F1;
            if (q == 2) M = ar[2] * F0 - ar[0] * F2;
            if (q == 3) M = ar[0] * F1 - ar[1] * F0;
        }
#pragma unroll
        for (int o = 16; o >= 4; o >>= 1) {
            F += __shfl_xor_sync(kFull, F, o);
            M += __shfl_xor_sync(kFull, M, o);
        }
        if (lane > 0 && lane < 4) {
            red[lane - 1][warp] = (double)F;
            red[lane + 2][warp] = (double)M;
        }
    } else {
#pragma unroll
        for (int o = 16; o >= 4; o >>= 1) vol += __shfl_xor_sync(kFull, vol, o);
        if (lane == 0) red[0][warp] = vol;
    }
    __syncthreads();
    if ((int)threadIdx.x < body_sums(B)) {
        double s = 0.0;
        for (int k = 0; k < kQuadThreads / 32; ++k) s += red[threadIdx.x][k];
        B.part[body_sums(B) * vb + threadIdx.x] = s;
    }
}

// The blocks take the nvb groups of points in turn (gridDim.x = nvb unless
// the launch caps the grid).
template <typename R>
__global__ void __launch_bounds__(mls_threads(sizeof(R) == 8 ? 0 : 1)) k_mls(const R *mom, Lattice L, BodyView B,
                                                     int *err, int nvb) {
    chain_release();  // the structure kernel may be scheduled beside this one
    for (int vb = blockIdx.x; vb < nvb; vb += gridDim.x) {
        // launched programmatically after the moments kernel, whose results
        // it waits for inside
        mls_body<R, true, true>(mom, L, B, err, vb);
        __syncthreads();  // the next group reuses the shared memory
    }
}

template <typename R>
__global__ void __launch_bounds__(kQuadThreads) k_mls_quad(const R *mom, Lattice L, BodyView B, int *err,
                                                           int nvb) {
    chain_release();  // the structure kernel may be scheduled beside this one
    for (int vb = blockIdx.x; vb < nvb; vb += gridDim.x) {
        mls_quad_body<R>(mom, L, B, err, vb);
        __syncthreads();  // the next group reuses the shared memory
    }
}

// Hydrodynamic force on triangle t from its two probes (Eqs. hydroForP,
// hydroForNu): F = [-(p+ - p-) n + (tau+ - tau-) . n] A.
template <typename R>
__device__ __forceinline__ void tri_hydro(const BodyView &B, int t, R *F) {
    const R *tg = (const R *)B.tri_geo + 8 * t;
    const R *pp = (const R *)B.probe + 8 * t, *pm = pp + 4;
    const R A = tg[3];
    for (int a = 0; a < 3; ++a) F[a] = (-(pp[0] - pm[0]) * tg[a] + (pp[1 + a] - pm[1 + a])) * A;
}

// Spreading by the 8 lanes of a marker: c phi_k F added to the force field
// at the support nodes with r_k <= 1 (the others have phi_k = 0), from the
// marker's transfer record; the tiles of the 27 nodes' 8 corners are flagged.
// These are all their tiles, but for a middle node that is a tile by itself:
// the last node of a periodic axis of 8 m + 1 nodes (Lattice::seam).
constexpr int kLanes = 8;  // lanes per marker in the structure kernels
template <typename R>
__device__ __forceinline__ void spread(const Lattice &L, const BodyView &B, int p, int l8, R c, const R *Fl,
                                       R *__restrict__ force, uint32_t *stamp, uint32_t step) {
    const R *rec = (const R *)B.phi + (size_t)kRec * p;
    const int4 bs = reinterpret_cast<const int4 *>(B.node)[p];
    const R r0 = rec[0], r1 = rec[1], r2 = rec[2], r3 = rec[3], fx = rec[4], fy = rec[5], fz = rec[6];
    const R F0 = c * Fl[0], F1 = c * Fl[1], F2 = c * Fl[2];
    const long long st = L.stride;
#pragma unroll
    for (int q = l8; q < 27; q += kLanes) {
        if (!((unsigned)bs.w >> q & 1u)) continue;
        const int i = q % 3, j = (q / 3) % 3, k = q / 9;
        const int node = support_coord(L, 0, bs.x + i - 1) +
                         L.nx * (support_coord(L, 1, bs.y + j - 1) + L.ny * support_coord(L, 2, bs.z + k - 1));
        const R phi = (rec[7 + i] * rec[10 + j] * rec[13 + k]) *
                      (r0 + r1 * (R(i - 1) - fx) + r2 * (R(j - 1) - fy) + r3 * (R(k - 1) - fz));
        atomicAdd(force + node, phi * F0);
        atomicAdd(force + st + node, phi * F1);
        atomicAdd(force + 2 * st + node, phi * F2);
    }
    auto flag = [&](int i, int j, int k) {
        const int x = support_coord(L, 0, bs.x + i), y = support_coord(L, 1, bs.y + j), z = support_coord(L, 2, bs.z + k);
        stamp[(x >> 3) + L.ntx * ((y >> 3) + L.nty * (z >> 3))] = step;
    };
    const bool seam = (L.seam & 1 && support_coord(L, 0, bs.x) == L.nx - 1) ||
                      (L.seam & 2 && support_coord(L, 1, bs.y) == L.ny - 1) ||
                      (L.seam & 4 && support_coord(L, 2, bs.z) == L.nz - 1);
    if (!seam) {
        flag(l8 & 1 ? 1 : -1, l8 & 2 ? 1 : -1, l8 & 4 ? 1 : -1);
    } else {
        for (int q = l8; q < 27; q += kLanes) flag(q % 3 - 1, (q / 3) % 3 - 1, q / 9 - 1);
    }
}
template <typename T>
__device__ __forceinline__ T lanes_sum(T v) {  // over the 8 lanes of a marker
#pragma unroll
    for (int o = kLanes / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// A body's sum q over the partials of its MLS blocks (called by whole warps;
// a fixed order).  Above kDirectParts partials k_body_sums has added them up
// into the slot behind them.
constexpr int kDirectParts = 512;
__device__ __forceinline__ double body_sum(const BodyView &B, int nparts, int q) {
    const int ns = body_sums(B), lane = threadIdx.x & 31;
    const double *part = B.part;
    if (nparts > kDirectParts) return __ldcg(part + (size_t)ns * nparts + q);
    double s = 0.0;
    for (int k = lane; k < nparts; k += 32) s += __ldcg(part + (size_t)ns * k + q);
    return warp_sum(s);
}
__device__ __forceinline__ void body_sums_body(const BodyView &B, int nparts) {
    const int ns = body_sums(B), lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    __shared__ double red[6][8];
    // every warp takes a share of the partials of all sums
    double s[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    const double *part = B.part;
    for (int k = threadIdx.x; k < nparts; k += blockDim.x)
        for (int q = 0; q < ns; ++q) s[q] += __ldcg(part + (size_t)ns * k + q);
    for (int q = 0; q < ns; ++q) {
        const double t = warp_sum(s[q]);
        if (lane == 0) red[q][threadIdx.x >> 5] = t;
    }
    __syncthreads();
    if ((int)threadIdx.x < ns) {
        double t = 0.0;
        for (int w = 0; w < nw; ++w) t += red[threadIdx.x][w];
        B.part[(size_t)ns * nparts + threadIdx.x] = t;
    }
}
__global__ void __launch_bounds__(256) k_body_sums(BodyView B, int nparts) {
    chain_release();
    chain_wait();
    body_sums_body(B, nparts);
}

// Node box of level n+1: each block reduces its markers' cells in shared
// memory and then updates the global box once (contention on the six
// global words stays at one update per block).
struct BlockBox {
    int v[6];
    __device__ void init() {
        if (threadIdx.x < 6) v[threadIdx.x] = threadIdx.x < 3 ? 0x7fffffff : (int)0x80000000;
    }
    __device__ void add(int a, double x) {
        const int c = __double2int_rd(x);
        atomicMin(&v[a], c - kBoxLo);
        atomicMax(&v[3 + a], c + kBoxHi);
    }
    __device__ void flush(int *box) {
        if (threadIdx.x < 3)
            atomicMin(box + threadIdx.x, v[threadIdx.x]);
        else if (threadIdx.x < 6)
            atomicMax(box + threadIdx.x, v[threadIdx.x]);
    }
};

// Membrane vertex update, 8 lanes per vertex: spring (Eq. strainFor),
// bending (gradient of k_b[1 - cos(theta - theta0)], reading of Eq. bendFor),
// volume penalty (restoring reading of Eq. volFor) and element hydrodynamic
// forces shared 1/3 per vertex (Eq. newtonSoft), with the lanes sharing the
// incident hinges (12 on a regular mesh) and triangles (6); Verlet positions
// (Eqs. verletPos, verletVel) in FP64, one thread per component; boundary
// velocity U_b = U + F/m_v dt; the Lagrangian force F_l = U_b - U spread with
// c_l = A_l (Eq. bodyforce).  The hinges need the positions only: launched
// programmatically behind the MLS kernel they run beside it, and chain_wait
// stands before the first use of its results.
template <typename R>
__device__ __forceinline__ void membrane_body(const Lattice &L, const BodyView &B, R *__restrict__ force,
                                              uint32_t *__restrict__ stamp, const uint32_t *__restrict__ dstep,
                                              const int vb, const int nparts) {
    __shared__ R s_cv;
    __shared__ BlockBox sbox;
    __shared__ R s_F[32][3];       // per vertex: total force
    __shared__ R s_Fl[32][3];      // per vertex: Lagrangian force
    __shared__ double s_U[32][3];  // centroid markers: the vertex velocity
    const int l8 = threadIdx.x & (kLanes - 1), g = threadIdx.x / kLanes;
    const int nvpb = blockDim.x / kLanes, v0 = vb * nvpb, v = v0 + g;
    R F[3] = {R(0), R(0), R(0)};
    sbox.init();
    if (v < B.nv) {
    const R *Xr = (const R *)B.Xrel;
    for (int q = B.vh_ptr[v] + l8; q < B.vh_ptr[v + 1]; q += kLanes) {
        const int role = B.vh_list[q] & 3;
        const int4 H = B.vh_verts[q];
        const R *par = (const R *)B.vh_par + 4 * q;  // k_s, l0, k_b, theta0
        const R ksh = par[0], l0h = par[1], kbh = par[2], th0h = par[3];
        R e[3], ac[3], ad[3];
        for (int a = 0; a < 3; ++a) {
            const R xa = __ldcg(Xr + 3 * H.x + a);
            e[a] = __ldcg(Xr + 3 * H.y + a) - xa;
            ac[a] = __ldcg(Xr + 3 * H.z + a) - xa;
            ad[a] = __ldcg(Xr + 3 * H.w + a) - xa;
        }
        if constexpr (sizeof(R) == 4) {
            // the FP32 coordinates carry an absolute error of half an ulp of
            // the body's size; their residuals restore the edges' own relative
            // precision, which the spring extensions l - l0 and the dihedral
            // angles (small differences of the edges) need
            const float *Xl = B.Xlo;
            for (int a = 0; a < 3; ++a) {
                const float la = __ldcg(Xl + 3 * H.x + a);
                e[a] += __ldcg(Xl + 3 * H.y + a) - la;
                ac[a] += __ldcg(Xl + 3 * H.z + a) - la;
                ad[a] += __ldcg(Xl + 3 * H.w + a) - la;
            }
        }
        const R le2 = e[0] * e[0] + e[1] * e[1] + e[2] * e[2];
        const R le = sqrt(le2), ile = rcp(le);
        if (role < 2) {
            // F_a = -k (l - l0) (x_a - x_b)/l = k (l - l0) e / l, F_b = -F_a
            const R c = ksh * (le - l0h) * ile;
            const R sg = role == 0 ? R(1) : R(-1);
            for (int a = 0; a < 3; ++a) F[a] += sg * c * e[a];
        }
        const R N1[3] = {e[1] * ac[2] - e[2] * ac[1], e[2] * ac[0] - e[0] * ac[2], e[0] * ac[1] - e[1] * ac[0]};
        const R N2[3] = {ad[1] * e[2] - ad[2] * e[1], ad[2] * e[0] - ad[0] * e[2], ad[0] * e[1] - ad[1] * e[0]};
        const R l1s = N1[0] * N1[0] + N1[1] * N1[1] + N1[2] * N1[2];
        const R l2s = N2[0] * N2[0] + N2[1] * N2[1] + N2[2] * N2[2];
        const R il1 = rcp(sqrt(l1s)), il2 = rcp(sqrt(l2s));
        R n1[3], n2[3];
        for (int a = 0; a < 3; ++a) {
            n1[a] = N1[a] * il1;
            n2[a] = N2[a] * il2;
        }
        const R cx[3] = {n1[1] * n2[2] - n1[2] * n2[1], n1[2] * n2[0] - n1[0] * n2[2], n1[0] * n2[1] - n1[1] * n2[0]};
        const R theta = atan2((cx[0] * e[0] + cx[1] * e[1] + cx[2] * e[2]) * ile,
                              n1[0] * n2[0] + n1[1] * n2[1] + n1[2] * n2[2]);
        const R dth = theta - th0h;
        const R dE = B.bend_variant ? kbh * dth : kbh * sin(dth);
        const R ile2 = ile * ile;
        const R tc = (ac[0] * e[0] + ac[1] * e[1] + ac[2] * e[2]) * ile2;
        const R td = (ad[0] * e[0] + ad[1] * e[1] + ad[2] * e[2]) * ile2;
        R c1, c2;  // dtheta/dx = c1 n1/h1 + c2 n2/h2, h = |N|/|e|
        if (role == 0) {
            c1 = R(1) - tc;
            c2 = R(1) - td;
        } else if (role == 1) {
            c1 = tc;
            c2 = td;
        } else if (role == 2) {
            c1 = R(-1);
            c2 = R(0);
        } else {
            c1 = R(0);
            c2 = R(-1);
        }
        const R g1 = c1 * le * il1, g2 = c2 * le * il2;  // c / h
        for (int a = 0; a < 3; ++a) F[a] -= dE * (g1 * n1[a] + g2 * n2[a]);
    }
    }
    const int q1 = v < B.nv ? B.vt_ptr[v + 1] : 0, q0 = v < B.nv ? B.vt_ptr[v] + l8 : 0;
    const int t0 = q0 < q1 ? B.vt_list[q0] / 3 : 0;
    // components of the block's vertices integrated below: thread 3 j + a
    const int j = threadIdx.x / 3, a = threadIdx.x % 3, vj = v0 + j;
    const bool mine = (int)threadIdx.x < 3 * nvpb && vj < B.nv;
    const double x = mine ? __ldcg(B.X + 3 * vj + a) : 0.0, xp = mine ? __ldcg(B.Xprev + 3 * vj + a) : 0.0;
    chain_wait();
    const uint32_t step = __ldcg(dstep);  // written by the moments kernel of the step
    const double U0 = mine && !B.centroid ? B.U[3 * vj + a] : 0.0;
    if ((int)threadIdx.x >= (int)blockDim.x - 32) {
        const double v6 = body_sum(B, nparts, 0);
        if ((threadIdx.x & 31) == 0) s_cv = R(B.kv * (1.0 - v6 * B.inv_6V0));
    }
    // element terms: volume penalty (G, the vertex's share of sum A n) and
    // hydrodynamic force, 1/3 per vertex
    R Al = R(0), G[3] = {R(0), R(0), R(0)};
    double Uv[3] = {0.0, 0.0, 0.0};
    for (int q = q0; q < q1; q += kLanes) {
        const int t = q == q0 ? t0 : B.vt_list[q] / 3;
        const R *tg = (const R *)B.tri_geo + 8 * t;
        const R A3 = tg[3] / R(3);
        Al += A3;
        R Fh[3] = {R(0), R(0), R(0)};
        if (!B.kinematic) tri_hydro<R>(B, t, Fh);  // kinematic IB: the fluid's stresses stay in the fluid
        for (int a = 0; a < 3; ++a) {
            G[a] += tg[a] * A3;
            F[a] += Fh[a] / R(3);
        }
        if (B.centroid)
            for (int a = 0; a < 3; ++a) Uv[a] += (double)A3 * B.Uc[3 * t + a];
    }
    for (int a = 0; a < 3; ++a) F[a] = lanes_sum(F[a]);
    for (int a = 0; a < 3; ++a) G[a] = lanes_sum(G[a]);
    Al = lanes_sum(Al);
    if (B.centroid) {
        // the vertex moves with the area-weighted mean of its triangles'
        // centroid velocities
        for (int a = 0; a < 3; ++a) Uv[a] = lanes_sum(Uv[a]);
        if (l8 == 0)
            for (int a = 0; a < 3; ++a) s_U[g][a] = Uv[a] / (double)Al;
    }
    __syncthreads();
    if (l8 == 0) {
        const R cv = s_cv;
        for (int a = 0; a < 3; ++a) s_F[g][a] = F[a] + cv * G[a];
    }
    __syncthreads();
    // Newton (Eq. newtonSoft) and Verlet (Eqs. verletPos, verletVel), dt = 1,
    // in FP64 for the block's vertices at once: thread 3 j + a integrates
    // component a of vertex j (FP64 issues per warp-instruction, so the
    // components fill whole warps)
    if (mine) {
        const double acc = (double)s_F[j][a] * B.inv_mv;
        double U = U0;
        if (B.centroid) {
            U = s_U[j][a];
            B.U[3 * vj + a] = U;
        }
        const double Ub = U + acc;
        const double Fla = Ub - U;
        double xn;
        if (B.kinematic) {
            xn = x + U;  // kinematic IB: advected with the interpolated fluid velocity
        } else {
            const double xt = x + U + 0.5 * acc;
            const double ubdf = 1.5 * xt - 2.0 * x + 0.5 * xp;
            xn = x + ubdf + 0.5 * acc;
        }
        // a vertex moving a lattice unit or more in one step (or a NaN) has
        // diverged
        if (!(fabs(xn - x) < kMaxMarkerStep)) atomicCAS(B.err, 0, kErrDiverged);
        B.Xnew[3 * vj + a] = xn;
        const double rel = xn - B.origin[a];
        ((R *)B.Xrel_next)[3 * vj + a] = R(rel);
        if constexpr (sizeof(R) == 4) B.Xlo_next[3 * vj + a] = float(rel - double(float(rel)));
        B.Ub[3 * vj + a] = Ub;
        B.Fl[3 * vj + a] = Fla;
        record(B.rec, step, 0, 3 * vj + a, xn);
        record(B.rec, step, 1, 3 * vj + a, Ub);
        record(B.rec, step, 2, 3 * vj + a, Fla);
        sbox.add(a, xn);
        s_Fl[j][a] = R(Fla);
    }
    __syncthreads();
    if (!B.centroid && v < B.nv) spread<R>(L, B, v, l8, Al, s_Fl[g], force, stamp, step);
    sbox.flush(B.bbox_next);
}

template <typename R>
__global__ void __launch_bounds__(kStructThreads) k_membrane(Lattice L, BodyView B, R *__restrict__ force,
                                                             uint32_t *__restrict__ stamp,
                                                             const uint32_t *__restrict__ dstep, int nvb, int nparts) {
    chain_release();
    for (int vb = blockIdx.x; vb < nvb; vb += gridDim.x) {
        membrane_body<R>(L, B, force, stamp, dstep, vb, nparts);
        __syncthreads();  // the next group of vertices reuses the shared memory
    }
}

// Rigid body: F = m du/dt and M = I dw/dt with I in the world frame and F
// the element stresses (or the momentum exchange) plus gravity minus
// buoyancy, second-order backward velocities (Eqs. linearVelRig,
// angularVelRig), centre and orientation advanced with the new velocities.
//
// Every block of the marker kernel does this for itself with one warp: FP64
// is a serial chain here (64 cycles per dependent operation, 16 per
// independent one, whatever the lanes), so a kernel of its own cost 10 us on
// 1280 triangles, most of it launch, cross-block reduction and the chain.
// What does not need the step's force is formed before the MLS kernel ends
// (rigid_prepare), the velocities follow in five operations
// (rigid_velocities), and the orientation (rigid_orientation) is advanced
// while the other warps form the markers' IB force.
struct RigidBlock {
    double S[RigidState::SIZE];  // state of level n, then of level n+1
    double W[9], T[9];           // R I_b^-1 R^T, and I_b^-1 R^T
    double c[6];                 // 2 v(t) - v(t - dt)/2 of u and w
    double add[6];               // force and moment besides the element sums
    double F[6];                 // the element sums
    double xo[3];                // centre of level n
    int last;
};
__device__ __forceinline__ void rigid_prepare(const BodyView &B, RigidBlock &r, const int lane) {
    for (int k = lane; k < RigidState::SIZE; k += 32) r.S[k] = __ldcg(B.rstate + k);
    __syncwarp();
    const double *S = r.S, *Rm = S + RigidState::ROT, *Ii = S + RigidState::IBINV;
    const int i = lane / 3, j = lane % 3;
    if (lane < 9) r.T[lane] = Ii[3 * i] * Rm[3 * j] + Ii[3 * i + 1] * Rm[3 * j + 1] + Ii[3 * i + 2] * Rm[3 * j + 2];
    if (lane < 6) {
        const int v = lane < 3 ? RigidState::U : RigidState::W, vp = lane < 3 ? RigidState::UP : RigidState::WP;
        r.c[lane] = 2.0 * S[v + j] - 0.5 * S[vp + j];
        double add = 0.0;
        if (lane < 3) {
            add = (S[RigidState::DENS] - 1.0) * S[RigidState::VOL] * S[RigidState::GRAV + lane];
            // momentum exchange: the fluid inside moves with the body, rho_f V du/dt
            if (B.rigid_force) add += S[RigidState::VOL] * (S[RigidState::U + lane] - S[RigidState::UP + lane]);
            r.xo[lane] = S[RigidState::XC + lane];
        }
        r.add[lane] = add;
    }
    __syncwarp();
    if (lane < 9) r.W[lane] = Rm[3 * i] * r.T[j] + Rm[3 * i + 1] * r.T[3 + j] + Rm[3 * i + 2] * r.T[6 + j];
    if (B.rigid_force) {
        // and I_f dw/dt = R I_b R^T (w - wp) rho_f / rho_s (r.T reused)
        const double *w = S + RigidState::W, *wp = S + RigidState::WP, *Ib = S + RigidState::IB;
        __syncwarp();
        if (lane < 3) r.T[lane] = Rm[lane] * (w[0] - wp[0]) + Rm[3 + lane] * (w[1] - wp[1]) + Rm[6 + lane] * (w[2] - wp[2]);
        __syncwarp();
        if (lane < 3) r.T[3 + lane] = Ib[3 * lane] * r.T[0] + Ib[3 * lane + 1] * r.T[1] + Ib[3 * lane + 2] * r.T[2];
        __syncwarp();
        if (lane < 3)
            r.add[3 + lane] =
                (Rm[3 * lane] * r.T[3] + Rm[3 * lane + 1] * r.T[4] + Rm[3 * lane + 2] * r.T[5]) / S[RigidState::DENS];
    }
    __syncwarp();
}
// The body's sums over the MLS blocks' partials, 16 lanes each.
__device__ __forceinline__ void rigid_sums(const BodyView &B, RigidBlock &r, const int nparts) {
    const int h = threadIdx.x >> 4, l = threadIdx.x & 15, nh = blockDim.x >> 4;
    const double *part = B.part;
    for (int q0 = 0; q0 < 6; q0 += nh) {
        const int q = q0 + h;
        double t = 0.0;
        if (q < 6) {
            if (nparts > kDirectParts)
                t = l == 0 ? __ldcg(part + 6 * (size_t)nparts + q) : 0.0;
            else
                for (int k = l; k < nparts; k += 16) t += __ldcg(part + 6 * (size_t)k + q);
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (q < 6 && l == 0) r.F[q] = t;
    }
}
__device__ __forceinline__ void rigid_velocities(RigidBlock &r, const int lane) {
    double *S = r.S;
    if (lane < 6) {
        const int a = lane % 3;
        double vdot;
        if (lane < 3) {
            vdot = (r.F[a] + r.add[a]) * S[RigidState::INVM];
        } else {
            vdot = r.W[3 * a] * (r.F[3] + r.add[3]) + r.W[3 * a + 1] * (r.F[4] + r.add[4]) +
                   r.W[3 * a + 2] * (r.F[5] + r.add[5]);
        }
        const double vn = 2.0 / 3.0 * (r.c[lane] + vdot);
        const int v = lane < 3 ? RigidState::U : RigidState::W, vp = lane < 3 ? RigidState::UP : RigidState::WP;
        S[vp + a] = S[v + a];
        S[v + a] = vn;
    }
    __syncwarp();
}
__device__ __forceinline__ void rigid_orientation(RigidBlock &r, const int lane) {
    double *S = r.S;
    if (lane < 3) {
        S[RigidState::XC_OLD + lane] = r.xo[lane];
        S[RigidState::XC + lane] = r.xo[lane] + S[RigidState::U + lane];
    }
    // rotation by |w| about w: dq = (cos(|w|/2), sin(|w|/2) w/|w|)
    const double w0 = S[RigidState::W], w1 = S[RigidState::W + 1], w2 = S[RigidState::W + 2];
    const double th2 = w0 * w0 + w1 * w1 + w2 * w2;
    double c, sth;  // cos(|w|/2) and sin(|w|/2)/|w|
    if (th2 < 1e-6) {
        // series in x^2 = |w|^2/4 (terms beyond x^8 are below double rounding)
        const double x2 = 0.25 * th2;
        c = 1.0 + x2 * (-0.5 + x2 * (1.0 / 24.0 + x2 * (-1.0 / 720.0 + x2 * (1.0 / 40320.0))));
        sth = 0.5 * (1.0 + x2 * (-1.0 / 6.0 + x2 * (1.0 / 120.0 + x2 * (-1.0 / 5040.0))));
    } else {
        const double wl = sqrt(th2);
        double sn;
        sincos(0.5 * wl, &sn, &c);
        sth = sn / wl;
    }
    // component l = lane & 3 of dq (x) q: sum over k of +-dq_k q_(l xor k), the
    // minus signs those of the quaternion product
    const int l = lane & 3;
    const double *q = S + RigidState::Q4;
    auto term = [&](int k, bool minus) { return minus ? -q[l ^ k] : q[l ^ k]; };
    double qn = c * q[l] + (sth * w0) * term(1, l == 0 || l == 2) + (sth * w1) * term(2, l == 0 || l == 3) +
                (sth * w2) * term(3, l == 0 || l == 1);
    if (!(th2 > 0.0)) qn = q[l];
    double qq = qn * qn;
    qq += __shfl_xor_sync(0xffffffffu, qq, 1);
    qq += __shfl_xor_sync(0xffffffffu, qq, 2);
    double rs = (double)rsqrtf((float)qq);  // 1/sqrt(qq), refined twice
    rs = rs * (1.5 - 0.5 * qq * rs * rs);
    rs = rs * (1.5 - 0.5 * qq * rs * rs);
    if (th2 > 0.0) qn *= rs;
    __syncwarp();
    if (lane < 4) S[RigidState::Q4 + lane] = qn;
    __syncwarp();
    if (lane < 9) {
        // entry (i, j): 1 - 2 (a^2 + b^2) of the other two components on the
        // diagonal, else 2 (u_i u_j -+ w u_k), k the third axis; one form for
        // both, base - 2 (f0 f1 + f2 f3)
        const int i = lane / 3, j = lane % 3;
        const int k = i == j ? (i + 2) % 3 : 3 - i - j;
        const bool plus = (j - i + 3) % 3 == 2;
        const double w = q[0], ui = q[1 + i], uj = q[1 + j], uk = q[1 + k], a = q[1 + (i + 1) % 3];
        const double f0 = i == j ? a : -ui, f1 = i == j ? a : uj;
        const double f2 = i == j ? uk : plus ? -w : w, f3 = uk;
        S[RigidState::ROT + lane] = (i == j ? 1.0 : 0.0) - 2.0 * (f0 * f1 + f2 * f3);
    }
    __syncwarp();
}
// After every warp's last read of the old state (a block barrier before):
// the last block of the kernel to get here writes the new one.
__device__ __forceinline__ void rigid_commit(const BodyView &B, RigidBlock &r, const int nblocks, const int lane) {
    if (lane == 0) {
        __threadfence();
        r.last = atomicAdd(B.vol_count, 1u) == (unsigned)nblocks - 1;
    }
    __syncwarp();
    if (r.last) {
        for (int k = lane; k < RigidState::SIZE; k += 32) B.rstate[k] = r.S[k];
        if (lane == 0) *B.vol_count = 0u;
    }
}

// Rigid markers, 8 lanes each: boundary velocity u + w x (X - x_c) of
// level n, IB force and spreading, then the markers of level n+1.  The
// block takes the groups vb, vb + stride, ... below nvb; nblocks blocks work
// on the body.
template <typename R>
__device__ __forceinline__ void rigid_markers_body(const Lattice &L, const BodyView &B, R *__restrict__ force,
                                                   uint32_t *__restrict__ stamp, const uint32_t *__restrict__ dstep,
                                                   int vb, const int stride, const int nvb, const int nparts,
                                                   const int nblocks) {
    __shared__ RigidBlock r;
    __shared__ BlockBox sbox;
    __shared__ R s_Fl[32][3];
    __shared__ double s_U[32][3];  // centroid markers: the vertex velocity
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int l8 = threadIdx.x & (kLanes - 1), g = threadIdx.x / kLanes, nvpb = blockDim.x / kLanes;
    // FP64 for the block's markers at once: thread 32 + 3 j + a handles
    // component a of marker j (warp 0 advances the body meanwhile)
    const int comp = (int)threadIdx.x - 32, j = comp / 3, a = comp % 3, a1 = (a + 1) % 3, a2 = (a + 2) % 3;
    if (warp == 0) rigid_prepare(B, r, lane);
    sbox.init();
    for (bool first = true; vb < nvb; vb += stride, first = false) {
        const int v0 = vb * nvpb, v = v0 + g, vj = v0 + j;
        const bool mine = comp >= 0 && comp < 3 * nvpb && vj < B.nv;
        // what the MLS kernel does not write
        double x[3] = {0.0, 0.0, 0.0}, xb[3] = {0.0, 0.0, 0.0};
        if (mine)
            for (int k = 0; k < 3; ++k) {
                x[k] = __ldcg(B.X + 3 * vj + (a + k) % 3);
                xb[k] = B.Xbody[3 * vj + k];
            }
        const int q1 = v < B.nv ? B.vt_ptr[v + 1] : 0, q0 = v < B.nv ? B.vt_ptr[v] + l8 : 0;
        const int t0 = q0 < q1 ? B.vt_list[q0] / 3 : 0;
        chain_wait();
        if (first) rigid_sums(B, r, nparts);
        const uint32_t step = __ldcg(dstep);  // written by the moments kernel of the step
        const double U0 = mine && !B.centroid ? B.U[3 * vj + a] : 0.0;
        R Al = R(0);
        double Uv[3] = {0.0, 0.0, 0.0};
        for (int q = q0; q < q1; q += kLanes) {
            const int t = q == q0 ? t0 : B.vt_list[q] / 3;
            const R At3 = ((const R *)B.tri_geo)[8 * t + 3] / R(3);
            Al += At3;
            if (B.centroid)
                for (int k = 0; k < 3; ++k) Uv[k] += (double)At3 * B.Uc[3 * t + k];
        }
        Al = lanes_sum(Al);
        if (B.centroid) {
            // the vertex velocity: area-weighted mean of its triangles'
            // centroid velocities
            for (int k = 0; k < 3; ++k) Uv[k] = lanes_sum(Uv[k]);
            if (l8 == 0)
                for (int k = 0; k < 3; ++k) s_U[g][k] = Uv[k] / (double)Al;
        }
        if (first) {
            __syncthreads();
            if (warp == 0) rigid_velocities(r, lane);
        }
        __syncthreads();
        const double *S = r.S;
        if (mine) {
            const double *un = S + RigidState::U, *wn = S + RigidState::W;
            const double r1 = x[1] - r.xo[a1], r2 = x[2] - r.xo[a2];
            const double ub = un[a] + (wn[a1] * r2 - wn[a2] * r1);  // (w x r)_a
            double U = U0;
            if (B.centroid) {
                U = s_U[j][a];
                B.U[3 * vj + a] = U;
            }
            const double Fla = ub - U;
            B.Ub[3 * vj + a] = ub;
            B.Fl[3 * vj + a] = Fla;
            record(B.rec, step, 1, 3 * vj + a, ub);
            record(B.rec, step, 2, 3 * vj + a, Fla);
            s_Fl[j][a] = R(Fla);
        } else if (first && warp == 0) {
            rigid_orientation(r, lane);
        }
        __syncthreads();
        if (!B.centroid && v < B.nv) spread<R>(L, B, v, l8, Al, s_Fl[g], force, stamp, step);
        if (mine) {
            const double *xc = S + RigidState::XC, *Rn = S + RigidState::ROT;
            const double xn = xc[a] + Rn[3 * a] * xb[0] + Rn[3 * a + 1] * xb[1] + Rn[3 * a + 2] * xb[2];
            // a marker moving a lattice unit or more in one step (or a NaN)
            // has diverged
            if (!(fabs(xn - x[0]) < kMaxMarkerStep)) atomicCAS(B.err, 0, kErrDiverged);
            B.Xnew[3 * vj + a] = xn;
            record(B.rec, step, 0, 3 * vj + a, xn);
            ((R *)B.Xrel_next)[3 * vj + a] = R(xn - B.origin[a]);
            sbox.add(a, xn);
        }
        if (first && warp == 0) rigid_commit(B, r, nblocks, lane);
        __syncthreads();
    }
    sbox.flush(B.bbox_next);
}

template <typename R>
__global__ void __launch_bounds__(kStructThreads) k_rigid_markers(Lattice L, BodyView B, R *__restrict__ force,
                                                                  uint32_t *__restrict__ stamp,
                                                                  const uint32_t *__restrict__ dstep, int nvb,
                                                                  int nparts) {
    chain_release();
    rigid_markers_body<R>(L, B, force, stamp, dstep, blockIdx.x, gridDim.x, nvb, nparts, gridDim.x);
}

// IB force of centroid markers, 8 lanes per triangle: the boundary
// velocity at the centroid (rigid: u + w x (X_c - x_c) of level n;
// membrane: the interpolated velocity advanced by the mean Newton
// acceleration of the triangle's vertices, which the structure kernel left
// as their Lagrangian force), F_l = U_b - U spread with c_l = A_t.
template <typename R>
__device__ __forceinline__ void centroid_body(const Lattice &L, const BodyView &B, R *__restrict__ force,
                                              uint32_t *__restrict__ stamp, const uint32_t *__restrict__ dstep,
                                              const int vb) {
    const uint32_t step = __ldcg(dstep);  // written by the moments kernel of the step
    __shared__ R s_Fl[32][3];
    const int l8 = threadIdx.x & (kLanes - 1), g = threadIdx.x / kLanes;
    const int ntpb = blockDim.x / kLanes, t0 = vb * ntpb, t = t0 + g;
    // FP64 for the block's markers at once: thread 3 j + a handles component
    // a of marker j
    if ((int)threadIdx.x < 3 * ntpb && t0 + (int)threadIdx.x / 3 < B.nt) {
        const int j = threadIdx.x / 3, a = threadIdx.x % 3, tj = t0 + j;
        const int *tv = B.tri + 3 * tj;
        const double uc = B.Uc[3 * tj + a];
        double ub;
        if (B.rigid) {
            const int a1 = (a + 1) % 3, a2 = (a + 2) % 3;
            const double *S = B.rstate;
            const double *un = S + RigidState::U, *wn = S + RigidState::W, *xo = S + RigidState::XC_OLD;
            const double r1 = (B.X[3 * tv[0] + a1] + B.X[3 * tv[1] + a1] + B.X[3 * tv[2] + a1]) / 3.0 - xo[a1];
            const double r2 = (B.X[3 * tv[0] + a2] + B.X[3 * tv[1] + a2] + B.X[3 * tv[2] + a2]) / 3.0 - xo[a2];
            ub = un[a] + (wn[a1] * r2 - wn[a2] * r1);
        } else {
            const double acc = B.Fl[3 * tv[0] + a] + B.Fl[3 * tv[1] + a] + B.Fl[3 * tv[2] + a];
            ub = uc + acc / 3.0;
        }
        const double Fla = ub - uc;
        B.Flc[3 * tj + a] = Fla;
        s_Fl[j][a] = R(Fla);
    }
    __syncthreads();
    if (t < B.nt)
        spread<R>(L, B, t, l8, ((const R *)B.tri_geo)[8 * t + 3], s_Fl[g], force, stamp, step);
}

template <typename R>
__global__ void __launch_bounds__(kStructThreads) k_centroid_spread(Lattice L, BodyView B, R *__restrict__ force,
                                                         uint32_t *__restrict__ stamp,
                                                         const uint32_t *__restrict__ dstep) {
    centroid_body<R>(L, B, force, stamp, dstep, blockIdx.x);
}

// ---- batch kernels: the bodies of all lattices of a batch per launch ----
// Each is launched programmatically behind the one before and waits for it
// once its tables are staged (and, MLS and membrane, the positions, weights
// and hinge forces formed).  Those early parts read, at the L2, what the
// previous step's structure kernels wrote: the sweep between releases its
// successor only after its own wait, so these have completed by then.
template <typename S, typename R>
__global__ void __launch_bounds__(256) kb_moments(BatchTables T, int phase) {
    __shared__ Lattice L;
    const int j = __ldg(T.mom_blk + blockIdx.x);
    const int vb = blockIdx.x - __ldg(T.mom_pre + j), nvb = __ldg(T.mom_pre + j + 1) - __ldg(T.mom_pre + j);
    const BodyRef &br = T.body[phase * T.nb + j];
    stage_shared(L, T.lat + br.lat);
    const LatRef &F = T.ref[phase * T.nl + br.lat];
    chain_release();
    chain_wait();
    moments_body<S, R, true>((const S *)F.fin, L, br.v.bbox, br.v.bbox_next, (R *)F.mom, br.inc_step ? F.d_step : nullptr,
                       vb, nvb);
}

// Five blocks an SM (96 registers instead of 130 and three blocks): the
// gathers of many bodies need warps in flight (64 lattices, 618 000 points:
// 1.091 -> 1.063 ms a step, in spite of 44 spilt bytes).
template <typename R>
__global__ void __launch_bounds__(kBatchMlsThreads, sizeof(R) == 4 ? 5 : 2) kb_mls(BatchTables T, int phase) {
    __shared__ Lattice L;
    __shared__ BodyRef br;
    const int j = __ldg(T.mls_blk + blockIdx.x);
    const int vb = blockIdx.x - __ldg(T.mls_pre + j), nvb = __ldg(T.mls_pre + j + 1) - __ldg(T.mls_pre + j);
    stage_shared(br, T.body + phase * T.nb + j);
    stage_shared(L, T.lat + br.lat);
    const LatRef &F = T.ref[phase * T.nl + br.lat];
    chain_release();
    mls_body<R, true, true>((const R *)F.mom, L, br.v, F.err, vb);
}

template <typename R>
__global__ void __launch_bounds__(256) kb_membrane(BatchTables T, int phase) {
    __shared__ Lattice L;
    __shared__ BodyRef br;
    const int m = __ldg(T.memb_blk + blockIdx.x);
    stage_shared(br, T.body + phase * T.nb + __ldg(T.memb_id + m));
    stage_shared(L, T.lat + br.lat);
    const LatRef &F = T.ref[phase * T.nl + br.lat];
    chain_release();
    membrane_body<R>(L, br.v, (R *)F.force, F.stamp, F.d_step, blockIdx.x - __ldg(T.memb_pre + m),
                     points_blocks(br.v, kBatchMlsThreads));
}

// One block per body with more MLS partials than the structure kernels add up
// by themselves.
__global__ void __launch_bounds__(256) kb_body_sums(BatchTables T, int phase) {
    const BodyRef &br = T.body[phase * T.nb + __ldg(T.sums_id + blockIdx.x)];
    chain_release();
    chain_wait();
    body_sums_body(br.v, points_blocks(br.v, kBatchMlsThreads));
}

template <typename R>
__global__ void __launch_bounds__(256) kb_rigid_markers(BatchTables T, int phase) {
    __shared__ Lattice L;
    __shared__ BodyRef br;
    const int m = __ldg(T.rm_blk + blockIdx.x);
    stage_shared(br, T.body + phase * T.nb + __ldg(T.rigid_id + m));
    stage_shared(L, T.lat + br.lat);
    const LatRef &F = T.ref[phase * T.nl + br.lat];
    const int b0 = __ldg(T.rm_pre + m), nvb = __ldg(T.rm_pre + m + 1) - b0;
    chain_release();
    rigid_markers_body<R>(L, br.v, (R *)F.force, F.stamp, F.d_step, blockIdx.x - b0, nvb, nvb,
                          points_blocks(br.v, kBatchMlsThreads), nvb);
}

template <typename R>
__global__ void __launch_bounds__(256) kb_centroid_spread(BatchTables T, int phase) {
    __shared__ Lattice L;
    __shared__ BodyRef br;
    const int m = __ldg(T.cen_blk + blockIdx.x);
    stage_shared(br, T.body + phase * T.nb + __ldg(T.cen_id + m));
    stage_shared(L, T.lat + br.lat);
    const LatRef &F = T.ref[phase * T.nl + br.lat];
    chain_release();
    chain_wait();
    centroid_body<R>(L, br.v, (R *)F.force, F.stamp, F.d_step, blockIdx.x - __ldg(T.cen_pre + m));
}

// ---- persistent batched step ----
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Thread 0: waits until every item of kind k of lattice l in steps 0..upto
// of this launch has finished (count (upto + 1) * need).  Gives up, and
// marks the launch aborted, once the wait has lasted P.wait_ns, or when
// another block has aborted.  The acquire load orders the item's later
// loads after the awaited items' stores.
__device__ bool wait_kind(const PersistTables &P, int l, int k, int upto, unsigned long long t0) {
    const unsigned need = __ldg(P.need + l * kPKinds + k);
    if (upto < 0 || need == 0) return true;
    const unsigned target = (unsigned)(upto + 1) * need;
    const unsigned *ctr = P.done + l * kPKinds + k;
    for (;;) {
        if (ld_acquire(ctr) >= target) return true;
        if (*(volatile unsigned *)P.abort) return false;
        if ((long long)(global_ns() - t0) >= P.wait_ns) {
            atomicExch(P.abort, 1u);
            return false;
        }
        __nanosleep(100);
    }
}

// The items an item of kind k, lattice l, step s waits for: its lattice's
// earlier phases of the step, and the previous step's sweep.
__device__ bool wait_deps(const PersistTables &P, int k, int l, int s) {
    const unsigned long long t0 = global_ns();
    asm volatile("fence.acq_rel.gpu;" ::: "memory");  // an acquire even when nothing is awaited
    switch (k) {
        case kPMom: return wait_kind(P, l, kPSweep, s - 1, t0);
        case kPMls: return wait_kind(P, l, kPMom, s, t0);
        case kPSum: return wait_kind(P, l, kPMls, s, t0);
        case kPMemb:
        case kPRm: return wait_kind(P, l, kPMls, s, t0) && wait_kind(P, l, kPSum, s, t0);
        case kPCen: return wait_kind(P, l, kPMemb, s, t0) && wait_kind(P, l, kPRm, s, t0);
        default:
            for (int j = kPMom; j < kPSweep; ++j)
                if (!wait_kind(P, l, j, s, t0)) return false;
            return wait_kind(P, l, kPSweep, s - 1, t0);
    }
}

// Several steps of every lattice of a batch in one launch: blocks take work
// items (support moments, MLS, structure updates, spreading, sweep tiles)
// in ticket order from a table that interleaves the lattices' chains (the
// host staggers them, so that each stretch of the queue mixes some
// lattices' sweeps with other lattices' IB phases), each item starting
// after the items it depends on (per-lattice completion counters).  A
// wait that exceeds its bound sets LBIB_ETIMEOUT on every lattice and ends
// the launch.
template <typename S, typename R, bool kOff32>
__global__ void __launch_bounds__(256, 4) kp_batch(BatchTables T, PersistTables P) {
    __shared__ Lattice L;
    __shared__ BodyRef br;
    __shared__ unsigned s_t[2];  // this item's ticket and the next one (taken early, double-buffered)
    __shared__ int s_ok;
    const unsigned total = (unsigned)P.nitems;
    if (threadIdx.x == 0) s_t[0] = atomicAdd(P.ticket, 1u);
    for (int k = 0;; k ^= 1) {
        __syncthreads();
        const unsigned t = s_t[k];
        if (t >= total) break;
        const int4 it = __ldg(P.items + t);
        const int kind = it.x & 0xff, s = it.x >> 8;
        const int phase = (P.phase0 + s) % 6;
        const int lat = kind == kPSweep ? it.y : __ldg(P.body_lat + it.y);
        if (threadIdx.x == 0) {
            s_ok = !*(volatile unsigned *)P.abort && wait_deps(P, kind, lat, s);
            if (!s_ok)
                for (int l = 0; l < T.nl; ++l) atomicCAS(T.ref[l].err, 0, kErrTimeout);
            s_t[k ^ 1] = atomicAdd(P.ticket, 1u);  // the next item's ticket, in flight during this one
        }
        // stage the lattice (and body) parameters; the barrier also
        // publishes s_ok
        {
            const uint32_t *srcL = reinterpret_cast<const uint32_t *>(T.lat + lat);
            uint32_t *dstL = reinterpret_cast<uint32_t *>(&L);
            for (int w = threadIdx.x; w < (int)(sizeof(Lattice) / 4); w += blockDim.x) dstL[w] = __ldg(srcL + w);
            if (kind != kPSweep) {
                const uint32_t *srcB = reinterpret_cast<const uint32_t *>(T.body + phase * T.nb + it.y);
                uint32_t *dstB = reinterpret_cast<uint32_t *>(&br);
                for (int w = threadIdx.x; w < (int)(sizeof(BodyRef) / 4); w += blockDim.x) dstB[w] = __ldg(srcB + w);
            }
        }
        __syncthreads();
        if (!s_ok) break;
        const LatRef &F = T.ref[phase * T.nl + lat];
        switch (kind) {
            case kPSweep: {
                const uint32_t step = F.stamp ? __ldcg(F.d_step) : 0u;
                const uint32_t seed = __ldcg(F.sr + F.parity);
                if (it.z == 0 && threadIdx.x == 0) F.sr[F.parity ^ 1] = seed + 1u;
                const int c0 = it.z * P.sweep_cells;
                const int c1 = min(c0 + P.sweep_cells, L.ncell);
                for (int c = c0 + (int)threadIdx.x; c < c1; c += blockDim.x) {
                    int x, y, z;
                    node_coords(L, c, x, y, z);
                    sweep_cell<S, R, kOff32, true>((const S *)F.fin, (S *)F.fout, (R *)F.force, F.stamp, step, L,
                                                   nullptr, x, y, z, seed);
                }
                break;
            }
            case kPMom:
                moments_body<S, R, true>((const S *)F.fin, L, br.v.bbox, br.v.bbox_next, (R *)F.mom,
                                         br.inc_step ? F.d_step : nullptr, it.z, it.w);
                break;
            case kPMls:
                mls_body<R, true>((const R *)F.mom, L, br.v, F.err, it.z);
                break;
            case kPSum: body_sums_body(br.v, points_blocks(br.v, kPersistThreads)); break;
            case kPMemb:
                membrane_body<R>(L, br.v, (R *)F.force, F.stamp, F.d_step, it.z, points_blocks(br.v, kPersistThreads));
                break;
            case kPRm:
                rigid_markers_body<R>(L, br.v, (R *)F.force, F.stamp, F.d_step, it.z, it.w, it.w,
                                      points_blocks(br.v, kPersistThreads), it.w);
                break;
            default: centroid_body<R>(L, br.v, (R *)F.force, F.stamp, F.d_step, it.z); break;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();  // the item's stores (every thread's, ordered by the barrier) before its count
            atomicAdd(P.done + lat * kPKinds + kind, 1u);
        }
    }
}

template <typename S, typename R>
static cudaError_t persistent_t(const BatchTables &T, const PersistTables &P, int grid, cudaStream_t s) {
    if (T.sweep_off32)
        kp_batch<S, R, true><<<grid, 256, 0, s>>>(T, P);
    else
        kp_batch<S, R, false><<<grid, 256, 0, s>>>(T, P);
    return cudaGetLastError();
}

cudaError_t launch_batch_persistent(int prec, const BatchTables &T, const PersistTables &P, int grid,
                                    cudaStream_t s) {
    switch (prec) {
        case 0: return persistent_t<double, double>(T, P, grid, s);
        case 1: return persistent_t<float, float>(T, P, grid, s);
        case 2: return persistent_t<__half, float>(T, P, grid, s);
        default: return persistent_t<__nv_bfloat16, float>(T, P, grid, s);
    }
}

// Resident blocks per SM of the persistent kernel, for the grid size.
template <typename S, typename R>
static int persistent_occ(bool off32) {
    int n = 0;
    if (off32)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kp_batch<S, R, true>, 256, 0);
    else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kp_batch<S, R, false>, 256, 0);
    return n;
}

int batch_persistent_blocks_per_sm(int prec, bool off32) {
    switch (prec) {
        case 0: return persistent_occ<double, double>(off32);
        case 1: return persistent_occ<float, float>(off32);
        case 2: return persistent_occ<__half, float>(off32);
        default: return persistent_occ<__nv_bfloat16, float>(off32);
    }
}

template <typename S, typename R>
static cudaError_t batch_ib_t(const BatchTables &T, const BatchGrid &G, int phase, bool chained, cudaStream_t s) {
    auto go = [&](auto kernel, int grid, int block) {
        if (grid <= 0) return cudaSuccess;
        return launch_chained(kernel, dim3(grid), dim3(block), 0, s, T, phase);
    };
    cudaError_t e = cudaSuccess;
    if (chained)
        e = go(kb_moments<S, R>, G.mom, 256);
    else if (G.mom > 0)
        kb_moments<S, R><<<G.mom, 256, 0, s>>>(T, phase);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) e = go(kb_mls<R>, G.mls, kBatchMlsThreads);
    if (e == cudaSuccess) e = go(kb_body_sums, G.sums, 256);
    if (e == cudaSuccess) e = go(kb_membrane<R>, G.memb, 256);
    if (e == cudaSuccess) e = go(kb_rigid_markers<R>, G.rm, 256);
    if (e == cudaSuccess) e = go(kb_centroid_spread<R>, G.cen, 256);  // after the structure kernels
    return e;
}

cudaError_t launch_batch_ib(int prec, const BatchTables &T, const BatchGrid &G, int phase, bool chained,
                            cudaStream_t s) {
    switch (prec) {
        case 0: return batch_ib_t<double, double>(T, G, phase, chained, s);
        case 1: return batch_ib_t<float, float>(T, G, phase, chained, s);
        case 2: return batch_ib_t<__half, float>(T, G, phase, chained, s);
        default: return batch_ib_t<__nv_bfloat16, float>(T, G, phase, chained, s);
    }
}

// ---- launchers ----
int mls_blocks(const BodyView &B, int threads) { return points_blocks(B, threads); }
bool needs_body_sums(const BodyView &B, int threads) { return points_blocks(B, threads) > kDirectParts; }

// Grid of n blocks' work under a cap (0: none).
static int capped(int n, int cap) { return cap > 0 && cap < n ? cap : n; }

template <typename S, typename R>
static cudaError_t ib_front_t(const void *fin, const Lattice &L, const BodyView &B, void *mom, int nsm,
                              int box_nodes, int *err, uint32_t *step_inc, int grid_cap, cudaStream_t s) {
    k_moments<S, R><<<node_blocks(box_nodes, kNodeThreads, nsm), kNodeThreads, 0, s>>>(
        (const S *)fin, L, B.bbox, B.bbox_next, (R *)mom, step_inc);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // the MLS kernel is scheduled while the moments kernel ends, and forms its
    // points' positions and weights meanwhile
    const int prec = sizeof(R) == 8 ? 0 : 1, nvb = mls_blocks(B, mls_points(prec, B));
    const dim3 g(capped(nvb, grid_cap));
    if (mls_quads(prec, B))
        return launch_chained(k_mls_quad<R>, g, dim3(kQuadThreads), 0, s, (const R *)mom, L, B, err, nvb);
    return launch_chained(k_mls<R>, g, dim3(mls_threads(prec)), 0, s, (const R *)mom, L, B, err, nvb);
}

cudaError_t launch_ib_front(int prec, const void *fin, const Lattice &L, const BodyView &B, void *mom, int nsm,
                            int box_nodes, int *err, uint32_t *step_inc, int grid_cap, cudaStream_t s) {
    switch (prec) {
        case 0: return ib_front_t<double, double>(fin, L, B, mom, nsm, box_nodes, err, step_inc, grid_cap, s);
        case 1: return ib_front_t<float, float>(fin, L, B, mom, nsm, box_nodes, err, step_inc, grid_cap, s);
        case 2: return ib_front_t<__half, float>(fin, L, B, mom, nsm, box_nodes, err, step_inc, grid_cap, s);
        default: return ib_front_t<__nv_bfloat16, float>(fin, L, B, mom, nsm, box_nodes, err, step_inc, grid_cap, s);
    }
}

static cudaError_t launch_centroid(int prec, const Lattice &L, const BodyView &B, void *force, uint32_t *stamp,
                                   const uint32_t *step, cudaStream_t s) {
    const unsigned g = (unsigned)((B.nt + kStructThreads / kLanes - 1) / (kStructThreads / kLanes));
    if (prec == 0)
        k_centroid_spread<double><<<g, kStructThreads, 0, s>>>(L, B, (double *)force, stamp, step);
    else
        k_centroid_spread<float><<<g, kStructThreads, 0, s>>>(L, B, (float *)force, stamp, step);
    return cudaGetLastError();
}

// The structure kernel is launched programmatically behind the MLS kernel:
// the membrane's hinge forces and the rigid body's preparation run beside
// it.  Its blocks hold their registers while they wait, on SMs that a
// far-field sweep could use, so only grids of at most this many blocks per SM
// are launched so.  Us a step, chained / not, FP32 sphere and capsule: 96^3
// 161 blocks 33.4 / 35.4 and 29.0 / 33.6, 257 35.0 / 36.2 and 30.4 / 34.6, 641
// 43.6 / 44.1 and 39.5 / 43.0; where the far field is the longer part 128^3 161
// 57.3 / 56.3 and 56.4 / 56.4, 257 59.0 / 56.6 and 57.8 / 56.5, 385 64.6 / 59.4 and
// 62.9 / 59.7, 160x160x480 641 305.8 / 298.6 and 301.3 / 297.6; FP64 72^3 97 blocks
// 147.0 / 147.5 and 149.7 / 173.9, 96^3 161 280.9 / 269.4 and 285.5 / 282.2, 257
// 315.4 / 288.5 and 316.8 / 309.5.
constexpr int kChainPerSm = 2;

template <typename... KArgs, typename... Args>
static cudaError_t launch_struct(void (*kernel)(KArgs...), bool chained, unsigned grid, unsigned block, cudaStream_t s,
                                 Args... args) {
    if (chained) return launch_chained(kernel, dim3(grid), dim3(block), 0, s, args...);
    kernel<<<grid, block, 0, s>>>(args...);
    return cudaGetLastError();
}

cudaError_t launch_structure(int prec, const Lattice &L, const BodyView &B, void *force, uint32_t *stamp,
                             const uint32_t *step, int nsm, int grid_cap, bool chained, cudaStream_t s) {
    const int nparts = points_blocks(B, mls_points(prec, B));
    cudaError_t e = cudaSuccess;
    if (nparts > kDirectParts) e = launch_struct(k_body_sums, chained, 1, 256, s, B, nparts);
    if (e != cudaSuccess) return e;
    const int per = kStructThreads / kLanes, nvb = (B.nv + per - 1) / per;
    const unsigned g = (unsigned)capped(nvb, grid_cap);
    chained = chained && (int)g <= kChainPerSm * nsm;
    if (B.rigid)
        e = prec == 0 ? launch_struct(k_rigid_markers<double>, chained, g, kStructThreads, s, L, B, (double *)force,
                                      stamp, step, nvb, nparts)
                      : launch_struct(k_rigid_markers<float>, chained, g, kStructThreads, s, L, B, (float *)force,
                                      stamp, step, nvb, nparts);
    else
        e = prec == 0 ? launch_struct(k_membrane<double>, chained, g, kStructThreads, s, L, B, (double *)force, stamp,
                                      step, nvb, nparts)
                      : launch_struct(k_membrane<float>, chained, g, kStructThreads, s, L, B, (float *)force, stamp,
                                      step, nvb, nparts);
    if (e != cudaSuccess || !B.centroid) return e;
    return launch_centroid(prec, L, B, force, stamp, step, s);
}

}  // namespace lbib
