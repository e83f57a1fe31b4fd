// fields.cuh -- grid kernels of libpic: Yee curl updates (standard and
// expanding box), the shearing-box implicit-midpoint sweep, guard-cell fill
// and current fold with the shearing-periodic shift, the shearing-box
// current advection, and FP64 reductions.  All kernels work on padded
// component arrays (see common.cuh); one thread per grid point.
//
// A step's grid work is few launches, each with all guard points it needs:
// the start (context, zero current), the current's conversion, fold and
// advection in one pass, then three curl updates that write their guard
// images themselves, or the shearing boxes' sweeps, which fetch the
// (shearing-)periodic neighbours in place, and one pass that writes the new
// fields with their guards.  Small boxes are bound by the number of dependent
// launches (2 - 3 us each): 7 a step in place of 16, and of a shearing box at
// four sweeps 9 (10 in FP32 with y active) in place of 46.
#pragma once

#include <type_traits>

#include "common.cuh"

namespace pic {

// Launch shape of the grid kernels: x (or the fastest index) over the
// threads of a block and over blockIdx.x, the other two indices over
// blockIdx.y and blockIdx.z, so no thread divides an index.
constexpr int CELL_THREADS = 128;
inline dim3 cell_grid(long long nfast, long long ny, long long nz) {
    return dim3((unsigned)((nfast + CELL_THREADS - 1) / CELL_THREADS), (unsigned)ny, (unsigned)nz);
}

// Launch shape of the point kernels of a step: rows of interior points (j, k),
// four to a block, 32 x points each; rows go over blockIdx.x (no limit on
// their number), x over blockIdx.y.
constexpr int PT_X = 32, PT_Y = 4;
inline dim3 point_block() { return dim3(PT_X, PT_Y); }
__host__ __device__ inline int point_rows(const Grid& g) { return (int)(((long long)g.ny * g.nz + PT_Y - 1) / PT_Y); }
inline dim3 point_grid(int row_blocks, int nx) { return dim3((unsigned)row_blocks, (unsigned)((nx + PT_X - 1) / PT_X)); }
// this thread's point for row block rb; i counts from 0 to ni - 1
__device__ __forceinline__ bool point_of(const Grid& g, int rb, int ni, int& i, int& j, int& k) {
    const int r = rb * PT_Y + threadIdx.y;
    i = blockIdx.y * PT_X + threadIdx.x;
    if (i >= ni || r >= g.ny * g.nz) return false;
    k = r / g.ny;
    j = r - k * g.ny;
    return true;
}

// Offsets from a point to its periodic images among the guards (0: none).
struct Images { long long x, y, z; };
template <int G> __device__ __forceinline__ long long image_y(const Grid& g, int j) {
    if (!GeomT<G>::AY) return 0;
    const int high = g.py - g.gy - g.ny;
    return j < high ? (long long)g.ny * g.px : (j >= g.ny - g.gy ? -(long long)g.ny * g.px : 0);
}
template <int G> __device__ __forceinline__ long long image_z(const Grid& g, int k) {
    if (!GeomT<G>::AZ) return 0;
    const int high = g.pz - g.gz - g.nz;
    const long long plane = (long long)g.px * g.py;
    return k < high ? g.nz * plane : (k >= g.nz - g.gz ? -g.nz * plane : 0);
}
__device__ __forceinline__ long long image_x(const Grid& g, int i) {
    const int high = g.px - g.gx - g.nx;
    return i < high ? g.nx : (i >= g.nx - g.gx ? -g.nx : 0);
}
// v to a point and its images
template <class T> __device__ __forceinline__ void put_images(T* F, long long o, const Images& m, T v) {
    F[o] = v;
    if (m.x) F[o + m.x] = v;
    if (m.y) {
        F[o + m.y] = v;
        if (m.x) F[o + m.y + m.x] = v;
    }
    if (m.z) {
        F[o + m.z] = v;
        if (m.x) F[o + m.z + m.x] = v;
        if (m.y) {
            F[o + m.z + m.y] = v;
            if (m.x) F[o + m.z + m.y + m.x] = v;
        }
    }
}

// w0 a + w1 b with one product rounded and the other in a fused multiply-add,
// which of the two being fixed (mix: w1 b rounded) so that every kernel that
// interpolates between two rows rounds alike.
__device__ __forceinline__ float mix(float w0, float a, float w1, float b) { return __fmaf_rn(w0, a, __fmul_rn(w1, b)); }
__device__ __forceinline__ double mix(double w0, double a, double w1, double b) { return __fma_rn(w0, a, __dmul_rn(w1, b)); }

// ---- start of a step ---------------------------------------------------------------------
// One launch: the step context (first warp of block 0), the shearing boxes'
// advection table (block 0) and a zero current.
//
// Advection of J' along y by v_{s,y} dt / 2 = -s Omega0 x dt / 2 per x column
// (x of each component's location from the box centre): row j takes
// y = j - d = j + m + f, 0 <= f < 1.  Entry i: components y and z; entry
// nx + i: component x, half a cell further.
template <class T> struct AdvCol { int m; T f; };

template <class T> __device__ __forceinline__ AdvCol<T> advect_col(double xc, double sO, int ny) {
    const double md = sO * xc * 0.5;  // -d
    const double fl = floor(md);
    AdvCol<T> a;
    a.f = T(md - fl);
    int m = (int)(fabs(fl) < (double)ny ? fl : fmod(fl, (double)ny));
    if (m < 0) m += ny;
    a.m = m;
    return a;
}

template <class T>
__device__ __forceinline__ void pre_body(JWord<T>* J, long long n, StepCtx* ctx, const CtxConst& cc, AdvCol<T>* adv, int nx,
                                         double half_nx, int b, int nb) {
    // zero the current, 16 bytes a store (component arrays are multiples of 16 bytes)
    const long long n16 = n * (long long)sizeof(JWord<T>) / 16;
    int4* z = reinterpret_cast<int4*>(J);
    for (long long q = b * (long long)blockDim.x + threadIdx.x; q < n16; q += (long long)nb * blockDim.x)
        z[q] = make_int4(0, 0, 0, 0);
    if (b != 0) return;
    if (threadIdx.x < 32) ctx_update(ctx, cc);
    __syncthreads();
    if (!adv) return;
    for (int q = threadIdx.x; q < 2 * nx; q += blockDim.x) {
        const int i = q < nx ? q : q - nx;
        adv[q] = advect_col<T>((double)i + (q < nx ? 0.0 : 0.5) - half_nx, ctx->sO_vf, cc.ny);
    }
}

template <class T>
__global__ void pre_kernel(JWord<T>* J, long long n, StepCtx* ctx, CtxConst cc, AdvCol<T>* adv, int nx, double half_nx) {
    pre_body<T>(J, n, ctx, cc, adv, nx, half_nx, blockIdx.x, gridDim.x);
}

// ---- Yee curl updates ------------------------------------------------------------------
// out_c <- alpha_c out_c + beta_c curl(sigma (.) in)_c + gam_c J_c over interior cells.
// CURL_E: curl of an E-located field, result at B locations; else curl of a
// B-located field, result at E locations.  The ignorable 2D axis contributes no
// differences.  Standard Yee: alpha = 1, sigma = 1; expanding box: the
// transforms X' = ell L^-1 X folded into alpha, beta, gam, sigma (Sec. 3.2).
// The result also goes to the point's periodic images among the guards (these
// boxes have no shear shift), so no fill pass follows.
template <class T, int G, bool CURL_E>
__device__ __forceinline__ void curl_update_body(const Grid& g, const T* __restrict__ in, T* __restrict__ out,
                                                 const T* __restrict__ J, const StepCtx* __restrict__ ctx, int which,
                                                 int i, int j, int k) {
    using GT = GeomT<G>;
    const CoefT<T> cf = CtxT<T>::curl(ctx, which);
    const Images im{image_x(g, i), image_y<G>(g, j), image_z<G>(g, k)};
    {
        long long c0 = g.idx(i, j, k);
        const long long sx = 1, sy = g.px, sz = (long long)g.px * g.py, cs = g.cstride;
        const T* X = in;
        const T* Y = in + cs;
        const T* Z = in + 2 * cs;
        T s0 = T(cf.s[0]), s1 = T(cf.s[1]), s2 = T(cf.s[2]);
        T cu[3];
        if (CURL_E) {
            // (curl E)_x = dy Ez - dz Ey, (curl E)_y = dz Ex - dx Ez, (curl E)_z = dx Ey - dy Ex, forward differences
            T dyEz = GT::AY ? s2 * (Z[c0 + sy] - Z[c0]) : T(0);
            T dzEy = GT::AZ ? s1 * (Y[c0 + sz] - Y[c0]) : T(0);
            T dzEx = GT::AZ ? s0 * (X[c0 + sz] - X[c0]) : T(0);
            T dxEz = s2 * (Z[c0 + sx] - Z[c0]);
            T dxEy = s1 * (Y[c0 + sx] - Y[c0]);
            T dyEx = GT::AY ? s0 * (X[c0 + sy] - X[c0]) : T(0);
            cu[0] = dyEz - dzEy;
            cu[1] = dzEx - dxEz;
            cu[2] = dxEy - dyEx;
        } else {
            // backward differences
            T dyBz = GT::AY ? s2 * (Z[c0] - Z[c0 - sy]) : T(0);
            T dzBy = GT::AZ ? s1 * (Y[c0] - Y[c0 - sz]) : T(0);
            T dzBx = GT::AZ ? s0 * (X[c0] - X[c0 - sz]) : T(0);
            T dxBz = s2 * (Z[c0] - Z[c0 - sx]);
            T dxBy = s1 * (Y[c0] - Y[c0 - sx]);
            T dyBx = GT::AY ? s0 * (X[c0] - X[c0 - sy]) : T(0);
            cu[0] = dyBz - dzBy;
            cu[1] = dzBx - dxBz;
            cu[2] = dxBy - dyBx;
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            T v = T(cf.a[c]) * out[c * cs + c0] + T(cf.b[c]) * cu[c];
            if (J) v += T(cf.g[c]) * J[c * cs + c0];
            put_images<T>(out + c * cs, c0, im, v);
        }
    }
}

template <class T, int G, bool CURL_E>
__global__ void curl_update_kernel(Grid g, const T* __restrict__ in, T* __restrict__ out, const T* __restrict__ J,
                                   const StepCtx* __restrict__ ctx, int which) {
    // launch: point_grid(point_rows(g), nx), point_block().  In place: a curl
    // reads the other field, and of its own only the point it writes.
    int i, j, k;
    if (point_of(g, blockIdx.x, g.nx, i, j, k)) curl_update_body<T, G, CURL_E>(g, in, out, J, ctx, which, i, j, k);
}

// ---- shearing-box implicit-midpoint sweep ---------------------------------------------
// X_out = X_n + dt F((X_n + X_k)/2), F the right-hand sides of the KSB-OA
// field equations (Sec. 2.1) with V(x) = -s Omega0 (x - nx/2):
//   F_B  = -c curl E' - V dy B - s Omega0 Bx e_y
//   F_Ex = c (curl B)_x - 4 pi J'_x + V dy E'_x - V dx E'_y
//   F_Ey = c (curl B)_y - 4 pi J'_y - V dy E'_y - V (dx E'_x + dz E'_z)
//   F_Ez = c (curl B)_z - 4 pi J'_z + V dy E'_z - V dz E'_y
// The advection term of each component is upwinded for its own transport
// velocity (V in the B and E'_y rows, -V in the E'_x and E'_z rows); the
// other V-terms are centred and averaged in y onto the component's location;
// Bx in the By row is the mean of its four neighbours.
//
// The shearing + expanding box sweeps the expanding-frame fields X^ = ell
// L^{-1} X (Sec. 3.1) with the factors of its coordinates from the step
// context: curls of (l_a^2 / ell) X^_a, the shear flow and shear term times
// l_1/l_2, the -V d_x E^_y and -V d_z E^_y terms times (l_2/l_1)^2 and
// (l_2/l_3)^2, all at t^{n+1/2}.  For the shearing box these are ones.
//
// The neighbours are fetched from the interior of X_n and X_k with periodic
// wraps in y and z; beyond the x faces they are the shearing-periodic images
// at t^{n+1/2}, interpolated between two rows as fill_x_body does.  So the
// iterates need no guards: a step takes one launch per sweep in place of one
// sweep and six guard passes, and no copy of X_n.
template <class T, int G, bool EDGE>
__device__ __forceinline__ void ksb_sweep_point(const Grid& g, const T* __restrict__ En, const T* __restrict__ Bn,
                                                const T* __restrict__ Ek, const T* __restrict__ Bk, const T* __restrict__ J,
                                                T* __restrict__ Eo, T* __restrict__ Bo, T c, T half_nx,
                                                const StepCtx* __restrict__ ctx, int i, int j, int k) {
    using GT = GeomT<G>;
    const T sO = CtxT<T>::sO(ctx);
    const T sg0 = CtxT<T>::sig(ctx, 0), sg1 = CtxT<T>::sig(ctx, 1), sg2 = CtxT<T>::sig(ctx, 2);
    const T rx = CtxT<T>::rx(ctx), rz = CtxT<T>::rz(ctx);
    const T FOUR_PI = T(12.566370614359172);
    const long long cs = g.cstride, plane = (long long)g.px * g.py;
    const long long c0 = g.idx(i, j, k);
    // offsets to the periodic neighbours (0 on an ignorable axis)
    const long long yp = GT::AY ? (j == g.ny - 1 ? -(long long)(g.ny - 1) * g.px : g.px) : 0;
    const long long ym = GT::AY ? (j == 0 ? (long long)(g.ny - 1) * g.px : -(long long)g.px) : 0;
    const long long zp = GT::AZ ? (k == g.nz - 1 ? -(g.nz - 1) * plane : plane) : 0;
    const long long zm = GT::AZ ? (k == 0 ? (g.nz - 1) * plane : -plane) : 0;
    // beyond an x face: column and rows of the shearing image (EDGE: this point
    // is in the first or last column, so only one of dx = -1, 1 leaves the box)
    const int side = i == 0 ? -1 : 1;
    const ShearShift<T> sh = EDGE ? CtxT<T>::shift(ctx, 0, side > 0) : ShearShift<T>{0, 0, T(1), T(0)};
    // field value at (i + dx, j + dy, k + dz)
    auto at = [&](const T* __restrict__ F, int dx, int dy, int dz) -> T {
        const long long o = c0 + (dy > 0 ? yp : (dy < 0 ? ym : 0)) + (dz > 0 ? zp : (dz < 0 ? zm : 0));
        if (!EDGE || dx == 0) return F[o + dx];
        const bool out = dx == side;
        const long long oi = o + (out ? -(long long)side * (g.nx - 1) : dx);
        if (!GT::AY) return F[oi];
        int jj = j + dy;
        if (jj >= g.ny) jj -= g.ny;
        if (jj < 0) jj += g.ny;
        const bool lerp = out && sh.on;
        int j0 = jj + sh.m;
        if (j0 >= g.ny) j0 -= g.ny;
        if (j0 < 0) j0 += g.ny;
        const int j1 = j0 + 1 >= g.ny ? 0 : j0 + 1;
        // both loads are made in any case: no branch orders them
        const T a = F[oi + (lerp ? (long long)(j0 - jj) * g.px : 0)], b = F[oi + (lerp ? (long long)(j1 - jj) * g.px : 0)];
        return lerp ? mix(sh.w0, a, sh.w1, b) : a;
    };
    // midpoint fields
    auto ME = [&](int comp, int dx, int dy, int dz) -> T {
        return T(0.5) * (at(En + comp * cs, dx, dy, dz) + at(Ek + comp * cs, dx, dy, dz));
    };
    auto MB = [&](int comp, int dx, int dy, int dz) -> T {
        return T(0.5) * (at(Bn + comp * cs, dx, dy, dz) + at(Bk + comp * cs, dx, dy, dz));
    };
    // x - nx/2 at nodes and half-points: exact in either precision
    const T VN = -sO * (T(i) - half_nx);
    const T VH = -sO * ((T(i) + T(0.5)) - half_nx);
    // curls (ignorable-axis differences vanish because its offsets are 0)
    T curlEx = sg2 * (ME(2, 0, 1, 0) - ME(2, 0, 0, 0)) - sg1 * (ME(1, 0, 0, 1) - ME(1, 0, 0, 0));
    T curlEy = sg0 * (ME(0, 0, 0, 1) - ME(0, 0, 0, 0)) - sg2 * (ME(2, 1, 0, 0) - ME(2, 0, 0, 0));
    T curlEz = sg1 * (ME(1, 1, 0, 0) - ME(1, 0, 0, 0)) - sg0 * (ME(0, 0, 1, 0) - ME(0, 0, 0, 0));
    T curlBx = sg2 * (MB(2, 0, 0, 0) - MB(2, 0, -1, 0)) - sg1 * (MB(1, 0, 0, 0) - MB(1, 0, 0, -1));
    T curlBy = sg0 * (MB(0, 0, 0, 0) - MB(0, 0, 0, -1)) - sg2 * (MB(2, 0, 0, 0) - MB(2, -1, 0, 0));
    T curlBz = sg1 * (MB(1, 0, 0, 0) - MB(1, -1, 0, 0)) - sg0 * (MB(0, 0, 0, 0) - MB(0, 0, -1, 0));
    auto upB = [&](int comp, T v) -> T {
        return v > T(0) ? MB(comp, 0, 0, 0) - MB(comp, 0, -1, 0) : MB(comp, 0, 1, 0) - MB(comp, 0, 0, 0);
    };
    auto upE = [&](int comp, T v) -> T {
        return v > T(0) ? ME(comp, 0, 0, 0) - ME(comp, 0, -1, 0) : ME(comp, 0, 1, 0) - ME(comp, 0, 0, 0);
    };
    T bx4 = T(0.25) * (MB(0, 0, 0, 0) + MB(0, 1, 0, 0) + MB(0, 0, -1, 0) + MB(0, 1, -1, 0));
    // the sums of two products with the rounding order spelled out (mix)
    const T FBx = -mix(c, curlEx, VN, upB(0, VN));
    const T FBy = -mix(c, curlEy, VH, upB(1, VH)) - sO * bx4;
    const T FBz = -mix(VH, upB(2, VH), c, curlEz);
    T dxEy = T(0.5) * ((ME(1, 1, 0, 0) - ME(1, 0, 0, 0)) + (ME(1, 1, -1, 0) - ME(1, 0, -1, 0)));
    T divxz = T(0.5) * ((ME(0, 0, 0, 0) - ME(0, -1, 0, 0)) + (ME(0, 0, 1, 0) - ME(0, -1, 1, 0)) +
                        (ME(2, 0, 0, 0) - ME(2, 0, 0, -1)) + (ME(2, 0, 1, 0) - ME(2, 0, 1, -1)));
    T dzEy = T(0.5) * ((ME(1, 0, 0, 1) - ME(1, 0, 0, 0)) + (ME(1, 0, -1, 1) - ME(1, 0, -1, 0)));
    T FEx = c * curlBx - FOUR_PI * J[c0] + VH * upE(0, -VH) - VH * (rx * dxEy);
    T FEy = c * curlBy - FOUR_PI * J[cs + c0] - VN * upE(1, VN) - VN * divxz;
    T FEz = c * curlBz - FOUR_PI * J[2 * cs + c0] + VN * upE(2, -VN) - VN * (rz * dzEy);
    Eo[c0] = En[c0] + FEx;
    Eo[cs + c0] = En[cs + c0] + FEy;
    Eo[2 * cs + c0] = En[2 * cs + c0] + FEz;
    Bo[c0] = Bn[c0] + FBx;
    Bo[cs + c0] = Bn[cs + c0] + FBy;
    Bo[2 * cs + c0] = Bn[2 * cs + c0] + FBz;
}

template <class T, int G>
__global__ void ksb_sweep_kernel(Grid g, const T* __restrict__ En, const T* __restrict__ Bn, const T* __restrict__ Ek,
                                 const T* __restrict__ Bk, const T* __restrict__ J, T* __restrict__ Eo, T* __restrict__ Bo,
                                 T c, T half_nx, const StepCtx* __restrict__ ctx) {
    // launch: sweep_grid(g), point_block().  The first and the last column take
    // the sheared path; blocks of their own hold them (lanes along y), or every
    // warp of a row shorter than 64 points would run both paths.
    const int rb = point_rows(g);
    if ((int)blockIdx.x >= rb) {
        const int q = (((int)blockIdx.x - rb) * PT_Y + threadIdx.y) * PT_X + threadIdx.x;
        const int n = g.ny * g.nz;
        if (blockIdx.y != 0 || q >= 2 * n) return;
        const int r = q < n ? q : q - n, k = r / g.ny;
        ksb_sweep_point<T, G, true>(g, En, Bn, Ek, Bk, J, Eo, Bo, c, half_nx, ctx, q < n ? 0 : g.nx - 1, r - k * g.ny, k);
        return;
    }
    int i, j, k;
    if (point_of(g, blockIdx.x, g.nx - 2, i, j, k))
        ksb_sweep_point<T, G, false>(g, En, Bn, Ek, Bk, J, Eo, Bo, c, half_nx, ctx, i + 1, j, k);
}
inline dim3 sweep_grid(const Grid& g) {
    dim3 d = point_grid(point_rows(g), g.nx - 2);
    d.x += (2 * g.ny * g.nz + PT_X * PT_Y - 1) / (PT_X * PT_Y);
    return d;
}

// End of a shearing box's field step: the last iterate to E and B with all
// their guards at t^{n+1} (x guards: the interior interpolated between the
// rows of the shear shift; y and z guards: images).  SCALE: the shearing +
// expanding box's X = L X^ / ell.  Launch: point_grid(point_rows(g), px).
template <class T, int G, bool SCALE>
__global__ void ksb_finish_kernel(Grid g, const T* __restrict__ Es, const T* __restrict__ Bs, T* __restrict__ E,
                                  T* __restrict__ B, const StepCtx* __restrict__ ctx) {
    using GT = GeomT<G>;
    int p, j, k;
    if (!point_of(g, blockIdx.x, g.px, p, j, k)) return;
    const int i = p - g.gx;  // physical column, guards included
    const Images im{0, image_y<G>(g, j), image_z<G>(g, k)};
    const long long o = g.idx(i, j, k);
    const int w = i < 0 ? -1 : (i >= g.nx ? 1 : 0);
    const long long oi = o - (long long)w * g.nx;
    long long o0 = oi, o1 = oi;
    ShearShift<T> sh{0, 0, T(1), T(0)};
    if (w != 0 && GT::AY) {
        sh = CtxT<T>::shift(ctx, 1, w > 0);
        int j0 = j + sh.m;
        if (j0 >= g.ny) j0 -= g.ny;
        if (j0 < 0) j0 += g.ny;
        const int j1 = j0 + 1 >= g.ny ? 0 : j0 + 1;
        if (sh.on) {
            o0 = oi + (long long)(j0 - j) * g.px;
            o1 = oi + (long long)(j1 - j) * g.px;
        }
    }
#pragma unroll
    for (int comp = 0; comp < 6; ++comp) {
        const T* S = (comp < 3 ? Es : Bs) + (comp % 3) * g.cstride;
        T* D = (comp < 3 ? E : B) + (comp % 3) * g.cstride;
        T v;
        if (sh.on) v = mix(sh.w0, S[o0], sh.w1, S[o1]);
        else v = S[oi];
        if (SCALE) v = T((double)v * ctx->sxe_post[comp % 3]);
        put_images<T>(D, o, im, v);
    }
}

// ---- guard fill -----------------------------------------------------------------------
// Axis passes: x first (interior y, z rows; with the shear shift dys for the
// shearing box: the ghost at (i >= nx, j) is the interior value at
// (i - nx, j + dys), linearly interpolated, and at (i < 0, j) the one at
// (i + nx, j - dys)), then y over all padded x, then z over all padded x, y.
// These passes run when fields or the time are set; a step writes its guards
// itself.
template <class T, int G>
__device__ __forceinline__ void fill_x_body(const Grid& g, T* F, int dys_i, double dys_f, int j, int k, int zs) {
    using GT = GeomT<G>;
    const int nguard = g.px - g.nx;  // gx low + the rest high
    {
        const int comp = zs / nguard, gi = zs - comp * nguard;
        int i = gi < g.gx ? gi - g.gx : g.nx + (gi - g.gx);  // physical ghost index
        int w = i < 0 ? -1 : 1;
        int is = i - w * g.nx;
        T* Fc = F + (long long)comp * g.cstride;
        T v;
        if (GT::AY && (dys_i != 0 || dys_f != 0.0)) {
            // y + w dys = j + w (dys_i + dys_f)
            int m;
            double f;
            if (w > 0) { m = dys_i; f = dys_f; }
            else { m = -dys_i; f = -dys_f; if (f < 0.0) { f += 1.0; m -= 1; } }
            int j0 = j + m, j1 = j0 + 1;
            j0 %= g.ny; if (j0 < 0) j0 += g.ny;
            j1 %= g.ny; if (j1 < 0) j1 += g.ny;
            v = T(1.0 - f) * Fc[g.idx(is, j0, k)] + T(f) * Fc[g.idx(is, j1, k)];
        } else {
            v = Fc[g.idx(is, j, k)];
        }
        Fc[g.idx(i, j, k)] = v;
    }
}

template <class T, int G>
__global__ void fill_x_kernel(Grid g, T* F, int ncomp, int dys_i, double dys_f) {
    // launch: cell_grid(ny, nz, ncomp * nguard)
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= g.ny) return;
    fill_x_body<T, G>(g, F, dys_i, dys_f, j, blockIdx.y, blockIdx.z);
}

template <class T>
__device__ __forceinline__ void fill_y_body(const Grid& g, T* F, int pi, int k, int zs) {
    const int nguard = g.py - g.ny;
    const int comp = zs / nguard, gj = zs - comp * nguard;
    int j = gj < g.gy ? gj - g.gy : g.ny + (gj - g.gy);
    int js = j < 0 ? j + g.ny : j - g.ny;
    T* Fc = F + (long long)comp * g.cstride;
    long long row = (long long)(k + g.gz) * g.py;
    Fc[(row + j + g.gy) * g.px + pi] = Fc[(row + js + g.gy) * g.px + pi];
}

template <class T>
__global__ void fill_y_kernel(Grid g, T* F, int ncomp) {
    // launch: cell_grid(px, nz, ncomp * nguard)
    const int pi = blockIdx.x * blockDim.x + threadIdx.x;
    if (pi >= g.px) return;
    fill_y_body<T>(g, F, pi, blockIdx.y, blockIdx.z);
}

template <class T>
__device__ __forceinline__ void fill_z_body(const Grid& g, T* F, int pi, int pj, int zs) {
    const int nguard = g.pz - g.nz;
    const long long plane = (long long)g.px * g.py;
    const long long pp = (long long)pj * g.px + pi;
    const int comp = zs / nguard, gk = zs - comp * nguard;
    int k = gk < g.gz ? gk - g.gz : g.nz + (gk - g.gz);
    int ks = k < 0 ? k + g.nz : k - g.nz;
    T* Fc = F + (long long)comp * g.cstride;
    Fc[(long long)(k + g.gz) * plane + pp] = Fc[(long long)(ks + g.gz) * plane + pp];
}

template <class T>
__global__ void fill_z_kernel(Grid g, T* F, int ncomp) {
    // launch: cell_grid(px, py, ncomp * nguard)
    const int pi = blockIdx.x * blockDim.x + threadIdx.x;
    if (pi >= g.px) return;
    fill_z_body<T>(g, F, pi, blockIdx.y, blockIdx.z);
}

// ---- current: conversion, fold (adjoint of the fill) and advection -------------------------
// The folded current of an interior point adds the guard values that map onto
// it, in the order z, y, x; a guard value at (i >= nx, j) belongs at
// (i - nx, j + dys), split (1 - f, f) between rows floor and floor + 1 (the
// shear shift at t^{n+1/2}); at (i < 0, j) at (i + nx, j - dys).  Points away
// from the faces read one word, so one pass over the raw accumulators
// converts (FP32: fixed point to float), folds and, in the shearing boxes,
// advects, where a conversion, three folds and the advection were five passes.
// The conversion is FP64 arithmetic (19 cycles per warp instruction and SM), so
// a word must be converted once: the advection, which reads two rows per
// point, works on floats that fixed_to_float_kernel made.
// A fixed-point sum that reached half of the int32 range (the only place a
// wrap could show) is flagged; every word is read by the point it folds onto.
__device__ __forceinline__ float fixed_value(int v, double unit, int* err) {
    if (v > (1 << 30) || v < -(1 << 30)) atomicOr(err, ERRB_J_RANGE);
    return (float)((double)v * unit);
}

__global__ void fixed_to_float_kernel(long long n, const int* __restrict__ src, float* __restrict__ dst, double unit,
                                      int* err) {
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x)
        dst[q] = fixed_value(src[q], unit, err);
}

template <class T, int G, class S> struct RawCurrent {
    const Grid& g;
    const S* __restrict__ J;  // one component
    double unit;
    int* err;
    __device__ __forceinline__ T value(S v) const {
        if constexpr (!std::is_same<S, T>::value) {
            return fixed_value(v, unit, err);
        } else {
            return v;
        }
    }
    // the words of padded column pi at (j, k) and its images among the y and z
    // guards; loaded together before any is used, so their latencies overlap
    struct Words { S w, z, y, yz; bool hy, hz; };
    __device__ __forceinline__ Words load(int pi, int j, int k) const {
        const long long plane = (long long)g.px * g.py, o = (long long)(k + g.gz) * plane + (long long)(j + g.gy) * g.px + pi;
        const long long dy = image_y<G>(g, j), dz = image_z<G>(g, k);
        Words r;
        r.hy = dy != 0;
        r.hz = dz != 0;
        r.w = J[o];
        r.z = r.hz ? J[o + dz] : S(0);
        r.y = r.hy ? J[o + dy] : S(0);
        r.yz = r.hy && r.hz ? J[o + dy + dz] : S(0);
        return r;
    }
    __device__ __forceinline__ T sum(const Words& r) const {
        T v = value(r.w);
        if (GeomT<G>::AZ && r.hz) v += value(r.z);
        if (GeomT<G>::AY && r.hy) {
            T u = value(r.y);
            if (GeomT<G>::AZ && r.hz) u += value(r.yz);
            v += u;
        }
        return v;
    }
};

// Component comp of the current at interior point (i, j, k) from the raw
// accumulators Jr to Jo.  ADV: advected along y by the column's shift
// (advect_col), linear between the rows, periodic.
template <class T, int G, bool ADV, class S>
__device__ __forceinline__ void fold_point(const Grid& g, const S* __restrict__ Jr, T* __restrict__ Jo, double unit,
                                           int* err, const StepCtx* __restrict__ ctx, const AdvCol<T>* __restrict__ adv,
                                           int comp, int i, int j, int k) {
    const RawCurrent<T, G, S> cur{g, Jr + comp * g.cstride, unit, err};
    using Words = typename RawCurrent<T, G, S>::Words;
    constexpr int NR = ADV ? 2 : 1;
    int row[NR] = {j};
    AdvCol<T> a{0, T(0)};
    if constexpr (ADV) {
        a = adv[comp == 0 ? g.nx + i : i];
        int ja = j + a.m;
        if (ja >= g.ny) ja -= g.ny;
        row[0] = ja;
        row[1] = ja + 1 >= g.ny ? 0 : ja + 1;
    }
    Words own[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) own[r] = cur.load(i + g.gx, row[r], k);
    T v[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) v[r] = cur.sum(own[r]);
    // a point near an x face also takes its guard column w nx away
    const int w = i < g.px - g.gx - g.nx ? 1 : (i >= g.nx - g.gx ? -1 : 0);
    if (w != 0) {
        const int ps = i + g.gx + w * g.nx;
        // sources: guard rows js with floor(js + w dys) = j (weight 1-f) or j - 1 (weight f)
        const ShearShift<T> sh = GeomT<G>::AY ? CtxT<T>::shift(ctx, 0, w > 0) : ShearShift<T>{0, 0, T(1), T(0)};
        const bool sheared = GeomT<G>::AY && sh.on;
        Words s0[NR], s1[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            int ja = row[r] - (sheared ? sh.m : 0);
            if (ja >= g.ny) ja -= g.ny;
            if (ja < 0) ja += g.ny;
            s0[r] = cur.load(ps, ja, k);
            if (GeomT<G>::AY) {
                const int jb = ja == 0 ? g.ny - 1 : ja - 1;
                s1[r] = cur.load(ps, sheared ? jb : ja, k);
            }
        }
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            T add = cur.sum(s0[r]);
            if (GeomT<G>::AY && sheared) add = mix(sh.w0, add, sh.w1, cur.sum(s1[r]));
            v[r] = v[r] + add;
        }
    }
    T out = v[0];
    if constexpr (ADV) out = mix(T(1) - a.f, v[0], a.f, v[NR - 1]);
    Jo[comp * g.cstride + g.idx(i, j, k)] = out;
}

// Particle bookkeeping after the particle kernels of a step, per species:
// clamp each tile's arrival count to the claims that got a slot (failed
// claims over-count), clamp the loose count to the list capacity, and zero
// the counters of the consumed buffer, which the next step writes.  occ_max
// keeps the largest tile occupancy since it was last reset, occ_loose the
// loose count after the step (the library's capacity check reads them).
struct TileCounts {
    const int* stay_in;
    int* arr_in;
    int* arr_out;
    int* lcount_in;
    int* lcount_out;
    long long tcap, lcap;
    int* occ_max;
    int* occ_loose;
};
struct FinalizeArgs {
    TileCounts s[4];
    int nsp, ntiles;
    int* err;
};

__device__ __forceinline__ void finalize_body(const FinalizeArgs& A, int b, int nb) {
    // block b: species b mod nsp, every (nb / nsp)-th chunk of its tiles
    const int tid = threadIdx.y * blockDim.x + threadIdx.x, nthr = blockDim.x * blockDim.y;
    if (A.nsp == 0) return;
    {
        const TileCounts& C = A.s[b % A.nsp];
        b /= A.nsp;
        nb /= A.nsp;
        int mx = 0;
        for (int t = b * nthr + tid; t < A.ntiles; t += nb * nthr) {
            const int cnt = C.stay_in[t] + C.arr_in[t];
            mx = max(mx, cnt);
            const int room = (int)(C.tcap - cnt);
            if (C.arr_out[t] > room) C.arr_out[t] = room;
            C.arr_in[t] = 0;
        }
        for (int sh = 16; sh > 0; sh >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, sh));
        if ((tid & 31) == 0 && mx > 0) atomicMax(C.occ_max, mx);
        if (b == 0 && tid == 0) {
            int lc = *C.lcount_out;
            if (lc > C.lcap) { atomicOr(A.err, ERRB_LOOSE_OVERFLOW); lc = (int)C.lcap; *C.lcount_out = lc; }
            *C.occ_loose = lc;
            *C.lcount_in = 0;
        }
    }
}

// Blocks [0, row_blocks) of x fold the current (component blockIdx.z), the
// rest (of blockIdx.y = z = 0) do the particle bookkeeping: neither reads what the other writes, and the
// bookkeeping's 2 us per species would be launches of their own.
template <class T, int G, bool ADV, class S>
__global__ void fold_kernel(Grid g, const S* __restrict__ Jr, T* __restrict__ Jo, double unit, int* err,
                            const StepCtx* __restrict__ ctx, const AdvCol<T>* __restrict__ adv, int row_blocks,
                            const __grid_constant__ FinalizeArgs fin) {
    if ((int)blockIdx.x >= row_blocks) {
        if (blockIdx.y == 0 && blockIdx.z == 0) finalize_body(fin, (int)blockIdx.x - row_blocks, (int)gridDim.x - row_blocks);
        return;
    }
    int i, j, k;
    if (point_of(g, blockIdx.x, g.nx, i, j, k)) fold_point<T, G, ADV, S>(g, Jr, Jo, unit, err, ctx, adv, blockIdx.z, i, j, k);
}

__global__ void finalize_kernel(const __grid_constant__ FinalizeArgs fin) { finalize_body(fin, blockIdx.x, gridDim.x); }

// Component-wise scaling of a padded 3-component field (guards included) by
// ctx->sxe_pre: X^ = ell L^{-1} X at t^n.  Launch: cell_grid(cstride, 1, 3).
template <class T>
__global__ void scale3_kernel(T* F, long long cstride, const StepCtx* __restrict__ ctx) {
    const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= cstride) return;
    const int comp = blockIdx.z;
    F[comp * cstride + q] = T((double)F[comp * cstride + q] * ctx->sxe_pre[comp]);
}

// ---- batched grid kernels -----------------------------------------------------------------
// The grid work of many (unsheared) boxes of one kind in one launch each: box
// b's row blocks are blockIdx.x in [roff[b], roff[b+1]), y covers the widest
// box's x points and threads beyond a box's own extent return.  The bodies
// are the single-box kernels', so results are the same bit for bit.
// Descriptors and the offset table live in device memory (fixed for the life
// of a batch).
template <class T> struct FieldBox {
    Grid g;
    T* E;
    T* B;
    T* J;           // the current the field update reads (the folded one)
    JWord<T>* Jraw; // the accumulators of the particle kernels
    StepCtx* ctx;
    int* err;
    double fx_unit;
    CtxConst cc;
};

__device__ __forceinline__ int box_of_row(const int* __restrict__ roff, int n, int r) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (roff[mid] <= r) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Start of a step for every box (pre_kernel).  Launch: grid (any, n); block
// row b serves box b.
template <class T>
__global__ void multi_pre_kernel(const FieldBox<T>* __restrict__ fb, int n) {
    const int b = blockIdx.y;
    if (b >= n) return;
    const FieldBox<T>& f = fb[b];
    pre_body<T>(f.Jraw, 3ll * f.g.cstride, f.ctx, f.cc, nullptr, 0, 0.0, blockIdx.x, gridDim.x);
}

template <class T, int G>
__global__ void multi_fold_kernel(const FieldBox<T>* __restrict__ fb, const int* __restrict__ roff, int n) {
    const int b = box_of_row(roff, n, blockIdx.x);
    const FieldBox<T>& f = fb[b];
    int i, j, k;
    if (point_of(f.g, blockIdx.x - roff[b], f.g.nx, i, j, k))
        fold_point<T, G, false, JWord<T>>(f.g, f.Jraw, f.J, f.fx_unit, f.err, f.ctx, nullptr, blockIdx.z, i, j, k);
}

template <class T, int G, bool CURL_E>
__global__ void multi_curl_kernel(const FieldBox<T>* __restrict__ fb, const int* __restrict__ roff, int n, int which) {
    const int b = box_of_row(roff, n, blockIdx.x);
    const FieldBox<T>& f = fb[b];
    int i, j, k;
    if (!point_of(f.g, blockIdx.x - roff[b], f.g.nx, i, j, k)) return;
    curl_update_body<T, G, CURL_E>(f.g, CURL_E ? f.E : f.B, CURL_E ? f.B : f.E, CURL_E ? nullptr : f.J, f.ctx, which, i, j,
                                   k);
}

// ---- host <-> padded layout -----------------------------------------------------------
template <class T>
__global__ void scatter_field_kernel(Grid g, const double* __restrict__ src, T* __restrict__ dst) {
    long long n = 3ll * g.nx * g.ny * g.nz;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        int i = (int)(q % g.nx);
        long long r = q / g.nx;
        int j = (int)(r % g.ny);
        r /= g.ny;
        int k = (int)(r % g.nz);
        int comp = (int)(r / g.nz);
        dst[(long long)comp * g.cstride + g.idx(i, j, k)] = T(src[q]);
    }
}

template <class T>
__global__ void gather_field_kernel(Grid g, const T* __restrict__ src, double* __restrict__ dst) {
    long long n = 3ll * g.nx * g.ny * g.nz;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        int i = (int)(q % g.nx);
        long long r = q / g.nx;
        int j = (int)(r % g.ny);
        r /= g.ny;
        int k = (int)(r % g.nz);
        int comp = (int)(r / g.nz);
        dst[q] = (double)src[(long long)comp * g.cstride + g.idx(i, j, k)];
    }
}

template <class T>
__global__ void uniform_field_kernel(Grid g, T* dst, double v0, double v1, double v2) {
    long long n = 3ll * g.cstride;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        int comp = (int)(q / g.cstride);
        dst[q] = T(comp == 0 ? v0 : (comp == 1 ? v1 : v2));
    }
}

// ---- FP64 reductions -------------------------------------------------------------------
// Sum of squares of each component over interior cells: block partials in
// `partial` ([gridDim.x][3]), then one block adds them (deterministic order).
template <class T>
__global__ void sumsq_partial_kernel(Grid g, const T* __restrict__ F, double* __restrict__ partial) {
    __shared__ double red[3][32];
    double acc[3] = {0.0, 0.0, 0.0};
    long long n = (long long)g.nx * g.ny * g.nz;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
        int i = (int)(q % g.nx);
        long long r = q / g.nx;
        int j = (int)(r % g.ny);
        int k = (int)(r / g.ny);
        long long c0 = g.idx(i, j, k);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            double v = (double)F[c * g.cstride + c0];
            acc[c] += v * v;
        }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        double v = acc[c];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0) red[c][threadIdx.x >> 5] = v;
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[threadIdx.x][w];
        partial[blockIdx.x * 3 + threadIdx.x] = s;
    }
}

__global__ void sum_partials_kernel(const double* __restrict__ partial, int nblocks, int width, double* __restrict__ out) {
    // one warp per output column: each lane adds every 32nd partial, then the
    // lanes in a fixed tree (deterministic; one thread per column took 65 us)
    const int c = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (c >= width) return;
    double s = 0.0;
    for (int b = lane; b < nblocks; b += 32) s += partial[b * width + c];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) out[c] = s;
}

// Everything pic_diagnostics reads, in one place for one copy.
struct DiagOut {
    double sums[10];  // sum E_c^2, sum B_c^2 (3 each), kinetic energies
    unsigned long long counters[2];
    int loose[4];
    int err;
};
struct DiagSrc { const int* loose[4]; };
__global__ void collect_diag_kernel(DiagOut* __restrict__ out, const unsigned long long* __restrict__ counters,
                                    const int* __restrict__ err, DiagSrc src) {
    const int i = threadIdx.x;
    if (i < 2) out->counters[i] = counters[i];
    if (i < 4) out->loose[i] = src.loose[i] ? *src.loose[i] : 0;
    if (i == 0) out->err = *err;
}

}  // namespace pic
