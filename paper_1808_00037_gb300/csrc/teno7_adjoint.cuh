// teno7_adjoint.cuh -- discrete adjoint of the 1D Euler right-hand side
// L(U) = -(F_{i+1/2} - F_{i-1/2})/dx of the TENO7-ext scheme, with the stencil
// selection (every Delta_i, taken from the forward kernels' codes) and the global
// Lax-Friedrichs alpha frozen at their values for the given state.
// out += scale (dL/dU)^T v.
//
// With the selection frozen the scheme is linear between frame and flux, so no
// characteristic value is needed again.  Per face j+1/2 (one lane; a_k(t) the
// frozen coefficients of field k, h_kc = sum_t a_k(t) G_c(t) over both splits):
//   f_k = L_k . h_k
//   lambda_F = (v_{j+1} - v_j)/dx                     (flux difference)
//   lambda_f = R^T lambda_F,  lambda_R = lambda_F f^T   (back-projection)
//   lambda_L = lambda_f h^T                             (projection)
//   M_kc = L_kc lambda_f,k, so that lambda_G,c(t) = sum_k a_k(t) M_kc
// and lambda_L, lambda_R go through the frame in reverse (Roe state, then the two
// cells).  Then the lanes turn to cells: cell l gathers lambda_G+- from the eight
// faces whose stencils hold it, applies the flux Jacobian once,
//   lambda_U = (A^T (lambda_G+ + lambda_G-) + alpha (lambda_G+ - lambda_G-))/2,
// adds its share of the two frames it takes part in, and is written once.  Where
// every stencil of a warp's faces is kept, the a_k are one row and M and h lose
// their field index.
#pragma once
#include "teno7_adjoint_params.h"
#include "teno7_kernels.cuh"

namespace t7 {

template <typename T>
__device__ __forceinline__ T adj_div(T a, T b) {
    if constexpr (sizeof(T) == 8) {
        return div64(a, b);
    } else {
        return a / b;
    }
}
template <typename T>
__device__ __forceinline__ T adj_sqrt(T a) {
    if constexpr (sizeof(T) == 8) {
        return sqrt64(a);
    } else {
        return sqrtf(a);
    }
}
__device__ __forceinline__ double fmaT(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float fmaT(float a, float b, float c) { return __fmaf_rn(a, b, c); }

// Bound in FP64 by its chain of some 270 FP64 instructions where every stencil
// is kept (64 cycles each from the lone warp an SM has at 4096 cells).  Gathering
// by cell instead of scattering 30 atomic sums per face, the linear form and the
// frame in reverse instead of as dual numbers took a launch at 4096 cells from 69
// to 15 us.  A tile is 32 faces and the AT = 25 cells that all eight of their
// faces belong to, among the n + 8 cells with their ghosts; a ghost cell's share
// goes to the cell it stands for, atomically, as do the cells near the ends.  The RK
// step's vector sums ride along (e1, e2, aux): four launches a recorded step instead of
// six, the gradient of 100 steps at 4096 cells FP32 6.77 -> 6.49 ms, FP64 13.25 -> 13.06.
constexpr int AT = 25, AWPB = 4;  // cells per tile, warps per CTA

template <typename T>
struct AdjTile {
    T gp[3][WC], gm[3][WC];  // 2 G+-
    T u[WC], H[WC], s[WC], ir[WC];  // velocity, enthalpy, sqrt(rho), 1/rho
    T M[3][3][32], A[32], B[32], E[32];
    unsigned code[32];  // Table co2 rows: 4 (k + 3 split) bits
};

template <typename T>
__global__ void __launch_bounds__(AWPB * 32, 2) rhs_adjoint1d_kernel(const Adjoint1D p) {
    __shared__ AdjTile<T> tiles[AWPB];
    __shared__ T s_coef[92];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int q = threadIdx.x; q < 91; q += blockDim.x) s_coef[q] = coef<T>(q);
    const T alpha = p.alpha_ptr ? T(*p.alpha_ptr) : T(__longlong_as_double((long long)p.ctl->amax[p.slot_in][0]));
    const T gm1 = T(p.gamma - 1.0), gam = gm1 + T(1), sdx = T(p.scale / p.dx);
    const T *U = static_cast<const T *>(p.U);
    const T *V = static_cast<const T *>(p.v);
    T *out = static_cast<T *>(p.out);
    const int n = p.n;
    const int ntiles = (n + 8 + AT - 1) / AT;
    AdjTile<T> &w = tiles[warp];
    __syncthreads();
    for (int tile = blockIdx.x * nw + warp; tile < ntiles; tile += gridDim.x * nw) {
        const int l0 = tile * AT - 4;  // first cell; faces l0 - 4 .., staged cells l0 - 7 ..
        for (int c = lane; c < WS; c += 32) {
            int gi = l0 - 7 + c;
            if (gi < 0 || gi >= n) gi = ghost_map(gi, n, p.bc_lo, p.bc_hi);
            gi = chk(p.ctl, gi, 0, n);
            const T U0 = U[gi], U1 = U[(size_t)n + gi], U2 = U[(size_t)2 * n + gi];
            const T ir = adj_div(T(1), U0), u = U1 * ir;
            const T pr = gm1 * fmaT(T(-0.5), U1 * u, U2), e = U2 + pr;
            const T F[3] = {U1, fmaT(U1, u, pr), u * e}, Uc[3] = {U0, U1, U2};
#pragma unroll
            for (int k = 0; k < 3; k++) {
                w.gp[k][c] = fmaT(alpha, Uc[k], F[k]);
                w.gm[k][c] = fmaT(-alpha, Uc[k], F[k]);
            }
            w.u[c] = u;
            w.H[c] = e * ir;
            w.s[c] = adj_sqrt(U0);
            w.ir[c] = ir;
        }
        // ---- faces: lane l, face j + 1/2 ----------------------------------
        const int j = l0 - 4 + lane;
        const bool face = j >= -1 && j <= n - 1;
        unsigned code = 0u;
        T lF[3] = {T(0), T(0), T(0)};
        if (face) {
#pragma unroll
            for (int q = 0; q < 6; q++) {
                int m = lut_select(p.masks[(size_t)q * (n + 1) + (j + 1)]);
                if (m == 15) m = 11;
                code |= (unsigned)m << (4 * q);
            }
#pragma unroll
            for (int c = 0; c < 3; c++) {
                const T vr = (j + 1 <= n - 1) ? V[(size_t)c * n + chk(p.ctl, j + 1, 0, n)] : T(0);
                const T vl = (j >= 0) ? V[(size_t)c * n + chk(p.ctl, j, 0, n)] : T(0);
                lF[c] = sdx * (vr - vl);
            }
        }
        w.code[lane] = code;
        const bool smooth = __all_sync(0xffffffffu, code == 0u);  // (orders the staging too)
        __syncwarp();
        const T sl = w.s[lane + 3], sr = w.s[lane + 4], iS = adj_div(T(1), sl + sr);
        const T ut = fmaT(sl, w.u[lane + 3], sr * w.u[lane + 4]) * iS;
        const T Ht = fmaT(sl, w.H[lane + 3], sr * w.H[lane + 4]) * iS;
        const T X = ut * ut, c2 = gm1 * fmaT(T(-0.5), X, Ht);
        const T cc = adj_sqrt(c2), rc = adj_div(T(1), cc), rc2 = rc * rc, b1 = gm1 * rc2;
        const T b2 = T(0.5) * X * b1, b1u = b1 * ut, uc = ut * rc;
        const T L[3][3] = {{T(0.5) * (b2 + uc), T(-0.5) * (b1u + rc), T(0.5) * b1},
                           {T(1) - b2, b1u, -b1},
                           {T(0.5) * (b2 - uc), T(-0.5) * (b1u - rc), T(0.5) * b1}};
        // h_kc (from 2 G+-)
        T h[3][3];
        if (smooth) {
#pragma unroll
            for (int c = 0; c < 3; c++) {
                T hp = T(0), hm = T(0);
#pragma unroll
                for (int t = 0; t < 7; t++) {
                    const T a = T(0.5) * row0<T>(t);
                    hp = fmaT(a, w.gp[c][lane + t], hp);
                    hm = fmaT(a, w.gm[c][lane + 7 - t], hm);
                }
                h[0][c] = h[1][c] = h[2][c] = hp + hm;
            }
        } else {
#pragma unroll
            for (int k = 0; k < 3; k++)
#pragma unroll
                for (int c = 0; c < 3; c++) h[k][c] = T(0);
            for (int t = 0; t < 7; t++) {
                T gp[3], gm[3];
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    gp[c] = w.gp[c][lane + t];
                    gm[c] = w.gm[c][lane + 7 - t];
                }
#pragma unroll
                for (int k = 0; k < 3; k++) {
                    const T ap = T(0.5) * s_coef[7 * ((code >> (4 * k)) & 15u) + t];
                    const T am = T(0.5) * s_coef[7 * ((code >> (4 * (3 + k))) & 15u) + t];
#pragma unroll
                    for (int c = 0; c < 3; c++) h[k][c] = fmaT(ap, gp[c], fmaT(am, gm[c], h[k][c]));
                }
            }
        }
        const T umc = ut - cc, upc = ut + cc, R20 = fmaT(-ut, cc, Ht), R21 = T(0.5) * X, R22 = fmaT(ut, cc, Ht);
        const T lf[3] = {fmaT(R20, lF[2], fmaT(umc, lF[1], lF[0])), fmaT(R21, lF[2], fmaT(ut, lF[1], lF[0])),
                         fmaT(R22, lF[2], fmaT(upc, lF[1], lF[0]))};
        T f[3];
#pragma unroll
        for (int k = 0; k < 3; k++) f[k] = fmaT(L[k][2], h[k][2], fmaT(L[k][1], h[k][1], L[k][0] * h[k][0]));
        if (smooth) {
#pragma unroll
            for (int c = 0; c < 3; c++)
                w.M[0][c][lane] = fmaT(L[2][c], lf[2], fmaT(L[1][c], lf[1], L[0][c] * lf[0]));
        } else {
#pragma unroll
            for (int k = 0; k < 3; k++)
#pragma unroll
                for (int c = 0; c < 3; c++) w.M[k][c][lane] = L[k][c] * lf[k];
        }
        // ---- the frame in reverse: lambda of the rows' common terms, then of c^2,
        // u~ and H~ ------------------------------------------------------------
        const T l00 = lf[0] * h[0][0], l01 = lf[0] * h[0][1], l02 = lf[0] * h[0][2];
        const T l10 = lf[1] * h[1][0], l11 = lf[1] * h[1][1], l12 = lf[1] * h[1][2];
        const T l20 = lf[2] * h[2][0], l21 = lf[2] * h[2][1], l22 = lf[2] * h[2][2];
        const T lb2 = fmaT(T(0.5), l00 + l20, -l10);
        const T lb1u = fmaT(T(-0.5), l01 + l21, l11);
        const T dif = T(0.5) * (l00 - l20);
        const T lrc = fmaT(ut, dif, T(0.5) * (l21 - l01));
        T lb1 = fmaT(ut, lb1u, fmaT(T(0.5), l02 + l22, -l12));
        lb1 = fmaT(T(0.5) * X, lb2, lb1);
        T lu = fmaT(b1, lb1u, fmaT(rc, dif, b1u * lb2));
        lu = fmaT(lF[1], f[0] + f[1] + f[2], lu);
        lu = fmaT(lF[2], fmaT(cc, f[2] - f[0], ut * f[1]), lu);
        T lc = fmaT(fmaT(ut, lF[2], lF[1]), f[2] - f[0], -(rc2 * lrc));
        const T lc2 = fmaT(T(0.5) * rc, lc, -(b1 * rc2 * lb1));
        const T lH = fmaT(gm1, lc2, lF[2] * (f[0] + f[2]));
        lu = fmaT(-gm1 * ut, lc2, lu);
        const T A_ = lu * iS, B_ = lH * iS;
        w.A[lane] = A_;
        w.B[lane] = B_;
        w.E[lane] = fmaT(A_, ut, B_ * Ht);
        __syncwarp();
        // ---- cells: lane q, cell l0 + q; its face of position t is lane q + 7 - t --
        const int l = l0 + lane;
        if (lane < AT && l < n + 4) {
            T gp[3] = {T(0), T(0), T(0)}, gm[3] = {T(0), T(0), T(0)};
            if (smooth) {
#pragma unroll
                for (int t = 0; t < 8; t++) {
                    const int fc = lane + 7 - t;
#pragma unroll
                    for (int c = 0; c < 3; c++) {
                        const T m = w.M[0][c][fc];
                        if (t <= 6) gp[c] = fmaT(row0<T>(t), m, gp[c]);
                        if (t >= 1) gm[c] = fmaT(row0<T>(7 - t), m, gm[c]);
                    }
                }
            } else {
                for (int t = 0; t < 8; t++) {
                    const int fc = lane + 7 - t;
                    const unsigned code_f = w.code[fc];
#pragma unroll
                    for (int k = 0; k < 3; k++) {
                        const T ap = t <= 6 ? s_coef[7 * ((code_f >> (4 * k)) & 15u) + t] : T(0);
                        const T am = t >= 1 ? s_coef[7 * ((code_f >> (4 * (3 + k))) & 15u) + 7 - t] : T(0);
#pragma unroll
                        for (int c = 0; c < 3; c++) {
                            const T m = w.M[k][c][fc];
                            gp[c] = fmaT(ap, m, gp[c]);
                            gm[c] = fmaT(am, m, gm[c]);
                        }
                    }
                }
            }
            const T u = w.u[lane + 7], H = w.H[lane + 7], s = w.s[lane + 7], ir = w.ir[lane + 7];
            const T s0 = gp[0] + gm[0], s1 = gp[1] + gm[1], s2 = gp[2] + gm[2];
            const T u2 = u * u, k2 = T(0.5) * gm1 * u2 - H;  // A_20 / u
            T o[3];
            // A = [[0,1,0],[(g-3)/2 u^2,(3-g)u,g-1],[u((g-1)/2 u^2 - H), H-(g-1)u^2, g u]]
            o[0] = T(0.5) * fmaT(T(0.5) * (gam - T(3)) * u2, s1, fmaT(u * k2, s2, alpha * (gp[0] - gm[0])));
            o[1] = T(0.5) * (fmaT((T(3) - gam) * u, s1, s0) + fmaT(fmaT(-gm1, u2, H), s2, alpha * (gp[1] - gm[1])));
            o[2] = T(0.5) * fmaT(gm1, s1, fmaT(gam * u, s2, alpha * (gp[2] - gm[2])));
            // the Roe averages of faces l - 1/2 (lane + 3) and l + 1/2 (lane + 4):
            // u~ = (s_l u_l + s_r u_r)/(s_l + s_r), H~ likewise, s = sqrt(rho)
            const T a = w.A[lane + 3] + w.A[lane + 4], bb = w.B[lane + 3] + w.B[lane + 4];
            const T ls = fmaT(a, u, fmaT(bb, H, -(w.E[lane + 3] + w.E[lane + 4])));
            const T lus = a * s, lHs = bb * s;
            o[0] = fmaT(ir, fmaT(lHs, k2, fmaT(-lus, u, T(0.5) * s * ls)), o[0]);
            o[1] = fmaT(ir, fmaT(-gm1 * u, lHs, lus), o[1]);
            o[2] = fmaT(ir, gam * lHs, o[2]);
            const int cell = chk(p.ctl, ghost_map(l, n, p.bc_lo, p.bc_hi), 0, n);
            if (l >= 0 && l < n) {  // the cell itself, not a ghost of it
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    const size_t i = (size_t)c * n + cell;
                    if (p.e1) o[c] = fmaT(T(p.c1), static_cast<const T *>(p.e1)[i], o[c]);
                    if (p.e2) o[c] = fmaT(T(p.c2), static_cast<const T *>(p.e2)[i], o[c]);
                    if (p.aux) {
                        T *x = static_cast<T *>(p.aux) + i;
                        *x = p.aux_c != 0.0 ? T(p.aux_c) * *x : T(0);
                    }
                }
            }
#pragma unroll
            for (int c = 0; c < 3; c++) {
                T *dst = &out[(size_t)c * n + cell];
                if (l >= 4 && l < n - 4) *dst += o[c];
                else atomicAdd(dst, o[c]);
            }
        }
        __syncwarp();  // the next tile overwrites this warp's arrays
    }
}

// out = c1 x + c2 (y + c3 z); x may be null.
template <typename T>
__global__ void combine_kernel(T *out, const T *x, const T *y, const T *z, T c1, T c2, T c3, size_t N) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x) {
        const T a = x ? c1 * x[i] : T(0);
        out[i] = a + c2 * (y[i] + c3 * z[i]);
    }
}

template <typename T>
cudaError_t launch_rhs_adjoint1d(const Adjoint1D &p, cudaStream_t st) {
    const int ntiles = (p.n + 8 + AT - 1) / AT;
    int nw = AWPB;
    while (nw > 1 && (ntiles + nw - 1) / nw < num_sms()) nw >>= 1;
    int grid = (ntiles + nw - 1) / nw;
    if (grid > num_sms() * 4 * (AWPB / nw)) grid = num_sms() * 4 * (AWPB / nw);
    rhs_adjoint1d_kernel<T><<<grid, nw * 32, 0, st>>>(p);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_combine(void *out, const void *x, const void *y, const void *z, double c1, double c2, double c3,
                           size_t N, cudaStream_t st) {
    int grid = (int)((N + 255) / 256);
    if (grid > num_sms() * 8) grid = num_sms() * 8;
    combine_kernel<T><<<grid, 256, 0, st>>>(static_cast<T *>(out), static_cast<const T *>(x),
                                            static_cast<const T *>(y), static_cast<const T *>(z), T(c1), T(c2),
                                            T(c3), N);
    return cudaGetLastError();
}

}  // namespace t7
