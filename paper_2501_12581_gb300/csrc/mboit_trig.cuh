// Trigonometric-moment variant of the moment bound (n = 3 or 4 complex
// moments, the "6 / 8 trigonometric moments" of Sec. 4.3 and Fig. 3).
//
// Depth z maps to the angle phi = z (1 - zeta) pi, leaving a wrapping zone of
// width 2 zeta pi between the farthest and the nearest depth.  Pass 1 sums
// b0 = sum a and t_j = sum a e^{i j phi}; the stored moments are
// tau_j = t_j / b0 (float16 / bfloat16).  The bias mixes them with the
// uniform measure on the circle: tau'_j = (1 - beta) tau_j, which keeps the
// Toeplitz matrix G[k][l] = tau'_{l-k} positive definite.
//
// Bound at u0 = e^{i phi0}: the canonical (Szego) representation through u0
// has its other nodes at the roots of K(u, u0) = v(u)^T G^-1 conj(v(u0))
// (v(u) = (1, u, .., u^n)) and every node u_i carries the Christoffel weight
// 1 / K(u_i, u_i).  Substituting u = u0 (s + i) / (s - i), which sends u0 to
// s = infinity, turns K(., u0) into a real polynomial in s of degree n whose
// leading coefficient is K(u0, u0) > 0, so after division it is monic and
// real; its n real roots come from closed forms (Viete for the cubic, Ferrari
// for the quartic) polished by Newton steps.  A node lies in front of u0
// (angle in (-pi, phi0)) exactly when s < tan(phi0 / 2).  The result is
// A = w0 rho0 + the weights of the nodes in front.
//
// The per-pixel factorisation G = L D L^H runs in FP64; per sample all
// arithmetic is FP32.  The conditioning of G is bounded by the bias (about
// 1 / beta); the 16-bit storages need beta >= 2e-3, where FP32 suffices.
#pragma once
#include "mboit_vec.cuh"

namespace mb {

struct cf {
    float x, y;
};
MB_HD cf cmul(cf a, cf b) { return {ffma(a.x, b.x, -a.y * b.y), ffma(a.x, b.y, a.y * b.x)}; }
MB_HD cf cconj(cf a) { return {a.x, -a.y}; }

// Complex numbers of one point or two (mboit_vec.cuh), by coefficients that the
// points of a pixel share.
template <class T>
struct cv {
    T x, y;
};
template <class T>
MB_HD cv<T> cmul(cv<T> a, cv<T> b) {
    return {vfma(a.x, b.x, vmul(vneg(a.y), b.y)), vfma(a.x, b.y, vmul(a.y, b.x))};
}
template <class T>
MB_HD cv<T> cconj(cv<T> a) { return {a.x, vneg(a.y)}; }
// a - b
template <class T>
MB_HD cv<T> csub_of(cv<T> a, cf b) { return {vadd(a.x, Vec<T>::splat(-b.x)), vadd(a.y, Vec<T>::splat(-b.y))}; }
// a - b * c
template <class T>
MB_HD cv<T> cfms(cv<T> a, cf b, cv<T> c) {
    const T nx = Vec<T>::splat(-b.x), y = Vec<T>::splat(b.y), ny = Vec<T>::splat(-b.y);
    return {vfma(nx, c.x, vfma(y, c.y, a.x)), vfma(nx, c.y, vfma(ny, c.x, a.y))};
}
// a - conj(b) * c
template <class T>
MB_HD cv<T> cfms_conj(cv<T> a, cf b, cv<T> c) {
    const T nx = Vec<T>::splat(-b.x), y = Vec<T>::splat(b.y), ny = Vec<T>::splat(-b.y);
    return {vfma(nx, c.x, vfma(ny, c.y, a.x)), vfma(nx, c.y, vfma(y, c.x, a.y))};
}

struct TrigFrame {
    int32_t n;            // 0: no absorber, or G not positive definite (then A = 0)
    float m0_log2e;
    cf L[10];             // strictly lower part of L, row i at i (i - 1) / 2
    float invD[5];
};

// FP64 factorisation of the biased Toeplitz matrix of one pixel.
MB_HD TrigFrame make_trig_frame(float b0, const cf* tau, int n, float beta) {
    TrigFrame F;
    F.n = 0;
    F.m0_log2e = 0.0f;
    for (int i = 0; i < 10; ++i) F.L[i] = {0.0f, 0.0f};
    for (int i = 0; i < 5; ++i) F.invD[i] = 0.0f;
    if (!(b0 > 0.0f)) return F;
    const int n1 = n + 1;
    double tr[5], ti[5];
    tr[0] = 1.0;
    ti[0] = 0.0;
    for (int j = 1; j <= n; ++j) {
        tr[j] = (1.0 - (double)beta) * (double)tau[j - 1].x;
        ti[j] = (1.0 - (double)beta) * (double)tau[j - 1].y;
    }
    double Lr[5][5], Li[5][5], D[5];
    for (int j = 0; j < n1; ++j) {
        // G[j][j] = 1
        double s = 1.0;
        for (int k = 0; k < j; ++k) s -= (Lr[j][k] * Lr[j][k] + Li[j][k] * Li[j][k]) * D[k];
        if (!(s > 0.0)) return F;
        D[j] = s;
        for (int i = j + 1; i < n1; ++i) {
            // G[i][j] = conj(tau'[i - j])
            double xr = tr[i - j], xi = -ti[i - j];
            for (int k = 0; k < j; ++k) {
                // L[i][k] conj(L[j][k]) D[k]
                const double pr = Lr[i][k] * Lr[j][k] + Li[i][k] * Li[j][k];
                const double pi = Li[i][k] * Lr[j][k] - Lr[i][k] * Li[j][k];
                xr -= pr * D[k];
                xi -= pi * D[k];
            }
            Lr[i][j] = xr / D[j];
            Li[i][j] = xi / D[j];
        }
    }
    for (int i = 1; i < n1; ++i)
        for (int j = 0; j < i; ++j) F.L[i * (i - 1) / 2 + j] = {(float)Lr[i][j], (float)Li[i][j]};
    for (int i = 0; i < n1; ++i) F.invD[i] = (float)(1.0 / D[i]);
    F.n = n;
    F.m0_log2e = (float)((double)b0 * 1.4426950408889634);
    return F;
}

MB_HD void sincos_fast(float x, float& sn, float& cs) {
#if defined(__CUDA_ARCH__)
    __sincosf(x, &sn, &cs);
#else
    sn = sinf(x);
    cs = cosf(x);
#endif
}
#if defined(__CUDACC__)
__device__ __forceinline__ void sincos_fast(float2 x, float2& sn, float2& cs) {
    sincos_fast(x.x, sn.x, cs.x);
    sincos_fast(x.y, sn.y, cs.y);
}
#endif

// K(u, u) = sum_k |x_k|^2 / D_k with L x = conj(v(u)).
template <int N, class T>
MB_HD T trig_kernel_diag(const TrigFrame& F, cv<T> u) {
    cv<T> x[N + 1];
    const cv<T> ub = cconj(u);
    cv<T> p = ub;
    T K = Vec<T>::splat(F.invD[0]);   // x_0 = 1
#pragma unroll
    for (int i = 1; i <= N; ++i) {
        cv<T> xi = csub_of(p, F.L[i * (i - 1) / 2]);
#pragma unroll
        for (int k = 1; k < i; ++k) xi = cfms(xi, F.L[i * (i - 1) / 2 + k], x[k]);
        x[i] = xi;
        K = vfma(vfma(xi.x, xi.x, vmul(xi.y, xi.y)), Vec<T>::splat(F.invD[i]), K);
        if (i < N) p = cmul(p, ub);
    }
    return K;
}

// Weight of the node at s: 1 / K(u, u) at u = u0 (s + i) / (s - i).
template <int N, class T>
MB_HD T trig_weight(const TrigFrame& F, cv<T> u0, T s) {
    const T inv = vrcp(vfma(s, s, Vec<T>::splat(1.0f)));
    const cv<T> e = {vmul(vfma(s, s, Vec<T>::splat(-1.0f)), inv), vmul(vtwice(s), inv)};
    return vrcp(trig_kernel_diag<N, T>(F, cmul(u0, e)));
}

// Sum of the weights of the nodes in front, r ascending, the first `front` of
// them in front; `weight` gives a root's.  The weights of all nodes and of the
// point itself (rho0) add up to 1, so the smaller side is summed: one weight
// of three nodes, at most two of four (the second only where a point of the
// warp has two nodes on either side), instead of every one in front.
template <int N, class T, class W>
MB_HD T front_weight(const T* r, Lanes<T> front, T rho0, T w0, const W& weight) {
    const T one = Vec<T>::splat(1.0f), zero = Vec<T>::splat(0.0f);
    const T hi = vfma(vsub(w0, one), rho0, one);
    // the side's outermost node, none where the other side holds all
    const T s = pick_gt(front, N / 2, r[N - 1], r[0]);
    T w = weight(s);
    w = pick_eq(front, 0, zero, pick_eq(front, N, zero, w));
    if (N == 4 && any_eq(front, 2)) w = vadd(w, pick_eq(front, 2, weight(r[1]), zero));
    return pick_gt(front, N / 2, vsub(hi, w), vfma(w0, rho0, w));
}

// Alg. 3 for trigonometric moments: fraction A of the optical depth in front
// of warped depth z0 (F.n > 0), for one depth (float) or two (float2).
template <int N, class T>
MB_HD T trig_fraction(const TrigFrame& F, const TrigTables& tab, T z0, float w0) {
    cv<T> u0;
    sincos_fast(vmul(z0, Vec<T>::splat(tab.zone_scale)), u0.y, u0.x);
    // y = G^-1 w, w = conj(v(u0)) = (1, conj(u0), conj(u0)^2, ..)
    cv<T> w[N + 1], y[N + 1];
    w[1] = cconj(u0);
#pragma unroll
    for (int k = 2; k <= N; ++k) w[k] = cmul(w[k - 1], w[1]);
#pragma unroll
    for (int i = 1; i <= N; ++i) {
        cv<T> t = csub_of(w[i], F.L[i * (i - 1) / 2]);   // y_0 = 1
#pragma unroll
        for (int k = 1; k < i; ++k) t = cfms(t, F.L[i * (i - 1) / 2 + k], y[k]);
        y[i] = t;
    }
    y[0] = {Vec<T>::splat(F.invD[0]), Vec<T>::splat(0.0f)};
#pragma unroll
    for (int i = 1; i <= N; ++i) {
        const T d = Vec<T>::splat(F.invD[i]);
        y[i] = {vmul(y[i].x, d), vmul(y[i].y, d)};
    }
#pragma unroll
    for (int i = N; i >= 0; --i) {
        cv<T> t = y[i];
#pragma unroll
        for (int k = i + 1; k <= N; ++k) t = cfms_conj(t, F.L[k * (k - 1) / 2 + i], y[k]);
        y[i] = t;
    }
    // z_k = y_k u0^k; K(u0, u0) = Re sum z_k; real polynomial coefficients
    T zr[N + 1], nzi[N + 1], K00 = y[0].x;
    zr[0] = y[0].x;
    nzi[0] = vneg(y[0].y);
#pragma unroll
    for (int k = 1; k <= N; ++k) {
        const cv<T> z = cmul(y[k], cconj(w[k]));
        zr[k] = z.x;
        nzi[k] = vneg(z.y);
        K00 = vadd(K00, z.x);
    }
    const T rho0 = vrcp(K00);
    T coef[N];
#pragma unroll
    for (int m = 0; m < N; ++m) {
        T acc = vfma(zr[0], Vec<T>::splat(tab.er[0][m]), vmul(nzi[0], Vec<T>::splat(tab.ei[0][m])));
#pragma unroll
        for (int k = 1; k <= N; ++k)
            acc = vfma(zr[k], Vec<T>::splat(tab.er[k][m]), vfma(nzi[k], Vec<T>::splat(tab.ei[k][m]), acc));
        coef[m] = vmul(acc, rho0);
    }
    T rts[N];
    if constexpr (N == 3)
        cubic3(coef[2], coef[1], coef[0], rts);
    else
        quartic4(coef[3], coef[2], coef[1], coef[0], rts);
    // tan(phi0 / 2); |phi0| < pi by the wrapping zone
    const T sp = vmul(u0.y, vrcp(vadd(Vec<T>::splat(1.0f), u0.x)));
    Lanes<T> front = below(rts[0], sp);
#pragma unroll
    for (int i = 1; i < N; ++i) front = front + below(rts[i], sp);
    return front_weight<N, T>(rts, front, rho0, Vec<T>::splat(w0), [&](T s) { return trig_weight<N, T>(F, u0, s); });
}

}  // namespace mb
