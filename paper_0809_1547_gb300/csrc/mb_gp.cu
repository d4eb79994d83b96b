// Bound states of the dimensionless spectral-envelope equation of the
// random-laser theory (the paper's Eq. g5, "Gross-Pitaevskii equation"
// paragraph):
//     -phi'' + tau^2 phi + phi^3 = E phi,   phi > 0,  phi(+-L) = 0,
// for a batch of eigenvalues E > 1, and the spectral waist and peak of each
// (Figs. 3, 5).  Second-order differences on tau_i = -L + i h (i = 1..n,
// h = 2L/(n+1)), Newton's method with a tridiagonal solve per iteration, all
// in FP64.  Newton starts from the larger of the Thomas-Fermi profile
// sqrt(max(E - tau^2, 0)) and the first-order solution near threshold
// 2^{1/4} sqrt(E - 1) exp(-tau^2 / 2) and stops when the residual is below
// 1e-13 max(1, E) or stagnates at rounding level; a result whose
// residual stays above 1e-9 max(1, E), or that collapses towards the trivial
// solution phi = 0, is reported as not converged.
#include "mb_host.h"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

namespace {

constexpr int kGpMaxIter = 100;
constexpr int kGpThreads = 128;
constexpr size_t kGpSharedMax = 200 * 1024;   // dynamic shared memory of a block's arrays

// Largest of the block's values of |x| (as bit patterns: the order of
// non-negative doubles is that of their bits, so the FP64 pipe has no part
// in it; a NaN comes out largest).
__device__ unsigned long long block_max(unsigned long long v, unsigned long long* red) {
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();   // red is free
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    v = red[0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) v = max(v, red[w]);
    return v;
}

__device__ double block_sum(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    v = red[0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) v += red[w];
    return v;
}

__device__ __forceinline__ unsigned long long abs_bits(double x) {
    return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}

// A block per eigenvalue.  Thread t owns points [t m, (t+1) m), m = ceil(n /
// threads) (at least 2; points past n are identity rows with phi = 0), kept
// interleaved (point i of thread t at i T + t): four arrays phi, b, f, v of m
// T doubles in shared memory, or in global scratch where they do not fit.
//
// Newton step by partition: a thread's last row is a separator.  It
// eliminates its other rows from the left, keeping the fill towards the
// separator of the thread before (v), so that x_i = f_i - b_i x_{i+1} - v_i
// s_{t-1}, and folds them into its first row (Y, V, W).  The separators form
// a tridiagonal system of one row per thread, solved by parallel cyclic
// reduction; back-substitution gives the rest.
//
// The residual takes phi'' from differences of neighbours, which are exact
// (their ratio is below 2 where phi matters), so that what is left of its
// rounding is of the size of phi'' and not of phi / h^2: with the sum of the
// neighbours against 2 phi the features at n = 2047 were off by up to 2e-11
// (p_phi; the tridiagonal solve in order of the points 1e-13), with the
// differences by 2e-14 (against extended precision, 1.05 <= E <= 60).
//
// The serial form (one thread per eigenvalue walking its n points through
// global memory, three dependent passes and two divisions per point and
// iteration) took 35 ms for 200 eigenvalues at n = 2047 (8 warps busy on the
// whole GPU); this takes 0.55 ms, 0.32 ms for one eigenvalue.  This form is
// bound by the FP64 pipe (2 operations per cycle and SM here): about 29 FP64
// operations per point and iteration plus the
// cyclic reduction's ~170 per thread.  128 threads put one warp on each of
// an SM's four schedulers, which the pipe's rate already fills: 64 threads took
// 0.45 ms for one eigenvalue and 1.6 against 1.0 ms for 64 at n = 8191, 256
// threads 0.65 against 0.55 ms for 200 at n = 2047 (longer reduction).
__global__ void __launch_bounds__(kGpThreads) k_gp_solve(const double* Es, int n, int m, double* scratch,
                                                         double* phi_out, double* w_out, double* p_out,
                                                         int* status) {
    extern __shared__ double gp_sh[];
    __shared__ double ra[2][kGpThreads], rb[2][kGpThreads], rc[2][kGpThreads], rf[2][kGpThreads];
    __shared__ double red[kGpThreads / 32];
    unsigned long long* redu = reinterpret_cast<unsigned long long*>(red);
    const int T = blockDim.x, t = threadIdx.x, q = blockIdx.x;
    const size_t len = (size_t)m * T;
    double* base = scratch ? scratch + 4 * len * q : gp_sh;
    double* phi = base + t;
    double* bb = base + len + t;
    double* ff = base + 2 * len + t;
    double* vv = base + 3 * len + t;
    const double E = Es[q];
    const double L = sqrt(E) + 8.0;
    const double h = 2.0 * L / (n + 1);
    const double ih2 = 1.0 / (h * h);
    const double off = -ih2;
    const double amp = pow(2.0, 0.25) * sqrt(E - 1.0);
    const double d0 = 2.0 * ih2;
    const int i0 = t * m;
    const int mine = min(m, max(0, n - i0));   // points of the grid among the thread's m
    for (int i = 0; i < m; ++i) {
        const double tau = -L + h * (i0 + i + 1);
        const double tf = sqrt(fmax(E - tau * tau, 0.0));
        phi[(size_t)i * T] = i < mine ? fmax(tf, amp * exp(-0.5 * tau * tau)) : 0.0;
    }
    // phi of the point before the thread's first and after its last
    auto left = [&]() { return t > 0 ? phi[(size_t)(m - 1) * T - 1] : 0.0; };
    auto right = [&]() { return t < T - 1 ? phi[1] : 0.0; };
    const double tol = 1e-13 * fmax(1.0, E), accept = 1e-9 * fmax(1.0, E);
    double rprev = 0.0;
    int ok = 0;
    for (int it = 0;; ++it) {
        // residual into f, the Jacobian's diagonal into b
        __syncthreads();
        unsigned long long rm = 0;
        {
            double c = phi[0], dl = c - left();
            const double after = right();
            for (int i = 0; i < mine; ++i) {
                const double r = i + 1 < m ? phi[(size_t)(i + 1) * T] : after;
                const double tau = fma(h, (double)(i0 + i + 1), -L);
                const double p2 = c * c;
                const double g = fma(tau, tau, -E) + p2;
                const double dr = r - c;
                const double f = fma(c, g, off * (dr - dl));
                ff[(size_t)i * T] = f;
                bb[(size_t)i * T] = fma(2.0, p2, g) + d0;
                rm = max(rm, abs_bits(f));
                dl = dr;
                c = r;
            }
        }
        const double rmax = __longlong_as_double((long long)block_max(rm, redu));
        if (rmax < tol) {
            ok = 1;
            break;
        }
        // rounding floor (~eps / h^2 can lie above tol): the residual no
        // longer falls and is already below what is accepted
        if (it > 0 && rmax < accept && rmax >= 0.5 * rprev) {
            ok = 1;
            break;
        }
        if (it == kGpMaxIter) {
            ok = rmax < accept;
            break;
        }
        rprev = rmax;
        // rows 0 .. m-2 eliminated from the left: cp in b, dp in f, fill in v
        double cp = 0.0, dp = 0.0, vp = 0.0;
        for (int i = 0; i < m - 1; ++i) {
            if (i < mine) {
                const double r = 1.0 / (i > 0 ? fma(-off, cp, bb[(size_t)i * T]) : bb[0]);
                dp = (i > 0 ? fma(-off, dp, ff[(size_t)i * T]) : ff[0]) * r;
                const double o = off * r;
                vp = i > 0 ? -o * vp : o;
                cp = o;
            } else {
                cp = dp = vp = 0.0;
            }
            bb[(size_t)i * T] = cp;
            ff[(size_t)i * T] = dp;
            vv[(size_t)i * T] = vp;
        }
        // first row in terms of the two separators: x_0 = Y + V s_{t-1} + W s_t
        double Y = dp, V = -vp, W = -cp;
        for (int i = m - 3; i >= 0; --i) {
            const double c = bb[(size_t)i * T];
            Y = fma(-c, Y, ff[(size_t)i * T]);
            V = fma(-c, V, -vv[(size_t)i * T]);
            W *= -c;
        }
        // separator rows: off x_{m-2} + b s_t + off x_0(t+1) = f
        __syncthreads();
        ra[0][t] = Y;
        rb[0][t] = V;
        rc[0][t] = W;
        __syncthreads();
        double A = 0.0, B = 1.0, C = 0.0, F = 0.0;
        if (mine == m) {
            const bool nx = t < T - 1;
            const double Yn = nx ? ra[0][t + 1] : 0.0, Vn = nx ? rb[0][t + 1] : 0.0, Wn = nx ? rc[0][t + 1] : 0.0;
            A = t > 0 ? -off * vp : 0.0;
            B = fma(off, Vn - cp, bb[(size_t)(m - 1) * T]);
            C = off * Wn;
            F = fma(-off, dp + Yn, ff[(size_t)(m - 1) * T]);
        }
        // parallel cyclic reduction over the separators
        int cur = 1;
        for (int s = 1; s < T; s <<= 1) {
            ra[cur][t] = A;
            rb[cur][t] = 1.0 / B;
            rc[cur][t] = C;
            rf[cur][t] = F;
            __syncthreads();
            double al = 0.0, ga = 0.0, Al = 0.0, Cl = 0.0, Fl = 0.0, Ar = 0.0, Cr = 0.0, Fr = 0.0;
            if (t >= s) {
                al = -A * rb[cur][t - s];
                Al = ra[cur][t - s];
                Cl = rc[cur][t - s];
                Fl = rf[cur][t - s];
            }
            if (t + s < T) {
                ga = -C * rb[cur][t + s];
                Ar = ra[cur][t + s];
                Cr = rc[cur][t + s];
                Fr = rf[cur][t + s];
            }
            B = fma(al, Cl, fma(ga, Ar, B));
            F = fma(al, Fl, fma(ga, Fr, F));
            A = al * Al;
            C = ga * Cr;
            cur ^= 1;   // the next step writes the other set
        }
        double x = F / B;   // the step at the thread's separator
        __syncthreads();
        ra[0][t] = x;
        __syncthreads();
        const double sl = t > 0 ? ra[0][t - 1] : 0.0;
        unsigned long long dm = abs_bits(x), pm;
        double pn = phi[(size_t)(m - 1) * T] - x;
        if (mine < m) pn = 0.0;
        phi[(size_t)(m - 1) * T] = pn;
        pm = pn > 0.0 ? abs_bits(pn) : 0ull;
        for (int i = m - 2; i >= 0; --i) {
            x = fma(-vv[(size_t)i * T], sl, fma(-bb[(size_t)i * T], x, ff[(size_t)i * T]));
            if (i < mine) {
                pn = phi[(size_t)i * T] - x;
                phi[(size_t)i * T] = pn;
                dm = max(dm, abs_bits(x));
                if (__double_as_longlong(pn) > 0) pm = max(pm, abs_bits(pn));
            }
        }
        const double dmax = __longlong_as_double((long long)block_max(dm, redu));
        const double pmx = __longlong_as_double((long long)block_max(pm, redu));
        if (dmax <= 1e-14 * fmax(1.0, pmx)) {   // stagnated: accepted by its residual
            rprev = 0.0;
            __syncthreads();
            unsigned long long r2 = 0;
            double c = phi[0], dl = c - left();
            const double after = right();
            for (int i = 0; i < mine; ++i) {
                const double r = i + 1 < m ? phi[(size_t)(i + 1) * T] : after;
                const double tau = fma(h, (double)(i0 + i + 1), -L);
                const double dr = r - c;
                r2 = max(r2, abs_bits(fma(c, fma(tau, tau, -E) + c * c, off * (dr - dl))));
                dl = dr;
                c = r;
            }
            ok = __longlong_as_double((long long)block_max(r2, redu)) < accept;
            break;
        }
    }
    // features: p = (h sum phi)^2 / (4 pi^2); w = sqrt(sum dphi^2 / sum phi^2) / (2 pi)
    __syncthreads();
    double s1 = 0.0, s2 = 0.0, sd = 0.0;
    unsigned long long pm = 0;
    {
        double prev = left();
        for (int i = 0; i < mine; ++i) {
            const double p = phi[(size_t)i * T];
            s1 += p;
            s2 = fma(p, p, s2);
            sd = fma(p - prev, p - prev, sd);
            prev = p;
            if (__double_as_longlong(p) > 0) pm = max(pm, abs_bits(p));
            if (phi_out) phi_out[(size_t)q * n + i0 + i] = p;
        }
        if (mine > 0 && i0 + mine == n) sd = fma(prev, prev, sd);   // the step to phi(L) = 0
    }
    s1 = block_sum(s1, red);
    s2 = block_sum(s2, red);
    sd = block_sum(sd, red);
    const double pmax = __longlong_as_double((long long)block_max(pm, redu));
    if (t == 0) {
        const double pi = 3.14159265358979323846;
        const double hs1 = h * s1;
        p_out[q] = hs1 * hs1 / (4.0 * pi * pi);
        w_out[q] = sqrt((sd / (h * h)) / s2) / (2.0 * pi);
        if (ok && pmax < 0.5 * amp) ok = 0;   // collapsed towards phi = 0
        status[q] = ok;
    }
}

}  // namespace

extern "C" int mb_gp_features(const double* E, int nE, int n_grid, double* w_phi, double* p_phi,
                              double* phi_out) {
    if (!E || nE < 1 || n_grid < 16 || n_grid > (1 << 20) || !w_phi || !p_phi) {
        mb::set_thread_error("bad arguments: nE >= 1, 16 <= n_grid <= 2^20, outputs non-null");
        return MB_ERR_ARG;
    }
    for (int q = 0; q < nE; ++q)
        if (!(E[q] > 1.0) || !std::isfinite(E[q])) {
            mb::set_thread_error("every E must be finite and > 1 (bound states exist above threshold)");
            return MB_ERR_ARG;
        }
    const size_t n = (size_t)n_grid;
    const int m = std::max(2, (n_grid + kGpThreads - 1) / kGpThreads);
    const size_t arrays = sizeof(double) * 4 * (size_t)m * kGpThreads;
    const bool shared = arrays <= kGpSharedMax;
    std::vector<int> st((size_t)nE);
    int rc = MB_OK;
    // one device buffer: E, w, p, status, then phi (when asked for) and the
    // blocks' arrays (when they do not fit in shared memory)
    double* buf = nullptr;
    const size_t head = 4 * (size_t)nE, phis = phi_out ? n * (size_t)nE : 0;
    // scratch for at most 2 GB of eigenvalues at a time
    const int batch = shared ? nE : (int)std::max<size_t>(1, std::min<size_t>(nE, (size_t(2) << 30) / arrays));
    cudaError_t e = cudaMalloc((void**)&buf, sizeof(double) * (head + phis) + (shared ? 0 : arrays * batch));
    double *dw = buf + nE, *dp = buf + 2 * (size_t)nE, *dphi = phi_out ? buf + head : nullptr;
    int* dst = reinterpret_cast<int*>(buf + 3 * (size_t)nE);
    std::vector<double> out(head);
    if (e == cudaSuccess) e = cudaMemcpy(buf, E, sizeof(double) * nE, cudaMemcpyHostToDevice);
    if (e == cudaSuccess && shared)
        e = cudaFuncSetAttribute(k_gp_solve, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGpSharedMax);
    for (int q = 0; q < nE && e == cudaSuccess; q += batch) {
        k_gp_solve<<<std::min(batch, nE - q), kGpThreads, shared ? arrays : 0>>>(
            buf + q, n_grid, m, shared ? nullptr : buf + head + phis, dphi ? dphi + n * q : nullptr, dw + q,
            dp + q, dst + q);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(out.data(), buf, sizeof(double) * head, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess && phi_out) e = cudaMemcpy(phi_out, dphi, sizeof(double) * phis, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) {
        std::copy(out.begin() + nE, out.begin() + 2 * (size_t)nE, w_phi);
        std::copy(out.begin() + 2 * (size_t)nE, out.begin() + 3 * (size_t)nE, p_phi);
        std::memcpy(st.data(), out.data() + 3 * (size_t)nE, sizeof(int) * nE);
    }
    if (e != cudaSuccess) {
        mb::set_thread_error(std::string("gp solve: ") + cudaGetErrorString(e));
        rc = e == cudaErrorMemoryAllocation ? MB_ERR_OOM : MB_ERR_CUDA;
    } else {
        for (int q = 0; q < nE; ++q)
            if (!st[q]) {
                mb::set_thread_error("Newton did not converge to a bound state for E = " + std::to_string(E[q]));
                rc = MB_ERR_STATE;
                break;
            }
    }
    if (buf) cudaFree(buf);
    return rc;
}
