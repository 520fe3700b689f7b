// Spectral functions for the observables of Sec. 5.2 (von Neumann entropy, fidelity) on reduced
// density matrices, which the GPU partial trace brings to the host (2^k x 2^k, k <= 6).
#include "hermitian.h"

#include <algorithm>
#include <cmath>
#include <numeric>
#include <vector>

namespace qcw {

using cd = std::complex<double>;

// Eigenvalues only: Householder reduction to a real tridiagonal matrix (Golub and Van Loan, "Matrix
// Computations", Sec. 8.3: A <- A - v w^H - w v^H with w = p - (beta / 2) (p^H v) v, p = beta A v),
// then implicit QR steps with Wilkinson's shift on it (Sec. 8.3.5).  O(N^3) once where each sweep
// of the Jacobi iteration below costs several times that: 64 x 64 took 6 ms with it.
static void eigenvalues_only(const cd *A_in, int N, double *w)
{
    // A in separate real and imaginary parts, lower right block k.. updated in place
    std::vector<double> Ar((size_t)N * N), Ai((size_t)N * N), vr(N), vi(N), pr(N), pi(N), d(N), e(N, 0.0);
    for (size_t i = 0; i < (size_t)N * N; i++) Ar[i] = A_in[i].real(), Ai[i] = A_in[i].imag();
    for (int k = 0; k + 1 < N; k++) {
        const int m0 = k + 1;
        double nrm = 0;
        for (int i = m0; i < N; i++) {
            vr[i] = Ar[(size_t)i * N + k], vi[i] = Ai[(size_t)i * N + k];
            nrm += vr[i] * vr[i] + vi[i] * vi[i];
        }
        nrm = std::sqrt(nrm);
        e[k] = nrm;  // |off-diagonal|: its phase is a diagonal similarity
        double tail = 0;
        for (int i = m0 + 1; i < N; i++) tail += vr[i] * vr[i] + vi[i] * vi[i];
        if (tail == 0 || nrm == 0) continue;  // already of the form (x0, 0, ..., 0)
        const double a0 = std::hypot(vr[m0], vi[m0]);
        // v = x + e^{i arg x0} |x| e_0
        const double cr = a0 > 0 ? vr[m0] / a0 : 1.0, ci = a0 > 0 ? vi[m0] / a0 : 0.0;
        vr[m0] += cr * nrm, vi[m0] += ci * nrm;
        const double beta = 1.0 / (nrm * (nrm + a0));  // 2 / v^H v
        for (int i = m0; i < N; i++) pr[i] = pi[i] = 0;
        for (int j = m0; j < N; j++) {  // p = A v, row by row of the conjugate (no reductions inside)
            const double *ar = &Ar[(size_t)j * N], *ai = &Ai[(size_t)j * N];
            const double xr = vr[j], xi = vi[j];
            for (int i = m0; i < N; i++) {
                pr[i] += ar[i] * xr + ai[i] * xi;
                pi[i] += ar[i] * xi - ai[i] * xr;
            }
        }
        double kr = 0;
        for (int i = m0; i < N; i++) {
            pr[i] *= beta, pi[i] *= beta;
            kr += pr[i] * vr[i] + pi[i] * vi[i];  // p^H v is real (A is Hermitian)
        }
        const double h = 0.5 * beta * kr;
        for (int i = m0; i < N; i++) pr[i] -= h * vr[i], pi[i] -= h * vi[i];
        for (int i = m0; i < N; i++) {
            double *ar = &Ar[(size_t)i * N], *ai = &Ai[(size_t)i * N];
            const double xr = vr[i], xi = vi[i], yr = pr[i], yi = pi[i];
            for (int j = m0; j < N; j++) {  // - v_i conj(w_j) - w_i conj(v_j)
                ar[j] -= xr * pr[j] + xi * pi[j] + yr * vr[j] + yi * vi[j];
                ai[j] -= xi * pr[j] - xr * pi[j] + yi * vr[j] - yr * vi[j];
            }
        }
    }
    double scale = 0;
    for (int i = 0; i < N; i++) d[i] = Ar[(size_t)i * N + i], scale = std::max(scale, std::fabs(d[i]) + e[i]);
    // QR steps on the last block lo..hi that does not split: T <- Q^T T Q with Q a product of plane
    // rotations (c, s) of rows k, k + 1, the first one that of T - mu, the others those that put back the
    // element (k + 1, k - 1) which the one before it has filled.
    for (int hi = N - 1, steps = 0; hi > 0;) {
        int lo = hi;
        while (lo > 0 && std::fabs(e[lo - 1]) > 1e-17 * scale &&
               std::fabs(e[lo - 1]) > 2.3e-16 * (std::fabs(d[lo - 1]) + std::fabs(d[lo])))
            lo--;
        if (lo == hi || steps == 60) {  // d[hi] is an eigenvalue
            hi--, steps = 0;
            continue;
        }
        steps++;
        // mu: of the eigenvalues of the last two rows the one nearer to d[hi]
        const double half = 0.5 * (d[hi - 1] - d[hi]), root = std::hypot(half, e[hi - 1]);
        double x = d[lo] - d[hi] + e[hi - 1] * (e[hi - 1] / (half + (half >= 0 ? root : -root))), z = e[lo];
        for (int k = lo; k < hi; k++) {
            const double r2 = x * x + z * z, r = r2 > 1e-280 && r2 < 1e280 ? std::sqrt(r2) : std::hypot(x, z);
            const double c = r > 0 ? x / r : 1.0, s = r > 0 ? z / r : 0.0;
            if (k > lo) e[k - 1] = r;
            const double p = c * d[k] + s * e[k], q = c * e[k] + s * d[k + 1];      // rows k and k + 1 rotated
            const double t = c * e[k] - s * d[k], u = c * d[k + 1] - s * e[k];
            d[k] = c * p + s * q;  // then the columns
            d[k + 1] = c * u - s * t;
            x = e[k] = c * t + s * u;
            if (k + 1 < hi) {
                z = s * e[k + 1];
                e[k + 1] *= c;
            }
        }
    }
    std::sort(d.begin(), d.end());
    for (int i = 0; i < N; i++) w[i] = d[i];
}

// Cyclic Jacobi: for each off-diagonal pair (p, q) with a_pq = r e^{i phi}, the unitary
// U = diag(1, e^{-i phi}) G on coordinates (p, q), G the plane rotation by
// theta = atan2(2 r, a_pp - a_qq) / 2, makes (U^dagger A U)_pq = 0 (the phase turns a_pq into r,
// G diagonalises the real 2 x 2 block).  Sweeps repeat until the off-diagonal part is below
// 1e-15 of the matrix norm (quadratic convergence: a handful of sweeps).
void herm_eig(const cd *A_in, int N, double *w, cd *V)
{
    if (!V) {
        eigenvalues_only(A_in, N, w);
        return;
    }
    std::vector<cd> A(A_in, A_in + (size_t)N * N);
    std::vector<cd> U;
    if (V) {
        U.assign((size_t)N * N, cd(0, 0));
        for (int i = 0; i < N; i++) U[(size_t)i * N + i] = 1.0;
    }
    double norm = 0;
    for (const cd &x : A) norm += std::norm(x);
    norm = std::sqrt(norm);
    for (int sweep = 0; sweep < 100 && norm > 0; sweep++) {
        double off = 0;
        for (int p = 0; p < N; p++)
            for (int q = p + 1; q < N; q++) off += std::norm(A[(size_t)p * N + q]);
        if (std::sqrt(2 * off) <= 1e-15 * norm) break;
        for (int p = 0; p < N; p++)
            for (int q = p + 1; q < N; q++) {
                const cd apq = A[(size_t)p * N + q];
                const double r = std::abs(apq);
                if (r == 0) continue;
                const cd e = std::conj(apq / r);  // e^{-i phi}
                const double th = 0.5 * std::atan2(2 * r, A[(size_t)p * N + p].real() - A[(size_t)q * N + q].real());
                const double c = std::cos(th), s = std::sin(th);
                const cd upp = c, upq = -s, uqp = e * s, uqq = e * c;
                for (int k = 0; k < N; k++) {  // A <- A U
                    const cd akp = A[(size_t)k * N + p], akq = A[(size_t)k * N + q];
                    A[(size_t)k * N + p] = akp * upp + akq * uqp;
                    A[(size_t)k * N + q] = akp * upq + akq * uqq;
                }
                for (int k = 0; k < N; k++) {  // A <- U^dagger A
                    const cd apk = A[(size_t)p * N + k], aqk = A[(size_t)q * N + k];
                    A[(size_t)p * N + k] = std::conj(upp) * apk + std::conj(uqp) * aqk;
                    A[(size_t)q * N + k] = std::conj(upq) * apk + std::conj(uqq) * aqk;
                }
                A[(size_t)p * N + q] = A[(size_t)q * N + p] = 0.0;
                A[(size_t)p * N + p] = A[(size_t)p * N + p].real();
                A[(size_t)q * N + q] = A[(size_t)q * N + q].real();
                if (V)
                    for (int k = 0; k < N; k++) {  // U_acc <- U_acc U
                        const cd vkp = U[(size_t)k * N + p], vkq = U[(size_t)k * N + q];
                        U[(size_t)k * N + p] = vkp * upp + vkq * uqp;
                        U[(size_t)k * N + q] = vkp * upq + vkq * uqq;
                    }
            }
    }
    std::vector<int> idx(N);
    std::iota(idx.begin(), idx.end(), 0);
    std::sort(idx.begin(), idx.end(),
              [&](int a, int b) { return A[(size_t)a * N + a].real() < A[(size_t)b * N + b].real(); });
    for (int i = 0; i < N; i++) w[i] = A[(size_t)idx[i] * N + idx[i]].real();
    if (V)
        for (int k = 0; k < N; k++)
            for (int i = 0; i < N; i++) V[(size_t)k * N + i] = U[(size_t)k * N + idx[i]];
}

double entropy_bits(const double *w, int N)
{
    double s = 0;
    for (int i = 0; i < N; i++)
        if (w[i] > 1e-15) s -= w[i] * std::log2(w[i]);
    return s;
}

double fidelity_root(const cd *rho, const cd *sigma, int N)
{
    std::vector<double> mu(N), nu(N);
    std::vector<cd> V((size_t)N * N), S((size_t)N * N, cd(0, 0)), T((size_t)N * N), M((size_t)N * N);
    herm_eig(sigma, N, mu.data(), V.data());
    for (int a = 0; a < N; a++)  // sqrt(sigma) = V diag(sqrt mu) V^dagger
        for (int b = 0; b < N; b++) {
            cd x = 0;
            for (int i = 0; i < N; i++)
                x += V[(size_t)a * N + i] * std::sqrt(std::max(mu[i], 0.0)) * std::conj(V[(size_t)b * N + i]);
            S[(size_t)a * N + b] = x;
        }
    for (int a = 0; a < N; a++)  // T = sqrt(sigma) rho
        for (int b = 0; b < N; b++) {
            cd x = 0;
            for (int i = 0; i < N; i++) x += S[(size_t)a * N + i] * rho[(size_t)i * N + b];
            T[(size_t)a * N + b] = x;
        }
    for (int a = 0; a < N; a++)  // M = T sqrt(sigma), made exactly Hermitian
        for (int b = 0; b < N; b++) {
            cd x = 0;
            for (int i = 0; i < N; i++) x += T[(size_t)a * N + i] * S[(size_t)i * N + b];
            M[(size_t)a * N + b] = x;
        }
    for (int a = 0; a < N; a++)
        for (int b = a; b < N; b++) {
            const cd h = 0.5 * (M[(size_t)a * N + b] + std::conj(M[(size_t)b * N + a]));
            M[(size_t)a * N + b] = h;
            M[(size_t)b * N + a] = std::conj(h);
        }
    herm_eig(M.data(), N, nu.data(), V.data());  // the Jacobi iteration: square roots of small eigenvalues follow
    double f = 0;
    for (int i = 0; i < N; i++) f += std::sqrt(std::max(nu[i], 0.0));
    return f;
}

}  // namespace qcw
