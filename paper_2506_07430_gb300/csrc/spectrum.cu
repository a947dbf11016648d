// Kernel damping and Chebyshev reconstruction of the spectrum (Eq. kpm,
// Eq. jackson) on the Chebyshev nodes x_k = cos(theta_k), theta_k = pi(k+1/2)/M:
//   I(x_k) = (g_0 Omega_0 + 2 sum_{n>=1} g_n Omega_n T_n(x_k)) / (pi sin theta_k)
// with the Jackson kernel g_n = [(N-n+1) cos(pi n/(N+1)) + sin(pi n/(N+1))
// cot(pi/(N+1))]/(N+1), or the Lorentz kernel g_n = sinh(lambda (1 - n/N)) /
// sinh(lambda) of the KPM review the paper cites (the Methods name "modified
// kernels like the Jackson kernel"; Lorentz broadening suits Green's functions).
// This is a type-III discrete cosine transform of the damped moments, evaluated as a
// direct FP64 sum.  What bounds it is FP64 operations (two per clock and SM) and the
// latency of a chain of them (70 clocks each), so the 32 lanes of a warp take
// n = lane, lane + 32, ... of one node, each by the three-term recurrence in steps of 32
// (its error grows with the square of the steps taken, N / 32 instead of N), and
//  - moments beyond the number of nodes fold onto the first M: T_n(x_k) = cos(n theta_k)
//    repeats, up to sign, with period 2M in n (k_fold);
//  - a node and its mirror image (T_n(-x) = (-1)^n T_n(x)) share the sums over even and
//    over odd n.
// Both hold at the exact nodes.  A node rounded to double is off by up to 1e-16, which
// T_n turns into n times that over sin theta: N M 1.4e-17 of the spectrum (measured: 9e-10
// at 8192 x 8191, 6e-9 at 60000 x 8192, no damping).  Up to N M = 2^24 that is below
// 3e-10 and the exact nodes are used; beyond, the sum is over all N moments at the
// rounded node itself, the x of the omega that is returned.
// A call with host arrays, 2048 moments at 2048 nodes: 232 us (334 in a process that has
// nothing else allocated) with one chain per node (16 blocks) and four allocations, 51 us here
// (22 us of it k_reconstruct); 60000 at 2048: 5.2 and 0.54 ms.
// Energy axis omega = a x + b, density per unit energy I/a, written in ascending omega.
#include "common.cuh"

namespace kpm {

__global__ void k_damp(const double* __restrict__ mom, int N, int kernel, double lambda,
                       double* __restrict__ mt) {
    int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    double g = 1.0;
    if (kernel == 1) {
        const double q = M_PI / (N + 1);
        double sn, cn;
        sincos(q * n, &sn, &cn);
        g = ((N - n + 1) * cn + sn * (cos(q) / sin(q))) / (N + 1);
    } else if (kernel == 2) {
        g = sinh(lambda * (1.0 - (double)n / N)) / sinh(lambda);
    }
    mt[n] = g * mom[n] * (n == 0 ? 1.0 : 2.0);
}

// c[m], m < M, gains every damped moment n >= M with T_n(x_k) = +-T_m(x_k) at all nodes:
// n = 4Mj + m (+), 2M(2j + 1) -+ m (-), 4M(j + 1) - m (+).  T_n vanishes at every node for
// n = M(2j + 1); those only pass on a moment that is not finite.
__global__ void __launch_bounds__(128)
k_fold(double* __restrict__ c, int N, int M) {
    const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    const int64_t P = 2 * (int64_t)M;
    double s = c[m];
    // images below, above and so on: 2M - m, 2M + m, 4M - m, 4M + m, ...
    for (int64_t q = P; q - m < N; q += P) {
        const double sg = (q / P) & 1 ? -1.0 : 1.0;
        if (m > 0) s += sg * c[q - m];
        if (q + m < N) s += sg * c[q + m];
    }
    if (m == 0)
        for (int64_t n = M; n < N; n += P) s += 0.0 * c[n];
    c[m] = s;
}

constexpr int REC_WARPS = 8;
constexpr int64_t REC_EXACT = (int64_t)1 << 24;

// EXACT: a warp per pair of mirror nodes, angles reduced in whole numbers; else a warp
// per rounded node.
template <bool EXACT>
__global__ void __launch_bounds__(32 * REC_WARPS)
k_reconstruct(const double* __restrict__ c, int N, double a, double b, int M,
              double* __restrict__ omega, double* __restrict__ inten) {
    const int64_t k = (int64_t)blockIdx.x * REC_WARPS + (threadIdx.x >> 5);   // node of the pair
    const int lane = threadIdx.x & 31;
    if ((EXACT ? 2 * k : k) >= M) return;
    double c32, t;
    if (EXACT) {
        const int64_t per = 4 * (int64_t)M, odd = 2 * k + 1;   // theta_k = pi (2k + 1) / (2M)
        c32 = cospi((double)(32 * odd % per) / (2.0 * M));
        t = cospi((double)(lane * odd % per) / (2.0 * M));
    } else {
        const double th = acos(cos(M_PI * (k + 0.5) / M));
        c32 = cos(32.0 * th);
        t = cos(lane * th);
    }
    // T at n - 32 for n = lane: cos((32 - lane) theta)
    double tm = __shfl_sync(0xffffffffu, t, (32 - lane) & 31);
    if (lane == 0) tm = c32;
    const double c2 = 2.0 * c32;
    double acc = 0.0;
    int n = lane;
    for (; n + 96 < N; n += 128) {
        double v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] = __ldg(c + n + 32 * u);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            acc = fma(v[u], t, acc);
            const double nx = fma(c2, t, -tm);
            tm = t;
            t = nx;
        }
    }
    for (; n < N; n += 32) {
        acc = fma(__ldg(c + n), t, acc);
        const double nx = fma(c2, t, -tm);
        tm = t;
        t = nx;
    }
    // sums over even n in the even lanes, over odd n in the odd ones
    for (int o = 16; o > 1; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    const double other = __shfl_xor_sync(0xffffffffu, acc, 1);
    const int64_t kk = EXACT && lane ? M - 1 - k : k;
    if (lane > (EXACT ? 1 : 0) || (lane == 1 && kk == k)) return;
    const double th = M_PI * (kk + 0.5) / M;
    const double sum = lane ? other - acc : acc + other;
    const int64_t o = M - 1 - kk;
    omega[o] = a * cos(th) + b;
    inten[o] = sum / (M_PI * sin(th)) / a;
}

void spectrum_dev(const double* moments, int N, double a, double b, int M, int kernel,
                  double* damped, double* omega, double* intensity, cudaStream_t st,
                  double lambda) {
    k_damp<<<(N + 127) / 128, 128, 0, st>>>(moments, N, kernel, lambda, damped);
    KPM_LAUNCHED();
    if ((int64_t)N * M > REC_EXACT) {
        k_reconstruct<false><<<(unsigned)((M + REC_WARPS - 1) / REC_WARPS), 32 * REC_WARPS, 0, st>>>(
            damped, N, a, b, M, omega, intensity);
        KPM_LAUNCHED();
        return;
    }
    if (N > M) {
        k_fold<<<(M + 127) / 128, 128, 0, st>>>(damped, N, M);
        KPM_LAUNCHED();
    }
    const int pairs = M / 2 + (M & 1);
    k_reconstruct<true><<<(unsigned)((pairs + REC_WARPS - 1) / REC_WARPS), 32 * REC_WARPS, 0, st>>>(
        damped, N < M ? N : M, a, b, M, omega, intensity);
    KPM_LAUNCHED();
}

}  // namespace kpm
