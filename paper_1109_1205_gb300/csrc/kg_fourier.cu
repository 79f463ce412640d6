// kg_fourier.cu -- the frequency-dependent Green's function from the
// time-dependent one (Section 3: G(omega) by Fourier transformation of G(t),
// the Lorentzian broadening eta entering as the damping e^{-eta t} that makes
// the time integral converge at t_max).  For samples t_k = k dt, k < n_t:
//
//   G(omega_j) = sum_k w_k e^{i (omega_j + i eta) t_k} G(t_k),
//   w_0 = w_{n_t-1} = dt/2, w_k = dt otherwise,
//
// the trapezoidal rule for the integral over [0, (n_t - 1) dt]; zero for one
// sample.  Transforming the particle part G^>(t) gives the particle part of
// Eq. (gomega), transforming -G^<(t) the hole part.
//
// Two evaluations on the caller's frequency grid, chosen by their FP64 work.
//
// Direct (short series, few frequencies or a wide range of them): one
// thread per frequency, the samples of one series staged in shared memory
// (every thread reads the same sample: a broadcast), and within each chunk of
// kFtChunk samples a Horner recurrence in z = e^{i (omega + i eta) dt},
//   S = g_0 + z (g_1 + z (g_2 + ...)),
// four FP64 FMAs per sample and frequency.  Each chunk is rotated into place
// by e^{i (omega + i eta) t_c}, computed from sincos/exp at the chunk start,
// so rounding does not build up over long series.  Long series are split
// over blockIdx.z to fill the GPU; a second kernel sums the splits in a fixed
// order (deterministic).
//
// Through nodes (long series): a run of B samples centred at t_c contributes
// e^{i omega t_c} F_c(omega), F_c(omega) = sum_q g_q e^{i omega (t_q - t_c)},
// and F_c has only frequencies up to B dt / 2 as a function of omega: on a
// window of omega of width D it is a polynomial of degree K - 1 through its
// values at K Chebyshev nodes up to 2 (D B dt / 8)^K / K!, below 2e-17 of
// sum |g_q| for K = 24 and D B dt <= 15.2.  So the sums are taken at the nodes
// only (168 of them instead of 4,001 frequencies on the paper's grid with
// B = 512), two real multiply-adds per sample, node and part, the cosines and
// sines being the same for every run (k_ft_nodes); then every frequency
// interpolates (24 real factors, the Lagrange polynomials of the window,
// k_ft_weights) and rotates each run into place (k_ft_eval).  The rotation is
// anchored on sincos every kFtGroup runs.  Two series of 100,001 samples onto
// 4,001 frequencies take 3.2e9 multiply-adds directly, 6.0 ms with the FP64
// pipe 97% busy, and 1.6e8 this way, 0.44 ms with the copy of the series
// (6.28 -> 0.63 ms for the call); the error against a plain sum stays 2e-14.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "kg_internal.h"

namespace kg {

constexpr int kFtThreads = 128;  // frequencies per block, one per thread
constexpr int kFtTile = 512;     // samples staged in shared memory per pass
constexpr int kFtChunk = 128;    // samples per Horner chunk (one rotation each)
constexpr int kFtMaxSeries = 65535;
constexpr long long kFtMaxSamples = 1ll << 30;

__global__ void __launch_bounds__(kFtThreads) k_fourier(const double2* __restrict__ Gt, int n_t, double dt,
                                                        const double* __restrict__ omega, int n_omega, double eta,
                                                        int tiles_per_split, double2* __restrict__ out) {
    __shared__ double2 g[kFtTile];
    const int j = blockIdx.x * kFtThreads + threadIdx.x;
    const int series = blockIdx.y, split = blockIdx.z;
    const double2* G = Gt + (size_t)series * n_t;
    const double w = j < n_omega ? omega[j] : 0.0;
    double s1, c1;
    sincos(w * dt, &s1, &c1);
    const double r1 = exp(-eta * dt);
    const double zr = r1 * c1, zi = r1 * s1;
    double ar = 0.0, ai = 0.0;
    const int k_begin = split * tiles_per_split * kFtTile;
    const long long k_lim = (long long)k_begin + (long long)tiles_per_split * kFtTile;
    const int k_end = k_lim < n_t ? (int)k_lim : n_t;
    for (int k0 = k_begin; k0 < k_end; k0 += kFtTile) {
        const int len = k_end - k0 < kFtTile ? k_end - k0 : kFtTile;
        __syncthreads();  // the previous tile is consumed
        for (int q = threadIdx.x; q < len; q += kFtThreads) {
            const int k = k0 + q;
            const double wk = (k == 0 || k == n_t - 1) ? 0.5 * dt : dt;
            const double2 v = G[k];
            g[q] = make_double2(wk * v.x, wk * v.y);
        }
        __syncthreads();
        for (int c0 = 0; c0 < len; c0 += kFtChunk) {
            const int cl = len - c0 < kFtChunk ? len - c0 : kFtChunk;
            double sr = 0.0, si = 0.0;
            if (cl == kFtChunk) {
#pragma unroll 16
                for (int q = kFtChunk - 1; q >= 0; --q) {
                    const double2 v = g[c0 + q];
                    const double nr = fma(zr, sr, fma(-zi, si, v.x));
                    const double ni = fma(zr, si, fma(zi, sr, v.y));
                    sr = nr;
                    si = ni;
                }
            } else {
                for (int q = cl - 1; q >= 0; --q) {
                    const double2 v = g[c0 + q];
                    const double nr = fma(zr, sr, fma(-zi, si, v.x));
                    const double ni = fma(zr, si, fma(zi, sr, v.y));
                    sr = nr;
                    si = ni;
                }
            }
            // rotate the chunk to its start time t_c
            const double tc = (double)(k0 + c0) * dt;
            double sa, ca;
            sincos(w * tc, &sa, &ca);
            const double ra = exp(-eta * tc);
            const double pr = ra * ca, pi = ra * sa;
            ar = fma(pr, sr, fma(-pi, si, ar));
            ai = fma(pr, si, fma(pi, sr, ai));
        }
    }
    if (j < n_omega) out[((size_t)split * gridDim.y + series) * n_omega + j] = make_double2(ar, ai);
}

// out[i] = sum over the n_split partial planes of part[s][i], in split order.
__global__ void __launch_bounds__(kThreads) k_fourier_sum(const double2* __restrict__ part, int n_split,
                                                          long long plane, double2* __restrict__ out) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < plane;
         i += (long long)gridDim.x * blockDim.x) {
        double r = 0.0, im = 0.0;
        for (int s = 0; s < n_split; ++s) {
            const double2 v = part[(size_t)s * plane + i];
            r += v.x;
            im += v.y;
        }
        out[i] = make_double2(r, im);
    }
}

// ------------------------------------------------------ through nodes
constexpr int kFtK = 24;            // Chebyshev nodes per window
constexpr double kFtPhase = 15.2;   // largest window width times run length
constexpr int kFtRuns = 4;          // runs per block of k_ft_nodes
constexpr int kFtPairs = 64;        // sample pairs staged at a time
constexpr int kFtGroup = 16;        // runs per anchor of the rotation
constexpr int kFtNodeThreads = 64;

// The plan: runs of B samples, W windows of width D from omega0.
struct FtPlan {
    int B = 0, W = 0, runs = 0, groups = 0;
    double omega0 = 0.0, D = 0.0, cost = 0.0;
};

__device__ __forceinline__ double ft_node(int m) { return cospi((2 * m + 1) * (0.5 / kFtK)); }

// Per frequency: its window, the K Lagrange factors at it (barycentric form on
// Chebyshev nodes of the first kind) and the rotation from run to run.
__global__ void __launch_bounds__(kFtThreads) k_ft_weights(const double* __restrict__ omega, int n_omega, FtPlan P,
                                                           double dt, int* __restrict__ window, double* __restrict__ L,
                                                           double2* __restrict__ turn) {
    __shared__ double xn[kFtK], wn[kFtK];
    if (threadIdx.x < kFtK) {
        xn[threadIdx.x] = ft_node(threadIdx.x);
        const double v = sinpi((2 * threadIdx.x + 1) * (0.5 / kFtK));
        wn[threadIdx.x] = threadIdx.x & 1 ? -v : v;
    }
    __syncthreads();
    const int j = blockIdx.x * kFtThreads + threadIdx.x;
    if (j >= n_omega) return;
    const double w = omega[j];
    const int win = max(0, min(P.W - 1, (int)((w - P.omega0) / P.D)));
    const double x = (w - (P.omega0 + (win + 0.5) * P.D)) * (2.0 / P.D);
    double t[kFtK], s = 0.0;
    int at = -1;
#pragma unroll
    for (int m = 0; m < kFtK; ++m) {
        const double d = x - xn[m];
        if (d == 0.0) at = m;
        t[m] = wn[m] / d;
        s += t[m];
    }
    const double r = 1.0 / s;
#pragma unroll
    for (int m = 0; m < kFtK; ++m) L[(size_t)m * n_omega + j] = at >= 0 ? (m == at ? 1.0 : 0.0) : t[m] * r;
    double sn, cn;
    sincos(w * (P.B * dt), &sn, &cn);
    turn[j] = make_double2(cn, sn);
    window[j] = win;
}

// cos and sin of nu_m tau_q (node m of all windows, tau_q = (q + 1/2) dt), and
// the damping from the run's start to the samples on both sides of its centre
// (at most 1, so that no sample overflows).
__global__ void __launch_bounds__(kFtThreads) k_ft_table(FtPlan P, double dt, double eta, double2* __restrict__ table,
                                                         double2* __restrict__ damp) {
    const int n = P.W * kFtK, half = P.B / 2;
    const int e = blockIdx.x * kFtThreads + threadIdx.x;
    if (e < half) {
        damp[e] = make_double2(exp(-eta * ((half + e) * dt)), exp(-eta * ((half - 1 - e) * dt)));
    }
    if (e >= n * half) return;
    const int q = e / n, m = e - q * n, win = m / kFtK;
    const double nu = P.omega0 + (win + 0.5) * P.D + 0.5 * P.D * ft_node(m - win * kFtK);
    double s, c;
    sincos(nu * ((q + 0.5) * dt), &s, &c);
    table[e] = make_double2(c, s);
}

// F[series][run][node] = sum over the run, damped, kFtRuns runs per block,
// one node per thread.  With a = g_+ + g_-, b = i (g_+ - g_-) of the samples at
// t_c +- tau_q: F = sum_q cos(nu tau_q) a_q + sin(nu tau_q) b_q.
__global__ void __launch_bounds__(kFtNodeThreads) k_ft_nodes(const double2* __restrict__ Gt, int n_t, double dt,
                                                             double eta, FtPlan P, const double2* __restrict__ table,
                                                             const double2* __restrict__ damp, double2* __restrict__ F) {
    __shared__ double2 sa[kFtRuns][kFtPairs], sb[kFtRuns][kFtPairs];
    const int nodes = P.W * kFtK, half = P.B / 2;
    const int m = blockIdx.x * kFtNodeThreads + threadIdx.x, c0 = blockIdx.y * kFtRuns, series = blockIdx.z;
    const double2* G = Gt + (size_t)series * n_t;
    double2 acc[kFtRuns];
#pragma unroll
    for (int r = 0; r < kFtRuns; ++r) acc[r] = make_double2(0.0, 0.0);
    for (int q0 = 0; q0 < half; q0 += kFtPairs) {
        __syncthreads();
        for (int e = threadIdx.x; e < kFtRuns * kFtPairs; e += kFtNodeThreads) {
            const int r = e / kFtPairs, q = e - r * kFtPairs;
            const long long mid = (long long)(c0 + r) * P.B + half, kp = mid + q0 + q, km = mid - 1 - q0 - q;
            const double2 dm = damp[q0 + q];
            double2 gp = make_double2(0.0, 0.0), gm = gp;
            if (kp < n_t) {
                const double w = (kp == n_t - 1 ? 0.5 * dt : dt) * dm.x;
                const double2 v = G[kp];
                gp = make_double2(w * v.x, w * v.y);
            }
            if (km < n_t) {
                const double w = (km == 0 || km == n_t - 1 ? 0.5 * dt : dt) * dm.y;
                const double2 v = G[km];
                gm = make_double2(w * v.x, w * v.y);
            }
            sa[r][q] = make_double2(gp.x + gm.x, gp.y + gm.y);
            sb[r][q] = make_double2(gm.y - gp.y, gp.x - gm.x);
        }
        __syncthreads();
        if (m < nodes) {
            const double2* T = table + (size_t)q0 * nodes + m;
#pragma unroll 8
            for (int q = 0; q < kFtPairs; ++q) {
                const double2 t = T[(size_t)q * nodes];
#pragma unroll
                for (int r = 0; r < kFtRuns; ++r) {
                    const double2 a = sa[r][q], b = sb[r][q];
                    acc[r].x = fma(t.x, a.x, fma(t.y, b.x, acc[r].x));
                    acc[r].y = fma(t.x, a.y, fma(t.y, b.y, acc[r].y));
                }
            }
        }
    }
    if (m < nodes)
#pragma unroll
        for (int r = 0; r < kFtRuns; ++r)
            if (c0 + r < P.runs) {
                const double d = exp(-eta * ((double)(c0 + r) * P.B * dt));
                F[((size_t)series * P.runs + c0 + r) * nodes + m] = make_double2(d * acc[r].x, d * acc[r].y);
            }
}

// out[group][series][j] = sum over the group's runs of e^{i omega_j t_c} F_c(omega_j).
__global__ void __launch_bounds__(kFtThreads) k_ft_eval(const double2* __restrict__ F, double dt,
                                                        const double* __restrict__ omega, int n_omega, FtPlan P,
                                                        const int* __restrict__ window, const double* __restrict__ L,
                                                        const double2* __restrict__ turn, double2* __restrict__ out) {
    const int j = blockIdx.x * kFtThreads + threadIdx.x, series = blockIdx.y, group = blockIdx.z;
    if (j >= n_omega) return;
    double l[kFtK];
#pragma unroll
    for (int m = 0; m < kFtK; ++m) l[m] = L[(size_t)m * n_omega + j];
    const int c0 = group * kFtGroup, c1 = min(P.runs, c0 + kFtGroup);
    double pr, pi;
    sincos(omega[j] * (((c0 + 0.5) * P.B - 0.5) * dt), &pi, &pr);
    const double2 z = turn[j];
    const double2* Fc = F + ((size_t)series * P.runs + c0) * (P.W * kFtK) + window[j] * kFtK;
    double ar = 0.0, ai = 0.0;
    for (int c = c0; c < c1; ++c, Fc += P.W * kFtK) {
        double fr = 0.0, fi = 0.0, gr = 0.0, gi = 0.0;
#pragma unroll
        for (int m = 0; m < kFtK; m += 2) {
            const double2 v = Fc[m], u = Fc[m + 1];
            fr = fma(l[m], v.x, fr);
            fi = fma(l[m], v.y, fi);
            gr = fma(l[m + 1], u.x, gr);
            gi = fma(l[m + 1], u.y, gi);
        }
        fr += gr;
        fi += gi;
        ar = fma(pr, fr, fma(-pi, fi, ar));
        ai = fma(pr, fi, fma(pi, fr, ai));
        const double t = pr;
        pr = fma(pr, z.x, -pi * z.y);
        pi = fma(t, z.y, pi * z.x);
    }
    out[((size_t)group * gridDim.y + series) * n_omega + j] = make_double2(ar, ai);
}

// The cheapest plan in FP64 multiply-adds, or B = 0 when the direct sum is
// (about 4.5 per sample and frequency with its rotations; the plan must halve
// it, for its launches and passes).  Runs whose damping spans more than e^40
// stay direct, like frequencies so far apart that the windows would multiply.
static FtPlan ft_plan(int n_series, int n_t, double dt, const double* omega, int n_omega, double eta) {
    double lo = omega[0], hi = omega[0];
    for (int j = 1; j < n_omega; ++j) {
        lo = std::min(lo, omega[j]);
        hi = std::max(hi, omega[j]);
    }
    FtPlan best;
    best.cost = 0.5 * 4.5 * n_series * (double)n_t * n_omega;
    for (int B = 2 * kFtPairs; B <= 4096; B *= 2) {
        const double T = B * dt, width = (hi - lo) * T / kFtPhase;
        if (!(width < 2048.0) || eta * T > 80.0) break;
        FtPlan P;
        P.B = B;
        P.W = std::max(1, (int)std::ceil(width));
        // a single window is as wide as it may be, around its frequencies: equal or
        // nearly equal ones would otherwise have nodes that FP64 cannot tell apart
        P.D = P.W > 1 ? (hi - lo) / P.W : kFtPhase / T;
        P.omega0 = P.W > 1 ? lo : 0.5 * lo + 0.5 * hi - 0.5 * P.D;
        // as when the frequencies are that large themselves
        if (P.D < 0x1p-40 * std::max(std::fabs(lo), std::fabs(hi))) break;
        P.runs = (int)((n_t + (long long)B - 1) / B);
        P.groups = (P.runs + kFtGroup - 1) / kFtGroup;
        const double nodes = (double)P.W * kFtK;
        // tables, and three more launches: about 10 us of the GPU's FP64 rate
        const double table = 60.0 * nodes * (B / 2) + 400.0 * n_omega + 4e6;
        P.cost = table + n_series * (2.0 * nodes * (double)P.runs * B + (double)P.runs * n_omega * (2 * kFtK + 8) +
                                     60.0 * P.groups * n_omega);
        if (P.groups <= 65535 && P.runs / kFtRuns < 65535 && P.cost < best.cost) best = P;
    }
    return best;
}

static int fourier_args(const double* G_t, int n_series, int n_t, double dt, const double* omega, int n_omega,
                        double eta, const double* G_w) {
    if (n_series < 0 || n_series > kFtMaxSeries || n_t < 1 || n_t > kFtMaxSamples || n_omega < 0 ||
        !(dt > 0.0) || !std::isfinite(dt) || !(eta >= 0.0) || !std::isfinite(eta)) {
        set_error("kg_green_fourier: need 0 <= n_series <= %d, 1 <= n_t <= 2^30, n_omega >= 0, finite dt > 0 and "
                  "finite eta >= 0", kFtMaxSeries);
        return KG_EINVAL;
    }
    if (n_series > 0 && n_omega > 0) {
        if (!G_t || !omega || !G_w) {
            set_error("kg_green_fourier: NULL buffer");
            return KG_EINVAL;
        }
        for (int j = 0; j < n_omega; ++j)
            if (!std::isfinite(omega[j])) {
                set_error("kg_green_fourier: omega[%d] is not finite", j);
                return KG_EINVAL;
            }
    }
    return KG_OK;
}

static int fourier_nodes(const double* G_t, int n_series, int n_t, double dt, const double* omega, int n_omega,
                         double eta, const FtPlan& P, cudaStream_t st, double* G_w) {
    const size_t plane = (size_t)n_series * n_omega, nodes = (size_t)P.W * kFtK;
    size_t at = 0;
    auto take = [&](size_t bytes) {
        const size_t a = at;
        at += (bytes + 255) & ~(size_t)255;
        return a;
    };
    const size_t o_gt = take(sizeof(double2) * (size_t)n_series * n_t), o_om = take(sizeof(double) * n_omega),
                 o_out = take(sizeof(double2) * plane), o_part = take(P.groups > 1 ? sizeof(double2) * plane * P.groups : 0),
                 o_win = take(sizeof(int) * n_omega), o_L = take(sizeof(double) * (size_t)kFtK * n_omega),
                 o_turn = take(sizeof(double2) * n_omega), o_tab = take(sizeof(double2) * nodes * (P.B / 2)),
                 o_damp = take(sizeof(double2) * (P.B / 2)), o_F = take(sizeof(double2) * nodes * P.runs * n_series);
    char* buf = nullptr;
    if (cudaMallocAsync((void**)&buf, at, st) != cudaSuccess) {
        cudaGetLastError();
        return KG_ENOMEM;
    }
    const double2* gt = reinterpret_cast<const double2*>(buf + o_gt);
    const double* om = reinterpret_cast<const double*>(buf + o_om);
    double2* out = reinterpret_cast<double2*>(buf + o_out);
    double2* part = P.groups > 1 ? reinterpret_cast<double2*>(buf + o_part) : out;
    int* win = reinterpret_cast<int*>(buf + o_win);
    double* L = reinterpret_cast<double*>(buf + o_L);
    double2* turn = reinterpret_cast<double2*>(buf + o_turn);
    double2* tab = reinterpret_cast<double2*>(buf + o_tab);
    double2* damp = reinterpret_cast<double2*>(buf + o_damp);
    double2* F = reinterpret_cast<double2*>(buf + o_F);
    int rc = KG_OK;
    // the tables need only the frequencies: they are made while the series is copied
    cudaError_t e = cudaMemcpyAsync(buf + o_om, omega, sizeof(double) * n_omega, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) {
        ProfScope ps("fourier", st);
        const int nbw = (n_omega + kFtThreads - 1) / kFtThreads;
        k_ft_weights<<<nbw, kFtThreads, 0, st>>>(om, n_omega, P, dt, win, L, turn);
        k_ft_table<<<(int)((nodes * (P.B / 2) + kFtThreads - 1) / kFtThreads), kFtThreads, 0, st>>>(P, dt, eta, tab, damp);
        e = cudaMemcpyAsync(buf + o_gt, G_t, sizeof(double2) * (size_t)n_series * n_t, cudaMemcpyHostToDevice, st);
        k_ft_nodes<<<dim3((unsigned)((nodes + kFtNodeThreads - 1) / kFtNodeThreads), (P.runs + kFtRuns - 1) / kFtRuns, n_series),
                     kFtNodeThreads, 0, st>>>(gt, n_t, dt, eta, P, tab, damp, F);
        k_ft_eval<<<dim3(nbw, n_series, P.groups), kFtThreads, 0, st>>>(F, dt, om, n_omega, P, win, L, turn, part);
        int launched = 4;
        if (P.groups > 1) {
            const int nb = (int)std::max<size_t>(1, std::min<size_t>((plane + kThreads - 1) / kThreads, 2048));
            k_fourier_sum<<<nb, kThreads, 0, st>>>(part, P.groups, (long long)plane, out);
            launched = 5;
        }
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e == cudaSuccess) count_launch(launched);
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(G_w, out, sizeof(double2) * plane, cudaMemcpyDeviceToHost, st);
    if (e != cudaSuccess) rc = cuda_fail(e, "kg_green_fourier", __FILE__, __LINE__);
    cudaFreeAsync(buf, st);
    e = cudaStreamSynchronize(st);
    if (rc == KG_OK && e != cudaSuccess) rc = cuda_fail(e, "kg_green_fourier", __FILE__, __LINE__);
    return rc;
}

static int green_fourier(const double* G_t, int n_series, int n_t, double dt, const double* omega, int n_omega,
                         double eta, cudaStream_t st, double* G_w) {
    KG_TRY(fourier_args(G_t, n_series, n_t, dt, omega, n_omega, eta, G_w));
    if (n_series == 0 || n_omega == 0) return KG_OK;
    const long long plane = (long long)n_series * n_omega;
    if (n_t == 1) {  // the integral over an empty interval
        std::memset(G_w, 0, sizeof(double2) * (size_t)plane);
        return KG_OK;
    }
    const FtPlan plan = ft_plan(n_series, n_t, dt, omega, n_omega, eta);
    if (plan.B) {
        const int rc = fourier_nodes(G_t, n_series, n_t, dt, omega, n_omega, eta, plan, st, G_w);
        if (rc != KG_ENOMEM) return rc;  // without room for the tables: the direct sum
    }
    int dev = 0, nsm = 148;
    KG_CUDA(cudaGetDevice(&dev));
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const int n_wtiles = (n_omega + kFtThreads - 1) / kFtThreads;
    const int n_tiles = (int)((n_t + kFtTile - 1) / kFtTile);
    const long long base = (long long)n_wtiles * n_series;
    // Split count: the resident blocks of an SM share its FP64 pipe, so an
    // SM's time is the number of tiles its blocks hold, and the launch ends
    // with the busiest SM, ceil(blocks / nsm) blocks of tiles_per_split tiles
    // (plus a small per-block cost).  Take the split count that minimises
    // this, the fewest splits among equals, over at most a few waves, with at
    // least 4 blocks (16 warps) per SM where the series is long enough: the
    // Horner chains need that many warps to keep the FP64 pipe busy.
    int per_sm = 1;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fourier, kFtThreads, 0) != cudaSuccess ||
        per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
    }
    const long long max_split = std::max(1LL, std::min<long long>(n_tiles, 4LL * per_sm * nsm / base + 1));
    const long long min_split = std::min(max_split, (4LL * nsm + base - 1) / base);
    int n_split = 1, tiles_per_split = n_tiles;
    double best = -1.0;
    for (int pass = 0; pass < 2 && best < 0.0; ++pass)
        for (long long ns = pass == 0 ? min_split : 1; ns <= max_split; ++ns) {
            const int tps = (int)((n_tiles + ns - 1) / ns);
            if ((n_tiles + tps - 1) / tps != ns) continue;  // would leave a split empty
            const long long busiest = (base * ns + nsm - 1) / nsm;
            const double cost = (double)busiest * (tps + 0.05);
            if (best < 0.0 || cost < best) {
                best = cost;
                n_split = (int)ns;
                tiles_per_split = tps;
            }
        }

    // device copies: the series, the frequencies, the partial planes, the result
    const size_t b_gt = sizeof(double2) * (size_t)n_series * n_t;
    const size_t b_om = (sizeof(double) * (size_t)n_omega + 255) & ~(size_t)255;
    const size_t b_out = sizeof(double2) * (size_t)plane;
    const size_t b_part = n_split > 1 ? b_out * n_split : 0;
    const size_t o_om = (b_gt + 255) & ~(size_t)255, o_out = o_om + b_om, o_part = o_out + ((b_out + 255) & ~(size_t)255);
    char* buf = nullptr;
    if (cudaMallocAsync((void**)&buf, o_part + b_part, st) != cudaSuccess) {
        cudaGetLastError();
        set_error("kg_green_fourier: cannot allocate %zu bytes on the device", o_part + b_part);
        return KG_ENOMEM;
    }
    const double2* d_gt = reinterpret_cast<const double2*>(buf);
    const double* d_om = reinterpret_cast<const double*>(buf + o_om);
    double2* d_out = reinterpret_cast<double2*>(buf + o_out);
    double2* d_part = n_split > 1 ? reinterpret_cast<double2*>(buf + o_part) : d_out;
    int rc = KG_OK;
    cudaError_t e = cudaMemcpyAsync(buf, G_t, b_gt, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(buf + o_om, omega, sizeof(double) * n_omega, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) rc = cuda_fail(e, "kg_green_fourier: copy in", __FILE__, __LINE__);
    if (rc == KG_OK) {
        ProfScope ps("fourier", st);
        k_fourier<<<dim3(n_wtiles, n_series, n_split), kFtThreads, 0, st>>>(d_gt, n_t, dt, d_om, n_omega, eta,
                                                                           tiles_per_split, d_part);
        int launched = 1;
        if (n_split > 1) {
            const int nb = (int)std::max(1LL, std::min<long long>((plane + kThreads - 1) / kThreads, 4LL * nsm));
            k_fourier_sum<<<nb, kThreads, 0, st>>>(d_part, n_split, plane, d_out);
            launched = 2;
        }
        e = cudaGetLastError();
        if (e != cudaSuccess) rc = cuda_fail(e, "kernel launch", __FILE__, __LINE__);
        else count_launch(launched);
    }
    if (rc == KG_OK) {
        e = cudaMemcpyAsync(G_w, d_out, b_out, cudaMemcpyDeviceToHost, st);
        if (e != cudaSuccess) rc = cuda_fail(e, "kg_green_fourier: copy out", __FILE__, __LINE__);
    }
    cudaFreeAsync(buf, st);
    e = cudaStreamSynchronize(st);
    if (rc == KG_OK && e != cudaSuccess) rc = cuda_fail(e, "kg_green_fourier", __FILE__, __LINE__);
    return rc;
}

}  // namespace kg

extern "C" int kg_green_fourier(const double* G_t, int n_series, int n_t, double dt, const double* omega,
                                int n_omega, double eta, void* stream, double* G_w) {
    return kg::green_fourier(G_t, n_series, n_t, dt, omega, n_omega, eta, (cudaStream_t)stream, G_w);
}
