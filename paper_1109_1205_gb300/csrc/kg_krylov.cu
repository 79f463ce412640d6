// kg_krylov.cu -- the Lanczos recursion with full
// reorthogonalisation, the small tridiagonal eigenproblem and exponential,
// and the basis combination (Section 2, Eqs. (recursion), (tmatrix),
// (tdiag), (eigen); Section 3, Eqs. (newstate) and (udelta)).
//
// Every kernel works on a batch of B independent columns, possibly of
// different sectors and dimensions (many instances, or many columns of one
// Green's-function calculation).  A launch walks a work list of (column,
// block, blocks-of-that-column) items, so one launch per phase serves the
// whole batch.  Lanczos vectors are stored unnormalised, V_k, with v_k = s_k
// V_k and s_k = 1/||V_k|| kept on the device, so normalisation never costs a
// separate pass.  Scalars (a_k, b_k, Gram-Schmidt and combination
// coefficients) never leave the device: a whole propagation step is a fixed
// launch sequence that a CUDA graph can replay.
#include <algorithm>
#include <array>
#include <utility>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>

#include "kg_internal.h"
#include "kg_stages.h"

namespace kg {

// ------------------------------------------------------------ workspace
size_t krylov_bytes(const std::vector<const kg_sector*>& cols, int M, bool planes, int schedule) {
    size_t nv = 0, nw = 0;
    for (auto* s : cols) {
        nv += (size_t)(M + 1) * (size_t)s->d;
        nw += (size_t)s->d;
    }
    // basis, W and U, fixed-point image; partial sums (at most 16 blocks per
    // SM of 72 doubles per column), work lists and descriptors
    size_t b = nv * sizeof(double2) + 3 * nw * sizeof(double2) + (cols.size() + 2) * (size_t(2) << 20);
    if (planes) b += nv * (sizeof(double) + sizeof(float2) + ((schedule & 4) ? 0 : sizeof(int4)));
    return b;
}

int krylov_alloc(Krylov& K, const std::vector<const kg_sector*>& cols, int M, int nsm, int schedule, bool planes) {
    K = Krylov();
    K.schedule = schedule;
    const bool int_hops = !(schedule & 1);
    K.B = (int)cols.size();
    K.M = M;
    K.nsm = nsm;
    if (K.B < 1) {
        set_error("empty Krylov batch");
        return KG_EINVAL;
    }
    size_t nv = 0, nw = 0, np = 0, nx = 0;
    for (auto* s : cols) K.total_d += s->d;
    K.hdesc.resize(K.B);
    K.hsec.resize(K.B);
    for (int b = 0; b < K.B; ++b) {
        const kg_sector* s = cols[b];
        ColDesc& D = K.hdesc[b];
        std::memset(&D, 0, sizeof D);
        D.d = (int)s->d;
        D.M = M;
        K.hsec[b] = s->view();
        const SecView& S = K.hsec[b];
        D.mode = S.hopmode == 0 ? ((int_hops && S.fix_pre >= 0) ? 3 : 0) : S.hopmode;
        D.Du = S.Du;
        D.Dd = S.Dd;
        D.fix_pre = S.fix_pre;
        if (D.mode == 3) nx += (size_t)D.d;
        nv += (size_t)(M + 1) * D.d;
        nw += (size_t)D.d;
    }
    // H*psi groups: consecutive columns of one mode while their inputs fit
    // kHpsiGroupBytes; then partial-sum rows for a one-wave list (<= 8 blocks
    // per SM) of any kernel at up to twice the wave, shared in proportion to
    // d over the batch or over the column's group, whichever is larger
    K.group.assign(K.B, 0);
    std::vector<long long> gbytes, gd;
    std::vector<int> slot(K.B);  // global group slot of each column
    {
        // balanced: as few groups as the budget allows, filled to the mean
        long long mbytes[4] = {0, 0, 0, 0};
        for (auto& D : K.hdesc) mbytes[D.mode] += 16LL * D.d;
        long long target[4];
        for (int m = 0; m < 4; ++m) {
            const long long ng = std::max(1LL, (mbytes[m] + kHpsiGroupBytes - 1) / kHpsiGroupBytes);
            target[m] = (mbytes[m] + ng - 1) / ng;
        }
        int cur[4] = {-1, -1, -1, -1};
        for (int b = 0; b < K.B; ++b) {
            ColDesc& D = K.hdesc[b];
            const long long bytes = 16LL * D.d;
            if (cur[D.mode] < 0 || gbytes[cur[D.mode]] + bytes > target[D.mode]) {
                cur[D.mode] = (int)gbytes.size();
                gbytes.push_back(0);
                gd.push_back(0);
                K.group[b] = K.ngroups[D.mode]++;
            } else {
                K.group[b] = K.ngroups[D.mode] - 1;
            }
            gbytes[cur[D.mode]] += bytes;
            gd[cur[D.mode]] += D.d;
            slot[b] = cur[D.mode];
        }
    }
    {
        std::vector<int> cl;
        small_plan(cols, M, schedule, cl);
        for (int b = 0; b < K.B; ++b) K.hdesc[b].small = cl[b];
    }
    np = 0;
    for (int b = 0; b < K.B; ++b) {
        ColDesc& D = K.hdesc[b];
        const double share = std::max((double)D.d / (double)K.total_d, (double)D.d / (double)gd[slot[b]]);
        const long long want = (long long)std::ceil(16.0 * nsm * share) + 2;
        D.nblk_max = (int)std::max(1LL, std::min(want, (long long)(D.d + kThreads - 1) / kThreads));
        np += (size_t)D.nblk_max * kPart;
    }
    // on any failure the workspace is released whole (krylov_free skips null)
    auto need = [&](cudaError_t e, const char* what) -> int {
        if (e == cudaSuccess) return KG_OK;
        cudaGetLastError();
        krylov_free(K);
        set_error("Krylov workspace: %s failed (%s)", what, cudaGetErrorString(e));
        return e == cudaErrorMemoryAllocation ? KG_ENOMEM : KG_ECUDA;
    };
    KG_TRY(need(cudaMalloc(&K.Vbuf, sizeof(double2) * nv), "basis allocation"));
    // Planes read by the Gram-Schmidt kernels (Re+Im for the three-multiply
    // dot products, a truncated FP32 copy for the small correction terms).
    // They are optional: without the memory the kernels use V alone.
    if (!planes || cudaMalloc(&K.Sbuf, sizeof(double) * nv) != cudaSuccess ||
        cudaMalloc(&K.V32buf, sizeof(float2) * nv) != cudaSuccess) {
        cudaGetLastError();
        cudaFree(K.Sbuf);
        cudaFree(K.V32buf);
        K.Sbuf = nullptr;
        K.V32buf = nullptr;
    }
    // fixed-point images for the exact integer Gram-Schmidt dots (schedule
    // bit 2 clear), optional like the planes
    if (K.Sbuf && !(schedule & 4) && cudaMalloc(&K.Ibuf, sizeof(int4) * nv) != cudaSuccess) {
        cudaGetLastError();
        K.Ibuf = nullptr;
    }
    // U = W - a_j v_j overwrites W, except for the FP64 dots, whose thread
    // groups each read W
    const bool inplace = K.Ibuf != nullptr;
    KG_TRY(need(cudaMalloc(&K.Wbuf, sizeof(double2) * (inplace ? 1 : 2) * nw), "work vector allocation"));
    if (nx) KG_TRY(need(cudaMalloc(&K.Xfbuf, sizeof(longlong2) * nx), "fixed-point image allocation"));
    KG_TRY(need(cudaMalloc(&K.partbuf, sizeof(double) * np), "partial-sum allocation"));
    KG_TRY(need(cudaMalloc(&K.pairbuf, sizeof(Partial) * 2 * (np / kPart)), "partial-sum allocation"));
    KG_TRY(need(cudaMalloc(&K.gaccbuf, sizeof(unsigned long long) * 8 * (size_t)K.B * (M + 1)), "dot allocation"));
    KG_TRY(need(cudaMalloc(&K.desc, sizeof(ColDesc) * K.B), "descriptor allocation"));
    KG_TRY(need(cudaMalloc(&K.secs, sizeof(SecView) * K.B), "sector view allocation"));
    KG_TRY(need(cudaMalloc(&K.cs, sizeof(ColScalars) * K.B), "scalar allocation"));
    KG_TRY(need(cudaMalloc(&K.cnt, sizeof(unsigned) * K.B), "ticket allocation"));
    KG_TRY(need(cudaMalloc(&K.Q, sizeof(double) * (size_t)K.B * M * M), "eigenvector allocation"));
    KG_TRY(need(cudaMemset(K.cs, 0, sizeof(ColScalars) * K.B), "scalar reset"));
    KG_TRY(need(cudaMemset(K.cnt, 0, sizeof(unsigned) * K.B), "ticket reset"));
    size_t ov = 0, ow = 0, op = 0, ox = 0;
    for (int b = 0; b < K.B; ++b) {
        ColDesc& D = K.hdesc[b];
        D.sec = K.secs + b;
        D.V = K.Vbuf + ov;
        D.S = K.Sbuf ? K.Sbuf + ov : nullptr;
        D.V32 = K.V32buf ? K.V32buf + ov : nullptr;
        D.I = K.Ibuf ? K.Ibuf + ov : nullptr;
        if (D.mode == 3) {
            D.Xf = K.Xfbuf + ox;
            ox += (size_t)D.d;
        }
        D.W = K.Wbuf + ow;
        D.U = inplace ? D.W : K.Wbuf + nw + ow;
        D.part = K.partbuf + op;
        D.part_a = K.pairbuf + 2 * (op / kPart);
        D.part_n = D.part_a + D.nblk_max;
        D.gacc = K.gaccbuf + 8 * (size_t)b * (M + 1);
        D.out = D.V;
        ov += (size_t)(M + 1) * D.d;
        ow += (size_t)D.d;
        op += (size_t)D.nblk_max * kPart;
    }
    {
        const int rc = small_alloc(K, cols);
        if (rc != KG_OK) {
            krylov_free(K);
            return rc;
        }
    }
    KG_TRY(need(cudaMemcpy(K.secs, K.hsec.data(), sizeof(SecView) * K.B, cudaMemcpyHostToDevice), "upload"));
    KG_TRY(need(cudaMemcpy(K.desc, K.hdesc.data(), sizeof(ColDesc) * K.B, cudaMemcpyHostToDevice), "upload"));
    KG_TRY(need(uploads_done(), "upload"));
    return KG_OK;
}

int krylov_upload(Krylov& K, cudaStream_t st) {
    KG_CUDA(cudaMemcpyAsync(K.desc, K.hdesc.data(), sizeof(ColDesc) * K.B, cudaMemcpyHostToDevice, st));
    return KG_OK;
}

int krylov_set_diag(Krylov& K, const double* diag) {
    for (auto& S : K.hsec) S.diag = diag;
    KG_CUDA(cudaMemcpy(K.secs, K.hsec.data(), sizeof(SecView) * K.B, cudaMemcpyHostToDevice));
    KG_CUDA(uploads_done());
    return KG_OK;
}

void krylov_free(Krylov& K) {
    small_free(K);
    for (auto& kv : K.lists) cudaFree(kv.second.first);
    cudaFree(K.Vbuf);
    cudaFree(K.Sbuf);
    cudaFree(K.V32buf);
    cudaFree(K.Ibuf);
    cudaFree(K.Xfbuf);
    cudaFree(K.Wbuf);
    cudaFree(K.partbuf);
    cudaFree(K.pairbuf);
    cudaFree(K.gaccbuf);
    cudaFree(K.desc);
    cudaFree(K.secs);
    cudaFree(K.cs);
    cudaFree(K.cnt);
    cudaFree(K.Q);
    K = Krylov();
}

static int occupancy(const void* kern, int threads, size_t smem) {
    static std::mutex mu;
    static std::map<std::pair<const void*, size_t>, int> occ;
    std::lock_guard<std::mutex> lk(mu);
    auto it = occ.find({kern, smem});
    if (it != occ.end()) return it->second;
    int bps = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kern, threads, smem) != cudaSuccess || bps < 1) bps = 1;
    occ[{kern, smem}] = bps;
    return bps;
}

// Work list of a kernel over the columns whose mode is `mode` (-1: all) and,
// with group >= 0, whose H*psi group is `group`: column b gets blocks in
// proportion to its dimension, one wave in total, with at least min_run
// elements per block (kThreads: the kernel keeps a partial-sum row per block).
int work_list(Krylov& K, const void* kern, int mode, const int4** items, int* n, int group, int threads, size_t smem,
              int min_run) {
    const int bps = occupancy(kern, threads, smem);
    const long long key = ((long long)bps << 8) + (mode + 1) + ((long long)std::lround(K.wave_scale * 64.0) << 20) +
                          ((long long)(group + 1) << 32) + ((long long)(min_run != kThreads) << 16);
    auto it = K.lists.find(key);
    if (it == K.lists.end()) {
        auto take = [&](const ColDesc& D, int b) {
            return (mode < 0 || D.mode == mode) && (group < 0 || K.group[b] == group);
        };
        long long dsel = 0;
        for (int b = 0; b < K.B; ++b)
            if (take(K.hdesc[b], b)) dsel += K.hdesc[b].d;
        const double total = std::max(1.0, K.wave_scale * K.nsm * bps);
        std::vector<int4> v;
        for (int b = 0; b < K.B; ++b) {
            const ColDesc& D = K.hdesc[b];
            if (!take(D, b)) continue;
            int nb = (int)std::lround(total * (double)D.d / (double)std::max(1LL, dsel));
            nb = std::max(1, std::min(nb, (D.d + min_run - 1) / min_run));
            if (min_run == kThreads) nb = std::min(nb, D.nblk_max);
            for (int k = 0; k < nb; ++k) v.push_back(make_int4(b, k, nb, 0));
        }
        int4* d = nullptr;
        if (!v.empty()) {
            KG_CUDA(cudaMalloc(&d, sizeof(int4) * v.size()));
            KG_CUDA(cudaMemcpy(d, v.data(), sizeof(int4) * v.size(), cudaMemcpyHostToDevice));
            KG_CUDA(uploads_done());
        }
        it = K.lists.emplace(key, std::make_pair(d, (int)v.size())).first;
    }
    *items = it->second.first;
    *n = it->second.second;
    return KG_OK;
}

// ------------------------------------------------- start-of-step norm
// beta0 = ||V_0||, s_0, the largest exponent of V_0, m_eff = M.
__global__ void __launch_bounds__(kThreads) k_colnorm(const ColDesc* desc, const int4* items, ColScalars* cs, int M,
                                                      unsigned* cnt) {
    __shared__ double sm[(kThreads / 32) * 2];
    __shared__ int smi[kThreads / 32];
    __shared__ double bs[2], red[2];
    KG_ITEM();
    chain_wait();
    const double2* x = D.V;
    double acc[1] = {0.0};
    int em = 0;
    KG_FOR(i) {
        const double2 v = x[i];
        acc[0] = fma(v.x, v.x, fma(v.y, v.y, acc[0]));
        em = max(em, max(exp_field(v.x), exp_field(v.y)));
        if (D.S) {
            D.S[i] = v.x + v.y;
            D.V32[i] = make_float2(f64_to_f32_trunc(v.x), f64_to_f32_trunc(v.y));
        }
    }
    em = block_max_int(em, smi);
    block_sum<1>(acc, 1, sm, bs);
    if (threadIdx.x == 0) bs[1] = (double)em;
    __syncthreads();
    if (grid_finish(bs, 1, D.part, cnt + b, blk, nblk, red, 1) && threadIdx.x == 0) {
        const double n = sqrt(red[0]);
        C->beta0 = n;
        C->beta[0] = 0.0;
        C->scale[0] = n > 0.0 ? 1.0 / n : 0.0;
        C->emax[0] = (int)red[1];
        C->eimg[0] = (int)red[1];  // I_0 is written by the first H*psi on this exponent
        C->m_eff = n > 0.0 ? M : 0;
        // the status is sticky over the steps of one call (reset by
        // launch_reset_status), so a non-finite column stays reported
        if (!isfinite(n)) {
            C->status = KG_ENUMERIC;
            C->m_eff = 0;
        }
    }
    if (blk == 0)  // totals of the exact dots of j = 0
        for (int q = threadIdx.x; q < 4 * (D.M + 1); q += blockDim.x) D.gacc[q] = 0ull;
}

int launch_colnorm(Krylov& K, cudaStream_t st) {
    ProfScope ps("colnorm", st);
    const int4* items;
    int n;
    KG_TRY(work_list(K, (const void*)k_colnorm, -1, &items, &n));
    return launch_chained(k_colnorm, n, kThreads, 0, st, K.desc, items, K.cs, K.M, K.cnt);
}

// ---------------------------------------- Gram-Schmidt coefficients
// First pass:  u = W - a_j v_j,  h_k = <v_k, u>   for k in [k0, k0+NK)
// Second pass: u = V_{j+1},      h_k = <v_k, u>
//
// With the plane S_k = Re V_k + Im V_k present, each complex product takes
// three FP64 multiply-adds instead of four (v = a + ib, u = c + id):
//   T1 = sum a c,  T2 = sum b d,  T3 = sum (a + b)(d - c),
//   Re <v,u> = T1 + T2,  Im <v,u> = T3 + T1 - T2,
// with d - c formed once per element and shared by all k.  The FP64 pipe
// bounds this kernel, so the extra 8 bytes per element of S cost less than
// the multiply-add they save.
//
// The accumulators live in registers.  For more than 12 vectors the two
// halves of the block take the two halves of the k range over the same
// elements (u is read twice, the second time from cache), which keeps the
// kernel at two blocks per SM without spilling.
template <int NK>
__global__ void __launch_bounds__(kThreads, 2) k_reorth_dots(const ColDesc* desc, const int4* items, ColScalars* cs,
                                                             int j, int k0, int nk, int second, unsigned* cnt) {
    constexpr int G = NK > 12 ? 2 : 1;         // thread groups splitting the k range
    constexpr int KH = (NK + G - 1) / G;       // vectors per group
    constexpr int TG = kThreads / G;           // threads per group
    __shared__ double sm[(kThreads / 32) * 3 * KH];
    __shared__ double bs[3 * NK], red[3 * NK];
    __shared__ HeadShared head;
    KG_ITEM();
    if (j >= C->m_eff) return;
    if (!second) resolve_alpha(D, C, j, blk == 0 && threadIdx.x == 0, head);
    const int d = D.d;
    const int grp = threadIdx.x / TG, t = threadIdx.x % TG;
    const int kb = grp * KH, kn = min(KH, NK - kb);
    const double2* Vb = D.V + (size_t)(k0 + kb) * d;
    const double2* w = second ? D.V + (size_t)(j + 1) * d : D.W;
    const double2* vj = D.V + (size_t)j * d;
    const double aj = second ? 0.0 : head.aj;
    double acc[3 * KH];
#pragma unroll
    for (int k = 0; k < 3 * KH; ++k) acc[k] = 0.0;
    const bool three = D.S != nullptr;
    // the last chunk of a first pass leaves u = W - a_j v_j in U for the update
    const bool keep = !second && k0 + NK == j + 1 && grp == 0;
    double2* wu = D.U;
    if (three) {
        const double* Sb = D.S + (size_t)(k0 + kb) * d;
        for (int i = blk * TG + t; i < d; i += nblk * TG) {
            double2 u = w[i];
            if (!second) {
                const double2 p = vj[i];
                u.x = fma(-aj, p.x, u.x);
                u.y = fma(-aj, p.y, u.y);
                if (keep) wu[i] = u;
            }
            const double dmc = u.y - u.x;
#pragma unroll
            for (int k = 0; k < KH; ++k) {
                if (k < kn) {
                    const size_t o = (size_t)k * d + i;
                    const double2 v = Vb[o];
                    const double sv = Sb[o];
                    acc[3 * k] = fma(v.x, u.x, acc[3 * k]);
                    acc[3 * k + 1] = fma(v.y, u.y, acc[3 * k + 1]);
                    acc[3 * k + 2] = fma(sv, dmc, acc[3 * k + 2]);
                }
            }
        }
    } else {
        for (int i = blk * TG + t; i < d; i += nblk * TG) {
            double2 u = w[i];
            if (!second) {
                const double2 p = vj[i];
                u.x = fma(-aj, p.x, u.x);
                u.y = fma(-aj, p.y, u.y);
            }
            if (keep) wu[i] = u;
#pragma unroll
            for (int k = 0; k < KH; ++k) {
                if (k < kn) {
                    const double2 v = Vb[(size_t)k * d + i];
                    acc[3 * k] = fma(v.x, u.x, fma(v.y, u.y, acc[3 * k]));
                    acc[3 * k + 1] = fma(v.x, u.y, fma(-v.y, u.x, acc[3 * k + 1]));
                }
            }
        }
    }
    // block sums: warps reduce their accumulators, then each group's warps
    // are added in warp order (fixed order, so results are reproducible)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 3 * KH; ++k) {
        const double v = warp_sum(acc[k]);
        if (lane == 0) sm[warp * 3 * KH + k] = v;
    }
    __syncthreads();
    constexpr int WG = TG / 32;  // warps per group
    for (int q = threadIdx.x; q < 3 * NK; q += blockDim.x) {
        const int g = q / (3 * KH), l = q - g * 3 * KH;
        double s = 0.0;
        for (int w2 = 0; w2 < WG; ++w2) s += sm[(g * WG + w2) * 3 * KH + l];
        bs[q] = s;
    }
    __syncthreads();
    if (grid_finish(bs, 3 * NK, D.part, cnt + b, blk, nblk, red)) {
        for (int k = threadIdx.x; k < NK; k += blockDim.x) {
            const double s = C->scale[k0 + k];
            const double t1 = red[3 * k], t2 = red[3 * k + 1], t3 = red[3 * k + 2];
            C->h[k0 + k] = three ? make_double2(s * (t1 + t2), s * (t3 + t1 - t2)) : make_double2(s * t1, s * t2);
        }
    }
}

// Exact-product Gram-Schmidt coefficients (first pass): h_k = s_k <V_k, u>
// with u = W - a_j v_j, from 52-bit fixed-point images.  Each V_k comes as
// its image I_k (written by the kernel that produced V_k, on the exponent
// bound eimg[k]); u is formed in FP64 here and converted on a bound E_u of
// its largest exponent.  With both numbers split into 26-bit halves, every
// partial product (hi*hi, hi*lo, lo*hi, lo*lo) is an exact 64-bit integer
// (one wide integer multiply-add), summed in three 64-bit accumulators (units
// 2^52, 2^26 and 1 of the full product).  Every further sum is an integer too:
// over a warp in 26-bit pieces (one warp-reduce instruction each), over the
// blocks by 64-bit atomic adds of two 46-bit limbs into gacc (in units of
// 2^26: the rest is dropped once per warp, below 2^-79 of the product of the
// two vectors' largest components).  Integer sums do not depend on the order, so the result is the
// same bits on every run without a last-block reduction, and the update that
// follows converts each total to FP64 once.  The FP64 pipe of this GPU issues
// about 2 multiply-adds per clock per SM, the integer pipe far more, so these
// dots are bounded by the 16 bytes of I_k per element and vector instead of
// the 3 FP64 multiply-adds per complex product of the Re+Im form.
//
// A block owns one run of elements and streams the NK images of it through a
// ring of shared-memory stages filled by bulk asynchronous copies (one per
// vector and tile; any run of 16-byte elements is a legal copy), so up to 90 KB
// per block are in flight without holding registers.  One warp only issues the
// copies.  The others meet once per kThreads elements, when every thread has
// formed its element of the next u and the image of it (W and V_j of it loaded
// one round ahead); within that round each warp walks the tiles on its own and
// reports a tile it is done with on the stage's second barrier, which the
// copying warp waits for before it refills the stage.  All waits are bounded;
// after one that ran out the computing warps wait no more, the copying warp
// issues no more copies and waits (bounded again) for those in flight
// (kg_stages.h), and the column's status says so.
//
// Measured on 12 columns of 731,808 states, mean over j < 20: 529 us per launch
// with per-thread loads, a barrier per tile and a last-block reduction; 382 us
// (5.0 TB/s of images) in this form.  On 300 states 20 -> 10 us.  Three or more
// vectors per warp leave too few warps to hide the multiply-adds' latency
// (491 us), a computing warp that also refills the stages holds up the others
// at the round's end (466 us).
//
// The update writes I_{j+1} on an exponent bounded before V_{j+1} exists.
// Near a breakdown (||V_{j+1}|| far below ||W||) that bound is loose and the
// image keeps too few of V_{j+1}'s own bits; a vector whose bound exceeds
// its true largest exponent by more than kFixSlack bits is therefore
// converted here from V_k on its exact exponent, the fresh image is stored
// back (each block its own elements) and its exponent updated by the update.
template <int NK>
struct IntDots {
    // Two vectors per warp: the accumulators stay at 24 registers per thread,
    // so that 16 to 28 warps per SM hide the latency of the multiply-adds; small
    // NK takes several warps per vector pair.
    static constexpr int KH = NK < 2 ? 1 : 2;           // vectors per group
    static constexpr int G = (NK + KH - 1) / KH;        // groups splitting k
    static constexpr int W = (8 + G - 1) / G;           // warps per group
    static constexpr int TG = 32 * W;                   // threads per group
    static constexpr int compute = TG * G;              // 256 to 448 threads per block
    static constexpr int threads = compute + 32;        // and the warp that issues the copies
    static constexpr int T = NK <= 6 ? 256 : (NK <= 12 ? 128 : 64);  // elements per tile
    static constexpr int kStage = NK * T * 16;
    static constexpr int kImage = 2 * kThreads * 24;  // two rounds of u's image
    static constexpr int fit = (104 * 1024 - kImage) / kStage;
    static constexpr int S = fit > 8 ? 8 : fit;  // stages; two blocks per SM
    static constexpr size_t smem = (size_t)S * kStage + kImage;
    static_assert(S >= 3, "at least three stages");
};

constexpr int kDotFlush = 256;   // elements a thread may add to its 64-bit sums
constexpr int kDotMinRun = 64;   // fewest elements worth a block

// The warp's total of s[0] 2^26 + s[1] + s[2] 2^-26 (|s[0]| < 2^62) as two
// limbs, total = l1 2^46 + l0.
__device__ __forceinline__ void warp_limbs(const long long (&s)[3], unsigned long long& l0, unsigned long long& l1) {
    constexpr long long m26 = (1ll << 26) - 1;
    const long long lo = s[1] + (s[2] >> 26), hi = s[0] + (lo >> 26);
    const unsigned s0 = __reduce_add_sync(0xffffffffu, (unsigned)(lo & m26));
    const unsigned s1 = __reduce_add_sync(0xffffffffu, (unsigned)(hi & m26));
    const unsigned s2 = __reduce_add_sync(0xffffffffu, (unsigned)((hi >> 26) & m26));
    const int s3 = __reduce_add_sync(0xffffffffu, (int)(hi >> 52));
    const unsigned long long a = (unsigned long long)s0 + ((unsigned long long)s1 << 26);   // < 2^58
    const long long b = (long long)s2 + ((long long)s3 << 26);                               // units of 2^52
    l0 = a & ((1ull << 46) - 1ull);
    l1 = (unsigned long long)((b << 6) + (long long)(a >> 46));
}

template <int NK>
__global__ void __launch_bounds__(IntDots<NK>::threads, 2) k_reorth_dots_int(const ColDesc* desc, const int4* items,
                                                                 ColScalars* cs, int j, int k0) {
    using P = IntDots<NK>;
    constexpr int KH = P::KH, TG = P::TG, T = P::T, S = P::S;
    extern __shared__ __align__(128) unsigned char dyn[];
    __shared__ __align__(8) unsigned long long full[S], empty[S];
    __shared__ HeadShared head;
    __shared__ int eu_s, any_s, fresh_s[NK], ek_s[NK];
    int4* const ua = reinterpret_cast<int4*>(dyn + S * P::kStage);  // [2][kThreads] image of u
    int2* const ub = reinterpret_cast<int2*>(dyn + S * P::kStage + 2 * kThreads * 16);
    KG_ITEM();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int q = 0; q < S; ++q) {
            mbar_init(full + q, 1);
            mbar_init(empty + q, P::compute / 32);
        }
        mbar_init_fence();
    }
    chain_wait();
    if (j >= C->m_eff) return;
    const int d = D.d;
    // this block's elements [e0, e0 + len), in tiles of T
    const int run = (int)(((long long)d + nblk - 1) / nblk);
    const size_t e0 = (size_t)min((long long)d, (long long)blk * run);
    const int len = (int)min((long long)run, (long long)d - (long long)e0);
    const int nt = (len + T - 1) / T, nr = (len + kThreads - 1) / kThreads;
    const int4* Ib = D.I + (size_t)k0 * d + e0;
    __syncthreads();  // the stages' barriers are ready
    const int lane = threadIdx.x & 31;
    const bool copies = threadIdx.x >= P::compute;
    auto issue = [&](int t) {  // by the copying warp: tile t into its stage
        const int q = t % S, n = min(T, len - t * T);
        if (lane == 0) mbar_expect(full + q, (unsigned)(NK * n * 16));
        __syncwarp();
        if (lane < NK)
            bulk_load(dyn + q * P::kStage + lane * T * 16, Ib + (size_t)lane * d + (size_t)t * T, (unsigned)(n * 16),
                      full + q);
    };
    if (copies)
        for (int t = 0; t < min(S, nt); ++t) issue(t);
    double2 wn = make_double2(0.0, 0.0), vn = wn;  // W and V_j of this thread's element of the next round
    const double2* wp = D.W + e0;
    const double2* vp = D.V + (size_t)j * d + e0;
    auto load_u = [&](int r) {
        const int e = r * kThreads + (int)threadIdx.x;
        if (threadIdx.x < kThreads && e < len) {
            wn = wp[e];
            vn = vp[e];
        }
    };
    if (nr > 0) load_u(0);
    const bool writer = blk == 0 && threadIdx.x == 0;
    resolve_alpha(D, C, j, writer, head);
    const double aj = head.aj;
    // the last chunk leaves u = W - a_j v_j in U (which may be W itself)
    const bool keep = k0 + NK == j + 1;
    if (threadIdx.x < NK) {
        ek_s[threadIdx.x] = C->emax[k0 + threadIdx.x];
        fresh_s[threadIdx.x] = C->eimg[k0 + threadIdx.x] - C->emax[k0 + threadIdx.x] > kFixSlack;
    }
    if (threadIdx.x < 32) {
        __syncwarp();
        const bool f = threadIdx.x < NK && fresh_s[threadIdx.x < NK ? threadIdx.x : 0];
        const unsigned any = __ballot_sync(0xffffffffu, f);
        if (threadIdx.x == 0) any_s = any != 0u;
    }
    if (threadIdx.x == 0) {
        // |u_i| <= |W_i| + |a_j| |V_j[i]| < (1 + |a_j| 2^(E_j - E_w)) 2^(E_w - 1022), with a margin
        const int ew = head.ew, ej = C->emax[j];
        const float r = (1.0f + scaled_abs(aj, ej - ew)) * (1.0f + 1.0f / 1024.0f);
        eu_s = r < 0x1p120f ? bound_exp(r, ew) : bound_exp((1.0 + fabs(aj) * ldexp(1.0, ej - ew)) * (1.0 + 1.0 / 1024.0), ew);
        if (writer) C->eu = eu_s;
    }
    __syncthreads();
    const int Eu = eu_s;
    const bool any_fresh = any_s != 0;
    const int grp = threadIdx.x / TG, tl = threadIdx.x % TG;
    const int kb = grp * KH, kn = min(KH, NK - kb);
    bool ok = true;
    if (copies) {
        // the warp's lanes agree on every wait
        auto landed = [&](int t) { return __all_sync(0xffffffffu, mbar_wait(full + t % S, (unsigned)((t / S) & 1))) != 0; };
        auto freed = [&](int t) { return __all_sync(0xffffffffu, mbar_wait(empty + t % S, (unsigned)((t / S) & 1))) != 0; };
        if (!feed_stages(nt, S, landed, freed, issue)) C->status = KG_ETIMEOUT;
        return;
    }
    double2* const up = D.U + e0;
    auto form_u = [&](int r) {
        const int e = r * kThreads + (int)threadIdx.x;
        if (threadIdx.x >= kThreads || e >= len) return;
        const double2 u = make_double2(fma(-aj, vn.x, wn.x), fma(-aj, vn.y, wn.y));
        if (keep) up[e] = u;
        const long long px = fix52(u.x, Eu), py = fix52(u.y, Eu);
        const int at = (r & 1) * kThreads + (int)threadIdx.x;
        ua[at] = make_int4(fix_hi(px), fix_lo(px), fix_hi(py), fix_lo(py));
        ub[at] = make_int2(fix_hi(-px), fix_lo(-px));
    };
    long long re[KH][3], im[KH][3];
#pragma unroll
    for (int k = 0; k < KH; ++k)
#pragma unroll
        for (int q = 0; q < 3; ++q) re[k][q] = im[k][q] = 0;
    int held = 0;  // elements in the sums
    unsigned long long* const acc = D.gacc + (size_t)(j & 1) * 4 * (D.M + 1) + 4 * (size_t)(k0 + kb);
    auto flush = [&]() {
        unsigned long long l0 = 0, l1 = 0;
#pragma unroll
        for (int k = 0; k < KH; ++k) {
            unsigned long long a0, a1;
            warp_limbs(re[k], a0, a1);
            if (lane == 2 * k) l0 = a0, l1 = a1;
            warp_limbs(im[k], a0, a1);
            if (lane == 2 * k + 1) l0 = a0, l1 = a1;
#pragma unroll
            for (int q = 0; q < 3; ++q) re[k][q] = im[k][q] = 0;
        }
        if (lane < 2 * kn) {
            atomicAdd(acc + 2 * lane, l0);
            atomicAdd(acc + 2 * lane + 1, l1);
        }
        held = 0;
    };
    if (nr > 0) form_u(0);
    block_bar(1, P::compute);
    int t = 0;
    for (int r = 0; r < nr; ++r) {
        if (r + 1 < nr) load_u(r + 1);
        const int tend = min(nt, (r + 1) * (kThreads / T));
        for (; t < tend; ++t) {
            ok = ok && mbar_wait(full + t % S, (unsigned)((t / S) & 1));
            int4* img = reinterpret_cast<int4*>(dyn + (t % S) * P::kStage) + kb * T;
            const int n = min(T, len - t * T), base = (r & 1) * kThreads + (t * T) % kThreads;
            if (any_fresh) {  // re-made images replace what was copied (each thread its own elements)
                for (int k = 0; k < kn; ++k)
                    for (int e = tl; fresh_s[kb + k] && e < n; e += TG) {
                        const size_t at = (size_t)(k0 + kb + k) * d + e0 + (size_t)t * T + e;
                        img[k * T + e] = D.I[at] = fix_image(D.V[at], ek_s[kb + k]);
                    }
                proxy_fence();  // ordinary stores to a stage that the next bulk copy fills again
            }
#pragma unroll 2
            for (int e = tl; e < n; e += TG) {
                const int4 u = ua[base + e];
                const int2 m = ub[base + e];
#pragma unroll
                for (int k = 0; k < KH; ++k)
                    if (k < kn) cdot_fix(img[k * T + e], u, m, re[k], im[k]);
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(empty + t % S);
        }
        held += (kThreads + TG - 1) / TG;
        if (held > kDotFlush - (kThreads + TG - 1) / TG) flush();
        if (r + 1 < nr) form_u(r + 1);
        block_bar(1, P::compute);
    }
    chain_next();
    flush();
    if (!ok) C->status = KG_ETIMEOUT;
}

// The accumulators of k_reorth_dots are compile-time sized and a kernel
// built for more vectors than a launch needs would still issue the FP64
// multiply-adds of the unused slots, so every count up to kChunk has its own
// instantiation (nk == NK in every launch).
using DotsKernel = void (*)(const ColDesc*, const int4*, ColScalars*, int, int, int, int, unsigned*);

template <int... N>
static constexpr std::array<DotsKernel, sizeof...(N)> dots_table(std::integer_sequence<int, N...>) {
    return {{&k_reorth_dots<N + 1>...}};
}

static DotsKernel dots_kernel(int nk) {
    static const std::array<DotsKernel, kChunk> exact = dots_table(std::make_integer_sequence<int, kChunk>{});
    return exact[nk - 1];
}

struct IntDotsKernel {
    void (*kern)(const ColDesc*, const int4*, ColScalars*, int, int);
    int threads;
    size_t smem;
};

template <int... N>
static std::array<IntDotsKernel, sizeof...(N)> int_dots_table(std::integer_sequence<int, N...>) {
    const std::array<IntDotsKernel, sizeof...(N)> t = {{{&k_reorth_dots_int<N + 1>, IntDots<N + 1>::threads, IntDots<N + 1>::smem}...}};
    for (auto& k : t)
        cudaFuncSetAttribute((const void*)k.kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k.smem);
    return t;
}

// Per device: the shared-memory attribute belongs to the device's context.
static IntDotsKernel int_dots_kernel(int nk) {
    static std::mutex mu;
    static std::map<int, std::array<IntDotsKernel, kChunk>> tables;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    auto it = tables.find(dev);
    if (it == tables.end()) it = tables.emplace(dev, int_dots_table(std::make_integer_sequence<int, kChunk>{})).first;
    return it->second[nk - 1];
}

// The exact integer dots serve first passes when every column has its images.
static bool use_int_dots(const Krylov& K, bool second) {
    if (second || (K.schedule & 4) || !K.Ibuf) return false;
    for (auto& D : K.hdesc)
        if (!D.I) return false;
    return true;
}

int launch_reorth_dots(Krylov& K, int j, int k0, int nk, bool second, cudaStream_t st) {
    ProfScope ps("reorth_dots", st);
    if (use_int_dots(K, second)) {
        const IntDotsKernel ik = int_dots_kernel(nk);
        const int4* items;
        int n;
        KG_TRY(work_list(K, (const void*)ik.kern, -1, &items, &n, -1, ik.threads, ik.smem, kDotMinRun));
        return launch_chained(ik.kern, n, ik.threads, ik.smem, st, K.desc, items, K.cs, j, k0);
    }
    const DotsKernel kern = dots_kernel(nk);
    const int4* items;
    int n;
    KG_TRY(work_list(K, (const void*)kern, -1, &items, &n));
    kern<<<n, kThreads, 0, st>>>(K.desc, items, K.cs, j, k0, nk, second ? 1 : 0, K.cnt);
    KG_LAUNCHED();
    return KG_OK;
}

// ------------------------------------------------------ the update
// First pass:  V_{j+1} = W - a_j v_j - [reorth] sum_{k<=j} h_k v_k
// Second pass: V_{j+1} -= sum_{k<=j} h_k v_k
// then b_{j+1} = ||V_{j+1}||, s_{j+1} = 1/b_{j+1}, a_j += Re h_j, the
// largest exponent of V_{j+1}, and the breakdown test (the Krylov space is
// invariant when b_{j+1} is at rounding level relative to |a_j| + b_j).
//
// After the three-term subtraction the Gram-Schmidt coefficients are at
// rounding level (|h_k| ~ 1e-14 for unit vectors).  A term whose coefficient
// is below kSmallCoef is accumulated in FP32 (FP32 FMA on the truncated
// vector): its error, < 2^-23 |h_k| |v_k[i]| < 1.2e-17 |v_k[i]|, is far
// below the FP64 rounding of the result, and the FP32 pipe is 64 times wider
// than the FP64 pipe on this GPU.  Larger coefficients use FP64.
// h_k = s_k <V_k, u> from the exact integer totals of the dots (units 2^26 of
// 2^(E_k - 1074) 2^(E_u - 1074), E_k the exponent of V_k's image; `keep`: also
// store E_k, which the dots changed if they re-made the image).
__device__ __forceinline__ double2 exact_dot(const ColDesc& D, ColScalars* C, int j, int k, bool keep) {
    const ulonglong2* t = reinterpret_cast<const ulonglong2*>(D.gacc + (size_t)(j & 1) * 4 * (D.M + 1) + 4 * (size_t)k);
    const int em = C->emax[k], ei = C->eimg[k], Ek = ei - em > kFixSlack ? em : ei;
    const double f = mul_pow2(C->scale[k], Ek + C->eu - 2122);
    auto val = [](ulonglong2 l) {
        const long long hi = (long long)l.y + (long long)(l.x >> 46);
        return fma((double)hi, 0x1p46, (double)(l.x & ((1ull << 46) - 1ull)));
    };
    if (keep) C->eimg[k] = Ek;
    return make_double2(f * val(t[0]), f * val(t[1]));
}

// Its first warp sorts the terms, one vector per lane: a serial pass by one
// thread costs two dependent L2 reads and a few FP64 operations per vector in
// every block.  With the sums reduced by the reader (resolve_norm) instead of
// by the last block to arrive, a Lanczos iteration on a 300-state column at
// M = 40 went from 53 to 38 us, on one 853,776-state column from 190 to 174 us.
__global__ void __launch_bounds__(kThreads) k_update(const ColDesc* desc, const int4* items, ColScalars* cs, int j,
                                                     int level, int second, int exact) {
    // block-uniform term lists: FP32 terms (small coefficients), FP64 terms
    __shared__ double2 coef64[kMaxMgs + 1];
    __shared__ float2 coef32[kMaxMgs + 1];
    __shared__ int idx32[kMaxMgs + 1], idx64[kMaxMgs + 1];
    __shared__ int n32, n64, efix_s;
    __shared__ double hre_s;
    __shared__ HeadShared head;
    KG_ITEM();
    chain_wait();
    if (j >= C->m_eff) return;
    const bool writer = blk == 0 && threadIdx.x == 0;
    const int d = D.d;
    double2* Vb = D.V;
    const int nk = (level >= 1 || second) ? j + 1 : 0;
    // a_j before the Gram-Schmidt correction: from the dots before a first
    // pass, else (no Gram-Schmidt) straight from the partial sums of H*psi
    int ew = 0;
    double araw = 0.0, aj = 0.0;
    if (second) {
        ew = C->emax[j + 1];
    } else if (nk) {
        araw = C->araw;
        ew = C->ew;
        if (threadIdx.x < 32) aj = araw * C->scale[j];  // the first warp's only (below)
    } else {
        resolve_alpha(D, C, j, writer, head);
        araw = head.araw;
        aj = head.aj;
        ew = head.ew;
    }
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        int a32 = 0, a64 = 0;
        // bound of the result's components, in units of 2^(ew - 1022) (below)
        float r = 0.0f;
        for (int k0 = 0; k0 < nk; k0 += 32) {
            const int k = k0 + lane;
            double2 h = make_double2(0.0, 0.0), c = h;
            int es = 0;
            if (k < nk) {
                const double s = C->scale[k];
                es = exp_field(s);
                h = exact ? exact_dot(D, C, j, k, blk == 0) : C->h[k];
                if (k == j) hre_s = h.x;
                c = make_double2(s * h.x, s * h.y);
                const int de = C->emax[k] - ew;
                r += scaled_abs(c.x, de) + scaled_abs(c.y, de);
            }
            // |h_k| for the unit vector v_k.  In FP64 where the FP32 copy of V_k leaves
            // FP32's range, or where c = s_k h_k or the sum could vanish (below
            // 2^-126) while they count beside w (above 2^-64 of its bound)
            const bool small = scaled_abs(h.x, 0) + scaled_abs(h.y, 0) < (float)kSmallCoef &&
                               (unsigned)(es - 963) <= 120u && es + ew >= 1983 && ew >= 960;
            const unsigned in = __ballot_sync(0xffffffffu, k < nk), ms = __ballot_sync(0xffffffffu, k < nk && small);
            const unsigned before = (1u << lane) - 1u;
            if (k < nk && small) {
                const int q = a32 + __popc(ms & before);
                coef32[q] = make_float2(f64_to_f32_near(c.x), f64_to_f32_near(c.y));
                idx32[q] = k;
            } else if (k < nk) {
                const int q = a64 + __popc(in & ~ms & before);
                coef64[q] = c;
                idx64[q] = k;
            }
            a32 += __popc(ms);
            a64 += __popc(in & ~ms);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
        __syncwarp();
        if (lane == 0) {
            n32 = a32;
            n64 = a64;
            // Every component of the result is below
            //   2^(E_u - 1022) + |a_j| 2^(E_j - 1022) + sum_k (|Re c_k| + |Im c_k|) 2^(E_k - 1022)
            // (E_u: largest exponent of W, or of V_{j+1} in a second pass),
            // times a margin for the rounding of the FP64 and FP32 arithmetic.
            r += 1.0f;
            if (!second) r += scaled_abs(aj, C->emax[j] - ew);
            r *= 1.0f + 1.0f / 1024.0f;
            if (r < 0x1p120f) {
                efix_s = bound_exp(r, ew);
            } else {  // coefficients out of FP32's range
                double rd = 1.0;
                if (!second) rd += fabs(aj) * ldexp(1.0, C->emax[j] - ew);
                for (int q = 0; q < a64; ++q)
                    rd += (fabs(coef64[q].x) + fabs(coef64[q].y)) * ldexp(1.0, C->emax[idx64[q]] - ew);
                for (int q = 0; q < a32; ++q)
                    rd += ((double)fabsf(coef32[q].x) + (double)fabsf(coef32[q].y)) * ldexp(1.0, C->emax[idx32[q]] - ew);
                efix_s = bound_exp(rd * (1.0 + 1.0 / 1024.0), ew);
            }
        }
    }
    __syncthreads();
    const int m32 = n32, m64 = n64;
    const double2* w = second ? Vb + (size_t)(j + 1) * d : D.W;
    const double2* vj = Vb + (size_t)j * d;
    double2* out = Vb + (size_t)(j + 1) * d;
    const float2* V32 = D.V32;
    double* S1 = D.S ? D.S + (size_t)(j + 1) * d : nullptr;
    float2* V32_1 = D.V32 ? D.V32 + (size_t)(j + 1) * d : nullptr;
    double acc = 0.0;
    int em = 0;
    // after a first-pass Gram-Schmidt (level >= 1) U holds W - a_j v_j
    const bool sub = !second && level < 1;
    const double2* win = (!second && level >= 1) ? D.U : w;
    auto element = [&](int i) {
        double2 u = win[i];
        if (sub) {
            const double2 p = vj[i];
            u.x = fma(-aj, p.x, u.x);
            u.y = fma(-aj, p.y, u.y);
        }
        float cx = 0.f, cy = 0.f;
        int q = 0;
        if (V32) {
            // eight loads in flight before their terms are applied
            for (; q + 8 <= m32; q += 8) {
                float2 v[8];
#pragma unroll
                for (int r = 0; r < 8; ++r) v[r] = V32[(size_t)idx32[q + r] * d + i];
#pragma unroll
                for (int r = 0; r < 8; ++r) {
                    const float2 c = coef32[q + r];
                    cx = fmaf(c.x, v[r].x, fmaf(-c.y, v[r].y, cx));
                    cy = fmaf(c.x, v[r].y, fmaf(c.y, v[r].x, cy));
                }
            }
            if (q + 4 <= m32) {
                float2 v[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) v[r] = V32[(size_t)idx32[q + r] * d + i];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const float2 c = coef32[q + r];
                    cx = fmaf(c.x, v[r].x, fmaf(-c.y, v[r].y, cx));
                    cy = fmaf(c.x, v[r].y, fmaf(c.y, v[r].x, cy));
                }
                q += 4;
            }
            for (; q < m32; ++q) {
                const float2 v = V32[(size_t)idx32[q] * d + i], c = coef32[q];
                cx = fmaf(c.x, v.x, fmaf(-c.y, v.y, cx));
                cy = fmaf(c.x, v.y, fmaf(c.y, v.x, cy));
            }
        } else {
            for (; q < m32; ++q) {
                const double2 v = Vb[(size_t)idx32[q] * d + i];
                const float2 c = coef32[q];
                const float vx = f64_to_f32_trunc(v.x), vy = f64_to_f32_trunc(v.y);
                cx = fmaf(c.x, vx, fmaf(-c.y, vy, cx));
                cy = fmaf(c.x, vy, fmaf(c.y, vx, cy));
            }
        }
        for (int r = 0; r < m64; ++r) {
            const double2 v = Vb[(size_t)idx64[r] * d + i], c = coef64[r];
            u.x -= fma(c.x, v.x, -c.y * v.y);
            u.y -= fma(c.x, v.y, c.y * v.x);
        }
        u.x -= f32_to_f64_int(cx);
        u.y -= f32_to_f64_int(cy);
        out[i] = u;
        if (S1) {
            S1[i] = u.x + u.y;
            V32_1[i] = make_float2(f64_to_f32_trunc(u.x), f64_to_f32_trunc(u.y));
        }
        acc = fma(u.x, u.x, fma(u.y, u.y, acc));
        em = max(em, max(exp_field(u.x), exp_field(u.y)));
        return u;
    };
    const bool img = D.I != nullptr && level >= 1;  // images for the exact Gram-Schmidt dots
    if ((D.Xf || img) && (second || level < 2)) {
        // Last pass of an exact-integer column: also write the fixed-point
        // image of V_{j+1} that the next H*psi reads, on the exponent efix;
        // with the exact dots, also its 52-bit image I_{j+1} on the same one.
        // The vector's largest exponent is only known after this kernel, so
        // efix bounds it from the inputs (the prologue).
        const int Ef = efix_s, P = D.fix_pre;
        int4* I1 = img ? D.I + (size_t)(j + 1) * d : nullptr;
        if (D.Xf && img) {
            KG_FOR(i) {
                const double2 u = element(i);
                D.Xf[i] = make_longlong2(fix_term(u.x, Ef, P, 0u), fix_term(u.y, Ef, P, 0u));
                I1[i] = fix_image(u, Ef);
            }
        } else if (D.Xf) {
            KG_FOR(i) {
                const double2 u = element(i);
                D.Xf[i] = make_longlong2(fix_term(u.x, Ef, P, 0u), fix_term(u.y, Ef, P, 0u));
            }
        } else {
            KG_FOR(i) I1[i] = fix_image(element(i), Ef);
        }
        if (blk == 0 && threadIdx.x == 0) {
            if (D.Xf) C->efix = Ef;
            if (img) C->eimg[j + 1] = Ef;
        }
    } else {
        KG_FOR(i) element(i);
    }
    chain_next();
    block_partial(acc, em, head.sum, D.part_n + blk);
    if (writer) {
        C->n_norm = nblk;
        C->abase = second ? C->alpha[j] : araw;
        C->hre = nk ? hre_s : 0.0;
    }
    // the other parity's totals are free: cleared for the dots of j + 1
    if (exact && blk == 0)
        for (int q = threadIdx.x; q < 4 * (D.M + 1); q += blockDim.x) D.gacc[((j + 1) & 1) * 4 * (D.M + 1) + q] = 0ull;
}

// resolve_norm by itself, one block per column.
__global__ void __launch_bounds__(kThreads) k_resolve(const ColDesc* desc, ColScalars* cs, int j) {
    __shared__ HeadShared head;
    const ColDesc D = desc[blockIdx.x];
    chain_wait();
    resolve_norm(D, cs + blockIdx.x, j, threadIdx.x == 0, head);
}

int launch_resolve(Krylov& K, int j, cudaStream_t st) {
    ProfScope ps("resolve", st);
    return launch_chained(k_resolve, K.B, kThreads, 0, st, K.desc, K.cs, j);
}

int launch_update(Krylov& K, int j, int level, bool second, cudaStream_t st) {
    ProfScope ps("update", st);
    const int4* items;
    int n;
    KG_TRY(work_list(K, (const void*)k_update, -1, &items, &n));
    const int exact = level >= 1 && use_int_dots(K, second);
    return launch_chained(k_update, n, kThreads, 0, st, K.desc, items, K.cs, j, level, second ? 1 : 0, exact);
}

// ------------------------------------------- tridiagonal eigenproblem
// One warp per column.  Implicit symmetric QR with Wilkinson shifts on the
// unreduced blocks of T (Golub and Van Loan, Section 8.3): lane 0 chases the
// bulge and records the Givens rotations of one sweep in shared memory, then
// all lanes apply them to their rows of Q (Q <- Q R_k).  On exit T = Q D Q^T.
//   mode 0 (propagation, Eq. (udelta)), with the column's tau:
//       c_k = beta0 * sum_m Q[k][m] e^{-i lambda_m tau} Q[0][m]
// The stored combination coefficient is c_k * s_k (Lanczos vectors are
// unnormalised).
//
// On this GPU a warp's FP64 instruction occupies the FP64 pipe for many
// cycles even with one active lane, so the serial chase is what costs: each
// rotation takes one reciprocal square root instead of a hypot and two
// divisions, and Q stays in shared memory for m <= 32 (every propagation
// step), so that applying a sweep's rotations does not wait on L2.
constexpr int kTriWarps = 2;
constexpr int kTriSmemQ = 32;

__global__ void __launch_bounds__(32 * kTriWarps) k_tridiag(const ColDesc* desc, ColScalars* cs, int B, int Mcap,
                                                           double* Qall, int mode, const double* taus, int ntau,
                                                           double2* cq) {
    __shared__ double sd[kTriWarps][kMaxMgs], se[kTriWarps][kMaxMgs];
    __shared__ double rc[kTriWarps][kMaxMgs], rs[kTriWarps][kMaxMgs];
    __shared__ int ctl[kTriWarps][4];
    __shared__ double sQ[kTriWarps][kTriSmemQ * kTriSmemQ];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b = blockIdx.x * kTriWarps + warp;
    if (b >= B) return;
    ColScalars* C = cs + b;
    const double tau = desc[b].tau;
    const int m = C->m_eff;
    double* Q = m <= kTriSmemQ ? sQ[warp] : Qall + (size_t)b * Mcap * Mcap;
    double* d = sd[warp];
    double* e = se[warp];
    if (m == 0) {
        for (int k = lane; k < Mcap; k += 32) C->c[k] = make_double2(0.0, 0.0);
        if (lane == 0) {
            C->lam0 = C->lam1 = 0.0;
            C->resest = 0.0;
        }
        return;
    }
    for (int k = lane; k < m; k += 32) {
        d[k] = C->alpha[k];
        e[k] = (k + 1 < m) ? C->beta[k + 1] : 0.0;
    }
    for (int r = lane; r < m; r += 32)
        for (int c = 0; c < m; ++c) Q[r * m + c] = (r == c) ? 1.0 : 0.0;
    __syncwarp();
    const double eps = 2.220446049250313e-16;
    int iter = 0;
    const int max_iter = 60 * m + 60;
    while (true) {
        if (lane == 0) {
            // deflate negligible off-diagonals, then locate the last unreduced block
            for (int i = 0; i + 1 < m; ++i)
                if (fabs(e[i]) <= eps * (fabs(d[i]) + fabs(d[i + 1]))) e[i] = 0.0;
            int hi = m - 1;
            while (hi > 0 && e[hi - 1] == 0.0) --hi;
            int lo = hi;
            while (lo > 0 && e[lo - 1] != 0.0) --lo;
            ctl[warp][0] = lo;
            ctl[warp][1] = hi;
            if (hi > 0 && iter < max_iter) {
                // Wilkinson shift from the trailing 2x2 of the block
                const double dd = 0.5 * (d[hi - 1] - d[hi]);
                const double bb = e[hi - 1];
                const double den = dd + copysign(hypot(dd, bb), dd == 0.0 ? 1.0 : dd);
                const double mu = d[hi] - bb * bb / den;
                double x = d[lo] - mu, z = e[lo];
                for (int k = lo; k < hi; ++k) {
                    // Givens rotation zeroing z against x: r = |(x, z)|
                    const double r2 = fma(x, x, z * z);
                    double c = 1.0, s = 0.0, r = 0.0;
                    if (r2 > 0.0) {
                        const double inv = rsqrt(r2);
                        c = x * inv;
                        s = z * inv;
                        r = r2 * inv;
                    }
                    if (k > lo) e[k - 1] = r;
                    const double ak = d[k], ak1 = d[k + 1], bk = e[k];
                    const double cc = c * c, ss = s * s, cs2 = 2.0 * c * s * bk;
                    d[k] = cc * ak + cs2 + ss * ak1;
                    d[k + 1] = ss * ak - cs2 + cc * ak1;
                    e[k] = c * s * (ak1 - ak) + (cc - ss) * bk;
                    if (k + 1 < hi) {
                        const double bulge = s * e[k + 1];
                        e[k + 1] *= c;
                        x = e[k];
                        z = bulge;
                    }
                    rc[warp][k] = c;
                    rs[warp][k] = s;
                }
            }
        }
        __syncwarp();
        const int lo = ctl[warp][0], hi = ctl[warp][1];
        if (hi == 0 || iter >= max_iter) break;
        for (int r = lane; r < m; r += 32) {
            double* row = Q + (size_t)r * m;
            double q0 = row[lo];
            for (int k = lo; k < hi; ++k) {
                const double c = rc[warp][k], s = rs[warp][k];
                const double q1 = row[k + 1];
                row[k] = c * q0 + s * q1;
                q0 = -s * q0 + c * q1;
            }
            row[hi] = q0;
        }
        __syncwarp();
        ++iter;
    }
    if (lane == 0 && iter >= max_iter && C->status == KG_OK) C->status = KG_ENOCONV;
    __syncwarp();
    if (mode == 0 || mode == 2) {
        // mode 0: the column's own tau into C->c; mode 2: ntau times
        // (quadrature nodes) into cq[b][t][k], from the same diagonalisation
        const double beta0 = C->beta0;
        double* pc = rc[warp];  // rotation buffers are free now: phases of e^{-i lambda tau}
        double* ps = rs[warp];
        const int nt = mode == 0 ? 1 : ntau;
        for (int t = 0; t < nt; ++t) {
            const double tt = mode == 0 ? tau : taus[(size_t)b * ntau + t];
            __syncwarp();
            for (int mm = lane; mm < m; mm += 32) {
                double sn, cn;
                sincos(d[mm] * tt, &sn, &cn);
                pc[mm] = cn * Q[mm];  // Q[0][mm] is Q[mm]
                ps[mm] = sn * Q[mm];
            }
            __syncwarp();
            for (int k = lane; k < m; k += 32) {
                double re = 0.0, im = 0.0;
                for (int mm = 0; mm < m; ++mm) {
                    const double q = Q[(size_t)k * m + mm];
                    re = fma(q, pc[mm], re);
                    im = fma(-q, ps[mm], im);
                }
                const double s = beta0 * C->scale[k];
                if (mode == 0)
                    C->c[k] = make_double2(s * re, s * im);
                else
                    cq[((size_t)b * ntau + t) * Mcap + k] = make_double2(s * re, s * im);
            }
        }
        if (mode == 2)
            for (int t = 0; t < ntau; ++t)
                for (int k = m + lane; k < Mcap; k += 32) cq[((size_t)b * ntau + t) * Mcap + k] = make_double2(0.0, 0.0);
    }
}

// The two lowest Ritz values and the lowest Ritz vector (ground state, Eq.
// (eigen)): lam0, lam1, c_k = q_k s_k, resest = |b_m q_{m-1}|; one block per
// column.  The eigenvalues by multisection with Sturm counts (the sign changes
// of the leading minors of T - x, by their three-term recurrence, scaled so
// that nothing overflows): two warps narrow the bracket of each, 64 points a
// round, nine rounds to full precision.  The vector by the twisted
// factorisation of T - lam0 (Parlett and Dhillon, Linear Algebra Appl. 267
// (1997) 247): one lane eliminates from the top, one from the bottom, and the
// vector starts where the two meet with the smallest pivot.  A warp's FP64
// instruction costs the same 64 cycles for one lane as for 32, so the 64
// points are free, while the implicit QR of k_tridiag spends them one by one:
// m = 100 takes 0.15 ms here and took 23 ms there.
constexpr int kLowThreads = 128;

__global__ void __launch_bounds__(kLowThreads) k_lowest(ColScalars* cs, int Mcap) {
    __shared__ double a[kMaxMgs], b[kMaxMgs + 1], b2[kMaxMgs + 1];  // scaled; b[i] couples i - 1 and i
    __shared__ double rp[kMaxMgs], rm[kMaxMgs], dp[kMaxMgs], dm[kMaxMgs], z[kMaxMgs];
    __shared__ double lo[2], hi[2], wlo[4], whi[4];
    __shared__ double gmax[4];
    __shared__ int rs;
    ColScalars* C = cs + blockIdx.x;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int m = C->m_eff;
    if (m == 0) {
        for (int k = tid; k < Mcap; k += kLowThreads) C->c[k] = make_double2(0.0, 0.0);
        if (tid == 0) {
            C->lam0 = C->lam1 = 0.0;
            C->resest = 0.0;
        }
        return;
    }
    // scale by a power of two so that the row sums are at most 1
    double g = 0.0;
    for (int k = tid; k < m; k += kLowThreads)
        g = fmax(g, fabs(C->alpha[k]) + (k > 0 ? fabs(C->beta[k]) : 0.0) + (k + 1 < m ? fabs(C->beta[k + 1]) : 0.0));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) g = fmax(g, __shfl_xor_sync(0xffffffffu, g, o));
    if (lane == 0) gmax[warp] = g;
    __syncthreads();
    g = fmax(fmax(gmax[0], gmax[1]), fmax(gmax[2], gmax[3]));
    const int e = g > 0.0 ? exp_field(g) - 1022 : 0;  // g < 2^e
    for (int k = tid; k < m; k += kLowThreads) {
        a[k] = ldexp(C->alpha[k], -e);
        b[k] = k > 0 ? ldexp(C->beta[k], -e) : 0.0;
        b2[k] = b[k] * b[k];
    }
    if (tid < 2) {
        lo[tid] = -1.0;
        hi[tid] = 1.0;
    }
    __syncthreads();
    const int which = warp >> 1;  // eigenvalue 0 or 1
    for (int round = 0; round < 9; ++round) {
        const double l = lo[which], h = hi[which];
        const int pt = tid & 63;
        const double x = fma(h - l, (pt + 1) * (1.0 / 65.0), l);
        double p0 = 1.0, p1 = a[0] - x;
        long long prev = 0;  // sign of p0
        int count = 0;
        for (int i = 0;;) {
            // a vanishing minor counts with the sign opposite to the one before
            const long long sg = p1 == 0.0 ? ~prev : __double_as_longlong(p1);
            count += (sg ^ prev) < 0;
            prev = sg;
            if (++i >= m) break;
            const double q = fma(a[i] - x, p1, -b2[i] * p0);
            p0 = p1;
            p1 = q;
            if ((i & 7) == 0) {
                const int top = max(exp_field(p0), exp_field(p1));
                if (top > 1323 || (top < 723 && top > 0)) {
                    const double f = __longlong_as_double((long long)(2046 - top) << 52);
                    p0 *= f;
                    p1 *= f;
                }
            }
        }
        // eigenvalue `which` lies below x exactly when more than `which` do
        const unsigned below = __ballot_sync(0xffffffffu, count > which);
        const int first = below ? __ffs(below) - 1 : 32;  // the counts grow with the point
        const double xl = __shfl_sync(0xffffffffu, x, first > 0 ? first - 1 : 0), xh = __shfl_sync(0xffffffffu, x, first & 31);
        if (lane == 0) {
            wlo[warp] = first > 0 ? xl : l;
            whi[warp] = first < 32 ? xh : h;
        }
        __syncthreads();
        if (tid < 2) {
            // the second warp's points follow the first's
            const double first_hi = whi[2 * tid], h0 = hi[tid];
            if (first_hi < h0) {
                lo[tid] = wlo[2 * tid];
                hi[tid] = first_hi;
            } else {
                lo[tid] = fmax(wlo[2 * tid], wlo[2 * tid + 1]);
                hi[tid] = whi[2 * tid + 1];
            }
        }
        __syncthreads();
    }
    const double lam = 0.5 * (lo[0] + hi[0]);
    if (warp == 0 && lane < 2) {
        const int s = lane == 0 ? 0 : m - 1, step = lane == 0 ? 1 : -1;
        double* d = lane == 0 ? dp : dm;
        double* r = lane == 0 ? rp : rm;
        double q = a[s] - lam;
        for (int i = 0, k = s;; k += step) {
            if (!(fabs(q) > 0x1p-900)) q = 0x1p-60;
            const double inv = 1.0 / q;
            d[k] = q;
            r[k] = inv;
            if (++i >= m) break;
            const int nx = k + step;
            q = (a[nx] - lam) - b2[lane == 0 ? nx : k] * inv;
        }
    }
    __syncthreads();
    if (warp == 0) {
        double best = INFINITY;
        int at = 0;
        for (int k = lane; k < m; k += 32) {
            const double v = fabs(dp[k] + dm[k] - (a[k] - lam));
            if (v < best) {
                best = v;
                at = k;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double ov = __shfl_xor_sync(0xffffffffu, best, o);
            const int oa = __shfl_xor_sync(0xffffffffu, at, o);
            if (ov < best || (ov == best && oa < at)) {
                best = ov;
                at = oa;
            }
        }
        if (lane == 0) rs = at;
    }
    __syncthreads();
    const int r = rs;
    // factors from z_r = 1 outwards: z_k = -b_{k+1} z_{k+1} / d+_k, z_k = -b_k z_{k-1} / d-_k
    for (int k = tid; k < m; k += kLowThreads) z[k] = k < r ? -b[k + 1] * rp[k] : (k > r ? -b[k] * rm[k] : 1.0);
    __syncthreads();
    if (warp == 0 && lane < 2) {
        double v = 1.0;
        if (lane == 0)
            for (int k = r - 1; k >= 0; --k) z[k] = v *= z[k];
        else
            for (int k = r + 1; k < m; ++k) z[k] = v *= z[k];
    }
    __syncthreads();
    if (warp == 0) {
        double s = 0.0;
        for (int k = lane; k < m; k += 32) s = fma(z[k], z[k], s);
        s = warp_sum(s);
        const double f = (z[0] < 0.0 ? -1.0 : 1.0) / sqrt(s);
        for (int k = lane; k < m; k += 32) C->c[k] = make_double2(f * z[k] * C->scale[k], 0.0);
        if (lane == 0) {
            C->lam0 = ldexp(lam, e);
            C->lam1 = m > 1 ? ldexp(0.5 * (lo[1] + hi[1]), e) : INFINITY;
            C->resest = fabs(C->beta[m] * f * z[m - 1]);
        }
    }
}

// ------------------------------------ step exponential by a Taylor series
// c = beta0 e^{-i T tau} e_1 (times s_k per component) by Tridiag::advance, one
// warp per column, and per time in mode 2.  Modes 0 and 2 as in
// k_tridiag.  A warp is a serial chain of FP64 instructions: taking the 10
// or 11 quadrature times of a column in order, each from the one before, took
// about 100 us a launch; side by side, all from e_1, it is about 15.
template <int R>
__global__ void __launch_bounds__(32 * kTriWarps) k_texp(const ColDesc* desc, ColScalars* cs, int B, int Mcap,
                                                        int mode, const double* taus, int ntau, double2* cq) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int item = blockIdx.x * kTriWarps + warp, t = item / B, b = item % B;
    chain_wait();
    if (t >= ntau) return;
    ColScalars* C = cs + b;
    const int m = C->m_eff;
    double2* const out = mode == 0 ? C->c : cq + ((size_t)b * ntau + t) * Mcap;
    const double tau = mode == 0 ? desc[b].tau : taus[(size_t)b * ntau + t];
    double2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = make_double2((lane + 32 * r) == 0 ? 1.0 : 0.0, 0.0);
    bool ok = m > 0;
    if (ok) {
        Tridiag<R> T;
        T.load(C->alpha, C->beta, m, lane);
        // a non-finite or absurdly large T (more than kMaxSub sub-steps)
        // cannot be exponentiated this way: report it instead of looping
        ok = T.advance(tau, v, lane, true);
        if (!ok && lane == 0) C->status = KG_ENUMERIC;
    }
    if (!ok) {
        for (int k = lane; k < Mcap; k += 32) C->c[k] = out[k] = make_double2(0.0, 0.0);
        return;
    }
    const double beta0 = C->beta0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int k = lane + 32 * r;
        if (k < m) {
            const double sc = beta0 * C->scale[k];
            out[k] = make_double2(sc * v[r].x, sc * v[r].y);
        } else if (k < Mcap && mode == 2) {
            out[k] = make_double2(0.0, 0.0);
        }
    }
}

static int launch_texp(Krylov& K, int mode, const double* taus, int ntau, double2* cq, cudaStream_t st) {
    const int nb = (K.B * ntau + kTriWarps - 1) / kTriWarps;
    return launch_chained(K.M <= 32 ? &k_texp<1> : &k_texp<2>, nb, 32 * kTriWarps, 0, st, K.desc, K.cs, K.B, K.M, mode,
                          taus, ntau, cq);
}

int launch_tridiag(Krylov& K, int mode, cudaStream_t st) {
    const int nb = (K.B + kTriWarps - 1) / kTriWarps;
    ProfScope ps("tridiag", st);
    if (mode == 0 && !(K.schedule & 2)) return launch_texp(K, 0, nullptr, 1, nullptr, st);
    if (mode == 1) {
        k_lowest<<<K.B, kLowThreads, 0, st>>>(K.cs, K.M);
        KG_LAUNCHED();
        return KG_OK;
    }
    k_tridiag<<<nb, 32 * kTriWarps, 0, st>>>(K.desc, K.cs, K.B, K.M, K.Q, mode, nullptr, 0, nullptr);
    KG_LAUNCHED();
    return KG_OK;
}

// ----------------------------------- combination and overlaps
// out = sum_{k<m} c_k V_k  (Eq. (udelta) in the form V x small vector), then
// ||out|| and <ov_a, out> for the column's n_ov overlap vectors, written to
// row cs[b].ov_slot of its overlap table (the slot advances by one).  NOV
// bounds n_ov at compile time so that the accumulators stay in registers.
//
// The Krylov coefficients decay quickly with k.  As in the update, a term
// whose coefficient on the unit vector v_k is below 1e-10 of the largest one
// (which bounds ||out||) is summed in FP32 from the truncated plane; the
// others use three FP64 multiply-adds per element with the Re+Im plane
// (c = p + iq, v = a + ib: T1 = p a, T2 = q b, T3 = (p + q)(a + b),
// Re = T1 - T2, Im = T3 - T1 - T2), or four without it.
template <int NOV>
__global__ void __launch_bounds__(kThreads) k_combine(const ColDesc* desc, const int4* items, ColScalars* cs,
                                                      unsigned* cnt, int fused) {
    __shared__ double2 coef[kMaxMgs];
    __shared__ double csum[kMaxMgs];
    __shared__ int idx64[kMaxMgs], idx32[kMaxMgs];
    __shared__ float2 coef32[kMaxMgs];
    __shared__ int n64, n32;
    __shared__ double sm[(kThreads / 32) * (2 * NOV + 2)];
    __shared__ double bs[2 * NOV + 2], red[2 * NOV + 2];
    KG_ITEM();
    chain_wait();
    const int m = C->m_eff;
    // a space from kg_small.cu comes without the planes
    const double* Sb = fused ? nullptr : D.S;
    const float2* V32 = fused ? nullptr : D.V32;
    if (threadIdx.x < 32) {  // the first warp sorts the terms, one per lane
        const int lane = threadIdx.x;
        double cmax = 0.0;
        for (int k = lane; k < m; k += 32) {
            const double2 c = C->c[k];
            const double sk = C->scale[k];
            if (sk > 0.0) cmax = fmax(cmax, (fabs(c.x) + fabs(c.y)) / sk);
        }
#pragma unroll
        for (int o_ = 16; o_ > 0; o_ >>= 1) cmax = fmax(cmax, __shfl_xor_sync(0xffffffffu, cmax, o_));
        int a64 = 0, a32 = 0;
        // norms, and their product (the coefficients), within 2^-60 .. 2^60: the FP32
        // copies and coefficients do not overflow, nor vanish above 2^-64 of the result
        const int ec = exp_field(cmax);
        const bool in32 = V32 && (unsigned)(ec - 963) <= 120u;
        for (int k0 = 0; k0 < m; k0 += 32) {
            const int k = k0 + lane;
            const double2 c = k < m ? C->c[k] : make_double2(0.0, 0.0);
            const double sk = k < m ? C->scale[k] : 0.0;
            const int es = exp_field(sk);
            const bool small = in32 && (unsigned)(es - 963) <= 120u && (unsigned)(ec + es - 1986) <= 120u &&
                               (fabs(c.x) + fabs(c.y)) < 1e-10 * cmax * sk;
            const unsigned in = __ballot_sync(0xffffffffu, k < m), ms = __ballot_sync(0xffffffffu, k < m && small);
            const unsigned before = (1u << lane) - 1u;
            if (k < m && small) {
                const int q = a32 + __popc(ms & before);
                coef32[q] = make_float2((float)c.x, (float)c.y);
                idx32[q] = k;
            } else if (k < m) {
                const int q = a64 + __popc(in & ~ms & before);
                coef[q] = c;
                csum[q] = c.x + c.y;
                idx64[q] = k;
            }
            a32 += __popc(ms);
            a64 += __popc(in & ~ms);
        }
        if (lane == 0) {
            n64 = a64;
            n32 = a32;
        }
    }
    __syncthreads();
    const int m64 = n64, m32 = n32;
    const int d = D.d;
    const int n_ov = D.n_ov;
    const double2* Vb = D.V;
    double2* o = D.out;
    double acc[2 * NOV + 2];
#pragma unroll
    for (int k = 0; k < 2 * NOV + 2; ++k) acc[k] = 0.0;
    KG_FOR(i) {
        double2 u;
        if (Sb) {
            double t1 = 0.0, t2 = 0.0, t3 = 0.0;
            for (int q = 0; q < m64; ++q) {
                const size_t o_ = (size_t)idx64[q] * d + i;
                const double2 v = Vb[o_];
                const double sv = Sb[o_];
                const double2 c = coef[q];
                t1 = fma(c.x, v.x, t1);
                t2 = fma(c.y, v.y, t2);
                t3 = fma(csum[q], sv, t3);
            }
            u = make_double2(t1 - t2, t3 - t1 - t2);
        } else {
            u = make_double2(0.0, 0.0);
            for (int q = 0; q < m64; ++q) {
                const double2 v = Vb[(size_t)idx64[q] * d + i];
                const double2 c = coef[q];
                u.x = fma(c.x, v.x, fma(-c.y, v.y, u.x));
                u.y = fma(c.x, v.y, fma(c.y, v.x, u.y));
            }
        }
        if (m32) {
            float cx = 0.f, cy = 0.f;
            int q = 0;
            for (; q + 4 <= m32; q += 4) {
                float2 v[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) v[r] = V32[(size_t)idx32[q + r] * d + i];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const float2 c = coef32[q + r];
                    cx = fmaf(c.x, v[r].x, fmaf(-c.y, v[r].y, cx));
                    cy = fmaf(c.x, v[r].y, fmaf(c.y, v[r].x, cy));
                }
            }
            for (; q < m32; ++q) {
                const float2 v = V32[(size_t)idx32[q] * d + i], c = coef32[q];
                cx = fmaf(c.x, v.x, fmaf(-c.y, v.y, cx));
                cy = fmaf(c.x, v.y, fmaf(c.y, v.x, cy));
            }
            u.x += (double)cx;
            u.y += (double)cy;
        }
        o[i] = u;
        acc[0] = fma(u.x, u.x, fma(u.y, u.y, acc[0]));
#pragma unroll
        for (int a = 0; a < NOV; ++a) {
            if (a < n_ov) {
                const double2 v = D.ov[(size_t)a * D.ov_stride + i];
                acc[2 + 2 * a] = fma(v.x, u.x, fma(v.y, u.y, acc[2 + 2 * a]));
                acc[3 + 2 * a] = fma(v.x, u.y, fma(-v.y, u.x, acc[3 + 2 * a]));
            }
        }
    }
    const int nv = 2 + 2 * n_ov;
    block_sum<2 * NOV + 2>(acc, nv, sm, bs);
    if (grid_finish(bs, nv, D.part, cnt + b, blk, nblk, red)) {
        const int slot = C->ov_slot;
        for (int a = threadIdx.x; a < n_ov; a += blockDim.x)
            if (slot < D.ov_rows) D.ov_out[(size_t)slot * n_ov + a] = make_double2(red[2 + 2 * a], red[3 + 2 * a]);
        __syncthreads();
        if (threadIdx.x == 0) {
            C->ovnorm = sqrt(red[0]);
            if (n_ov > 0) C->ov_slot = slot + 1;
        }
    }
}

int launch_combine(Krylov& K, cudaStream_t st) {
    int n_ov = 0;
    for (auto& D : K.hdesc) n_ov = std::max(n_ov, D.n_ov);
    if (n_ov > kMaxOv) {
        set_error("at most %d overlap vectors per combination pass", kMaxOv);
        return KG_EINVAL;
    }
    ProfScope ps("combine", st);
    const int4* items;
    int n;
    const auto kern = n_ov == 0 ? &k_combine<0> : n_ov <= 4 ? &k_combine<4> : n_ov <= 12 ? &k_combine<12> : &k_combine<32>;
    KG_TRY(work_list(K, (const void*)kern, -1, &items, &n));
    return launch_chained(kern, n, kThreads, 0, st, K.desc, items, K.cs, K.cnt, K.fused ? 1 : 0);
}

// -------------------------------------------- ground-state residual
// rq = <x, y> (x normalised), then rnorm = ||y - rq x||.
__global__ void __launch_bounds__(kThreads) k_rq(const double2* x, const double2* y, int d, ColScalars* cs,
                                                 int phase, double* part, unsigned* cnt) {
    __shared__ double sm[(kThreads / 32) * 2];
    __shared__ double bs[2], red[2];
    const double rq = phase ? cs->rq : 0.0;
    double acc[1] = {0.0};
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < d; i += gridDim.x * blockDim.x) {
        const double2 a = x[i], b = y[i];
        if (phase == 0) {
            acc[0] = fma(a.x, b.x, fma(a.y, b.y, acc[0]));
        } else {
            const double rx = fma(-rq, a.x, b.x), ry = fma(-rq, a.y, b.y);
            acc[0] = fma(rx, rx, fma(ry, ry, acc[0]));
        }
    }
    block_sum<1>(acc, 1, sm, bs);
    if (grid_finish(bs, 1, part, cnt, blockIdx.x, gridDim.x, red) && threadIdx.x == 0) {
        if (phase == 0)
            cs->rq = red[0];
        else
            cs->rnorm = sqrt(red[0]);
    }
}

// Coefficients of exp(-i H t) v_0 for ntau times per column (taus[b][t]),
// into cq[b][t][0..M) (already times the scales of the stored vectors).
constexpr int kMaxTaus = 32;  // times per column in one launch
int launch_tridiag_multi(Krylov& K, const double* taus, int ntau, double2* cq, cudaStream_t st) {
    if (ntau < 1 || ntau > kMaxTaus) {
        set_error("between 1 and %d times per column", kMaxTaus);
        return KG_EINVAL;
    }
    const int nb = (K.B + kTriWarps - 1) / kTriWarps;
    ProfScope ps("tridiag", st);
    if (!(K.schedule & 2)) return launch_texp(K, 2, taus, ntau, cq, st);
    k_tridiag<<<nb, 32 * kTriWarps, 0, st>>>(K.desc, K.cs, K.B, K.M, K.Q, 2, taus, ntau, cq);
    KG_LAUNCHED();
    return KG_OK;
}

// -------------------------------------------------- step sequencing
__global__ void k_set_slots(ColScalars* cs, int B, int value) {
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < B; b += gridDim.x * blockDim.x) cs[b].ov_slot = value;
}

__global__ void k_reset_status(ColScalars* cs, int B) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < B) cs[b].status = KG_OK;
}

int launch_reset_status(Krylov& K, cudaStream_t st) {
    k_reset_status<<<(K.B + 127) / 128, 128, 0, st>>>(K.cs, K.B);
    KG_LAUNCHED();
    return KG_OK;
}

int launch_set_slots(Krylov& K, int value, cudaStream_t st) {
    k_set_slots<<<(K.B + 127) / 128, 128, 0, st>>>(K.cs, K.B, value);
    KG_LAUNCHED();
    return KG_OK;
}

int prepare_step(Krylov& K, int reorth) {
    const int4* items;
    int n;
    K.fused = small_steps(K, reorth);
    if (K.fused) return KG_OK;
    KG_TRY(prepare_hpsi_lists(K));
    KG_TRY(work_list(K, (const void*)k_colnorm, -1, &items, &n));
    KG_TRY(work_list(K, (const void*)k_update, -1, &items, &n));
    if (reorth >= 1) {
        // every vector count of one step (and of the ground-state restarts)
        for (int nk = 1; nk <= std::min(kChunk, K.M + 1); ++nk) {
            KG_TRY(work_list(K, (const void*)dots_kernel(nk), -1, &items, &n));
            if (use_int_dots(K, false)) {
                const IntDotsKernel ik = int_dots_kernel(nk);
                KG_TRY(work_list(K, (const void*)ik.kern, -1, &items, &n, -1, ik.threads, ik.smem, kDotMinRun));
            }
        }
    }
    const void* comb[4] = {(const void*)k_combine<0>, (const void*)k_combine<4>, (const void*)k_combine<12>,
                           (const void*)k_combine<32>};
    for (auto* k : comb) KG_TRY(work_list(K, k, -1, &items, &n));
    return KG_OK;
}

// Lanczos space of every column's V_0.
int build_space(Krylov& K, int reorth, cudaStream_t st) {
    K.fused = small_steps(K, reorth);
    if (K.fused) return launch_small(K, false, st);
    KG_TRY(launch_colnorm(K, st));
    for (int j = 0; j < K.M; ++j) {
        KG_TRY(launch_lanczos_hpsi(K, j, st));
        if (reorth >= 1)
            for (int k0 = 0; k0 <= j; k0 += kChunk)
                KG_TRY(launch_reorth_dots(K, j, k0, std::min(kChunk, j + 1 - k0), false, st));
        KG_TRY(launch_update(K, j, reorth, false, st));
        if (reorth >= 2) {
            KG_TRY(launch_resolve(K, j + 1, st));
            for (int k0 = 0; k0 <= j; k0 += kChunk)
                KG_TRY(launch_reorth_dots(K, j, k0, std::min(kChunk, j + 1 - k0), true, st));
            KG_TRY(launch_update(K, j, reorth, true, st));
        }
    }
    return launch_resolve(K, K.M, st);
}

int enqueue_step(Krylov& K, int reorth, cudaStream_t st) {
    if (small_steps(K, reorth)) {
        K.fused = true;
        return launch_small(K, true, st);
    }
    KG_TRY(build_space(K, reorth, st));
    KG_TRY(launch_tridiag(K, 0, st));
    return launch_combine(K, st);
}

int read_scalars(const Krylov& K, std::vector<ColScalars>& h, cudaStream_t st) {
    h.resize(K.B);
    KG_CUDA(cudaMemcpyAsync(h.data(), K.cs, sizeof(ColScalars) * K.B, cudaMemcpyDeviceToHost, st));
    KG_CUDA(cudaStreamSynchronize(st));
    return KG_OK;
}

int column_rc(int status, const char* what) {
    if (status == KG_ENUMERIC) set_error("non-finite value during %s", what);
    else if (status == KG_ETIMEOUT) set_error("a bounded device wait ran out during %s", what);
    else return KG_OK;
    return status;
}

// ------------------------------------------------------ ground state
int ground_state(kg_sector* s, const kg_opts* o) {
    cudaStream_t st = pick_stream(s, o);
    const int d = (int)s->d;
    if (o->M_gs < 2 || o->M_gs > kMaxMgs) {
        set_error("M_gs must be in [2, %d]", kMaxMgs);
        return KG_EINVAL;
    }
    const int M = std::max(1, std::min(o->M_gs, d));
    if (!s->gs) KG_CUDA(cudaMalloc(&s->gs, sizeof(double2) * d));
    Krylov K;
    int rc = krylov_alloc(K, {s}, M, s->nsm, o->schedule);
    if (rc != KG_OK) {
        krylov_free(K);
        return rc;
    }
    auto done = [&](int r) {
        krylov_free(K);
        return r;
    };
    K.hdesc[0].out = s->gs;  // the Ritz vector of each restart goes to the cache
    rc = krylov_upload(K, st);
    const SecView S = s->view();
    double2* V0 = K.vec(0, 0);
    double2* W0 = K.hdesc[0].W;
    double* part = K.hdesc[0].part;
    const int nrq = std::max(1, std::min(K.hdesc[0].nblk_max, (d + kThreads - 1) / kThreads));
    if (rc == KG_OK) rc = launch_random_start(V0, d, o->seed, st);
    ColScalars h;
    bool converged = false;
    for (int r = 0; rc == KG_OK && r < o->max_restarts; ++r) {
        rc = build_space(K, std::max(1, o->reorth), st);
        if (rc == KG_OK) rc = launch_tridiag(K, 1, st);
        if (rc == KG_OK) rc = launch_combine(K, st);
        if (rc != KG_OK) break;
        if (cudaMemcpyAsync(&h, K.cs, sizeof(ColScalars), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess) {
            rc = cuda_fail(cudaGetLastError(), "ground-state readback", __FILE__, __LINE__);
            break;
        }
        if ((rc = column_rc(h.status, "the ground-state Lanczos recursion")) != KG_OK) break;
        if (!(h.ovnorm > 0.0) || !std::isfinite(h.ovnorm)) {
            set_error("non-finite value in the ground-state Lanczos recursion");
            rc = KG_ENUMERIC;
            break;
        }
        if ((rc = launch_scale_copy(s->gs, s->gs, d, 1.0 / h.ovnorm, st)) != KG_OK) break;
        if ((rc = launch_hpsi(s, s->gs, W0, st)) != KG_OK) break;
        k_rq<<<nrq, kThreads, 0, st>>>(s->gs, W0, d, K.cs, 0, part, K.cnt);
        count_launch();
        k_rq<<<nrq, kThreads, 0, st>>>(s->gs, W0, d, K.cs, 1, part, K.cnt);
        count_launch();
        if (cudaGetLastError() != cudaSuccess) {
            rc = KG_ECUDA;
            break;
        }
        if (cudaMemcpyAsync(&h, K.cs, sizeof(ColScalars), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess) {
            rc = cuda_fail(cudaGetLastError(), "ground-state readback", __FILE__, __LINE__);
            break;
        }
        s->E0 = h.rq;
        s->resid = h.rnorm;
        s->gap = h.lam1 - h.lam0;
        if (!std::isfinite(h.rq) || !std::isfinite(h.rnorm)) {
            set_error("non-finite Rayleigh quotient");
            rc = KG_ENUMERIC;
            break;
        }
        if (h.rnorm <= o->tol_resid * std::max(1.0, std::fabs(h.rq)) || M >= d) {
            converged = true;
            break;
        }
        // restart from the Ritz vector
        if (cudaMemcpyAsync(V0, s->gs, sizeof(double2) * d, cudaMemcpyDeviceToDevice, st) != cudaSuccess) {
            rc = KG_ECUDA;
            break;
        }
    }
    if (rc != KG_OK) return done(rc);
    s->has_gs = converged;
    if (!converged) {
        set_error("ground state not converged: residual %.3e after %d restarts", s->resid, o->max_restarts);
        return done(KG_ENOCONV);
    }
    if (s->gap < 1e-8 * std::max(1.0, std::fabs(s->E0))) {
        set_error("ground state looks degenerate: Ritz gap %.3e", s->gap);
        return done(KG_EDEGEN);
    }
    return done(KG_OK);
}

}  // namespace kg
