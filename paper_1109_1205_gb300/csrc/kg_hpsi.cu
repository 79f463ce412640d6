// kg_hpsi.cu -- the Hamiltonian applied on the fly in the
// occupation-number basis (Section 2, H_jj'; model Hamiltonians of Sections 3
// and 4).  One thread produces one output element y[s], s = i_dn*D_up + i_up:
//
//   y[s] = (e_up[i_up] + e_dn[i_dn] + U(b_up & b_dn)) x[s]
//        + sum_{up hops of i_up}  (+-h_ab) x[i_dn*D_up + j]     (same row)
//        + sum_{down hops of i_dn}(+-h_ab) x[j*D_up + i_up]     (other rows)
//
// Up hops gather inside one row (L1/L2 resident); down hops read whole rows
// at a stride of D_up, so a warp (consecutive i_up, one i_dn) walks the same
// down-hop list and its loads are coalesced.
//
// Hop sums.  The FP64 pipe of this GPU issues about two lanes per clock per
// SM, 64 times fewer than the integer pipe.  When every hop has the same
// amplitude h0 (the Hubbard ring and the SIAM chain), the hop part is h0 times
// a signed sum of gathered components, which is computed exactly on the
// integer pipe: each component becomes the 64-bit fixed-point number
// round(x * 2^(1075 + P - E)), E the largest exponent field of the vector and
// P = 9 - ceil(log2(hops + 1)) the head room, so no sum can overflow.  The
// sum is exact; the only rounding is the conversion of each term, at most
// 2^-57 of the vector's largest component, and one conversion back to FP64.
// Other hoppings (site-dependent or complex amplitudes) use FP64 FMAs.
#include <algorithm>

#include "kg_internal.h"

namespace kg {

__device__ __forceinline__ double flip(double v, uint32_t code) {
    return __longlong_as_double(__double_as_longlong(v) ^ ((long long)(code >> 31) << 63));
}

template <int MODE>
__device__ __forceinline__ void hop_acc(double2& acc, uint32_t code, double2 xs, const double2* amp) {
    if (MODE == 0) {
        acc.x += flip(xs.x, code);
        acc.y += flip(xs.y, code);
    } else if (MODE == 1) {
        const double a = flip(amp[code & 1023u].x, code);
        acc.x = fma(a, xs.x, acc.x);
        acc.y = fma(a, xs.y, acc.y);
    } else {
        double2 a = amp[code & 1023u];
        a.x = flip(a.x, code);
        a.y = flip(a.y, code);
        acc.x = fma(a.x, xs.x, fma(-a.y, xs.y, acc.x));
        acc.y = fma(a.x, xs.y, fma(a.y, xs.x, acc.y));
    }
}

__device__ __forceinline__ double diag_energy(const SecView& S, int i_dn, int i_up, const double* utab) {
    const uint32_t both = __ldg(S.up_bits + i_up) & __ldg(S.dn_bits + i_dn);
    double diag = __ldg(S.up_e + i_up) + __ldg(S.dn_e + i_dn);
    for (int c = 0; c < S.nchunk; ++c) diag += utab[c * 256 + ((both >> (8 * c)) & 255u)];
    return diag;
}

// Hop part of (H x)[i_dn, i_up].  MODE 0-2: FP64 accumulation (MODE 0 without
// the amplitude, applied by the caller); MODE 3: exact integer accumulation,
// returned in (ix, iy) as fixed-point sums.
template <int MODE>
__device__ __forceinline__ void hop_sum(const SecView& S, const double2* __restrict__ x, int i_dn, int i_up,
                                        const double2* amp, int E, double2& hop, long long& ix, long long& iy) {
    const double2* row = x + (size_t)i_dn * S.Du;
    const int u0 = __ldg(S.up_off + i_up), u1 = __ldg(S.up_off + i_up + 1);
    const int d0 = __ldg(S.dn_off + i_dn), d1 = __ldg(S.dn_off + i_dn + 1);
    if (MODE == 3) {
        const int P = S.fix_pre;
#pragma unroll 4
        for (int e = u0; e < u1; ++e) {
            const uint2 en = __ldg(S.up_ent + e);
            const double2 xs = row[en.x];
            ix += fix_term(xs.x, E, P, en.y >> 31);
            iy += fix_term(xs.y, E, P, en.y >> 31);
        }
#pragma unroll 4
        for (int e = d0; e < d1; ++e) {
            const uint2 en = __ldg(S.dn_ent + e);
            const double2 xs = x[(size_t)en.x * S.Du + i_up];
            ix += fix_term(xs.x, E, P, en.y >> 31);
            iy += fix_term(xs.y, E, P, en.y >> 31);
        }
    } else {
#pragma unroll 4
        for (int e = u0; e < u1; ++e) {
            const uint2 en = __ldg(S.up_ent + e);
            hop_acc<MODE>(hop, en.y, row[en.x], amp);
        }
#pragma unroll 4
        for (int e = d0; e < d1; ++e) {
            const uint2 en = __ldg(S.dn_ent + e);
            hop_acc<MODE>(hop, en.y, x[(size_t)en.x * S.Du + i_up], amp);
        }
    }
}

// Hop part of (H x)[i_dn, i_up] from the fixed-point image Xf of x (all
// components on one exponent, written by the kernel that produced x): the
// same signed sums as the on-the-fly path, without the conversions.
__device__ __forceinline__ void hop_sum_pre(const SecView& S, const longlong2* __restrict__ Xf, int i_dn, int i_up,
                                            long long& ix, long long& iy) {
    // each string's hop list holds its +1-sign hops first, then the -1 ones
    const int u0 = __ldg(S.up_off + i_up), us = __ldg(S.up_split + i_up), u1 = __ldg(S.up_off + i_up + 1);
    const int d0 = __ldg(S.dn_off + i_dn), ds = __ldg(S.dn_split + i_dn), d1 = __ldg(S.dn_off + i_dn + 1);
    const longlong2* row = Xf + (size_t)i_dn * S.Du;
    const longlong2* col = Xf + i_up;
    const unsigned* upx = reinterpret_cast<const unsigned*>(S.up_ent);  // .x of entry e at [2e]
    const unsigned* dnx = reinterpret_cast<const unsigned*>(S.dn_ent);
    long long px = 0, py = 0, nx = 0, ny = 0;
#pragma unroll 4
    for (int e = u0; e < us; ++e) {
        const longlong2 v = row[__ldg(upx + 2 * e)];
        px += v.x;
        py += v.y;
    }
#pragma unroll 4
    for (int e = us; e < u1; ++e) {
        const longlong2 v = row[__ldg(upx + 2 * e)];
        nx += v.x;
        ny += v.y;
    }
#pragma unroll 4
    for (int e = d0; e < ds; ++e) {
        const longlong2 v = col[(size_t)__ldg(dnx + 2 * e) * S.Du];
        px += v.x;
        py += v.y;
    }
#pragma unroll 4
    for (int e = ds; e < d1; ++e) {
        const longlong2 v = col[(size_t)__ldg(dnx + 2 * e) * S.Du];
        nx += v.x;
        ny += v.y;
    }
    ix += px - nx;
    iy += py - ny;
}

__device__ __forceinline__ void stage_amplitudes(const SecView& S, double2* amp) {
    for (int k = threadIdx.x; k < S.L * S.L; k += blockDim.x) amp[k] = S.hamp[k];
    __syncthreads();
}

__global__ void __launch_bounds__(kThreads) k_diag_table(SecView S, double* diag) {
    __shared__ double utab[4 * 256];
    for (int k = threadIdx.x; k < S.nchunk * 256; k += blockDim.x) utab[k] = S.Utab[k];
    __syncthreads();
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < S.d; idx += gridDim.x * blockDim.x) {
        int i_dn, i_up;
        split_index(S, idx, i_dn, i_up);
        diag[idx] = diag_energy(S, i_dn, i_up, utab);
    }
}

int launch_diag_table(const SecView& S, double* diag, cudaStream_t st) {
    const int nb = std::max(1, std::min((S.d + kThreads - 1) / kThreads, 148 * 16));
    k_diag_table<<<nb, kThreads, 0, st>>>(S, diag);
    KG_LAUNCHED();
    return KG_OK;
}

// Per-string and per-byte tables of a sector with on-site offsets added:
// e_up'[i] = e_up[i] + sum over the set bits p of string i of dp[p] (spin up),
// e_dn' likewise with dp[L + p], U'[c][v] = U[c][v] + sum over the set bits
// b of byte v of dp[2L + 8c + b].  H is linear in eps and U, so the diagonal
// built from these tables is that of the offset Hamiltonian.
__global__ void k_drive_tables(SecView S, const double* dp, double* e_up, double* e_dn, double* utab) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < S.Du) {
        double acc = S.up_e[i];
        for (uint32_t b = S.up_bits[i]; b; b &= b - 1u) acc += dp[__ffs(b) - 1];
        e_up[i] = acc;
    }
    if (i < S.Dd) {
        double acc = S.dn_e[i];
        for (uint32_t b = S.dn_bits[i]; b; b &= b - 1u) acc += dp[S.L + __ffs(b) - 1];
        e_dn[i] = acc;
    }
    if (i < S.nchunk * 256) {
        const int c = i >> 8;
        double acc = S.Utab[i];
        for (uint32_t b = (uint32_t)(i & 255); b; b &= b - 1u) {
            const int site = 8 * c + __ffs(b) - 1;
            if (site < S.L) acc += dp[2 * S.L + site];
        }
        utab[i] = acc;
    }
}

size_t drive_work_doubles(const kg_sector* s) {
    return (size_t)s->d + (size_t)s->Du + (size_t)s->Dd + (size_t)s->nchunk * 256;
}

int launch_drive_diag(const SecView& S, const double* dp, double* work, cudaStream_t st) {
    double* e_up = work + S.d;
    double* e_dn = e_up + S.Du;
    double* utab = e_dn + S.Dd;
    const int n = std::max(std::max(S.Du, S.Dd), S.nchunk * 256);
    k_drive_tables<<<(n + 255) / 256, 256, 0, st>>>(S, dp, e_up, e_dn, utab);
    KG_LAUNCHED();
    SecView T = S;
    T.up_e = e_up;
    T.dn_e = e_dn;
    T.Utab = utab;
    return launch_diag_table(T, work, st);
}

// H*psi of uniform hopping takes three short kernels: the largest exponent of
// x, its fixed-point image, the hop sums.  Chained by programmatic dependent
// launch, and with one exponent per block for the next kernel to reduce
// instead of an atomic on a cleared word, 731,808 states take 34.8 us (39.4
// with a clear and plain launches).
// Largest exponent field over the components of x, one value per block.
__global__ void __launch_bounds__(kThreads) k_maxexp(const double2* __restrict__ x, int d, int* emax) {
    __shared__ int sm[kThreads / 32];
    int m = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < d; i += gridDim.x * blockDim.x) {
        const double2 v = x[i];
        m = max(m, max(exp_field(v.x), exp_field(v.y)));
    }
    chain_next();
    m = block_max_int(m, sm);
    if (threadIdx.x == 0) emax[blockIdx.x] = m;
}

// Fixed-point image of x on the largest of the n exponents of k_maxexp, which
// is left in emax[n] (for the exact hop sums).  Launched while k_maxexp ends:
// x itself is older than both.
__global__ void __launch_bounds__(kThreads) k_tofix(const double2* __restrict__ x, int d, int* emax, int n, int P,
                                                    longlong2* __restrict__ xf) {
    __shared__ int sm[kThreads / 32];
    const int i0 = blockIdx.x * blockDim.x + threadIdx.x;
    double2 v = make_double2(0.0, 0.0);
    if (i0 < d) v = x[i0];
    chain_wait();
    int m = 0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) m = max(m, emax[i]);
    const int E = block_max_all(m, sm);
    if (i0 == 0) emax[n] = E;
    for (int i = i0; i < d; i += gridDim.x * blockDim.x) {
        if (i != i0) v = x[i];
        xf[i] = make_longlong2(fix_term(v.x, E, P, 0u), fix_term(v.y, E, P, 0u));
    }
    chain_next();
}

// y = H x with the hop sums read from the fixed-point image xf of x.
__global__ void __launch_bounds__(kThreads) k_hpsi_pre(SecView S, const double2* __restrict__ x,
                                                       const longlong2* xf, double2* __restrict__ y,
                                                       const int* emax) {
    chain_wait();
    const int E = *emax;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < S.d; idx += gridDim.x * blockDim.x) {
        int i_dn, i_up;
        split_index(S, idx, i_dn, i_up);
        const double2 xv = x[idx];
        const double diag = __ldg(S.diag + idx);
        long long ix = 0, iy = 0;
        hop_sum_pre(S, xf, i_dn, i_up, ix, iy);
        y[idx] = make_double2(fma(diag, xv.x, S.h0 * fix_to_double(ix, E, S.fix_pre)),
                              fma(diag, xv.y, S.h0 * fix_to_double(iy, E, S.fix_pre)));
    }
}

template <int MODE>
__global__ void __launch_bounds__(kThreads) k_hpsi(SecView S, const double2* __restrict__ x,
                                                   double2* __restrict__ y, const int* emax) {
    __shared__ double2 amp[kMaxL * kMaxL];
    stage_amplitudes(S, amp);
    const int E = (MODE == 3) ? *emax : 0;
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < S.d; idx += gridDim.x * blockDim.x) {
        int i_dn, i_up;
        split_index(S, idx, i_dn, i_up);
        const double2 xv = x[idx];
        const double diag = __ldg(S.diag + idx);
        double2 hop = make_double2(0.0, 0.0);
        long long ix = 0, iy = 0;
        hop_sum<MODE>(S, x, i_dn, i_up, amp, E, hop, ix, iy);
        double2 r;
        if (MODE == 3) {
            r.x = fma(diag, xv.x, S.h0 * fix_to_double(ix, E, S.fix_pre));
            r.y = fma(diag, xv.y, S.h0 * fix_to_double(iy, E, S.fix_pre));
        } else if (MODE == 0) {
            r.x = fma(diag, xv.x, S.h0 * hop.x);
            r.y = fma(diag, xv.y, S.h0 * hop.y);
        } else {
            r.x = fma(diag, xv.x, hop.x);
            r.y = fma(diag, xv.y, hop.y);
        }
        y[idx] = r;
    }
}

// Lanczos step j for column b of a work-list launch:
//   w = s_j H V_j - b_j s_{j-1} V_{j-1},   a_j = Re <s_j V_j, w>
// (Eq. (recursion) with normalised v_k = s_k V_k).
//
// It starts by finishing what the update that made V_j left (resolve_norm),
// and leaves the partial sums of a_j to the kernel after it: a reduction by
// the reader costs one pass over a few hundred partials that every block does
// at once, where a last block to arrive would add a fence, an atomic and a
// serial tail to every launch.
struct HpsiShared {
    double2 amp[kMaxL * kMaxL];
    HeadShared head;
    SecView S;
};

template <int MODE>
__device__ __forceinline__ void lanczos_hpsi_item(const ColDesc* desc, ColScalars* cs, int j, const int4 it_,
                                                  HpsiShared& sh) {
    const int b = it_.x, blk = it_.y, nblk = it_.z;
    const ColDesc D = desc[b];
    ColScalars* C = cs + b;
    SecView& S = sh.S;
    double2* amp = sh.amp;
    {
        // the sector's view, word by word, and its amplitudes
        static_assert(sizeof(SecView) % 8 == 0, "SecView is copied in 8-byte words");
        const unsigned long long* src = reinterpret_cast<const unsigned long long*>(D.sec);
        for (int k = threadIdx.x; k < (int)(sizeof(SecView) / 8); k += blockDim.x)
            reinterpret_cast<unsigned long long*>(&S)[k] = src[k];
        if (MODE == 1 || MODE == 2) {
            const int n = D.sec->L * D.sec->L;
            const double2* ha = D.sec->hamp;
            for (int k = threadIdx.x; k < n; k += blockDim.x) amp[k] = ha[k];
        }
    }
    chain_wait();
    const bool writer = blk == 0 && threadIdx.x == 0;
    HeadShared& H = sh.head;
    if (j > 0) {
        resolve_norm(D, C, j, writer, H);
    } else {  // the start vector's norm is k_colnorm's
        if (threadIdx.x == 0) {
            H.m_eff = C->m_eff;
            H.scale = C->scale[0];
            H.emax = C->emax[0];
            H.cprev = 0.0;
        }
        __syncthreads();
    }
    if (j >= H.m_eff) return;
    const double sj = H.scale, cprev = H.cprev;
    const int E = (MODE == 3) ? H.emax : 0;
    const double hs = S.h0 * sj;
    // V_j in fixed point, written by the update that produced it (not V_0),
    // used when its exponent bound is tight enough
    const int Ef = C->efix;
    const bool pre = MODE == 3 && j > 0 && D.Xf != nullptr && Ef >= E && Ef - E <= kFixSlack;
    const double2* x = D.V + (size_t)j * D.d;
    const double2* xp = D.V + (size_t)(j > 0 ? j - 1 : 0) * D.d;
    const int E0img = C->eimg[0];
    double2* w = D.W;
    double acc = 0.0;
    int ew = 0;
    KG_FOR(idx) {
        int i_dn, i_up;
        split_index(S, idx, i_dn, i_up);
        const double2 xv = x[idx];
        const double sdiag = sj * __ldg(S.diag + idx);
        double2 hop = make_double2(0.0, 0.0);
        long long ix = 0, iy = 0;
        const int Eu = pre ? Ef : E;
        if (MODE == 3 && pre)
            hop_sum_pre(S, D.Xf, i_dn, i_up, ix, iy);
        else
            hop_sum<MODE>(S, x, i_dn, i_up, amp, E, hop, ix, iy);
        double2 p = make_double2(0.0, 0.0);
        if (j > 0) p = xp[idx];
        double2 r;
        if (MODE == 3) {
            r.x = fma(sdiag, xv.x, fma(hs, fix_to_double(ix, Eu, S.fix_pre), -cprev * p.x));
            r.y = fma(sdiag, xv.y, fma(hs, fix_to_double(iy, Eu, S.fix_pre), -cprev * p.y));
        } else if (MODE == 0) {
            r.x = fma(sdiag, xv.x, fma(hs, hop.x, -cprev * p.x));
            r.y = fma(sdiag, xv.y, fma(hs, hop.y, -cprev * p.y));
        } else {
            r.x = fma(sdiag, xv.x, fma(sj, hop.x, -cprev * p.x));
            r.y = fma(sdiag, xv.y, fma(sj, hop.y, -cprev * p.y));
        }
        w[idx] = r;
        if (j == 0 && D.I) D.I[idx] = fix_image(xv, E0img);  // image of V_0 for the exact dots
        acc = fma(xv.x, r.x, fma(xv.y, r.y, acc));  // Re conj(x) r
        ew = max(ew, max(exp_field(r.x), exp_field(r.y)));
    }
    chain_next();
    block_partial(sj * acc, ew, sh.head.sum, D.part_a + blk);
    if (writer) C->n_alpha = nblk;
}

// One item per block (one-wave work lists, batches of any mix of sizes).
template <int MODE>
__global__ void __launch_bounds__(kThreads, 4) k_lanczos_hpsi(const ColDesc* desc, const int4* items, ColScalars* cs,
                                                           int j) {
    __shared__ HpsiShared sh;
    lanczos_hpsi_item<MODE>(desc, cs, j, items[blockIdx.x], sh);
}

int launch_hpsi(kg_sector* s, const double2* x, double2* y, cudaStream_t st) {
    const SecView S = s->view();
    const int nb = std::max(1, std::min((S.d + kThreads - 1) / kThreads, s->nsm * 8));
    if (S.hopmode == 0 && S.fix_pre >= 0) {
        // largest exponent of x, the fixed-point image of x on it, then exact
        // hop sums that add the image's integers.  The scratch belongs to the
        // sector (allocated once, on the first call), so calls with one
        // sector must be ordered, like every use of a handle.
        const int nmax = std::min(nb, s->nsm * 4);
        if (!s->hp_xf) {
            if (cudaMalloc(&s->hp_emax, sizeof(int) * (size_t)(nmax + 1)) != cudaSuccess ||
                cudaMalloc(&s->hp_xf, sizeof(longlong2) * (size_t)S.d) != cudaSuccess) {
                cudaGetLastError();
                cudaFree(s->hp_emax);
                s->hp_emax = nullptr;
                s->hp_xf = nullptr;
                set_error("H*psi scratch of %d elements", S.d);
                return KG_ENOMEM;
            }
        }
        ProfScope ps("hpsi", st);
        k_maxexp<<<nmax, kThreads, 0, st>>>(x, S.d, s->hp_emax);
        KG_LAUNCHED();
        KG_TRY(launch_chained(k_tofix, nb, kThreads, 0, st, x, S.d, s->hp_emax, nmax, S.fix_pre, s->hp_xf));
        return launch_chained(k_hpsi_pre, nb, kThreads, 0, st, S, x, s->hp_xf, y, s->hp_emax + nmax);
    }
    ProfScope ps("hpsi", st);
    if (S.hopmode == 0)
        k_hpsi<0><<<nb, kThreads, 0, st>>>(S, x, y, nullptr);
    else if (S.hopmode == 1)
        k_hpsi<1><<<nb, kThreads, 0, st>>>(S, x, y, nullptr);
    else
        k_hpsi<2><<<nb, kThreads, 0, st>>>(S, x, y, nullptr);
    KG_LAUNCHED();
    return KG_OK;
}

int prepare_hpsi_lists(Krylov& K) {
    bool present[4] = {false, false, false, false};
    for (auto& D : K.hdesc) present[D.mode] = true;
    const void* kerns[4] = {(const void*)k_lanczos_hpsi<0>, (const void*)k_lanczos_hpsi<1>,
                            (const void*)k_lanczos_hpsi<2>, (const void*)k_lanczos_hpsi<3>};
    for (int mode = 0; mode < 4; ++mode) {
        if (!present[mode]) continue;
        const int4* items;
        int n;
        for (int g = 0; g < K.ngroups[mode]; ++g) KG_TRY(work_list(K, kerns[mode], mode, &items, &n, g));
    }
    return KG_OK;
}

int launch_lanczos_hpsi(Krylov& K, int j, cudaStream_t st) {
    bool present[4] = {false, false, false, false};
    for (auto& D : K.hdesc) present[D.mode] = true;
    ProfScope ps("lanczos_hpsi", st);
    for (int mode = 0; mode < 4; ++mode) {
        if (!present[mode]) continue;
        const void* kern = mode == 3   ? (const void*)k_lanczos_hpsi<3>
                           : mode == 0 ? (const void*)k_lanczos_hpsi<0>
                           : mode == 1 ? (const void*)k_lanczos_hpsi<1>
                                       : (const void*)k_lanczos_hpsi<2>;
        const int4* items;
        int n;
        // one launch per group of columns whose gathered vectors fit in L2
        for (int g = 0; g < K.ngroups[mode]; ++g) {
            KG_TRY(work_list(K, kern, mode, &items, &n, g));
            const auto k = mode == 3 ? &k_lanczos_hpsi<3> : mode == 0 ? &k_lanczos_hpsi<0> : mode == 1 ? &k_lanczos_hpsi<1>
                                                                                                       : &k_lanczos_hpsi<2>;
            KG_TRY(launch_chained(k, n, kThreads, 0, st, K.desc, items, K.cs, j));
        }
    }
    return KG_OK;
}

}  // namespace kg
