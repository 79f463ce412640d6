// kg_small.cu -- a whole Krylov step of a small column in one launch.
//
// The streaming kernels of kg_hpsi.cu and kg_krylov.cu take three launches
// per Lanczos vector.  On a column of a few thousand states each of them is
// nothing but latency (launch, descriptor, reduction), and the FP64 pipe of
// the few SMs that a short launch reaches.  Here one thread-block cluster owns
// the column for the whole step: the blocks split its elements, keep the
// fixed-point images of their part of every Lanczos vector in shared memory
// and meet at the cluster's hardware barrier, three times per vector:
//
//   w = s_j H V_j - b_j s_{j-1} V_{j-1}, partial sums of a_j = <v_j, w>    | 1
//   u = w - a_j v_j, its image, exact dots h_k = <v_k, u>, k <= j           | 2
//   V_{j+1} = u - sum_k h_k v_k, its image, partial sums of its norm        | 3
//
// the recursion of Eq. (recursion) with the Gram-Schmidt pass of the
// streaming kernels, then the step exponential (Eq. (udelta)), the combination
// and the overlaps.  Partial sums go straight into the shared memory of every
// block of the cluster, which all add them up in the same order: no atomics,
// no polling, the same bits in every block.
//
// Arithmetic.  FP64 issues about two lanes per clock per SM here, integer
// multiply-adds about fifty, so every sum over elements is an integer sum:
// vectors are held as 56-bit fixed-point images on a bound of their largest
// exponent, split into 28-bit halves, and dots, norms and hop sums are exact
// sums of products of halves (32 x 32 -> 64 bit multiply-adds).  Hop
// amplitudes have such images too, so that real and complex hoppings cost 8
// and 16 integer multiply-adds per hop instead of 2 and 4 FP64 ones.  FP64 is
// left with about 11 operations per element and vector.
//
// Measured, one step: 300 states at M = 40 (two columns, clusters of 4) 330 us
// against 1,030 us by the streaming kernels; 4,900 states with complex hopping
// at M = 20 (cluster of 16) 340 against 690 us; 3,920 states on the chain 245
// against 550 us.  What bounds it is latency: about 8 us per Lanczos vector,
// of which the hop gathers take 1.5 (star) to 7 us (32 complex hops), the
// three barriers 1.1, the scalars 1.5.
#include <algorithm>
#include <array>
#include <map>
#include <mutex>
#include <type_traits>

#include "kg_internal.h"

namespace kg {

constexpr int kSmWarps = 15;                     // warps that own elements
constexpr int kSmOwn = 32 * kSmWarps;            // threads that own elements
constexpr int kSmThreads = kSmOwn + 32;          // and one warp for the column's scalars
constexpr int kSmMaxEpt = 2;                     // elements per thread
constexpr int kSmBatch = 8;                      // hops whose gathers are in flight together
constexpr int kSmSlack = 3;                      // bits an image's exponent bound may be loose
constexpr int kSmMaxCluster = 16;
constexpr size_t kSmSmem = 220 * 1024;           // dynamic shared memory a block may take

// Offsets of a block's dynamic shared memory.
struct SmallLayout {
    unsigned img, ua, amp, dots, sa, sn, up_off, dn_off, up_ent, dn_ent, scal, total;
};

__host__ __device__ inline SmallLayout small_layout(int M, int n_own, int C, int L, int mode, int Du, int Dd,
                                                    long long nnz) {
    SmallLayout o;
    unsigned at = 0;
    auto take = [&](long long bytes) {
        const unsigned a = at;
        at += (unsigned)((bytes + 15) & ~15ll);
        return a;
    };
    o.img = take(std::max(16ll * (M + 1) * n_own, 8ll * kSmWarps * (2 * kMaxOv + 2)));
    o.ua = take(16ll * n_own);
    o.amp = take(mode == 1 || mode == 2 ? 16ll * L * L : 0);
    o.dots = take(std::max(32ll * M * C, 8ll * C * (2 * kMaxOv + 2)));
    o.sa = take(16ll * C * kSmWarps);
    o.sn = take(16ll * C * kSmWarps);
    o.up_off = take(4ll * (Du + 1));
    o.dn_off = take(4ll * (Dd + 1));
    o.up_ent = take(4 * nnz);  // both spins' entries, up first
    o.dn_ent = o.up_ent;
    o.scal = take(64ll * (M + 2));
    o.total = at;
    return o;
}

// ------------------------------------------------------- cluster helpers
__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cluster_size() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
// Barrier of the cluster; shared, distributed shared and global writes before
// it are visible to the cluster's threads after it.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() {
    cluster_arrive();
    cluster_wait();
}
__device__ __forceinline__ void remote_store(const void* p, unsigned rank, unsigned long long a, unsigned long long b) {
    unsigned addr;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(smem_addr(p)), "r"(rank));
    asm volatile("st.shared::cluster.v2.b64 [%0], {%1, %2};" ::"r"(addr), "l"(a), "l"(b) : "memory");
}

__device__ __forceinline__ void remote_store(const double* p, unsigned rank, double v) {
    unsigned addr;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(smem_addr(p)), "r"(rank));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}

// ------------------------------------------------------ 28-bit halves
constexpr long long kM28 = (1ll << 28) - 1;

__device__ __forceinline__ int4 fix56(double2 u, int E) {  // round(x 2^(1078 - E)), halves hi 2^28 + lo
    const long long x = fix_term(u.x, E, 3, 0u), y = fix_term(u.y, E, 3, 0u);
    return make_int4((int)(x >> 28), (int)(x & kM28), (int)(y >> 28), (int)(y & kM28));
}

// A sum of products of halves: s0 2^56 + (s1 + t1) 2^28 + s2.  A wide
// multiply-add takes 28 cycles to the next one on the same sum, hence two
// sums of the cross terms.
struct Sum3 {
    long long s0 = 0, s1 = 0, t1 = 0, s2 = 0;
    __device__ __forceinline__ void add(int ah, int al, int bh, int bl) {
        s0 += (long long)ah * bh;
        s1 += (long long)ah * bl;
        t1 += (long long)al * bh;
        s2 += (long long)al * bl;
    }
    __device__ __forceinline__ void fold() {  // the carries, so that many more products fit
        s1 += t1 + (s2 >> 28);
        t1 = 0;
        s2 &= kM28;
        s0 += s1 >> 28;
        s1 &= kM28;
    }
    __device__ __forceinline__ long long top() const {  // rounded to units of 2^56
        return s0 + ((s1 + t1 + (s2 >> 28) + (1ll << 27)) >> 28);
    }
};

// conj(v) u
__device__ __forceinline__ void cdot_halves(const int4 v, const int4 u, Sum3& re, Sum3& im) {
    re.add(v.x, v.y, u.x, u.y);
    re.add(v.z, v.w, u.z, u.w);
    im.add(v.x, v.y, u.z, u.w);
    im.add(v.z, v.w, -u.x, -u.y);
}

// The warp's sum in units of 2^28 as two limbs, l1 2^46 + l0 (l0 < 2^46).
__device__ __forceinline__ void sum3_limbs(const Sum3& t, unsigned long long& l0, unsigned long long& l1) {
    constexpr unsigned m26 = (1u << 26) - 1u;
    const long long mid = t.s1 + t.t1 + (t.s2 >> 28), hi = t.s0 + (mid >> 28);
    // hi 2^28 + (mid mod 2^28) in pieces of 26 bits, the top one signed
    const unsigned long long low = (unsigned long long)(mid & kM28) | (unsigned long long)(hi & ((1ll << 34) - 1)) << 28;
    const long long high = hi >> 34;  // units of 2^62
    const unsigned q2 = (unsigned)(low >> 52) | ((unsigned)(high & 0xffff) << 10);
    const unsigned s0 = __reduce_add_sync(0xffffffffu, (unsigned)low & m26);
    const unsigned s1 = __reduce_add_sync(0xffffffffu, (unsigned)(low >> 26) & m26);
    const unsigned s2 = __reduce_add_sync(0xffffffffu, q2);
    const int s3 = __reduce_add_sync(0xffffffffu, (int)(high >> 16));
    const unsigned long long a = (unsigned long long)s0 + ((unsigned long long)s1 << 26);
    const long long b = (long long)s2 + ((long long)s3 << 26);
    l0 = a & ((1ull << 46) - 1ull);
    l1 = (unsigned long long)((b << 6) + (long long)(a >> 46));
}

__device__ __forceinline__ double limbs_value(unsigned long long l0, unsigned long long l1) {
    const long long hi = (long long)l1 + (long long)(l0 >> 46);
    return fma((double)hi, 0x1p46, (double)(l0 & ((1ull << 46) - 1ull)));
}

// Sum over n slots {l0 | e << 48, l1} by one warp: limbs and the largest e.
// (l0 < 2^46 per slot, at most 2^8 slots: pieces of 27 bits, then warp sums.)
__device__ __forceinline__ void sum_slots(const ulonglong2* slot, int n, unsigned long long& l0, unsigned long long& l1,
                                          int& e) {
    unsigned long long a = 0, b = 0;
    e = 0;
    for (int i = threadIdx.x & 31; i < n; i += 32) {
        const ulonglong2 v = slot[i];
        a += v.x & ((1ull << 48) - 1ull);
        b += v.y;
        e = max(e, (int)(v.x >> 48));
    }
    constexpr unsigned m27 = (1u << 27) - 1u;
    const unsigned a0 = __reduce_add_sync(0xffffffffu, (unsigned)a & m27);
    const unsigned a1 = __reduce_add_sync(0xffffffffu, (unsigned)(a >> 27));
    const unsigned b0 = __reduce_add_sync(0xffffffffu, (unsigned)b & m27);
    const unsigned b1 = __reduce_add_sync(0xffffffffu, (unsigned)(b >> 27) & m27);
    const unsigned b2 = __reduce_add_sync(0xffffffffu, (unsigned)(b >> 54));
    e = __reduce_max_sync(0xffffffffu, e);
    l0 = (unsigned long long)a0 + ((unsigned long long)a1 << 27);
    l1 = (unsigned long long)b0 + ((unsigned long long)b1 << 27) + ((unsigned long long)b2 << 54);
}

// What the scalar warp tells the block.
struct SmallShared {
    SecView S;
    double sj, cprev, aj, araw, hre;
    float r0;
    int Ew, Eu, Ef, m_eff, status, loose, n32, n64, ec;
    int any64[8], eh[8];  // per warp of coefficients
    int E0, Ed, Ea;
};

// ---------------------------------------------------------------- kernel
// finish: 0 the Lanczos space only, 1 the whole step.
template <int EPT>
__global__ void __launch_bounds__(kSmThreads, 1) k_small_step(const ColDesc* desc, const int* cols, ColScalars* cs,
                                                              int M, int finish) {
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ SmallShared sh;
    // a block's shared memory may be written by another block only once it has
    // started: waited for before the first remote_store
    cluster_arrive();
    const int C = (int)cluster_size(), rank = (int)cluster_rank();
    const int b = cols[blockIdx.x / C];
    const ColDesc D = desc[b];
    ColScalars* Cs = cs + b;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool owner = warp < kSmWarps, scalar = warp == kSmWarps;
    const int d = D.d, mode = D.mode == 3 ? 0 : D.mode;
    const int n_own = (d + C - 1) / C, e0 = rank * n_own, n = max(0, min(n_own, d - e0));
    const int nw = min(kSmWarps, (n_own + 31) / 32), ns = C * nw;  // warps with elements, slots of a sum
    const bool posts = warp < nw;
    {
        const unsigned long long* src = reinterpret_cast<const unsigned long long*>(D.sec);
        for (int k = tid; k < (int)(sizeof(SecView) / 8); k += kSmThreads)
            reinterpret_cast<unsigned long long*>(&sh.S)[k] = src[k];
    }
    __syncthreads();
    const SecView& S = sh.S;
    const int Du = S.Du, Dd = S.Dd, nnz_up = S.up_off[Du], nnz_dn = S.dn_off[Dd];
    const SmallLayout lay = small_layout(M, n_own, C, S.L, mode, Du, Dd, (long long)nnz_up + nnz_dn);
    int4* const img = reinterpret_cast<int4*>(dyn + lay.img);  // [M + 1][n_own]
    int4* const ua = reinterpret_cast<int4*>(dyn + lay.ua);
    int4* const amp = reinterpret_cast<int4*>(dyn + lay.amp);
    ulonglong2* const dots = reinterpret_cast<ulonglong2*>(dyn + lay.dots);  // [block][re, im][M]
    ulonglong2* const sa = reinterpret_cast<ulonglong2*>(dyn + lay.sa);
    ulonglong2* const sn = reinterpret_cast<ulonglong2*>(dyn + lay.sn);
    int* const up_off = reinterpret_cast<int*>(dyn + lay.up_off);
    int* const dn_off = reinterpret_cast<int*>(dyn + lay.dn_off);
    unsigned* const up_ent = reinterpret_cast<unsigned*>(dyn + lay.up_ent);
    unsigned* const dn_ent = up_ent + nnz_up;
    double2* const coef64 = reinterpret_cast<double2*>(dyn + lay.scal);  // [M + 2] each
    double* const alpha = reinterpret_cast<double*>(coef64 + (M + 2));
    double* const beta = alpha + (M + 2);
    double* const scale = beta + (M + 2);
    float2* const coef32 = reinterpret_cast<float2*>(scale + (M + 2));
    int* const emax = reinterpret_cast<int*>(coef32 + (M + 2));
    int* const eimg = emax + (M + 2);
    short* const idx32 = reinterpret_cast<short*>(eimg + (M + 2));
    short* const idx64 = idx32 + (M + 2);
    double2* const V = D.V;
    // hop tables: source rank | amplitude index << 16 | sign << 31
    for (int k = tid; k <= Du; k += kSmThreads) up_off[k] = S.up_off[k];
    for (int k = tid; k <= Dd; k += kSmThreads) dn_off[k] = S.dn_off[k];
    auto pack = [](uint2 en) { return en.x | ((en.y & 1023u) << 16) | (en.y & 0x80000000u); };
    for (int k = tid; k < nnz_up; k += kSmThreads) up_ent[k] = pack(S.up_ent[k]);
    for (int k = tid; k < nnz_dn; k += kSmThreads) dn_ent[k] = pack(S.dn_ent[k]);
    if (scalar && mode != 0) {  // amplitudes on the largest of their exponents
        const int LL = S.L * S.L;
        int e = 0;
        for (int k = lane; k < LL; k += 32)
            if (k / S.L != k % S.L) e = max(e, max(exp_field(S.hamp[k].x), exp_field(S.hamp[k].y)));
        e = __reduce_max_sync(0xffffffffu, e);
        for (int k = lane; k < LL; k += 32)
            amp[k] = k / S.L != k % S.L ? fix56(S.hamp[k], e) : make_int4(0, 0, 0, 0);
        if (lane == 0) sh.Ea = e;
    } else if (scalar && lane == 0) {
        sh.Ea = exp_field(S.h0);
    }
    // ---- the start vector: exponent, image, norm
    double2 x[EPT], p[EPT], w[EPT];
    double dg[EPT];
    int em = 0, ed = 0;
#pragma unroll
    for (int q = 0; q < EPT; ++q) {
        x[q] = p[q] = w[q] = make_double2(0.0, 0.0);
        dg[q] = 0.0;
        const int i = tid + q * kSmOwn;
        if (owner && i < n) {
            x[q] = V[e0 + i];
            dg[q] = S.diag[e0 + i];
            em = max(em, max(exp_field(x[q].x), exp_field(x[q].y)));
            ed = max(ed, exp_field(dg[q]));
        }
    }
    cluster_wait();  // every block of the cluster runs
    if (posts) {
        em = __reduce_max_sync(0xffffffffu, em);
        ed = __reduce_max_sync(0xffffffffu, ed);
        if (lane < C)
            remote_store(sa + rank * nw + warp, lane, (unsigned long long)em << 48, (unsigned long long)ed);
    }
    cluster_sync();
    if (scalar) {
        int a = 0, c = 0;
        for (int i = lane; i < ns; i += 32) {
            a = max(a, (int)(sa[i].x >> 48));
            c = max(c, (int)sa[i].y);
        }
        a = __reduce_max_sync(0xffffffffu, a);
        c = __reduce_max_sync(0xffffffffu, c);
        if (lane == 0) {
            sh.E0 = a;
            sh.Ed = c;
            sh.status = KG_OK;
            sh.m_eff = M;
            sh.araw = sh.hre = 0.0;
            eimg[0] = a;
        }
    }
    __syncthreads();
    // the image of x (this thread's elements) on exponent E, as vector k
    auto store_image = [&](int k, const double2 (&v)[EPT], int E, bool norm) {
        Sum3 t;
        int e = 0;
#pragma unroll
        for (int q = 0; q < EPT; ++q) {
            const int i = tid + q * kSmOwn;
            if (owner && i < n) {
                const int4 f = fix56(v[q], E);
                img[(size_t)k * n_own + i] = f;
                D.Xs[e0 + i] = f;
                t.add(f.x, f.y, f.x, f.y);
                t.add(f.z, f.w, f.z, f.w);
                e = max(e, max(exp_field(v[q].x), exp_field(v[q].y)));
            }
        }
        if (posts && norm) {
            unsigned long long l0, l1;
            sum3_limbs(t, l0, l1);
            e = __reduce_max_sync(0xffffffffu, e);
            if (lane < C) remote_store(sn + rank * nw + warp, lane, l0 | (unsigned long long)e << 48, l1);
        }
    };
    store_image(0, x, sh.E0, true);
    cluster_sync();
    // hop part of H V_j at this thread's elements, in the units of hop_value
    long long hx[EPT], hy[EPT];
    auto hop_sums = [&]() {
#pragma unroll
        for (int q = 0; q < EPT; ++q) {
            hx[q] = hy[q] = 0;
            const int i = tid + q * kSmOwn;
            if (!owner || i >= n) continue;
            int i_dn, i_up;
            split_index(S, e0 + i, i_dn, i_up);
            // both spins' hops as one list, in batches whose gathers are all in flight
            const int u0 = up_off[i_up], nu = up_off[i_up + 1] - u0, d0 = dn_off[i_dn], nh = nu + dn_off[i_dn + 1] - d0;
            const int4 *row = D.Xs + i_dn * Du, *col = D.Xs + i_up;
            Sum3 tx, ty;
            auto batch = [&](auto size, int c0, auto&& use) {
                constexpr int NB = decltype(size)::value;
                int4 v[NB];
                unsigned en[NB];
#pragma unroll
                for (int r = 0; r < NB; ++r) {
                    const int e = c0 + r;
                    v[r] = make_int4(0, 0, 0, 0);
                    en[r] = 0;
                    if (e < nu) {
                        en[r] = up_ent[u0 + e];
                        v[r] = row[en[r] & 0xffffu];
                    } else if (e < nh) {
                        en[r] = dn_ent[d0 + e - nu];
                        v[r] = col[(int)(en[r] & 0xffffu) * Du];
                    }
                }
#pragma unroll
                for (int r = 0; r < NB; ++r) use(v[r], en[r]);
            };
            if (mode == 0) {
                for (int c0 = 0; c0 < nh; c0 += kSmBatch)
                    batch(std::integral_constant<int, kSmBatch>(), c0, [&](const int4 v, unsigned en) {
                        const int sg = 1 - 2 * (int)(en >> 31);
                        tx.s0 += (long long)v.x * sg;
                        tx.s1 += (long long)v.y * sg;
                        ty.s0 += (long long)v.z * sg;
                        ty.s1 += (long long)v.w * sg;
                    });
            } else if (mode == 1) {
                for (int c0 = 0; c0 < nh; c0 += kSmBatch) {
                    batch(std::integral_constant<int, kSmBatch>(), c0, [&](const int4 v, unsigned en) {
                        const int4 a = amp[(en >> 16) & 1023u];
                        const int sg = 1 - 2 * (int)(en >> 31), ah = a.x * sg, al = a.y * sg;
                        tx.add(v.x, v.y, ah, al);
                        ty.add(v.z, v.w, ah, al);
                    });
                    tx.fold();
                    ty.fold();
                }
            } else {
                for (int c0 = 0; c0 < nh; c0 += kSmBatch / 2) {
                    batch(std::integral_constant<int, kSmBatch / 2>(), c0, [&](const int4 v, unsigned en) {
                        const int4 a = amp[(en >> 16) & 1023u];
                        const int sg = 1 - 2 * (int)(en >> 31);
                        const int ah = a.x * sg, al = a.y * sg, bh = a.z * sg, bl = a.w * sg;
                        tx.add(v.x, v.y, ah, al);
                        tx.add(v.z, v.w, -bh, -bl);
                        ty.add(v.z, v.w, ah, al);
                        ty.add(v.x, v.y, bh, bl);
                    });
                    tx.fold();
                    ty.fold();
                }
            }
            hx[q] = mode == 0 ? (tx.s0 << 28) + tx.s1 : tx.top();
            hy[q] = mode == 0 ? (ty.s0 << 28) + ty.s1 : ty.top();
        }
    };
    // by the scalar warp: what the sums over V_j say (b_j, s_j, a_{j-1}, breakdown);
    // what the others wait for first, the rest by resolve_rest
    double q_n2 = 0.0, q_rs = 0.0, q_a = 0.0, q_ref = 0.0;
    int q_e = 0;
    // a_{j-1} and the breakdown threshold, as soon as the dots are in
    auto resolve_alpha_j = [&](int j) {
        q_a = sh.araw + sh.hre;
        q_ref = 1e-12 * fmax(fabs(q_a) + (j > 1 ? beta[j - 1] : 0.0), 1e-300);
    };
    auto resolve = [&](int j) {
        unsigned long long l0, l1;
        int e;
        const double sprev = j > 0 ? scale[j - 1] : 0.0;
        sum_slots(sn, ns, l0, l1, e);
        const int E = eimg[j];
        const bool bad = e == 2047;  // images of a non-finite vector mean nothing
        // n2 = b_j^2 2^(2128 - 2 E)
        const double n2 = limbs_value(l0, l1);
        const bool some = n2 > 0.0 && !bad;
        const double rs = some ? rsqrt3(n2) : 0.0;
        const double b = mul_pow2(n2 * rs, E - 1064), sj = mul_pow2(rs, 1064 - E);
        // norms of 2^512 and above, whose squares FP64 does not hold, are refused as
        // by the streaming kernels: products of two scales would leave its range
        const bool fin = !bad && exp_field(b) < 1023 + 512 && (j == 0 || exp_field(q_a) != 2047);
        int m = M;
        // happy breakdown: K_j is invariant (positive doubles compare like their bits)
        if (j == 0 ? !some : __double_as_longlong(b) <= __double_as_longlong(q_ref)) m = j;
        if (!fin) m = min(m, j);
        const double cp = b * sprev;
        if (lane == 0) {
            if (!fin) sh.status = KG_ENUMERIC;
            sh.m_eff = m;
            sh.loose = E - e > kSmSlack && e > 0 && !bad;
            sh.sj = sj;
            sh.cprev = cp;
            // |w_i| <= s_j (|diag| + sum |h|) 2^(E_j - 1022) + c 2^(E_{j-1} - 1022), at most 60 hops
            const int e1 = e + exp_field(sj) - 2044 + max(sh.Ed, sh.Ea + 7) + 1;
            const int e2 = j > 0 ? exp_field(cp) - 1022 + emax[j - 1] : 0;
            sh.Ew = max(e1, e2) + 1;
            emax[j] = e;
            scale[j] = sj;
        }
        q_n2 = n2;
        q_rs = rs;
        q_e = E;
    };
    double fa = 0.0, faj = 0.0;
    auto resolve_rest = [&](int j) {
        const double b = q_rs != 0.0 ? sqrt_from(q_n2, q_rs) : 0.0;
        if (lane == 0) {
            if (j > 0) alpha[j - 1] = q_a;
            beta[j] = mul_pow2(b, q_e - 1064);  // beta[0]: ||V_0||
        }
        // <v_j, w> = s_j 2^(E_j + E_w - 2128) times its integer sum
        fa = mul_pow2(sh.sj, q_e + sh.Ew - 2128);
        faj = sh.sj * fa;
    };
    int j = 0;
    for (;; ++j) {
        // ---- w and the sums of a_j
        for (;;) {
            if (scalar) resolve(j);
            else if (j < M) hop_sums();
            __syncthreads();
            if (!sh.loose) break;
            // near a breakdown: V_j's image and norm again, on its own exponent
            cluster_sync();
            const int E = emax[j];
            if (tid == 0) eimg[j] = E;
            store_image(j, x, E, true);
            cluster_sync();
        }
        if (scalar) resolve_rest(j);
        if (j == M || j >= sh.m_eff) break;
        {
            const int E = eimg[j], Ew = sh.Ew;
            const double sj = sh.sj, cprev = sh.cprev, hs = mode == 0 ? S.h0 * sj : sj;
            const int Eh = mode == 0 ? E : E + sh.Ea - 1025, Ph = mode == 0 ? 3 : 0;
            Sum3 t;
            int ew = 0;
#pragma unroll
            for (int q = 0; q < EPT; ++q) {
                const int i = tid + q * kSmOwn;
                if (!owner || i >= n) continue;
                const double sd = sj * dg[q];
                w[q].x = fma(sd, x[q].x, fma(hs, fix_to_double(hx[q], Eh, Ph), -cprev * p[q].x));
                w[q].y = fma(sd, x[q].y, fma(hs, fix_to_double(hy[q], Eh, Ph), -cprev * p[q].y));
                const int4 f = fix56(w[q], Ew), v = img[(size_t)j * n_own + i];
                t.add(v.x, v.y, f.x, f.y);
                t.add(v.z, v.w, f.z, f.w);
                ew = max(ew, max(exp_field(w[q].x), exp_field(w[q].y)));
            }
            if (posts) {
                unsigned long long l0, l1;
                sum3_limbs(t, l0, l1);
                ew = __reduce_max_sync(0xffffffffu, ew);
                if (lane < C) remote_store(sa + rank * nw + warp, lane, l0 | (unsigned long long)ew << 48, l1);
            }
        }
        cluster_sync();
        // ---- u = w - a_j v_j and the exact dots
        if (scalar) {
            unsigned long long l0, l1;
            int ew;
            sum_slots(sa, ns, l0, l1, ew);
            const double t = ew == 2047 ? nan("") : limbs_value(l0, l1);
            const double aj = faj * t;
            if (lane == 0) {
                sh.aj = aj;
                sh.araw = fa * t;
                sh.Ew = ew;
                sh.Eu = max(ew, exp_field(aj) - 1022 + emax[j]) + 1;
                // V_{j+1} before its Gram-Schmidt terms is below r0 2^(E_w - 1022)
                sh.r0 = 1.0f + scaled_abs(aj, emax[j] - ew);
            }
        }
        __syncthreads();
        {
            const double aj = sh.aj;
            const int Eu = sh.Eu;
#pragma unroll
            for (int q = 0; q < EPT; ++q) {
                const int i = tid + q * kSmOwn;
                if (!owner || i >= n) continue;
                w[q].x = fma(-aj, x[q].x, w[q].x);
                w[q].y = fma(-aj, x[q].y, w[q].y);
                ua[i] = fix56(w[q], Eu);
            }
        }
        __syncthreads();
        // G lanes per vector, so that the block's threads cover all of them at once:
        // their sums over this block's elements go to every block
        {
            const int nk = j + 1;
            const int G = nk <= 16 ? 32 : (nk <= 32 ? 16 : 8);
            for (int k = tid / G; k - lane / G < nk; k += kSmThreads / G) {  // warp-uniform trip count
                const int g = tid & (G - 1);
                Sum3 tr, ti;
                if (k < nk) {
                    const int4* row = img + (size_t)k * n_own;
                    for (int i0 = g; i0 < n; i0 += 16 * G) {
                        const int i1 = min(n, i0 + 16 * G);
#pragma unroll 4
                        for (int i = i0; i < i1; i += G) cdot_halves(row[i], ua[i], tr, ti);
                        tr.fold();
                        ti.fold();
                    }
                }
                unsigned long long r0 = (unsigned long long)((tr.s0 & 0x3ffffll) << 28 | tr.s1), r1 = (unsigned long long)(tr.s0 >> 18);
                unsigned long long q0 = (unsigned long long)((ti.s0 & 0x3ffffll) << 28 | ti.s1), q1 = (unsigned long long)(ti.s0 >> 18);
                for (int o = G / 2; o > 0; o >>= 1) {
                    r0 += __shfl_xor_sync(0xffffffffu, r0, o);
                    r1 += __shfl_xor_sync(0xffffffffu, r1, o);
                    q0 += __shfl_xor_sync(0xffffffffu, q0, o);
                    q1 += __shfl_xor_sync(0xffffffffu, q1, o);
                }
                if (k < nk)
                    for (int c = g; c < C; c += G) {
                        remote_store(dots + (2 * rank) * M + k, c, r0, r1);
                        remote_store(dots + (2 * rank + 1) * M + k, c, q0, q1);
                    }
            }
        }
        cluster_sync();
        // ---- the Gram-Schmidt coefficients, one thread per vector: FP32 factors on
        // the upper halves of the images, the (rare) larger ones kept in FP64
        if (warp <= j / 32) {
            const int k = tid;
            int eh = 0;
            bool big = false;
            if (k <= j) {
                unsigned long long r0 = 0, r1 = 0, i0 = 0, i1 = 0;
                const double s = scale[k];
                const int Ek = eimg[k];
#pragma unroll 4
                for (int q = 0; q < C; ++q) {
                    const ulonglong2 re = dots[2 * q * M + k], im = dots[(2 * q + 1) * M + k];
                    r0 += re.x;
                    r1 += re.y;
                    i0 += im.x;
                    i1 += im.y;
                }
                // h_k = f times the integer sums; c_k = s_k h_k; x = hi 2^(E_k - 1050)
                const double f = mul_pow2(s, Ek + sh.Eu - 2128), fc = s * f, f32 = mul_pow2(fc, Ek - 1050);
                const double vr = limbs_value(r0, r1), vi = limbs_value(i0, i1);
                const double hx = f * vr, hy = f * vi;
                if (k == j) sh.hre = hx;
                // in FP64 also where the term or its factor on the upper halves (28 bits
                // below) could vanish, below 2^-126, while the term counts beside w
                // (above 2^-64 of it)
                big = !(scaled_abs(hx, 0) + scaled_abs(hy, 0) < (float)kSmallCoef) || sh.Ew < 988;
                coef32[k] = big ? make_float2(0.f, 0.f) : make_float2(f64_to_f32_near(f32 * vr), f64_to_f32_near(f32 * vi));
                coef64[k] = make_double2(big ? fc * vr : 0.0, big ? fc * vi : 0.0);
                // |c_k V_k| < 2^(eh - 1022)
                eh = max(exp_field(hx), exp_field(hy)) + exp_field(s) - 2044 + emax[k] + 3;
            }
            const unsigned any = __ballot_sync(0xffffffffu, big);
            eh = __reduce_max_sync(0xffffffffu, eh);
            if (lane == 0) {
                sh.any64[warp] = any != 0u;
                sh.eh[warp] = eh;
            }
        }
        __syncthreads();
        int Ef, any64 = 0;
        {
            int eh = 0;
            for (int q = 0; q <= j / 32; ++q) {
                any64 |= sh.any64[q];
                eh = max(eh, sh.eh[q]);
            }
            // at most 2^8 terms: below 2^-12 of 2^(E_w - 1022) they disappear in the margin of r
            const int ew = sh.Ew;
            const float r = sh.r0 * (1.0f + 1.0f / 1024.0f);
            if (eh + 8 < ew - 12 && r < 0x1p120f) {
                Ef = bound_exp(r, ew);
            } else {
                double rd = 1.0 + fabs(sh.aj) * ldexp(1.0, emax[j] - ew);
                rd += 256.0 * ldexp(1.0, eh - ew);
                Ef = bound_exp(rd * (1.0 + 1.0 / 1024.0), ew);
            }
            if (tid == 0) eimg[j + 1] = Ef;
        }
        // ---- V_{j+1}, its image and norm
        if (scalar) resolve_alpha_j(j + 1);
        {
#pragma unroll
            for (int q = 0; q < EPT; ++q) {
                const int i = tid + q * kSmOwn;
                if (!owner || i >= n) continue;
                double2 u = w[q];
                float cx = 0.f, cy = 0.f, dx = 0.f, dy = 0.f;
#pragma unroll 8
                for (int t = 0; t <= j; ++t) {
                    const int4 v = img[(size_t)t * n_own + i];
                    const float2 c = coef32[t];
                    const float vx = (float)v.x, vy = (float)v.z;
                    cx = fmaf(c.x, vx, cx);
                    dx = fmaf(-c.y, vy, dx);
                    cy = fmaf(c.x, vy, cy);
                    dy = fmaf(c.y, vx, dy);
                }
                cx += dx;
                cy += dy;
                if (any64)
                    for (int t = 0; t <= j; ++t) {
                        const double2 c = coef64[t];
                        if (c.x == 0.0 && c.y == 0.0) continue;
                        const double2 v = V[(size_t)t * d + e0 + i];
                        u.x -= fma(c.x, v.x, -c.y * v.y);
                        u.y -= fma(c.x, v.y, c.y * v.x);
                    }
                u.x -= f32_to_f64_int(cx);
                u.y -= f32_to_f64_int(cy);
                V[(size_t)(j + 1) * d + e0 + i] = u;
                p[q] = x[q];
                x[q] = u;
            }
        }
        store_image(j + 1, x, Ef, true);
        cluster_sync();
    }
    __syncthreads();
    const int m = sh.m_eff;
    if (rank == 0) {
        for (int k = tid; k <= min(m, M); k += kSmThreads) {
            if (k < m) Cs->alpha[k] = alpha[k];
            Cs->beta[k] = k == 0 ? 0.0 : beta[k];
            Cs->scale[k] = scale[k];
            Cs->emax[k] = emax[k];
        }
        if (tid == 0) {
            Cs->beta0 = beta[0];
            Cs->m_eff = m;
            if (sh.status != KG_OK) Cs->status = sh.status;
        }
    }
    if (!finish) return;
    // ---- e^{-iT tau} e_1 (every block by its scalar warp), then the combination
    if (scalar) {
        const double beta0 = beta[0];
        double2 v[2] = {make_double2(lane == 0 ? 1.0 : 0.0, 0.0), make_double2(0.0, 0.0)};
        bool ok = true;
        if (m > 32) {
            Tridiag<2> T;
            T.load(alpha, beta, m, lane);
            ok = T.advance(D.tau, v, lane, true);
        } else if (m > 0) {
            Tridiag<1> T;
            T.load(alpha, beta, m, lane);
            double2 v1[1] = {v[0]};
            ok = T.advance(D.tau, v1, lane, true);
            v[0] = v1[0];
        }
        if (!ok && rank == 0 && lane == 0) Cs->status = KG_ENUMERIC;
        double2 c[2];
        double cmax = 0.0;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int k = lane + 32 * r;
            const double s = k < m ? beta0 * scale[k] : 0.0;
            c[r] = ok ? make_double2(s * v[r].x, s * v[r].y) : make_double2(0.0, 0.0);
            if (k < m && scale[k] > 0.0) cmax = fmax(cmax, (fabs(c[r].x) + fabs(c[r].y)) / scale[k]);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) cmax = fmax(cmax, __shfl_xor_sync(0xffffffffu, cmax, o));
        // the FP32 terms in units of 2^(ec - 1023), so that none vanishes or overflows
        const int ec = exp_field(cmax);
        int a32 = 0, a64 = 0;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int k = lane + 32 * r;
            const bool small = k < m && scale[k] > 0.0 && (fabs(c[r].x) + fabs(c[r].y)) < 1e-10 * cmax * scale[k];
            const unsigned in = __ballot_sync(0xffffffffu, k < m), ms = __ballot_sync(0xffffffffu, small);
            const unsigned before = (1u << lane) - 1u;
            if (small) {
                const int q = a32 + __popc(ms & before);
                const int de = eimg[k] - 1050 + 1023 - ec;
                coef32[q] = make_float2(f64_to_f32_near(mul_pow2(c[r].x, de)), f64_to_f32_near(mul_pow2(c[r].y, de)));
                idx32[q] = (short)k;
            } else if (k < m) {
                const int q = a64 + __popc(in & ~ms & before);
                coef64[q] = c[r];
                idx64[q] = (short)k;
            }
            a32 += __popc(ms);
            a64 += __popc(in & ~ms);
        }
        if (lane == 0) {
            sh.n32 = a32;
            sh.n64 = a64;
            sh.ec = ec;
        }
    }
    __syncthreads();
    const int n_ov = D.n_ov;
    double nrm = 0.0;
#pragma unroll
    for (int q = 0; q < EPT; ++q) {
        const int i = tid + q * kSmOwn;
        w[q] = make_double2(0.0, 0.0);
        if (!owner || i >= n) continue;
        const int m32 = sh.n32, m64 = sh.n64;
        double2 u = make_double2(0.0, 0.0);
        double2 u2 = u;  // two chains
#pragma unroll 4
        for (int t = 0; t + 1 < m64; t += 2) {
            const double2 v = V[(size_t)idx64[t] * d + e0 + i], c = coef64[t];
            const double2 v2 = V[(size_t)idx64[t + 1] * d + e0 + i], c2 = coef64[t + 1];
            u.x = fma(c.x, v.x, fma(-c.y, v.y, u.x));
            u.y = fma(c.x, v.y, fma(c.y, v.x, u.y));
            u2.x = fma(c2.x, v2.x, fma(-c2.y, v2.y, u2.x));
            u2.y = fma(c2.x, v2.y, fma(c2.y, v2.x, u2.y));
        }
        if (m64 & 1) {
            const double2 v = V[(size_t)idx64[m64 - 1] * d + e0 + i], c = coef64[m64 - 1];
            u.x = fma(c.x, v.x, fma(-c.y, v.y, u.x));
            u.y = fma(c.x, v.y, fma(c.y, v.x, u.y));
        }
        u.x += u2.x;
        u.y += u2.y;
        float cx = 0.f, cy = 0.f;
#pragma unroll 4
        for (int t = 0; t < m32; ++t) {
            const int4 v = img[(size_t)idx32[t] * n_own + i];
            const float2 c = coef32[t];
            const float vx = (float)v.x, vy = (float)v.z;
            cx = fmaf(c.x, vx, fmaf(-c.y, vy, cx));
            cy = fmaf(c.x, vy, fmaf(c.y, vx, cy));
        }
        u.x += mul_pow2(f32_to_f64_int(cx), sh.ec - 1023);
        u.y += mul_pow2(f32_to_f64_int(cy), sh.ec - 1023);
        D.out[e0 + i] = u;
        w[q] = u;
        nrm = fma(u.x, u.x, fma(u.y, u.y, nrm));
    }
    __syncthreads();  // the images are no longer read: their place takes the overlaps' partial sums
    double* const ps = reinterpret_cast<double*>(img);                        // [warp][2 n_ov + 1]
    double* const pc = reinterpret_cast<double*>(dots);                       // [block][2 n_ov + 1], in block 0
    const int nv = 2 * n_ov + 1;
    if (owner) {
        const double t = warp_sum(nrm);
        if (lane == 0) ps[warp * nv] = t;
        for (int a = 0; a < n_ov; ++a) {
            double re = 0.0, im = 0.0;
#pragma unroll
            for (int q = 0; q < EPT; ++q) {
                const int i = tid + q * kSmOwn;
                if (i >= n) continue;
                const double2 v = D.ov[(size_t)a * D.ov_stride + e0 + i];
                re = fma(v.x, w[q].x, fma(v.y, w[q].y, re));
                im = fma(v.x, w[q].y, fma(-v.y, w[q].x, im));
            }
            re = warp_sum(re);
            im = warp_sum(im);
            if (lane == 0) {
                ps[warp * nv + 1 + 2 * a] = re;
                ps[warp * nv + 2 + 2 * a] = im;
            }
        }
    }
    __syncthreads();
    for (int k = tid; k < nv; k += kSmThreads) {
        double t = 0.0;
        for (int q = 0; q < kSmWarps; ++q) t += ps[q * nv + k];
        remote_store(pc + rank * nv + k, 0, t);
    }
    cluster_sync();
    if (rank == 0) {
        const int slot = Cs->ov_slot;
        __syncthreads();
        for (int k = tid; k < nv; k += kSmThreads) {
            double t = 0.0;
            for (int q = 0; q < C; ++q) t += pc[q * nv + k];
            if (k == 0) {
                Cs->ovnorm = sqrt(t);
                if (n_ov > 0) Cs->ov_slot = slot + 1;
            } else if (slot < D.ov_rows) {
                reinterpret_cast<double*>(D.ov_out)[2 * ((size_t)slot * n_ov) + k - 1] = t;
            }
        }
    }
}

// -------------------------------------------------------------- host side
using SmallKernel = void (*)(const ColDesc*, const int*, ColScalars*, int, int);

static SmallKernel small_kernel(int ept) { return ept == 1 ? &k_small_step<1> : &k_small_step<2>; }

// How many clusters of 1, 2, 4, 8, 16 blocks this device holds at once (0:
// none), per device.
static std::array<int, 5> small_resident() {
    static std::mutex mu;
    static std::map<int, std::array<int, 5>> known;
    std::array<int, 5> r = {{0, 0, 0, 0, 0}};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return r;
    std::lock_guard<std::mutex> lk(mu);
    auto it = known.find(dev);
    if (it != known.end()) return it->second;
    for (int ept = 1; ept <= kSmMaxEpt; ++ept) {
        const void* k = (const void*)small_kernel(ept);
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmSmem) != cudaSuccess ||
            cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
            cudaGetLastError();
        for (int i = 0; i < 5; ++i) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(1 << i);
            cfg.blockDim = dim3(kSmThreads);
            cfg.dynamicSmemBytes = kSmSmem;
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = 1 << i;
            at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            int nc = 0;
            if (cudaOccupancyMaxActiveClusters(&nc, k, &cfg) != cudaSuccess) {
                cudaGetLastError();
                nc = 0;
            }
            r[i] = ept == 1 ? nc : std::min(r[i], nc);
        }
    }
    known[dev] = r;
    return r;
}

static size_t small_bytes(const kg_sector* s, int M, int C) {
    const int n_own = ((int)s->d + C - 1) / C;
    return small_layout(M, n_own, C, s->L, s->hopmode, s->Du, s->Dd, s->up.nnz + s->dn.nnz).total;
}

// Cluster size per column (0: the streaming kernels, for the whole batch).  A
// column is small when some cluster holds its images.  The streaming kernels
// cost about 20 us of latency per Lanczos vector whatever the number of
// columns, and share the GPU evenly, so small columns beside a large one, or
// more of them than the GPU holds clusters at once, are better off there
// (96 columns of 6 to 52,920 states: 2.5 ms per step streaming, 2.6 with the
// small ones in clusters beside the others).  Otherwise more blocks shorten a
// step until a block is left with about 96 elements, as long as all clusters
// stay resident.
void small_plan(const std::vector<const kg_sector*>& cols, int M, int schedule, std::vector<int>& cluster) {
    cluster.assign(cols.size(), 0);
    if (schedule != 0) return;
    const std::array<int, 5> room = small_resident();
    std::vector<int> least(cols.size(), 0);
    auto log2i = [](int c) { return c == 1 ? 0 : c == 2 ? 1 : c == 4 ? 2 : c == 8 ? 3 : 4; };
    double share = 0.0, share_least = 0.0;  // of the clusters resident at once
    for (size_t b = 0; b < cols.size(); ++b) {
        const kg_sector* s = cols[b];
        if (s->Du <= 65535 && s->Dd <= 65535 && s->up.max_row + s->dn.max_row <= 60)
            for (int c = 1; c <= kSmMaxCluster; c *= 2) {
                const long long n_own = (s->d + c - 1) / c;
                if (n_own > kSmMaxEpt * kSmOwn || small_bytes(s, M, c) > kSmSmem || room[log2i(c)] < 1) continue;
                if (!least[b]) least[b] = c;
                cluster[b] = c;
                if (n_own <= 96) break;
            }
        if (cluster[b]) {
            share += 1.0 / room[log2i(cluster[b])];
            share_least += 1.0 / room[log2i(least[b])];
        }
        if (!cluster[b] || share_least > 1.0) {
            cluster.assign(cols.size(), 0);
            return;
        }
    }
    while (share > 1.0) {
        bool any = false;
        for (size_t b = 0; b < cols.size(); ++b)
            if (cluster[b] > least[b] && room[log2i(cluster[b] / 2)] > 0) {
                share += 1.0 / room[log2i(cluster[b] / 2)] - 1.0 / room[log2i(cluster[b])];
                cluster[b] /= 2;
                any = true;
            }
        if (!any) return;
    }
}

int small_alloc(Krylov& K, const std::vector<const kg_sector*>& cols) {
    size_t nx = 0;
    for (auto& D : K.hdesc)
        if (D.small) nx += (size_t)D.d;
    if (!nx) return KG_OK;
    KG_CUDA(cudaMalloc(&K.Xsbuf, sizeof(int4) * nx));
    size_t ox = 0;
    for (auto& D : K.hdesc)
        if (D.small) {
            D.Xs = K.Xsbuf + ox;
            ox += (size_t)D.d;
        }
    for (int c = kSmMaxCluster; c >= 1; c /= 2)
        for (int ept = kSmMaxEpt; ept >= 1; --ept) {
            std::vector<int> v;
            size_t smem = 0;
            for (int b = 0; b < K.B; ++b) {
                if (K.hdesc[b].small != c || ((K.hdesc[b].d + c - 1) / c + kSmOwn - 1) / kSmOwn != ept) continue;
                v.push_back(b);
                smem = std::max(smem, small_bytes(cols[b], K.M, c));
            }
            if (v.empty()) continue;
            K.small.emplace_back();
            Krylov::SmallGroup& g = K.small.back();
            g.cluster = c;
            g.ept = ept;
            g.n = (int)v.size();
            g.smem = smem;
            KG_CUDA(cudaMalloc(&g.cols, sizeof(int) * v.size()));
            KG_CUDA(cudaMemcpy(g.cols, v.data(), sizeof(int) * v.size(), cudaMemcpyHostToDevice));
        }
    if (K.small.size() > 1) {  // the groups run beside each other
        KG_CUDA(cudaEventCreateWithFlags(&K.fork, cudaEventDisableTiming));
        for (size_t i = 1; i < K.small.size(); ++i) {
            KG_CUDA(cudaStreamCreateWithFlags(&K.small[i].side, cudaStreamNonBlocking));
            KG_CUDA(cudaEventCreateWithFlags(&K.small[i].done, cudaEventDisableTiming));
        }
    }
    return KG_OK;
}

void small_free(Krylov& K) {
    for (auto& g : K.small) {
        if (g.side) cudaStreamDestroy(g.side);
        if (g.done) cudaEventDestroy(g.done);
        cudaFree(g.cols);
    }
    if (K.fork) cudaEventDestroy(K.fork);
    cudaFree(K.Xsbuf);
    K.small.clear();
    K.fork = nullptr;
    K.Xsbuf = nullptr;
}

int launch_small(Krylov& K, bool finish, cudaStream_t st) {
    if (K.fork) KG_CUDA(cudaEventRecord(K.fork, st));
    // the groups on their side streams first, so that none queues behind `st`
    for (size_t i = K.small.size(); i-- > 0;) {
        Krylov::SmallGroup& g = K.small[i];
        cudaStream_t s = g.side ? g.side : st;
        if (g.side) KG_CUDA(cudaStreamWaitEvent(g.side, K.fork, 0));
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(g.n * g.cluster);
        cfg.blockDim = dim3(kSmThreads);
        cfg.dynamicSmemBytes = g.smem;
        cfg.stream = s;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = g.cluster;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        ProfScope ps("small_step", s);
        KG_CUDA(cudaLaunchKernelEx(&cfg, small_kernel(g.ept), (const ColDesc*)K.desc, (const int*)g.cols, K.cs, K.M,
                                   finish ? 1 : 0));
        count_launch();
        if (g.side) KG_CUDA(cudaEventRecord(g.done, g.side));
    }
    for (auto& g : K.small)
        if (g.side) KG_CUDA(cudaStreamWaitEvent(st, g.done, 0));
    return KG_OK;
}

}  // namespace kg
