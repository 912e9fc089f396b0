// k_sbr.cu -- S2 for a banded H_F: reduction of the band straight to real tridiagonal form by
// Householder bulge chasing, and the back-transform of the chase's reflectors (S5).
//
// H_F is block-banded (Eq. 6, Appendix A): every nonzero lies within b of the diagonal, with
// b = max over the couplings' nonzero entries V^{l,h}[i][i'] of D h S_l + i' - i (and the width
// of H0).  The dense reduction (k_hetrd) would destroy that structure after one panel; the band
// reduction of Schwarz / Bischof, Lang & Sun keeps the work inside a band of width 2b and costs
// O(n^2 b) instead of O(n^3).  This is the "one column per sweep" chase:
//   sweep j (j = 0 .. n-2), step 0: the reflector H(j,0) of rows R0 = [j+1, j+b] annihilates
//     A(j+2.., j) (A(j+1, j) becomes the real beta = e_j) and is applied from both sides to the
//     diagonal block A(R0, R0);
//   step s >= 1: the previous reflector, applied from the right to the block B = A(Rs, Rs-1)
//     below it (Rs = Rs-1 + b), fills B's lower triangle (the bulge); H(j,s) annihilates B's
//     first column below its first row, is applied from the left to B's other columns and from
//     both sides to A(Rs, Rs).  The rest of the bulge is removed by sweep j+1.
// All reflectors satisfy H^H x = beta e_1 with beta real (H = I - tau v v^H, v[0] = 1; the
// convention of k_hetrd), so T = Q^H H_F Q is real and Q = prod_j prod_s H(j, s).
//
// Pipelining: sweep j+1 may run its step s once sweep j has finished step s and the first row of
// its step s+1 (their later steps touch disjoint entries), so several sweeps are in flight at once,
// each with a group of threads of its own that publishes its progress and waits (bounded) for its
// predecessor's.  The
// band itself stays in the dense matrix's lower triangle (global memory, L2-resident: about n x 2b
// entries are ever touched).
//
// Back-transform: Z = Q Y.  Reflectors of one sweep touch disjoint rows, and H(j', s') must
// precede H(j, s) only if j' > j and s' in {s-1, s}, so the order "s ascending, j descending"
// is valid.  In pass s consecutive reflectors overlap in all but one row: one thread per column
// of Z keeps a window of BMAX rows in registers, applies the reflector (a length-BMAX dot
// product and update), and slides the window up one row.  Z is kept row-major so that the
// threads of a warp (consecutive columns) load and store consecutive addresses.
#include <cooperative_groups.h>
#include <cstdlib>

#include "mmf_internal.h"

namespace cg = cooperative_groups;

// ------------------------------------------------------------------ reflector store
// (layout and Z's place: sbr_off / sbr_zbase in mmf_internal.h)
int64_t mmf_sbr_store_elems(int n, int b) { return sbr_nref(n, b) * (b + 1); }

#define SBR_WAIT_LIMIT (1 << 26)
// bytes before the groups' blocks in dynamic shared memory (progress keys, abort flag), rounded to
// 256 so that the blocks' 16-byte complex elements stay aligned
__host__ __device__ constexpr int sbr_hdr(int ng) { return (16 * ng + 16 + 255) / 256 * 256; }

// A vector entry in shared memory as the multiplier of packed products: (x, x), (y, y).  With it
// acc1 += a (x, x) and acc2 += a (y, y) are two packed FP32 instructions, and
// a v = (acc1.x - acc2.y, acc1.y + acc2.x), conj(v) a = (acc1.x + acc2.y, acc1.y - acc2.x).  The
// FP64 path keeps plain entries.
template <class C> struct SbrDup;
template <> struct SbrDup<float2> {
    typedef float4 T;
    static __device__ __forceinline__ T of(float2 v) { return make_float4(v.x, v.x, v.y, v.y); }
    static __device__ __forceinline__ float2 val(T t) { return make_float2(t.x, t.z); }
};
template <> struct SbrDup<double2> {
    typedef double2 T;
    static __device__ __forceinline__ T of(double2 v) { return v; }
    static __device__ __forceinline__ double2 val(T t) { return t; }
};
// running sum of a v and of conj(v) a over entries v
template <class C> struct SbrAcc;
template <> struct SbrAcc<float2> {
    float2 p, q;
    __device__ __forceinline__ SbrAcc() : p(make_float2(0.f, 0.f)), q(make_float2(0.f, 0.f)) {}
    __device__ __forceinline__ void add(float2 a, float4 v) {
        p = __ffma2_rn(a, make_float2(v.x, v.y), p);
        q = __ffma2_rn(a, make_float2(v.z, v.w), q);
    }
    __device__ __forceinline__ void addc(float2 a, float4 v) { add(a, v); }
    __device__ __forceinline__ float2 mul() const { return make_float2(p.x - q.y, p.y + q.x); }
    __device__ __forceinline__ float2 mulc() const { return make_float2(p.x + q.y, p.y - q.x); }
};
template <> struct SbrAcc<double2> {
    double2 p;
    __device__ __forceinline__ SbrAcc() : p(make_double2(0.0, 0.0)) {}
    __device__ __forceinline__ void add(double2 a, double2 v) { p = cmac(p, a, v); }
    __device__ __forceinline__ void addc(double2 a, double2 v) { p = cmacc(p, v, a); }
    __device__ __forceinline__ double2 mul() const { return p; }
    __device__ __forceinline__ double2 mulc() const { return p; }
};
// a - f conj(v) (rank-1 update by a row of conjugated entries) and a - f v
__device__ __forceinline__ float2 sbr_sub_conj(float2 a, float2 f, float4 v) {
    a = __ffma2_rn(make_float2(-f.x, -f.y), make_float2(v.x, v.y), a);
    return __ffma2_rn(make_float2(-f.y, f.x), make_float2(v.z, v.w), a);
}
__device__ __forceinline__ double2 sbr_sub_conj(double2 a, double2 f, double2 v) { return cmsubc(a, v, f); }
__device__ __forceinline__ float2 sbr_sub(float2 a, float2 f, float4 v) {
    a = __ffma2_rn(make_float2(-f.x, -f.y), make_float2(v.x, v.y), a);
    return __ffma2_rn(make_float2(f.y, -f.x), make_float2(v.z, v.w), a);
}
__device__ __forceinline__ double2 sbr_sub(double2 a, double2 f, double2 v) { return cmsub(a, f, v); }

// Shared memory of one group.  B and D: the step's two blocks, column-major with a padded column
// (LD even: two rows of a column are one aligned 16-byte read, and consecutive columns fall in
// other banks).
template <class C, int BMAX, bool EARLY> struct SbrLate {};
template <class C, int BMAX> struct SbrLate<C, BMAX, true> {
    C dl[BMAX];          // D's last row and B's last entry, taken from the predecessor's published row
    C bl, d00;
};
template <class C, int BMAX, int P, bool EARLY>
struct __align__(16) SbrGroup {
    static constexpr int LD = BMAX + 2;
    typedef typename SbrDup<C>::T Dup;
    Dup v[2][BMAX];      // current and previous reflector
    Dup wu[BMAX], wd[BMAX];
    C B[BMAX * LD];
    C D[BMAX * LD];
    C red[3][P][BMAX];   // partial sums: B v_p, v^H B, D v
    C c0[BMAX];          // B(:, 0)
    C ty[BMAX];
    C beta, pad;
    SbrLate<C, BMAX, EARLY> late;
};

__host__ __device__ constexpr bool sbr_early(int cl, int ng) { return cl >= 4 || ng >= 8; }

// Predicated load (zero where !ok) and store of one complex element, without a branch around each.
// CG reads L2 only: the CTAs of a cluster run on different SMs, whose L1 caches are not coherent, so
// band data written by one must not be read by another from a stale L1 line.
template <bool CG>
__device__ __forceinline__ float2 ld_if(const float2* p, bool ok) {
    float2 r;
    if (CG)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\tmov.f32 %0, 0f00000000;\n\t"
                     "mov.f32 %1, 0f00000000;\n\t@p ld.global.cg.v2.f32 {%0, %1}, [%2];\n\t}"
                     : "=&f"(r.x), "=&f"(r.y) : "l"(p), "r"((int)ok) : "memory");
    else
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\tmov.f32 %0, 0f00000000;\n\t"
                     "mov.f32 %1, 0f00000000;\n\t@p ld.global.v2.f32 {%0, %1}, [%2];\n\t}"
                     : "=&f"(r.x), "=&f"(r.y) : "l"(p), "r"((int)ok) : "memory");
    return r;
}
template <bool CG>
__device__ __forceinline__ double2 ld_if(const double2* p, bool ok) {
    double2 r;
    if (CG)
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\tmov.f64 %0, 0d0000000000000000;\n\t"
                     "mov.f64 %1, 0d0000000000000000;\n\t@p ld.global.cg.v2.f64 {%0, %1}, [%2];\n\t}"
                     : "=&d"(r.x), "=&d"(r.y) : "l"(p), "r"((int)ok) : "memory");
    else
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\tmov.f64 %0, 0d0000000000000000;\n\t"
                     "mov.f64 %1, 0d0000000000000000;\n\t@p ld.global.v2.f64 {%0, %1}, [%2];\n\t}"
                     : "=&d"(r.x), "=&d"(r.y) : "l"(p), "r"((int)ok) : "memory");
    return r;
}
__device__ __forceinline__ void st_if(float2* p, float2 v, bool ok) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\t@p st.global.v2.f32 [%0], {%1, %2};\n\t}" ::"l"(p),
                 "f"(v.x), "f"(v.y), "r"((int)ok)
                 : "memory");
}
__device__ __forceinline__ void st_if(double2* p, double2 v, bool ok) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\t@p st.global.v2.f64 [%0], {%1, %2};\n\t}" ::"l"(p),
                 "d"(v.x), "d"(v.y), "r"((int)ok)
                 : "memory");
}

// progress key of a group, in its CTA's shared memory (addressed as shared::cluster)
__device__ __forceinline__ long long key_load(uint32_t a) {
    long long v;
    asm volatile("ld.acquire.cluster.shared::cluster.b64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ int flag_load(uint32_t a) {
    int v;
    asm volatile("ld.relaxed.cluster.shared::cluster.b32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void key_store(uint32_t a, long long v) {
    asm volatile("st.release.cluster.shared::cluster.b64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}
// address of this CTA's shared memory location in the CTA of the given rank
__device__ __forceinline__ uint32_t map_rank(const void* p, int rank) {
    uint32_t a = (uint32_t)__cvta_generic_to_shared(p), r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}

template <int G>
__device__ __forceinline__ void gbar(int g) {
    if (G == 32) {
        __syncwarp();
    } else {
        asm volatile("bar.sync %0, %1;" ::"r"(1 + g), "r"(G) : "memory");
    }
}

// sum over the lanes that hold different entries of a vector of BMAX (all 32, or BMAX of them when
// the vector is repeated over the warp); every lane gets the result
template <int BMAX, class R>
__device__ __forceinline__ R lane_sum(R v) {
#pragma unroll
    for (int o = BMAX < 32 ? BMAX / 2 : 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// two consecutive complex entries of a column
__device__ __forceinline__ void ld_pair(const float2* p, float2& a, float2& b) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    a = make_float2(t.x, t.y);
    b = make_float2(t.z, t.w);
}
__device__ __forceinline__ void ld_pair(const double2* p, double2& a, double2& b) {
    a = p[0];
    b = p[1];
}

// One group of G = BMAX P threads per sweep: thread (i, p) keeps row i, columns p EL .. p EL + EL - 1
// of the step's two blocks B = A(R_s, R_{s-1}) and D = A(R_s, R_s) (lower triangle) in registers,
// from its loads to its stores; a copy in shared memory serves the sums down the columns.  A step is
//   load | y = B v_p (partial sums) | x = B(:,0) - tau_p y gives v, tau, beta | u = v^H B and D v
//   (rows from registers, columns from shared memory) | w vectors | rank-2 updates, store
// with five group barriers; one warp computes the vectors.  A successor's step s needs all but its last
// row from the predecessor's step s, and that row (B's is zero but for its last entry, beta) from the
// first row of the predecessor's step s + 1: one warp computes and publishes that row as soon as the
// step's vectors are known, so a sweep follows its predecessor by a step and the part of a step up to
// there, with its loads and B v_p done beforehand, where it waited for two whole steps (one FP32 system
// of n = 1323 15.1 -> 13.2 ms, eight in FP64 99 -> 87).  With few groups per system (CL <= 2 and wide
// windows) the SMs are busy anyway (64 systems: 24.9 ms with the publication, 23.7 without): there a sweep
// waits for all of the predecessor's step s + 1, and the publication's code, its shared memory and its
// terms in the stores' conditions are compiled out (left to run-time conditions that are constant they cost
// 64 systems 1 %).
//
// What bounds it: the critical path of one sweep after another (about 1.5 n steps), so the latency of a
// step; on the FP64 path the 2 FP64 FMAs per clock
// of an SM (24 b^2 FMAs a step).  NG groups per CTA and CL CTAs (SMs) per system hold
// CL x NG sweeps in flight (how many have work: see launch_chase).  Measured at n = 1323,
// b = 63 (128 threads per sweep with both blocks in shared memory, at most two CTAs per system -> this
// kernel): one system in FP32 36.2 -> 13.2 ms, 64 systems 37.4 -> 23.7 ms; eight systems in FP64
// 455 -> 87 ms.
//
// CL = 1: one CTA per system.  CL > 1: a cluster of CL CTAs per system, the sweeps dealt round-robin
// over all groups; a group reads its predecessor's progress key from that CTA's shared memory
// (distributed shared memory; the key is stored with release and read with acquire semantics, each
// warp polling for itself), and the band is read from L2 only (ld.cg).  A wait that gives up marks
// the system and makes every group run on without waiting (its results are void, every access stays
// in bounds), so that the group's warps pass the same barriers.
template <class R, int BMAX, int P, int NG, int CL>
__global__ void __launch_bounds__(BMAX* P* NG) k_sbr_chase(const MmfDesc* __restrict__ descs,
                                                          const int* __restrict__ idx,
                                                          typename Cx<R>::T* __restrict__ Hbase,
                                                          typename Cx<R>::T* __restrict__ store_base,
                                                          double* __restrict__ dvec, double* __restrict__ evec,
                                                          int* __restrict__ status) {
    typedef typename Cx<R>::T C;
    constexpr bool EARLY = sbr_early(CL, NG);       // first rows published ahead
    typedef SbrGroup<C, BMAX, P, EARLY> Grp;
    typedef SbrDup<C> DupC;
    constexpr int G = BMAX * P, EL = BMAX / P, LD = Grp::LD;
    constexpr int SL = BMAX >= 32 ? BMAX / 32 : 1;  // entries of a vector per lane
    constexpr bool F64 = sizeof(R) == 8;            // FP64 units are scarce: skip padding
    constexpr int NGT = CL * NG;                    // groups per system
    static_assert(G % 32 == 0 && EL * P == BMAX && EL % 2 == 0, "group shape");
    extern __shared__ __align__(16) unsigned char sbr_smem[];
    long long* key = reinterpret_cast<long long*>(sbr_smem);
    long long* pub = key + NG;
    int* abort_flag = reinterpret_cast<int*>(sbr_smem + 16 * NG);
    Grp* groups = reinterpret_cast<Grp*>(sbr_smem + sbr_hdr(NG));
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = CL > 1 ? (int)cluster.block_rank() : 0;

    const int sid = idx[blockIdx.x / CL];
    const MmfDesc d = descs[sid];
    const int n = d.n, b = d.band;
    const int ldi = d.ld;  // in-system offsets fit 32 bits (n ld < 2^31, checked by the host)
    C* Hg = Hbase + d.mat_off;
    // the store lives in the system's FP64 complex matrix slot
    C* V = reinterpret_cast<C*>(store_base + (sizeof(R) == 4 ? 2 : 1) * d.mat_off);
    C* T = V + sbr_nref(n, b) * b;
    double* dd = dvec + d.vec_off;
    double* ee = evec + d.vec_off;
    const int g = threadIdx.x / G, tid = threadIdx.x % G;
    const int lane = tid & 31, warp = tid >> 5;
    const int gg = rank * NG + g;  // the group's number within the system
    Grp& S = groups[g];
    const long long KK = sbr_passes(n, b) + 3;
    // the predecessor sweep's group, its progress key and its CTA's abort flag
    const int ggp = (gg + NGT - 1) % NGT;
    const uint32_t pkey = map_rank(key + ggp % NG, ggp / NG), ppub = map_rank(pub + ggp % NG, ggp / NG);
    const uint32_t pabort = map_rank(abort_flag, ggp / NG);
    const uint32_t mykey = map_rank(key + g, rank), mypub = map_rank(pub + g, rank);

    if (threadIdx.x < 2 * NG) key[threadIdx.x] = -1;
    if (threadIdx.x == 0) *abort_flag = 0;
    if (CL > 1) cluster.sync(); else __syncthreads();
    if (threadIdx.x == 0 && rank == 0) dd[0] = (double)Hg[0].x;

    const C zero = mk(R(0), R(0));
    const int i = tid % BMAX, p = tid / BMAX;
    const int k0 = p * EL;                     // this thread's columns (and rows, in the column sums)
    const int i0 = BMAX >= 32 ? (i & ~31) : 0; // the warp's first row
    const bool low = k0 + EL - 1 > i0, row = k0 <= i0 + 31;  // the warp's share of D: column / row sums
    int cur = 0;  // buffer of the current reflector in S.v
    bool stopped = false;
    C tau = zero, taup = zero;
    // a warp's bounded wait for a predecessor's progress (acquire); after one gave up nobody waits (the
    // caller asks: an early return in here costs a spilled flag in every step, 64 systems 25.6 ms for 23.9)
    auto wait_for = [&](uint32_t where, long long need) {
        if (lane == 0) {
            int it = 0;
            while (key_load(where) < need) {
                const int gave_up = ++it > SBR_WAIT_LIMIT;
                if (gave_up || flag_load(pabort) || *(volatile int*)abort_flag) {
                    *(volatile int*)abort_flag = 1;  // the successors' CTAs see it too
                    status[sid] = MMF_ST_NOCONV;
                    stopped = true;
                    break;
                }
                __nanosleep(32);
            }
        }
        stopped = __shfl_sync(0xffffffffu, stopped, 0);
        __syncwarp();  // orders the other lanes' loads after lane 0's acquire (a shuffle orders no memory)
    };
    for (int j = gg; j <= n - 2; j += NGT) {
        const int nsteps = (n - 2 - j) / b + 1;
        for (int s = 0; s < nsteps; ++s) {
            // rows r .. r + b - 2 are the predecessor's of its step s, which it has to have finished;
            // row r + b - 1, if there is one, is the first row of its step s + 1, published during it
            // (without publication: all of step s + 1)
            if (j > 0 && !stopped)
                wait_for(pkey, (long long)(j - 1) * KK + (EARLY ? s + 1 : s + 2 < KK - 1 ? s + 2 : KK - 1));
            const int r = j + 1 + s * b, rp = r - b;
            const int l = min(b, n - r);
            const bool late = EARLY && j > 0 && l == b;
            const int lim = late ? b - 1 : l;
            // (a) the step's entries: all loads in flight together, zeros outside the blocks
            C B[EL], D[EL], x[SL];
            {
                const C* h = Hg + (r + k0) * ldi + r + i;
#pragma unroll
                for (int q = 0; q < EL; ++q)
                    D[q] = ld_if<(CL > 1)>(h + q * ldi, i < lim && i >= k0 + q);
            }
            if (s > 0) {
                const C* h = Hg + (rp + k0) * ldi + r + i;
#pragma unroll
                for (int q = 0; q < EL; ++q)
                    B[q] = ld_if<(CL > 1)>(h + q * ldi, i < lim && k0 + q < b);
            } else if (warp == 0) {
#pragma unroll
                for (int u = 0; u < SL; ++u) {
                    const int e = BMAX >= 32 ? lane + 32 * u : lane % BMAX;
                    x[u] = ld_if<(CL > 1)>(Hg + j * ldi + r + e, e < lim);
                }
            }
#pragma unroll
            for (int q = 0; q < EL; ++q) S.D[(k0 + q) * LD + i] = i == k0 + q ? zero : D[q];
            if constexpr (EARLY) {
                if (tid == 0) S.late.d00 = D[0];
            }
            if (s > 0) {
                // y = B v_p over this thread's columns
                const auto* vp = S.v[cur ^ 1] + k0;
                SbrAcc<C> a0, a1;  // two partial sums: independent FMA chains
#pragma unroll
                for (int q = 0; q < EL; q += 2) {
                    S.B[(k0 + q) * LD + i] = B[q];
                    S.B[(k0 + q + 1) * LD + i] = B[q + 1];
                    if (!F64 || k0 + q < b) {
                        a0.add(B[q], vp[q]);
                        a1.add(B[q + 1], vp[q + 1]);
                    }
                }
                S.red[0][p][i] = a0.mul() + a1.mul();
                if (p == 0) S.c0[i] = B[0];
            }
            gbar<G>(g);
            // (b) the reflector.  With C1 = B H(j,s-1) = B - tau_p y v_p^H, x = C1(:, 0) gives H(j,s);
            // then H^H C1 = B - tau_p y v_p^H - conj(tau) v r with r_k = (v^H B)_k - gamma conj(v_p,k),
            // gamma = v^H (tau_p y).  At s = 0 x is column j below the diagonal.
            C vl[SL], ty[SL];
            R beta = R(0);
            if (warp == 0) {
                R part = R(0);
                C bl = zero;  // B(b-1, b-1), the only nonzero of B's last row; at s = 0 x(b-1)
                if constexpr (EARLY) if (late) {
                    if (!stopped) wait_for(ppub, (long long)(j - 1) * KK + (s + 2));
                    const C* h = Hg + r + b - 1;
                    bl = ld_if<(CL > 1)>(h + (r - 1) * ldi, true);
#pragma unroll
                    for (int u = 0; u < SL; ++u) {
                        const int e = BMAX >= 32 ? lane + 32 * u : lane % BMAX;
                        const C dl = ld_if<(CL > 1)>(h + (r + (e < b ? e : 0)) * ldi, e < b);
                        S.late.dl[e] = dl;
                        if (e < b - 1) S.D[e * LD + b - 1] = dl;
                        if (s == 0 && e == b - 1) x[u] = bl;
                    }
                    if (lane == 0) {
                        S.late.bl = bl;
                        if (s > 0) S.B[(b - 1) * LD + b - 1] = bl;
                    }
                }
                if (s > 0) {
#pragma unroll
                    for (int u = 0; u < SL; ++u) {
                        const int e = BMAX >= 32 ? lane + 32 * u : lane % BMAX;
                        C y = S.red[0][0][e];
#pragma unroll
                        for (int q = 1; q < P; ++q) y = y + S.red[0][q][e];
                        C c0 = S.c0[e];
                        if constexpr (EARLY) {
                            if (late && e == b - 1) {
                                y = y + bl * DupC::val(S.v[cur ^ 1][b - 1]);
                                if (b == 1) c0 = bl;
                            }
                        }
                        ty[u] = taup * y;
                        x[u] = c0 - ty[u];   // v_p[0] = 1
                        S.ty[e] = ty[u];
                    }
                }
#pragma unroll
                for (int u = 0; u < SL; ++u)
                    if (u > 0 || (BMAX >= 32 ? lane : lane % BMAX) > 0) part += abs2(x[u]);
                const R xn2 = lane_sum<BMAX>(part);
                const C alpha = mk(__shfl_sync(0xffffffffu, x[0].x, 0), __shfl_sync(0xffffffffu, x[0].y, 0));
                C scale;
                warp_reflector<R, C>(alpha, xn2, lane, tau, beta, scale);
#pragma unroll
                for (int u = 0; u < SL; ++u) {
                    const int e = BMAX >= 32 ? lane + 32 * u : lane % BMAX;
                    vl[u] = e == 0 ? mk(R(1), R(0)) : x[u] * scale;
                    S.v[cur][e] = DupC::of(vl[u]);
                }
                if (lane == 0) S.beta = mk(beta, R(0));
            }
            gbar<G>(g);
            const auto* v = S.v[cur];
            if constexpr (EARLY) if (late && i == b - 1) {  // the owners of the last row
#pragma unroll
                for (int q = 0; q < EL; ++q) {
                    if (k0 + q < b) D[q] = S.late.dl[k0 + q];
                    if (s > 0 && k0 + q == b - 1) B[q] = S.late.bl;
                }
            }
            // (c) column i over rows k0 .. k0 + EL - 1 of B and of D's strict lower triangle, and row i
            // of D's lower triangle over columns k0 .. (warps whose share is zero skip it)
            {
                SbrAcc<C> zu0, zu1, zc0, zc1, zr0, zr1;
#pragma unroll
                for (int q = 0; q < EL; q += 2) {
                    if (F64 && k0 + q >= l) continue;
                    const auto v0 = v[k0 + q], v1 = v[k0 + q + 1];
                    C b0, b1;
                    if (s > 0) {
                        ld_pair(&S.B[i * LD + k0 + q], b0, b1);
                        zu0.addc(b0, v0);
                        zu1.addc(b1, v1);
                    }
                    if (low) {
                        ld_pair(&S.D[i * LD + k0 + q], b0, b1);
                        zc0.addc(b0, v0);
                        zc1.addc(b1, v1);
                    }
                    if (row) {
                        zr0.add(D[q], v0);
                        zr1.add(D[q + 1], v1);
                    }
                }
                if (s > 0) S.red[1][p][i] = zu0.mulc() + zu1.mulc();
                S.red[2][p][i] = (zr0.mul() + zr1.mul()) + conj(zc0.mulc() + zc1.mulc());
            }
            C gam = zero;
            if (warp == 0 && s > 0) {  // gamma, while the other warps are at their sums
                R gre = R(0), gim = R(0);
#pragma unroll
                for (int u = 0; u < SL; ++u) {
                    const C gc = cmulc(vl[u], ty[u]);
                    gre += gc.x;
                    gim += gc.y;
                }
                gam = mk(lane_sum<BMAX>(gre), lane_sum<BMAX>(gim));
            }
            gbar<G>(g);
            // (d) w_u = conj(tau) r for B; D <- H^H D H = D - v w^H - w v^H with y = D v,
            // w = tau y - |tau|^2 (v^H y) / 2 v
            if (warp == 0) {
                C y2[SL];
                R part = R(0);
#pragma unroll
                for (int u = 0; u < SL; ++u) {
                    const int e = BMAX >= 32 ? lane + 32 * u : lane % BMAX;
                    y2[u] = S.red[2][0][e];
#pragma unroll
                    for (int q = 1; q < P; ++q) y2[u] = y2[u] + S.red[2][q][e];
                    part += vl[u].x * y2[u].x + vl[u].y * y2[u].y;  // Re(conj(v) y)
                    if (s > 0) {
                        C z = S.red[1][0][e];
#pragma unroll
                        for (int q = 1; q < P; ++q) z = z + S.red[1][q][e];
                        S.wu[e] = DupC::of(conj(tau) * (z - gam * conj(DupC::val(S.v[cur ^ 1][e]))));
                    }
                }
                const R t2 = R(0.5) * abs2(tau) * lane_sum<BMAX>(part);
#pragma unroll
                for (int u = 0; u < SL; ++u) {
                    const int e = BMAX >= 32 ? lane + 32 * u : lane % BMAX;
                    S.wd[e] = DupC::of(tau * y2[u] - t2 * vl[u]);
                }
            }
            gbar<G>(g);
            // the first row of both blocks, published at once for the successor, whose step s - 1 has it
            // as its last row
            if constexpr (EARLY) if (warp == G / 32 - 1) {
                const auto* vp = S.v[cur ^ 1];
#pragma unroll
                for (int u = 0; u < SL; ++u) {
                    const int e = BMAX >= 32 ? lane + 32 * u : lane % BMAX;
                    C a = S.beta;
                    if (s > 0 && e > 0)
                        a = sbr_sub(sbr_sub_conj(S.B[e * LD], S.ty[0], vp[e]), mk(R(1), R(0)), S.wu[e]);
                    st_if(Hg + (r - (s > 0 ? b - (e < b ? e : 0) : 1)) * ldi + r, a,
                          (BMAX >= 32 || lane < BMAX) && e < b && (s > 0 || e == 0));
                }
                if (lane == 0) {
                    const C w0 = DupC::val(S.wd[0]);
                    C a = late && b == 1 ? S.late.dl[0] : S.late.d00;
                    a = mk(a.x - R(2) * w0.x, R(0));  // v_0 = 1
                    st_if(Hg + r * ldi + r, a, true);
                    if (s == 0) {
                        dd[j + 1] = (double)a.x;
                        ee[j] = (double)S.beta.x;
                    }
                }
                __syncwarp();
                if (lane == 0) key_store(mypub, (long long)j * KK + (s + 1));
            }
            // (e) rank-2 updates of this thread's other entries, back to global memory
            const C vi = DupC::val(v[i]), wi = DupC::val(S.wd[i]);
            if (s > 0) {
                const C tyi = S.ty[i];
                const auto *vp = S.v[cur ^ 1] + k0, *wu = S.wu + k0;
                C* h = Hg + (rp + k0) * ldi + r + i;
#pragma unroll
                for (int q = 0; q < EL; ++q) {
                    if (F64 && k0 + q >= b) continue;
                    C a = sbr_sub(sbr_sub_conj(B[q], tyi, vp[q]), vi, wu[q]);
                    if (q == 0 && p == 0) a = i == 0 ? S.beta : zero;
                    if constexpr (EARLY) st_if(h + q * ldi, a, i > 0 && i < l && k0 + q < b);
                    else st_if(h + q * ldi, a, i < l && k0 + q < b);
                }
            }
            if (row) {
                const auto *vk = v + k0, *wd = S.wd + k0;
                C* h = Hg + (r + k0) * ldi + r + i;
#pragma unroll
                for (int q = 0; q < EL; ++q) {
                    const int k = k0 + q;
                    if (F64 && k >= l) continue;
                    // v_i conj(w_k) + w_i conj(v_k)
                    C a = sbr_sub_conj(sbr_sub_conj(D[q], vi, wd[q]), wi, vk[q]);
                    if (i == k) a.y = R(0);
                    if constexpr (EARLY) st_if(h + q * ldi, a, i > 0 && i < l && i >= k);
                    else st_if(h + q * ldi, a, i >= k && i < l);
                    if (!EARLY && q == 0 && s == 0 && tid == 0) dd[j + 1] = (double)a.x;
                }
            }
            if (warp == 0) {
                if (s == 0) {
#pragma unroll
                    for (int u = 0; u < SL; ++u) {
                        const int e = BMAX >= 32 ? lane + 32 * u : lane % BMAX;
                        if (EARLY ? e > 0 && e < l : e < l) Hg[j * ldi + r + e] = e == 0 ? mk(beta, R(0)) : zero;
                    }
                    if (!EARLY && lane == 0) ee[j] = (double)beta;
                }
                // store the reflector for the back-transform, marked evict-first: the store is
                // written once and read only after the chase, and L2 should keep the band's lines
#pragma unroll
                for (int u = 0; u < SL; ++u) {
                    const int e = BMAX >= 32 ? lane + 32 * u : lane % BMAX;
                    if (e < b) __stcs(&V[(sbr_off(n, b, s) + j) * b + e], vl[u]);
                }
                if (lane == 0) __stcs(&T[sbr_off(n, b, s) + j], tau);
            }
            taup = tau;
            cur ^= 1;
            gbar<G>(g);  // the group's writes, then (release) its key
            if (tid == G - 1) key_store(mykey, (long long)j * KK + (s + 1 == nsteps ? KK - 1 : s + 1));
        }
    }
    // other CTAs may still read this CTA's keys and abort flag: leave together
    if (CL > 1) cluster.sync();
}

// ------------------------------------------------------------------ back-transform
// Window of the column in registers (FP32) -- one thread per column of Z (row-major, row stride n).
template <int BMAX>
__global__ void __launch_bounds__(128) k_sbr_bt_f32(const MmfDesc* __restrict__ descs, const int* __restrict__ idx,
                                                   const double2* __restrict__ store_base,
                                                   const double* __restrict__ Yg, double* __restrict__ work) {
    __shared__ __align__(16) float2 vs[2][BMAX];
    __shared__ float2 ts[2];
    const MmfDesc d = descs[idx[blockIdx.y]];
    const int n = d.n, b = d.band;
    const int c = blockIdx.x * 128 + threadIdx.x;
    if (blockIdx.x * 128 >= n) return;
    const bool act = c < n;
    const float2* V = reinterpret_cast<const float2*>(store_base + d.mat_off);
    const float2* T = V + sbr_nref(n, b) * b;
    const double* Y = Yg + d.sq_off;
    float2* Z = reinterpret_cast<float2*>(sbr_zbase(work, d));
    if (act) Z[c] = make_float2((float)Y[c], 0.f);  // row 0: no reflector touches it
    const int np = sbr_passes(n, b);
    float2 zr[BMAX];
    for (int s = 0; s < np; ++s) {
        const int jtop = n - 2 - s * b;
        const int64_t off = sbr_off(n, b, s);
        // window rows [r, r + BMAX), r = jtop + 1 + s b = n - 1
#pragma unroll
        for (int q = 0; q < BMAX; ++q) zr[q] = make_float2(0.f, 0.f);
        if (act) zr[0] = s == 0 ? make_float2((float)Y[(int64_t)(n - 1) * n + c], 0.f) : Z[(int64_t)(n - 1) * n + c];
        if (threadIdx.x < BMAX)
            vs[0][threadIdx.x] = threadIdx.x < b ? V[(off + jtop) * b + threadIdx.x] : make_float2(0.f, 0.f);
        if (threadIdx.x == 0) ts[0] = T[off + jtop];
        __syncthreads();
        int buf = 0;
#pragma unroll 1
        for (int j = jtop; j >= 0; --j) {
            float2 vn = make_float2(0.f, 0.f), tn = make_float2(0.f, 0.f);
            if (j > 0) {
                if (threadIdx.x < b) vn = V[(off + j - 1) * b + threadIdx.x];
                if (threadIdx.x == 0) tn = T[off + j - 1];
            }
            // w = v^H z, z -= tau w v; the dot product runs from the window's bottom up, so that
            // the row loaded last (zr[0]) is needed last
            float wr0 = 0.f, wi0 = 0.f, wr1 = 0.f, wi1 = 0.f;
#pragma unroll
            for (int q = BMAX - 2; q >= 0; q -= 2) {
                const float4 v2 = *reinterpret_cast<const float4*>(&vs[buf][q]);
                wr0 = fmaf(v2.x, zr[q].x, wr0);
                wr0 = fmaf(v2.y, zr[q].y, wr0);
                wi0 = fmaf(v2.x, zr[q].y, wi0);
                wi0 = fmaf(-v2.y, zr[q].x, wi0);
                wr1 = fmaf(v2.z, zr[q + 1].x, wr1);
                wr1 = fmaf(v2.w, zr[q + 1].y, wr1);
                wi1 = fmaf(v2.z, zr[q + 1].y, wi1);
                wi1 = fmaf(-v2.w, zr[q + 1].x, wi1);
            }
            const float2 t = ts[buf];
            const float wr = wr0 + wr1, wi = wi0 + wi1;
            // reload v from shared memory below rather than keep all of it in registers
            asm volatile("" ::: "memory");
            const float twr = t.x * wr - t.y * wi, twi = t.x * wi + t.y * wr;
            // (volatile: a second read of v, so that v need not stay in registers)
            const volatile float4* vv = reinterpret_cast<const volatile float4*>(&vs[buf][0]);
#pragma unroll
            for (int q = 0; q < BMAX; q += 2) {
                const float4 v2 = make_float4(vv[q / 2].x, vv[q / 2].y, vv[q / 2].z, vv[q / 2].w);
                zr[q].x = fmaf(-twr, v2.x, fmaf(twi, v2.y, zr[q].x));
                zr[q].y = fmaf(-twr, v2.y, fmaf(-twi, v2.x, zr[q].y));
                zr[q + 1].x = fmaf(-twr, v2.z, fmaf(twi, v2.w, zr[q + 1].x));
                zr[q + 1].y = fmaf(-twr, v2.w, fmaf(-twi, v2.z, zr[q + 1].y));
            }
            if (j > 0) {
                const int r = j + 1 + s * b;
                if (act && r + BMAX - 1 < n) Z[(int64_t)(r + BMAX - 1) * n + c] = zr[BMAX - 1];
#pragma unroll
                for (int q = BMAX - 1; q > 0; --q) zr[q] = zr[q - 1];
                if (act) {
                    const int64_t row = r - 1;
                    zr[0] = s == 0 ? make_float2((float)Y[row * n + c], 0.f) : Z[row * n + c];
                }
                if (threadIdx.x < BMAX) vs[buf ^ 1][threadIdx.x] = vn;
                if (threadIdx.x == 0) ts[buf ^ 1] = tn;
            }
            __syncthreads();
            buf ^= 1;
        }
        const int r0 = 1 + s * b;
        if (act) {
#pragma unroll
            for (int q = 0; q < BMAX; ++q)
                if (r0 + q < n) Z[(int64_t)(r0 + q) * n + c] = zr[q];
        }
    }
}

// FP64: the same with the window in shared memory; a CTA of 128 threads takes NC columns, each
// column's window rows dealt over RG = 128 / NC threads.  The SM's FP64 units bound it (a warp-wide
// FP64 instruction takes 64 cycles on its scheduler, 19 over the four): 8 n^3 flops per system at
// least, which 8 systems of n = 1323 spread over the whole GPU do in 120 ms.  One column per thread
// (128 columns per CTA) left 64 of 152 SMs idle there and took 417 ms; slabs of 32 and 16 columns keep
// all four schedulers of a CTA's SM busy and spread evenly: 213 ms.  Rows past the band's b are skipped.
template <int BMAX, int NC>
__global__ void __launch_bounds__(128) k_sbr_bt_f64(const MmfDesc* __restrict__ descs, const int* __restrict__ idx,
                                                   const double2* __restrict__ store_base,
                                                   const double* __restrict__ Yg, double* __restrict__ work) {
    constexpr int RG = 128 / NC, WG = 32 / NC > 0 ? 32 / NC : 1, NP = RG / WG;  // row groups: all, per warp; partial sums
    __shared__ double2 vs[2][BMAX], ts[2], red[NP][NC], win[BMAX][NC];
    const MmfDesc d = descs[idx[blockIdx.y]];
    const int n = d.n, b = d.band;
    if (blockIdx.x * NC >= n) return;
    const int tx = threadIdx.x, cl = tx % NC, g = tx / NC, warp = tx >> 5;
    const int c = blockIdx.x * NC + cl;
    const bool act = c < n;
    const double2* V = store_base + d.mat_off;
    const double2* T = V + sbr_nref(n, b) * b;
    const double* Y = Yg + d.sq_off;
    double2* Z = reinterpret_cast<double2*>(sbr_zbase(work, d));
    const double2 z0 = make_double2(0.0, 0.0);
    if (act && g == 0) Z[c] = make_double2(Y[c], 0.0);  // row 0: no reflector touches it
    const int np = sbr_passes(n, b);
    for (int s = 0; s < np; ++s) {
        const int jtop = n - 2 - s * b;
        const int64_t off = sbr_off(n, b, s);
        int top = 0;  // window slot of the window's first row (circular over b slots)
        for (int q = g; q < b; q += RG) win[q][cl] = z0;
        __syncthreads();
        if (g == 0 && act)
            win[0][cl] = s == 0 ? make_double2(Y[(int64_t)(n - 1) * n + c], 0.0) : Z[(int64_t)(n - 1) * n + c];
        if (tx < b) vs[0][tx] = V[(off + jtop) * b + tx];
        if (tx == 0) ts[0] = T[off + jtop];
        __syncthreads();
        int buf = 0;
        for (int j = jtop; j >= 0; --j) {
            double2 vn = z0, tn = z0, zn = z0;  // the next step's reflector and row, loading meanwhile
            const int r = j + 1 + s * b;        // first row of the window
            if (j > 0) {
                if (tx < b) vn = V[(off + j - 1) * b + tx];
                if (tx == 0) tn = T[off + j - 1];
                if (g == 0 && act)
                    zn = s == 0 ? make_double2(Y[(int64_t)(r - 1) * n + c], 0.0) : Z[(int64_t)(r - 1) * n + c];
            }
            // w = v^H z over this thread's rows, then over the groups
            double2 w = z0;
            for (int q = g; q < b; q += RG) {
                int sl = top + q;
                sl -= sl >= b ? b : 0;
                w = cmacc(w, vs[buf][q], win[sl][cl]);
            }
#pragma unroll
            for (int o = NC; o < 32; o <<= 1) {
                w.x += __shfl_xor_sync(0xffffffffu, w.x, o);
                w.y += __shfl_xor_sync(0xffffffffu, w.y, o);
            }
            if ((tx & 31) < NC) red[warp % NP][cl] = w;
            __syncthreads();
            w = red[0][cl];
#pragma unroll
            for (int q = 1; q < NP; ++q) w = w + red[q][cl];
            const double2 tw = ts[buf] * w;
            const int bot = top == 0 ? b - 1 : top - 1;  // slot of the window's last row, the one that leaves
            for (int q = g; q < b; q += RG) {
                int sl = top + q;
                sl -= sl >= b ? b : 0;
                const double2 z = cmsub(win[sl][cl], tw, vs[buf][q]);
                if (j > 0 && q == b - 1) {
                    if (act && r + q < n) Z[(int64_t)(r + q) * n + c] = z;
                } else {
                    win[sl][cl] = z;
                }
            }
            if (j > 0) {
                __syncthreads();  // the last row's slot has been read
                if (g == 0) win[bot][cl] = zn;
                top = bot;
                if (tx < b) vs[buf ^ 1][tx] = vn;
                if (tx == 0) ts[buf ^ 1] = tn;
            }
            __syncthreads();
            buf ^= 1;
        }
        const int r0 = 1 + s * b;
        for (int q = g; q < b; q += RG) {
            int sl = top + q;
            sl -= sl >= b ? b : 0;
            if (act && r0 + q < n) Z[(int64_t)(r0 + q) * n + c] = win[sl][cl];
        }
        __syncthreads();
    }
}

// Z (row-major, work slot) -> the back-transform's output (column-major, ld; FP32 for the mixed
// path, FP64 otherwise), 32 x 32 tiles through shared memory.
template <class R>
__global__ void __launch_bounds__(256) k_sbr_out(const MmfDesc* __restrict__ descs, const int* __restrict__ idx,
                                                const double* __restrict__ work, typename Cx<R>::T* __restrict__ out) {
    typedef typename Cx<R>::T C;
    __shared__ C tile[32][33];
    const MmfDesc d = descs[idx[blockIdx.z]];
    const int n = d.n;
    const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
    if (r0 >= n || c0 >= n) return;
    const C* Z = reinterpret_cast<const C*>(sbr_zbase(const_cast<double*>(work), d));
    C* O = out + d.mat_off;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int q = ty; q < 32; q += 8) {
        const int r = r0 + q, c = c0 + tx;
        if (r < n && c < n) tile[q][tx] = Z[(int64_t)r * n + c];
    }
    __syncthreads();
    for (int q = ty; q < 32; q += 8) {
        const int c = c0 + q, r = r0 + tx;
        if (r < n && c < n) O[(int64_t)c * d.ld + r] = tile[tx][q];
    }
}

// ------------------------------------------------------------------ launchers
// The chase with CL CTAs per system; *fits (if given) only reports whether count clusters of that
// size are resident at once (a second wave would double the time).
template <class R, int BMAX, int P, int NG, int CL>
static cudaError_t launch_chase_cl(const MmfLaunch& L, void* H, double2* store, double* dvec, double* evec,
                                   int* status, bool* fits) {
    typedef typename Cx<R>::T C;
    static_assert(sizeof(SbrGroup<C, BMAX, P, sbr_early(CL, NG)>) % 16 == 0, "group blocks keep 16-byte alignment");
    const size_t sm = sbr_hdr(NG) + sizeof(SbrGroup<C, BMAX, P, sbr_early(CL, NG)>) * NG;
    auto kern = k_sbr_chase<R, BMAX, P, NG, CL>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(L.count * CL);
    cfg.blockDim = dim3(BMAX * P * NG);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = L.stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = CL;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (fits) {
        int nc = 0;
        e = cudaOccupancyMaxActiveClusters(&nc, kern, &cfg);
        *fits = e == cudaSuccess && L.count <= nc;
        return e;
    }
    return cudaLaunchKernelEx(&cfg, kern, L.desc, L.idx, (C*)H, (C*)store, dvec, evec, status);
}

// The most CTAs per system (1, 2, 4 or 8) that run in one wave, doubled while the sweeps in flight
// exceed the groups of half of them.  A sweep has up to n / b steps and starts two steps behind its
// predecessor, about one and a half where first rows are published ahead: n / (2 b) to n / (1.5 b) in
// flight, for which the rule takes n / BMAX (b lies in the upper half of a window class, but anywhere in
// the smallest one).  Twice that estimate gives the same times within 1 % from b = 7 to 63, n = 244 to 800,
// 1 to 12 systems, in both precisions; b = 3 at n = 242 would be 10 % (FP32) or 12 % (FP64) faster with the
// 8 CTAs it then takes for 4.  One system of n = 1323, b = 63 in FP32 with 2 CTAs per system takes the 24 ms that
// 64 such systems take, with 8 it takes 13.2.
template <class R, int BMAX, int P, int NG>
static cudaError_t launch_chase(const MmfLaunch& L, void* H, double2* store, double* dvec, double* evec,
                                int* status) {
    const int sweeps = L.nmax / BMAX + 1;
    bool fits = false;
    cudaError_t e = cudaSuccess;
    if (sweeps > 4 * NG) {
        e = launch_chase_cl<R, BMAX, P, NG, 8>(L, H, store, dvec, evec, status, &fits);
        if (e != cudaSuccess) return e;
        if (fits) return launch_chase_cl<R, BMAX, P, NG, 8>(L, H, store, dvec, evec, status, nullptr);
    }
    if (sweeps > 2 * NG) {
        e = launch_chase_cl<R, BMAX, P, NG, 4>(L, H, store, dvec, evec, status, &fits);
        if (e != cudaSuccess) return e;
        if (fits) return launch_chase_cl<R, BMAX, P, NG, 4>(L, H, store, dvec, evec, status, nullptr);
    }
    if (sweeps > NG) {
        e = launch_chase_cl<R, BMAX, P, NG, 2>(L, H, store, dvec, evec, status, &fits);
        if (e != cudaSuccess) return e;
        if (fits) return launch_chase_cl<R, BMAX, P, NG, 2>(L, H, store, dvec, evec, status, nullptr);
    }
    return launch_chase_cl<R, BMAX, P, NG, 1>(L, H, store, dvec, evec, status, nullptr);
}

template <int BMAX>
static cudaError_t launch_bt(const MmfLaunch& L, const double2* store, const double* Y, double* work, int fp32) {
    if (fp32) {
        k_sbr_bt_f32<BMAX><<<dim3((L.nmax + 127) / 128, L.count), 128, 0, L.stream>>>(L.desc, L.idx, store, Y, work);
        return cudaGetLastError();
    }
    // 32 columns per CTA once that gives every SM several CTAs (fewer exchanges per column), else 16
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if ((int64_t)((L.nmax + 31) / 32) * L.count >= 8 * (int64_t)sms)
        k_sbr_bt_f64<BMAX, 32><<<dim3((L.nmax + 31) / 32, L.count), 128, 0, L.stream>>>(L.desc, L.idx, store, Y, work);
    else
        k_sbr_bt_f64<BMAX, 16><<<dim3((L.nmax + 15) / 16, L.count), 128, 0, L.stream>>>(L.desc, L.idx, store, Y, work);
    return cudaGetLastError();
}

int mmf_sbr_class(int b) { return b <= 8 ? 8 : b <= 16 ? 16 : b <= 32 ? 32 : b <= 64 ? 64 : 0; }

cudaError_t mmf_launch_sbr_chase(const MmfLaunch& L, int bmax, void* H, double2* store, double* dvec, double* evec,
                                 int* status, int fp32) {
    if (L.count <= 0) return cudaSuccess;
    if (fp32) {
        switch (bmax) {
            case 8: return launch_chase<float, 8, 4, 16>(L, H, store, dvec, evec, status);
            case 16: return launch_chase<float, 16, 2, 16>(L, H, store, dvec, evec, status);
            case 32: return launch_chase<float, 32, 4, 4>(L, H, store, dvec, evec, status);
            case 64: return launch_chase<float, 64, 4, 2>(L, H, store, dvec, evec, status);
        }
    } else {
        switch (bmax) {
            case 8: return launch_chase<double, 8, 4, 16>(L, H, store, dvec, evec, status);
            case 16: return launch_chase<double, 16, 2, 8>(L, H, store, dvec, evec, status);
            case 32: return launch_chase<double, 32, 4, 4>(L, H, store, dvec, evec, status);
            case 64: return launch_chase<double, 64, 4, 1>(L, H, store, dvec, evec, status);
        }
    }
    return cudaErrorInvalidValue;
}

cudaError_t mmf_launch_sbr_out(const MmfLaunch& L, double* work, float2* Zout) {
    if (L.count <= 0) return cudaSuccess;
    const int t = (L.nmax + 31) / 32;
    k_sbr_out<float><<<dim3(t, t, L.count), 256, 0, L.stream>>>(L.desc, L.idx, work, Zout);
    return cudaGetLastError();
}

cudaError_t mmf_launch_sbr_bt(const MmfLaunch& L, int bmax, const double2* store, const double* Y, double* work,
                              void* Zout, int fp32) {
    if (L.count <= 0) return cudaSuccess;
    cudaError_t e;
    switch (bmax) {
        case 8: e = launch_bt<8>(L, store, Y, work, fp32); break;
        case 16: e = launch_bt<16>(L, store, Y, work, fp32); break;
        case 32: e = launch_bt<32>(L, store, Y, work, fp32); break;
        case 64: e = launch_bt<64>(L, store, Y, work, fp32); break;
        default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    const int t = (L.nmax + 31) / 32;
    dim3 g(t, t, L.count);
    if (fp32) k_sbr_out<float><<<g, 256, 0, L.stream>>>(L.desc, L.idx, work, (float2*)Zout);
    else k_sbr_out<double><<<g, 256, 0, L.stream>>>(L.desc, L.idx, work, (double2*)Zout);
    return cudaGetLastError();
}
