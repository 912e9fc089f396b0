// k_hetrd.cu -- S2: blocked complex Householder reduction of H_F to real tridiagonal form.
//
// The paper hands this step to LAPACK (Sec. 3.2); this is our own GPU formulation of the
// standard blocked reduction (Dongarra, Sorensen & Hammarling 1989).  Lower storage,
// column-major; only the lower triangle is read or updated.
//
// For column k the reflector P_k = I - tau_k v v^H (v[k+1] = 1, v[r] = 0 for r <= k)
// satisfies P_k^H A(k+1:, k) = beta_k e_1 with beta_k real:
//     beta = -sign(Re alpha) sqrt(|alpha|^2 + ||x||^2),  tau = (beta - alpha) / beta,
//     v[k+2:] = x / (alpha - beta)        (alpha = A(k+1, k), x = A(k+2:, k)).
// Two-sided update A <- P^H A P = A - v w^H - w v^H with
//     y = A v,   w = tau y - (1/2) |tau|^2 (v^H y) v.
// Within a panel of NB columns the updates are deferred (V, W kept in global workspace):
// before its reflector, column k receives A(k:, k) -= V W(k,:)^H + W V(k,:)^H, and
// y = A22 v - V (W^H v) - W (V^H v).  After the panel the trailing lower triangle
// receives A -= V W^H + W V^H (her2k).
// Result: d (diagonal), e = beta (sub-diagonal, real), tau, and v[k+2:] stored in
// A(k+2:, k).  Q = P_0 P_1 ... P_{n-2}, Q^H H_F Q = tridiag(e, d, e).
//
// One thread-block cluster of CL CTAs (512 threads each, CL = 1, 2, 4, 6 or 8) per system.  The hemv
// streams the lower triangle of the trailing matrix once per column with coalesced column reads: a
// warp takes tasks of rows (dealt over its lanes) x columns, sums the row part in registers and the
// column part by an exchange over the lanes, and adds both to y in shared memory.  The CTAs split the column blocks of the hemv and the
// tiles of the trailing update; everything of length m is split by rows (chunks of 32 rows dealt
// round-robin): the pending panel updates of the column, the dot products W^H v and V^H v, and the
// corrections of y.  Per column three cluster barriers: the column and its norm reach every CTA
// (pushed through distributed shared memory); the partial hemv results and dot products are
// complete; the scalar w^H v is complete.
//
// What bounds it: with one system per two SMs the hemv's L2 reads and the 2i column reads of the
// panel, repeated by each CTA; with 8 SMs a system the barriers and L2 latencies of a column (a few
// microseconds), which is why the split reaches the O(m i) steps too.  Two systems of n = 1792 in FP32 on 8
// SMs each: 40 ms, of 10.9 warp cycles per instruction 3.2 wait at barriers and 1.4 for loads, L2 at 2 % of
// its rate.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "mmf_internal.h"
#include "umma_common.h"

namespace cg = cooperative_groups;

#define HT_THREADS 512
#define HT_TILE 64
#define HT_CL4_N 256   // smallest n reduced by 4 / 8 CTAs per system
#define HT_CL8_N 384
template <class R>
__device__ __forceinline__ R block_sum(R v, R* red) {
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        R s = (threadIdx.x < HT_THREADS / 32) ? red[threadIdx.x] : R(0);
        s = warp_sum(s);
        if (threadIdx.x == 0) red[32] = s;
    }
    __syncthreads();
    R r = red[32];
    __syncthreads();
    return r;
}


template <class R>
__host__ __device__ constexpr size_t ht_fixed_bytes() {
    return sizeof(typename Cx<R>::T) * (4 * MMF_NB + 4) + sizeof(R) * 72;
}
template <class R>
__host__ __device__ inline size_t ht_big_offset(int nmax) {
    const size_t o = sizeof(typename Cx<R>::T) * 3 * (size_t)nmax + ht_fixed_bytes<R>();
    return (o + 15) & ~(size_t)15;
}
// the partial sums of the O(m i) steps, or the trailing update's operands: FP32 two stages of 64 KB
// at a 1024-byte boundary (tensor cores), FP64 four 32 x 64 tiles
#define HT_TC_STAGE 65536u
template <class R>
__host__ __device__ constexpr size_t ht_big_bytes() {
    return sizeof(R) == 4 ? (size_t)2 * HT_TC_STAGE + 1024
                          : (size_t)4 * MMF_NB * HT_TILE * sizeof(typename Cx<R>::T);
}
static_assert(4 * MMF_NB * HT_TILE * sizeof(float2) <= 2 * HT_TC_STAGE, "FP32-unit tiles fit");

// two block-wide sums in one pass (red holds 2 x 33 values)
template <class R>
__device__ __forceinline__ void block_sum2(R a, R b, R* red, R& sa, R& sb) {
    a = warp_sum(a);
    b = warp_sum(b);
    if ((threadIdx.x & 31) == 0) {
        red[threadIdx.x >> 5] = a;
        red[33 + (threadIdx.x >> 5)] = b;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        R x = (threadIdx.x < HT_THREADS / 32) ? red[threadIdx.x] : R(0);
        R y = (threadIdx.x < HT_THREADS / 32) ? red[33 + threadIdx.x] : R(0);
        x = warp_sum(x);
        y = warp_sum(y);
        if (threadIdx.x == 0) {
            red[32] = x;
            red[65] = y;
        }
    }
    __syncthreads();
    sa = red[32];
    sb = red[65];
    __syncthreads();
}

__device__ __forceinline__ void atomic_add_c(double2* p, double2 v) {
    atomicAdd(&p->x, v.x);
    atomicAdd(&p->y, v.y);
}
__device__ __forceinline__ void atomic_add_c(float2* p, float2 v) {
    atomicAdd(&p->x, v.x);
    atomicAdd(&p->y, v.y);
}


// One warp's share of y = A22 v: tasks of 32 RPL rows (RPL rows per lane: 4 in FP32, 2 in FP64) x cw
// columns on and below the diagonal, dealt round-robin over the warps of all CTAs.  A task goes by in
// blocks of 8 columns, HT_NL columns loading (L2) at a time.  The row part stays in registers over
// the task; the column parts of a block are summed over the lanes by one butterfly that halves the
// values at each exchange.  A warp's time is the latency of its chain
// of loads and exchanges (L2 latency near 1000 cycles), so few long steps beat many short ones: at
// m = 1000 on 8 SMs 9 us, 27 bytes a clock and SM (this product alone, in a loop), where blocks of 4 columns with an exchange and two
// in flight take 12; a ring of cp.async pieces 7 columns deep takes 15 (its instructions per column).
// (HT_NL = 8 measures the same and needs more registers.)  cw is chosen so that every warp gets a few
// tasks.
// FP32: complex products as packed pair FMAs with split accumulators p = sum (a.x v.x, a.y v.y) and
// q = sum (a.x v.y, a.y v.x): sum a v = (p.x - p.y, q.x + q.y), sum conj(a) v = (p.x + p.y, q.x - q.y).
#define HT_NL 4
template <class C> struct HtAcc;  // running sum of products of entries with entries of v
template <> struct HtAcc<float2> {
    float2 p, q;
    __device__ __forceinline__ HtAcc() : p(make_float2(0.f, 0.f)), q(make_float2(0.f, 0.f)) {}
    __device__ __forceinline__ void add(float2 a, float2 v, float2 vs) {  // vs = (v.y, v.x)
        p = __ffma2_rn(a, v, p);
        q = __ffma2_rn(a, vs, q);
    }
    __device__ __forceinline__ void addc(float2 a, float2 v, float2 vs) { add(a, v, vs); }
    __device__ __forceinline__ float2 mul() const { return make_float2(p.x - p.y, q.x + q.y); }   // sum a v
    __device__ __forceinline__ float2 mulc() const { return make_float2(p.x + p.y, q.x - q.y); }  // sum conj(a) v
};
template <> struct HtAcc<double2> {
    double2 p;
    __device__ __forceinline__ HtAcc() : p(make_double2(0.0, 0.0)) {}
    __device__ __forceinline__ void add(double2 a, double2 v, double2) { p = cmac(p, a, v); }
    __device__ __forceinline__ void addc(double2 a, double2 v, double2) { p = cmacc(p, a, v); }
    __device__ __forceinline__ double2 mul() const { return p; }
    __device__ __forceinline__ double2 mulc() const { return p; }
};

// a lane's entries of columns c .. c + NL - 1, rows r + 32 h; a task on the diagonal takes the lower
// triangle and the (real) diagonal only
template <class C, int RPL, int NL, bool DIAG>
__device__ __forceinline__ void ht_load(const C* __restrict__ p, int ld, int m, int r, int c, C (&a)[NL * RPL]) {
#pragma unroll
    for (int j = 0; j < NL; ++j)
#pragma unroll
        for (int h = 0; h < RPL; ++h) {
            C x = czero<C>();
            if (r + 32 * h < m && (!DIAG || r + 32 * h >= c + j)) x = __ldcg(p + (int64_t)j * ld + 32 * h);
            if (DIAG && r + 32 * h == c + j) x.y = 0;
            a[j * RPL + h] = x;
        }
}

template <class R, class C, int RPL, bool DIAG>
__device__ __forceinline__ void ht_task(const C* __restrict__ a22, int ld, int m, const C* __restrict__ vS, C* yS,
                                        int r, int c0, int cw, int lane) {
    constexpr int NL = HT_NL;
    C v[RPL], vs[RPL], a[NL * RPL];
    HtAcc<C> y[RPL];
    const C* p = a22 + (int64_t)c0 * ld + r;
#pragma unroll
    for (int h = 0; h < RPL; ++h) {
        v[h] = r + 32 * h < m ? vS[r + 32 * h] : czero<C>();
        vs[h] = mk(v[h].y, v[h].x);
    }
#pragma unroll 1
    for (int cb = c0; cb < c0 + cw; cb += 8) {
        R z[16];
#pragma unroll
        for (int b = 0; b < 8; b += NL) {
            ht_load<C, RPL, NL, DIAG>(p, ld, m, r, cb + b, a);
            p += NL * (int64_t)ld;
#pragma unroll
            for (int j = 0; j < NL; ++j) {
                const int c = cb + b + j;
                const C vc = vS[DIAG ? min(c, m - 1) : c];
                const C vcs = mk(vc.y, vc.x);
                HtAcc<C> s;
#pragma unroll
                for (int h = 0; h < RPL; ++h) {
                    y[h].add(a[j * RPL + h], vc, vcs);
                    // the diagonal entry counts once, in the row part
                    s.addc(DIAG && r + 32 * h == c ? czero<C>() : a[j * RPL + h], v[h], vs[h]);
                }
                const C f = s.mulc();
                z[2 * (b + j)] = f.x;
                z[2 * (b + j) + 1] = f.y;
            }
        }
        // lanes with bit o of their number set keep the upper half of the values
#pragma unroll
        for (int o = 16; o >= 2; o >>= 1) {
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int e = 0; e < o / 2; ++e) {
                const R keep = up ? z[e + o / 2] : z[e], send = up ? z[e] : z[e + o / 2];
                z[e] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        }
        z[0] += __shfl_xor_sync(0xffffffffu, z[0], 1);
        // lanes 2 q and 2 q + 1 hold value q: re / im (bit 0) of column cb + q / 2
        const int c = cb + (lane >> 2);
        if (!(lane & 1) && (!DIAG || c < m)) atomicAdd(reinterpret_cast<R*>(&yS[c]) + ((lane >> 1) & 1), z[0]);
    }
#pragma unroll
    for (int h = 0; h < RPL; ++h)
        if (r + 32 * h < m) atomic_add_c(&yS[r + 32 * h], y[h].mul());
}

template <class R, class C>
__device__ __forceinline__ void ht_hemv(const C* __restrict__ a22, int ld, int m, const C* __restrict__ vS, C* yS,
                                        int wid, int nw, int lane) {
    constexpr int RPL = sizeof(R) == 4 ? 4 : 2, TR = 32 * RPL;
    // columns per task: about three tasks for each warp, within 16 .. 64
    const int want = (int)((int64_t)m * m / (2 * TR * 3) / nw);
    const int cw = want < 24 ? 16 : want < 48 ? 32 : 64, G = TR / cw;
    const int nt = (m + TR - 1) / TR;
    const int ntask = nt * (nt + 1) / 2 * G;
    for (int t = wid; t < ntask; t += nw) {
        const int tt = t / G;
        int ti = (int)((sqrtf(8.0f * (float)tt + 1.0f) - 1.0f) * 0.5f);
        while ((ti + 1) * (ti + 2) / 2 <= tt) ++ti;
        while (ti * (ti + 1) / 2 > tt) --ti;
        const int tj = tt - ti * (ti + 1) / 2;
        const int c0 = tj * TR + (t - tt * G) * cw, r = ti * TR + lane;
        if (c0 >= m) continue;
        if (ti == tj) ht_task<R, C, RPL, true>(a22, ld, m, vS, yS, r, c0, cw, lane);
        else ht_task<R, C, RPL, false>(a22, ld, m, vS, yS, r, c0, cw, lane);
    }
}

// ------------------------------------------------------------------ trailing update, tensor cores
// A(c0:, c0:) -= V W^H + W V^H on the lower triangle (FP32 path), as real split-TF32 products on
// the tcgen05 engine.  Tiles of 128 rows x 64 complex columns: column block cb = c0 + 64 tj, row
// blocks rb = cb + 128 ti (the first holds the block's diagonal; entries above it are dropped).
// With K' = 128 real entries per row in four chunks of 32 (the panel's columns), ordered
// (Re V, Im V, Re W, Im W),
//     A'(r)       = [Re V(r,:), Im V(r,:), Re W(r,:), Im W(r,:)]
//     B'(2j)      = [Re W(c,:), Im W(c,:), Re V(c,:), Im V(c,:)]        (c = cb + j)
//     B'(2j + 1)  = [-Im W(c,:), Re W(c,:), -Im V(c,:), Re V(c,:)]
// the product D = A' B'^T holds Re and Im of (V W^H + W V^H)(r, c) in columns 2j and 2j + 1
// (Re(a conj b) = ar br + ai bi, Im(a conj b) = ai br - ar bi).  Each operand is split into TF32
// pieces x = x1 + x2 and each chunk's D = A1 B1^T + A1 B2^T + A2 B1^T goes to its own TMEM
// accumulator (4 x 128 columns), which the epilogue sums in FP32 registers: the tensor cores'
// accumulation is cut to 96 terms, and the result stays within a few FP32 roundings of the
// FP32 units' update.  Chunks 0-1 (the V pass) and 2-3 (the W pass) take the same complex
// values: a thread loads its pass's values once (L2) and builds both chunks from registers into
// one of two 64 KB stages, in the tensor cores' layout (K-major, 128-byte swizzle); one thread
// issues each chunk's 12 tcgen05.mma (M = 128, N = 128, K = 8) and commits them to the stage's
// mbarrier, so that the next chunk is built while they run.  Epilogue: warp w reads TMEM lanes
// 32 (w % 4) .. +31 (rows) and columns 32 (w / 4) .. +31 (16 complex columns) of each
// accumulator and subtracts the sum from A, whose old values it loaded when the tile began.
// Every wait is bounded; a wait that gives up makes the routine return false.
#define HT_TC_COLS 512u   // TMEM columns: four 128-column accumulators
struct HtTc {
    unsigned char* st;   // two stages of HT_TC_STAGE bytes (1024-byte aligned)
    uint64_t* bar;       // [0], [1]: stage free; [2]: tile's products done
    uint32_t tmem;
    uint32_t used[2], waited[2], pacc;
};

__device__ __forceinline__ void ht_split4(float* hi, float* lo, int off, float x0, float x1, float x2, float x3) {
    const float4 h = make_float4(tf32_round(x0), tf32_round(x1), tf32_round(x2), tf32_round(x3));
    *reinterpret_cast<float4*>(hi + off) = h;
    *reinterpret_cast<float4*>(lo + off) =
        make_float4(tf32_round(x0 - h.x), tf32_round(x1 - h.y), tf32_round(x2 - h.z), tf32_round(x3 - h.w));
}

__device__ __forceinline__ void ht_tmem_ld32(uint32_t ta, uint32_t* v) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
          "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
          "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(ta));
}

// Tiles are dealt round-robin over nshare CTAs (this one takes those with index % nshare ==
// share).
__device__ bool her2k_tc(float2* __restrict__ A, int ld, int n, int c0, const float2* __restrict__ V,
                         const float2* __restrict__ W, int nb, int nshare, int share, HtTc& T) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t idesc = umma_idesc_mn(2, 128u, 128u);  // TF32 x TF32 -> F32, M = N = 128
    const int ncb = (n - c0 + 63) / 64;
    int tcount = 0;
    bool ok = true;
    for (int tj = 0; tj < ncb && ok; ++tj) {
        const int cb = c0 + 64 * tj;
        for (int rb = cb; rb < n && ok; rb += 128) {
            if ((tcount++ % nshare) != share) continue;
            // old values of this thread's 16 entries (row r, columns cc .. cc + 15), in flight
            // while the operands are built
            const int r = rb + 32 * (warp & 3) + lane, cc = cb + 16 * (warp >> 2);
            float2 old[16];
#pragma unroll
            for (int q = 0; q < 16; ++q)
                old[q] = (r < n && cc + q < n && r >= cc + q) ? A[r + (int64_t)(cc + q) * ld]
                                                                 : make_float2(0.f, 0.f);
            for (int pass = 0; pass < 2 && ok; ++pass) {
                const float2* P = pass ? W : V;   // A' source
                const float2* Q = pass ? V : W;   // B' source
                // items e = tid, tid + 512: operand row rr = e % 128 (lanes over rows: coalesced
                // column reads), K group kq = e / 128 (4 panel columns)
                float2 a[2][4], b[2][4];
#pragma unroll
                for (int it = 0; it < 2; ++it) {
                    const int e = tid + it * HT_THREADS, rr = e & 127, kq = e >> 7;
                    const int ra = rb + rr, cbr = cb + (rr >> 1);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int p = 4 * kq + u;
                        a[it][u] = (p < nb && ra < n) ? P[ra + (int64_t)p * ld] : make_float2(0.f, 0.f);
                        b[it][u] = (p < nb && cbr < n) ? Q[cbr + (int64_t)p * ld] : make_float2(0.f, 0.f);
                    }
                }
                for (int half = 0; half < 2 && ok; ++half) {
                    const int kc = 2 * pass + half, s = half;
                    if (T.used[s] > T.waited[s]) {  // the products that last read this stage are done
                        ok = __syncthreads_and(mbar_wait(&T.bar[s], T.waited[s] & 1u) ? 1 : 0) != 0;
                        ++T.waited[s];
                        if (!ok) break;
                    }
                    float* ahi = reinterpret_cast<float*>(T.st + s * HT_TC_STAGE);
                    float* alo = ahi + 4096;
                    float* bhi = alo + 4096;
                    float* blo = bhi + 4096;
#pragma unroll
                    for (int it = 0; it < 2; ++it) {
                        const int e = tid + it * HT_THREADS, rr = e & 127, kq = e >> 7;
                        const int off = (rr >> 3) * 256 + (rr & 7) * 32 + ((kq ^ (rr & 7)) << 2);
                        // A': Re (half 0) or Im (half 1) of the pass's matrix; B' row rr (column
                        // cb + rr / 2): Re row (rr even) [Re, Im] of the other matrix over the two
                        // halves, Im row (rr odd) [-Im, Re]
                        const int h = rr & 1;
                        float x[4], y[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            x[u] = half ? a[it][u].y : a[it][u].x;
                            y[u] = h ? (half ? b[it][u].x : -b[it][u].y) : (half ? b[it][u].y : b[it][u].x);
                        }
                        ht_split4(ahi, alo, off, x[0], x[1], x[2], x[3]);
                        ht_split4(bhi, blo, off, y[0], y[1], y[2], y[3]);
                    }
                    // the stores above are read by the tensor cores' async proxy
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncthreads();
                    if (tid == 0) {
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const uint32_t sa = smem_u32(ahi);
                        const uint64_t a1 = umma_desc(sa), a2 = umma_desc(sa + 16384u);
                        const uint64_t b1 = umma_desc(sa + 32768u), b2 = umma_desc(sa + 49152u);
                        const uint32_t dacc = T.tmem + 128u * (uint32_t)kc;
#pragma unroll
                        for (int q = 0; q < 4; ++q) {  // 32 bytes (8 TF32) of K per instruction
                            const uint64_t adv = (uint64_t)((q * 32) >> 4);
                            const uint64_t pa[3] = {a1, a1, a2}, pb[3] = {b1, b2, b1};
#pragma unroll
                            for (int pp = 0; pp < 3; ++pp) {
                                const uint32_t accf = (q > 0 || pp > 0) ? 1u : 0u;
                                asm volatile(
                                    "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                                    "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(dacc),
                                    "l"(pa[pp] + adv), "l"(pb[pp] + adv), "r"(idesc), "r"(accf)
                                    : "memory");
                            }
                        }
                        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                         smem_u32(&T.bar[s]))
                                     : "memory");
                        if (kc == 3)
                            asm volatile(
                                "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                                    smem_u32(&T.bar[2]))
                                : "memory");
                    }
                    ++T.used[s];
                }
            }
            if (!ok) break;
            ok = __syncthreads_and(mbar_wait(&T.bar[2], T.pacc) ? 1 : 0) != 0;
            T.pacc ^= 1u;
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t ta = T.tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(32 * (warp >> 2));
            float2 acc[16];
#pragma unroll
            for (int q = 0; q < 16; ++q) acc[q] = make_float2(0.f, 0.f);
#pragma unroll
            for (int kc = 0; kc < 4; ++kc) {
                uint32_t v[32];
                ht_tmem_ld32(ta + 128u * (uint32_t)kc, v);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    acc[q].x += __uint_as_float(v[2 * q]);
                    acc[q].y += __uint_as_float(v[2 * q + 1]);
                }
            }
#pragma unroll
            for (int q = 0; q < 16; ++q)
                if (r < n && cc + q < n && r >= cc + q)
                    A[r + (int64_t)(cc + q) * ld] = make_float2(old[q].x - acc[q].x, old[q].y - acc[q].y);
            // the next tile's first products overwrite the accumulators after the next barrier
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        }
    }
    return ok;
}

template <class R, int CL, bool TC>
__global__ void __launch_bounds__(HT_THREADS, 1)
k_hetrd(const MmfDesc* __restrict__ descs, const int* __restrict__ idx,
        typename Cx<R>::T* __restrict__ H, typename Cx<R>::T* __restrict__ Vpool,
        typename Cx<R>::T* __restrict__ Wpool, double* __restrict__ dvec,
        double* __restrict__ evec, typename Cx<R>::T* __restrict__ taupool, int nmax,
        int* __restrict__ status) {
    static_assert(!TC || sizeof(R) == 4, "tensor-core trailing update on the FP32 path only");
    static_assert(MMF_NB <= 2 * (HT_THREADS / 32), "two columns of the panel per warp");
    typedef typename Cx<R>::T C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint64_t tc_bar[3];
    __shared__ uint32_t tc_tmem;
    // x, then v: the partners push the next column into one buffer while this CTA still reads the other
    C* vBuf = reinterpret_cast<C*>(smem_raw);  // 2 x nmax
    C* yS = vBuf + 2 * (size_t)nmax;            // nmax: this CTA's partial y = A22 v, then its rows of w
    C* wk = yS + nmax;                          // MMF_NB: row k of W, then W^H v
    C* vk = wk + MMF_NB;                        // MMF_NB: row k of V, then V^H v
    C* xw = vk + MMF_NB;                        // MMF_NB: this CTA's part of W^H v
    C* xv = xw + MMF_NB;                        // MMF_NB: this CTA's part of V^H v
    C* sc = xv + MMF_NB;                        // 4 scalars: tau, scale, alpha2
    R* red = reinterpret_cast<R*>(sc + 4);      // 72: 0-15, 32, 33-48, 65 block sums; the rest is pushed
    R* nrmP = red + 16;                         // by the partners: parts of ||x||^2 (8),
    R* dotP = red + 49;                         // parts of w^H v (8 complex),
    R* wnxt = red + 66;                         // w at row k + 1 before its last correction (complex)
    // one region shared by the partial sums of the O(m i) steps and the trailing update's operands
    C* big = reinterpret_cast<C*>(smem_raw + ht_big_offset<R>(nmax));
    C* tVr = big;                               // MMF_NB x HT_TILE (her2k staging, transposed)
    C* tWr = tVr + MMF_NB * HT_TILE;
    C* tVc = tWr + MMF_NB * HT_TILE;
    C* tWc = tVc + MMF_NB * HT_TILE;

    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (CL > 1) ? (int)cluster.block_rank() : 0;
    const MmfDesc d = descs[idx[blockIdx.x / CL]];
    const int n = d.n, ld = d.ld;
    C* A = H + d.mat_off;
    C* V = Vpool + d.pan_off;
    C* W = Wpool + d.pan_off;
    double* dd = dvec + d.vec_off;
    double* ee = evec + d.vec_off;
    C* tau = taupool + d.vec_off;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int NW = HT_THREADS / 32;
    HtTc T = {};
    bool tc_ok = true;
    if constexpr (TC) {
        if (tid == 0) {
            for (int q = 0; q < 3; ++q) mbar_init(&tc_bar[q], 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        if (warp == 0) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tc_tmem)),
                         "r"(HT_TC_COLS)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        T.st = reinterpret_cast<unsigned char*>(((uintptr_t)big + 1023) & ~(uintptr_t)1023);
        T.bar = tc_bar;
        T.tmem = tc_tmem;
    }

    // The first column pushes into the partners' shared memory: every CTA of the cluster has to be running
    // before any of them does.
    if (CL > 1) cluster.sync();

    // Rows in chunks of 32, chunk q with CTA q % CL.  In the O(m i) steps the warps split into CG
    // groups over the panel's columns, each group's NCW warps over this CTA's chunks.
    constexpr int CG = CL >= 6 ? 4 : CL >= 4 ? 2 : 1;
    constexpr int NCW = (HT_THREADS / 32) / CG;
    const int cw = warp % NCW, grp = warp / NCW;
    C* pS = big;  // CG x (32 chunks of this CTA) partial sums (CG > 1)
    C a2 = czero<C>();  // alpha2 of the previous column
    for (int j0 = 0; j0 < n; j0 += MMF_NB) {
        const int nb = min(MMF_NB, n - j0);
        for (int i = 0; i < nb; ++i) {
            const int k = j0 + i, m = n - k - 1;
            C* vS = vBuf + (k & 1) * nmax;           // this column's x, then v, from row k + 1 on
            const C* vP = vBuf + ((k & 1) ^ 1) * nmax;  // the previous column's v, from row k on
            int q0 = k >> 5;                         // this CTA's first chunk with rows >= k
            q0 += (rank - q0 % CL + CL) % CL;
            const int nch = (n - 1) / 32 >= q0 ? ((n - 1) / 32 - q0) / CL + 1 : 0;
            C* col = A + (int64_t)k * ld;
            // (a) pending panel updates of column k; row k of the newest W is formed here
            if (tid < i) {
                wk[tid] = tid == i - 1 ? conj(mk(wnxt[0], wnxt[1]) + a2 * vP[0]) : conj(W[k + (int64_t)tid * ld]);
                vk[tid] = tid == i - 1 ? conj(vP[0]) : conj(V[k + (int64_t)tid * ld]);
            }
            // (CG > 1: the column's entry this thread finishes below, loaded ahead)
            C xpre = czero<C>();
            if (CG > 1 && tid < nch * 32) {
                const int r = (q0 + CL * (tid >> 5)) * 32 + (tid & 31);
                if (r >= k && r < n) xpre = col[r];
            }
            __syncthreads();
            R part = 0;
            auto finish = [&](int r, C x0, C acc) {  // row r of the updated column
                const C x = x0 - acc;
                if (r == k) {
                    dd[k] = (double)x.x;
                } else {
#pragma unroll
                    for (int q = 0; q < CL; ++q) (CL > 1 ? cluster.map_shared_rank(vS, q) : vS)[r - k - 1] = x;
                    if (r >= k + 2) part += abs2(x);
                }
            };
            for (int t = cw; t < nch; t += NCW) {
                const int r = (q0 + CL * t) * 32 + lane;
                // unrolled so that the panel's loads (L2 latency each) are in flight together
                C acc = czero<C>(), acc2 = czero<C>();
                if (r >= k && r < n) {
                    const C x0 = CG == 1 ? col[r] : acc;
#pragma unroll 8
                    for (int c = grp; c < i; c += CG) {
                        acc = cmac(acc, V[r + (int64_t)c * ld], wk[c]);
                        acc2 = cmac(acc2, W[r + (int64_t)c * ld], vk[c]);
                    }
                    if (CG == 1) finish(r, x0, acc + acc2);
                }
                if (CG > 1) pS[(grp * nch + t) * 32 + lane] = acc + acc2;
            }
            if (CG > 1) {
                __syncthreads();
                for (int o = tid; o < nch * 32; o += HT_THREADS) {
                    const int r = (q0 + CL * (o >> 5)) * 32 + (o & 31);
                    if (r < k || r >= n) continue;
                    C acc = pS[o];
#pragma unroll
                    for (int q = 1; q < CG; ++q) acc = acc + pS[q * nch * 32 + o];
                    finish(r, o == tid ? xpre : col[r], acc);
                }
            }
            if (k == n - 1) break;

            // (b) reflector, the same in every CTA
            const R xpart = block_sum(part, red);
            if (CL > 1) {
                if (tid < CL) cluster.map_shared_rank(nrmP, tid)[rank] = xpart;
                cluster.sync();
            }
            if (tid == 0) {
                R xn2 = xpart;
                if (CL > 1) {
                    xn2 = nrmP[0];
#pragma unroll
                    for (int q = 1; q < CL; ++q) xn2 += nrmP[q];
                }
                const C alpha = vS[0];
                C t, s;
                R beta;
                if (xn2 == R(0) && alpha.y == R(0)) {
                    t = czero<C>();
                    s = czero<C>();
                    beta = alpha.x;
                } else {
                    beta = -copysign(sqrt(alpha.x * alpha.x + alpha.y * alpha.y + xn2), alpha.x);
                    t = mk((beta - alpha.x) / beta, -alpha.y / beta);
                    C den = mk(alpha.x - beta, alpha.y);  // 1 / (alpha - beta)
                    R dn = abs2(den);
                    s = mk(den.x / dn, -den.y / dn);
                }
                if (rank == 0) {
                    ee[k] = (double)beta;
                    tau[k] = t;
                }
                sc[0] = t;
                sc[1] = s;
            }
            __syncthreads();
            const C tk = sc[0], scale = sc[1];
            for (int rp = tid; rp < m; rp += HT_THREADS) {
                const C v = rp == 0 ? mk(R(1), R(0)) : vS[rp] * scale;
                const int r = rp + k + 1;
                vS[rp] = v;
                yS[rp] = czero<C>();
                if (CL == 1 || (r >> 5) % CL == rank) {
                    V[r + (int64_t)i * ld] = v;
                    if (rp > 0) col[r] = v;
                }
            }
            __syncthreads();

            // (c) y = A22 v (lower triangle; this CTA's share) and (d) x_w = W^H v, x_v = V^H v (its rows)
            const C* a22 = A + (k + 1) + (int64_t)(k + 1) * ld;
            if (warp < i) {  // columns warp and warp + 16 of both matrices: all loads in flight together
                const int ca = warp, cb = warp + NW < i ? warp + NW : warp;
                const C *Wa = W + (int64_t)ca * ld, *Va = V + (int64_t)ca * ld, *Wb = W + (int64_t)cb * ld,
                        *Vb = V + (int64_t)cb * ld;
                C s0 = czero<C>(), s1 = s0, s2 = s0, s3 = s0;
#pragma unroll 2
                for (int t = 0; t < nch; ++t) {
                    const int r = (q0 + CL * t) * 32 + lane;
                    if (r > k && r < n) {
                        const C v = vS[r - k - 1];
                        s0 = cmacc(s0, Wa[r], v);
                        s1 = cmacc(s1, Va[r], v);
                        s2 = cmacc(s2, Wb[r], v);
                        s3 = cmacc(s3, Vb[r], v);
                    }
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    s0 = s0 + mk(__shfl_xor_sync(0xffffffffu, s0.x, o), __shfl_xor_sync(0xffffffffu, s0.y, o));
                    s1 = s1 + mk(__shfl_xor_sync(0xffffffffu, s1.x, o), __shfl_xor_sync(0xffffffffu, s1.y, o));
                    s2 = s2 + mk(__shfl_xor_sync(0xffffffffu, s2.x, o), __shfl_xor_sync(0xffffffffu, s2.y, o));
                    s3 = s3 + mk(__shfl_xor_sync(0xffffffffu, s3.x, o), __shfl_xor_sync(0xffffffffu, s3.y, o));
                }
                if (lane == 0) {
                    xw[ca] = s0;
                    xv[ca] = s1;
                    xw[cb] = s2;
                    xv[cb] = s3;
                }
            }
            ht_hemv<R, C>(a22, ld, m, vS, yS, warp * CL + rank, NW * CL, lane);
            if (CL > 1) cluster.sync(); else __syncthreads();  // every part of y, x_w and x_v complete
            for (int e = tid; e < 2 * i; e += HT_THREADS) {
                const int c = e >> 1;
                C* src = (e & 1) ? xv : xw;
                C acc = src[c];
                if (CL > 1) {
                    acc = cluster.map_shared_rank(src, 0)[c];
#pragma unroll
                    for (int q = 1; q < CL; ++q) acc = acc + cluster.map_shared_rank(src, q)[c];
                }
                ((e & 1) ? vk : wk)[c] = acc;
            }
            __syncthreads();

            // (d) corrections, (e) w = tau y - (1/2) tau (w^H v) v, on this CTA's rows
            C dpart = czero<C>();
            auto form_w = [&](int rp, C corr) {
                C y = yS[rp];
                if (CL > 1) {
                    y = cluster.map_shared_rank(yS, 0)[rp];
#pragma unroll
                    for (int q = 1; q < CL; ++q) y = y + cluster.map_shared_rank(yS, q)[rp];
                }
                const C w = tk * (y - corr);
                yS[rp] = w;  // (the partners read only their own rows of this CTA's part)
                dpart = dpart + cmulc(w, vS[rp]);
                if (rp == 0) {
#pragma unroll
                    for (int q = 0; q < CL; ++q) {
                        R* pn = CL > 1 ? cluster.map_shared_rank(wnxt, q) : wnxt;
                        pn[0] = w.x;
                        pn[1] = w.y;
                    }
                }
            };
            for (int t = cw; t < nch; t += NCW) {
                const int r = (q0 + CL * t) * 32 + lane;
                C acc = czero<C>(), acc2 = czero<C>();
                if (r > k && r < n) {
#pragma unroll 8
                    for (int c = grp; c < i; c += CG) {
                        acc = cmac(acc, V[r + (int64_t)c * ld], wk[c]);
                        acc2 = cmac(acc2, W[r + (int64_t)c * ld], vk[c]);
                    }
                    if (CG == 1) form_w(r - k - 1, acc + acc2);
                }
                if (CG > 1) pS[(grp * nch + t) * 32 + lane] = acc + acc2;
            }
            if (CG > 1) {
                __syncthreads();
                for (int o = tid; o < nch * 32; o += HT_THREADS) {
                    const int r = (q0 + CL * (o >> 5)) * 32 + (o & 31);
                    if (r <= k || r >= n) continue;
                    C acc = pS[o];
#pragma unroll
                    for (int q = 1; q < CG; ++q) acc = acc + pS[q * nch * 32 + o];
                    form_w(r - k - 1, acc);
                }
            }
            R dx, dy;
            block_sum2(dpart.x, dpart.y, red, dx, dy);
            if (CL > 1) {
                if (tid < CL) {
                    R* pd = cluster.map_shared_rank(dotP, tid);
                    pd[2 * rank] = dx;
                    pd[2 * rank + 1] = dy;
                }
                cluster.sync();
                dx = dotP[0];
                dy = dotP[1];
#pragma unroll
                for (int q = 1; q < CL; ++q) {
                    dx += dotP[2 * q];
                    dy += dotP[2 * q + 1];
                }
            }
            a2 = R(-0.5) * (tk * mk(dx, dy));
            for (int o = tid; o < nch * 32; o += HT_THREADS) {
                const int r = (q0 + CL * (o >> 5)) * 32 + (o & 31);
                if (r > k && r < n) W[r + (int64_t)i * ld] = yS[r - k - 1] + a2 * vS[r - k - 1];
            }
        }
        if (CL > 1) cluster.sync(); else __syncthreads();  // the panel is complete

        // trailing her2k on the lower triangle of A(c0:, c0:)
        const int c0 = j0 + nb;
        if constexpr (TC) {
            if (c0 < n) {
                if (tc_ok)
                    tc_ok = her2k_tc(reinterpret_cast<float2*>(A), ld, n, c0, reinterpret_cast<const float2*>(V),
                                     reinterpret_cast<const float2*>(W), nb, CL, rank, T);
                if (CL > 1) cluster.sync();
            }
        } else if (c0 < n) {
            const int nt = (n - c0 + HT_TILE - 1) / HT_TILE;
            const int rr = tid & (HT_TILE - 1), cg = tid / HT_TILE;  // 8 column groups
            int tcount = 0;
            for (int ti = 0; ti < nt; ++ti) {
                for (int tj = 0; tj <= ti; ++tj) {
                    if ((tcount++ % CL) != rank) continue;
                    const int rbase = c0 + ti * HT_TILE, cbase = c0 + tj * HT_TILE;
                    for (int e = tid; e < nb * HT_TILE; e += HT_THREADS) {
                        const int p = e / HT_TILE, q = e - p * HT_TILE;
                        const int r = rbase + q, c = cbase + q;
                        tVr[e] = (r < n) ? V[r + (int64_t)p * ld] : czero<C>();
                        tWr[e] = (r < n) ? W[r + (int64_t)p * ld] : czero<C>();
                        tVc[e] = (c < n) ? conj(V[c + (int64_t)p * ld]) : czero<C>();
                        tWc[e] = (c < n) ? conj(W[c + (int64_t)p * ld]) : czero<C>();
                    }
                    __syncthreads();
                    C acc[8];
                    if constexpr (sizeof(R) == 4) {
                        // packed FP32 pairs: s1 += (a.x, a.x) c + (b.x, b.x) d, s2 += (a.y, a.y) c + (b.y, b.y) d,
                        // so that a c + b d = (s1.x - s2.y, s1.y + s2.x)
                        float2 s1[8], s2[8];
#pragma unroll
                        for (int q = 0; q < 8; ++q) s1[q] = s2[q] = make_float2(0.f, 0.f);
                        for (int p = 0; p < nb; ++p) {
                            const float2 a = tVr[p * HT_TILE + rr], b = tWr[p * HT_TILE + rr];
                            const float2 ax = make_float2(a.x, a.x), ay = make_float2(a.y, a.y);
                            const float2 bx = make_float2(b.x, b.x), by = make_float2(b.y, b.y);
#pragma unroll
                            for (int q = 0; q < 8; ++q) {
                                const int cc = cg + 8 * q;
                                const float2 c = tWc[p * HT_TILE + cc], dv = tVc[p * HT_TILE + cc];
                                s1[q] = __ffma2_rn(ax, c, s1[q]);
                                s1[q] = __ffma2_rn(bx, dv, s1[q]);
                                s2[q] = __ffma2_rn(ay, c, s2[q]);
                                s2[q] = __ffma2_rn(by, dv, s2[q]);
                            }
                        }
#pragma unroll
                        for (int q = 0; q < 8; ++q) acc[q] = mk(s1[q].x - s2[q].y, s1[q].y + s2[q].x);
                    } else {
#pragma unroll
                        for (int q = 0; q < 8; ++q) acc[q] = czero<C>();
                        for (int p = 0; p < nb; ++p) {
                            const C a = tVr[p * HT_TILE + rr], b = tWr[p * HT_TILE + rr];
#pragma unroll
                            for (int q = 0; q < 8; ++q) {
                                const int cc = cg + 8 * q;
                                acc[q] = cmac(cmac(acc[q], a, tWc[p * HT_TILE + cc]), b, tVc[p * HT_TILE + cc]);
                            }
                        }
                    }
                    const int r = rbase + rr;
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        const int c = cbase + cg + 8 * q;
                        if (r < n && c < n && r >= c) {
                            C* pa = A + r + (int64_t)c * ld;
                            *pa = *pa - acc[q];
                        }
                    }
                    __syncthreads();
                }
            }
            if (CL > 1) cluster.sync();
        }
    }
    if (CL > 1) cluster.sync();  // no CTA leaves while a partner may still read its shared memory
    if constexpr (TC) {
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (warp == 0)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(T.tmem), "r"(HT_TC_COLS) : "memory");
        // a wait of the tensor-core update that gave up (the system's reduction is then incomplete)
        if (!tc_ok && tid == 0) status[idx[blockIdx.x / CL]] = MMF_ST_NOCONV;
    }
}

static size_t hetrd_smem(int nmax, int fp32) {
    return fp32 ? ht_big_offset<float>(nmax) + ht_big_bytes<float>()
                : ht_big_offset<double>(nmax) + ht_big_bytes<double>();
}

int mmf_hetrd_max_n(int fp32) {
    const size_t cs = fp32 ? 8 : 16;
    const size_t fixed = fp32 ? ht_fixed_bytes<float>() + ht_big_bytes<float>()
                              : ht_fixed_bytes<double>() + ht_big_bytes<double>();
    // 64 bytes for the kernel's static shared variables (tensor-core mbarriers, TMEM address) and
    // the 16-byte rounding of the operand region
    return (int)((227 * 1024 - fixed - 64) / (3 * cs));
}

// CL CTAs per system; *fits (if given) only reports whether one wave holds all the clusters.
template <class R, int CL, bool TC>
static cudaError_t launch_hetrd_cl(const MmfLaunch& L, void* H, void* Vp, void* Wp, double* dvec,
                                   double* evec, void* tau, int* status, bool* fits) {
    typedef typename Cx<R>::T C;
    const size_t sm = hetrd_smem(L.nmax, sizeof(R) == 4);
    cudaError_t err = cudaFuncSetAttribute(k_hetrd<R, CL, TC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (err != cudaSuccess) return err;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(L.count * CL);
    cfg.blockDim = dim3(HT_THREADS);
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
        err = cudaOccupancyMaxActiveClusters(&nc, k_hetrd<R, CL, TC>, &cfg);
        *fits = err == cudaSuccess && L.count <= nc;
        return err;
    }
    return cudaLaunchKernelEx(&cfg, k_hetrd<R, CL, TC>, L.desc, L.idx, (C*)H, (C*)Vp, (C*)Wp, dvec, evec,
                              (C*)tau, L.nmax, status);
}

// The most CTAs per system that run in one wave (a GB300 holds 15 clusters of 8, 23 of 6, 36 of 4);
// from 4 on only for systems long enough that each CTA keeps a few row chunks (the barriers of a larger
// cluster cost more than a small column's work).  *ctas (if given) only reports the choice.
template <class R, bool TC>
static cudaError_t launch_hetrd(const MmfLaunch& L, void* H, void* Vp, void* Wp, double* dvec,
                                double* evec, void* tau, int* status, int* ctas) {
    cudaError_t e = cudaSuccess;
    bool done = false;
    auto attempt = [&](auto cl) {  // taken if its clusters fit one wave, and at the latest with one CTA per system
        constexpr int CL = decltype(cl)::value;
        if (done || e != cudaSuccess) return;
        bool fits = CL == 1;
        if (!fits) e = launch_hetrd_cl<R, CL, TC>(L, H, Vp, Wp, dvec, evec, tau, status, &fits);
        if (e != cudaSuccess || !fits) return;
        done = true;
        if (ctas) *ctas = CL;
        else e = launch_hetrd_cl<R, CL, TC>(L, H, Vp, Wp, dvec, evec, tau, status, nullptr);
    };
    if (L.nmax >= HT_CL8_N) {
        attempt(std::integral_constant<int, 8>());
        attempt(std::integral_constant<int, 6>());
    }
    if (L.nmax >= HT_CL4_N) attempt(std::integral_constant<int, 4>());
    attempt(std::integral_constant<int, 2>());
    attempt(std::integral_constant<int, 1>());
    return e;
}

static cudaError_t hetrd(const MmfLaunch& L, void* H, void* Vp, void* Wp, double* dvec, double* evec, void* tau,
                         int fp32, int tc, int* status, int* ctas) {
    if (L.nmax > mmf_hetrd_max_n(fp32)) return cudaErrorInvalidValue;
    if (fp32 && tc) return launch_hetrd<float, true>(L, H, Vp, Wp, dvec, evec, tau, status, ctas);
    if (fp32) return launch_hetrd<float, false>(L, H, Vp, Wp, dvec, evec, tau, status, ctas);
    return launch_hetrd<double, false>(L, H, Vp, Wp, dvec, evec, tau, status, ctas);
}

cudaError_t mmf_launch_hetrd(const MmfLaunch& L, void* H, void* Vp, void* Wp, double* dvec,
                             double* evec, void* tau, int fp32, int tc, int* status) {
    if (L.count <= 0) return cudaSuccess;
    return hetrd(L, H, Vp, Wp, dvec, evec, tau, fp32, tc, status, nullptr);
}

// CTAs per system that a launch of `count` systems, the largest of dimension n, takes
cudaError_t mmf_hetrd_ctas(int n, int count, int fp32, int tc, int* ctas) {
    MmfLaunch L = {};
    L.count = count;
    L.nmax = n;
    return hetrd(L, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, fp32, tc, nullptr, ctas);
}

// ------------------------------------------------------------------ self-test
// `count` seeded Hermitian n x n FP32 matrices (entries uniform in the unit square, full
// mantissas; leading dimension n rounded up to 8) reduced in one launch (at any n, also where a plan
// takes the one-CTA kernel), with the trailing update on the tensor cores (tc = 1) or the
// FP32 units (tc = 0).  For the first two systems the host applies the stored reflectors to the
// input in FP64, B = P_{n-2}^H ... P_0^H A P_0 ... P_{n-2}, and returns max |B - tridiag(e, d, e)|
// (every entry) and max |A|.  Returns 0, -1 (bad sizes), -4 (CUDA failure) or 1 (a wait gave up).
int mmf_hetrd_selftest_impl(int n, int count, int tc, double* max_err, double* max_ref) {
    if (n < 2 || n > mmf_hetrd_max_n(1) || count < 1 || count > 512 || (int64_t)n * n * count > (1 << 27)) return -1;
    const int ld = (n + 7) & ~7;
    const int64_t mat = (int64_t)n * ld, pan = (int64_t)ld * MMF_NB;
    std::vector<MmfDesc> hd(count);
    std::vector<int> hidx(count);
    for (int s = 0; s < count; ++s) {
        MmfDesc d = {};
        d.n = n;
        d.ld = ld;
        d.D = n;
        d.M = 1;
        d.mat_off = s * mat;
        d.pan_off = s * pan;
        d.vec_off = (int64_t)s * n;
        hd[s] = d;
        hidx[s] = s;
    }
    std::vector<float2> hA((size_t)mat * count, make_float2(0.f, 0.f));
    uint64_t x = 0x9E3779B97F4A7C15ull;
    auto unif = [&x]() {  // xorshift64*, uniform in [-1, 1)
        x ^= x >> 12;
        x ^= x << 25;
        x ^= x >> 27;
        return (double)((x * 0x2545F4914F6CDD1Dull) >> 11) * (2.0 / 9007199254740992.0) - 1.0;
    };
    for (int s = 0; s < count; ++s)
        for (int c = 0; c < n; ++c)
            for (int r = c; r < n; ++r) {
                const float re = (float)unif(), im = r == c ? 0.f : (float)unif();
                hA[s * mat + r + (int64_t)c * ld] = make_float2(re, im);
                hA[s * mat + c + (int64_t)r * ld] = make_float2(re, -im);
            }
    MmfDesc* dd = nullptr;
    int *didx = nullptr, *dst = nullptr;
    float2 *dA = nullptr, *dV = nullptr, *dW = nullptr, *dtau = nullptr;
    double *dD = nullptr, *dE = nullptr;
    int rc = 0;
    cudaStream_t st = nullptr;
    if (cudaStreamCreate(&st) != cudaSuccess) return -4;
    bool ok = cudaMalloc(&dd, sizeof(MmfDesc) * count) == cudaSuccess &&
              cudaMalloc(&didx, sizeof(int) * count) == cudaSuccess &&
              cudaMalloc(&dst, sizeof(int) * count) == cudaSuccess &&
              cudaMalloc(&dA, sizeof(float2) * mat * count) == cudaSuccess &&
              cudaMalloc(&dV, sizeof(float2) * pan * count) == cudaSuccess &&
              cudaMalloc(&dW, sizeof(float2) * pan * count) == cudaSuccess &&
              cudaMalloc(&dtau, sizeof(float2) * n * count) == cudaSuccess &&
              cudaMalloc(&dD, sizeof(double) * n * count) == cudaSuccess &&
              cudaMalloc(&dE, sizeof(double) * n * count) == cudaSuccess;
    std::vector<double> hD((size_t)n * count), hE((size_t)n * count);
    std::vector<float2> htau((size_t)n * count);
    std::vector<int> hst(count);
    if (ok) {
        ok = cudaMemcpy(dd, hd.data(), sizeof(MmfDesc) * count, cudaMemcpyHostToDevice) == cudaSuccess &&
             cudaMemcpy(didx, hidx.data(), sizeof(int) * count, cudaMemcpyHostToDevice) == cudaSuccess &&
             cudaMemset(dst, 0, sizeof(int) * count) == cudaSuccess &&
             cudaMemcpy(dA, hA.data(), sizeof(float2) * mat * count, cudaMemcpyHostToDevice) == cudaSuccess &&
             cudaMemset(dV, 0, sizeof(float2) * pan * count) == cudaSuccess &&
             cudaMemset(dW, 0, sizeof(float2) * pan * count) == cudaSuccess;
        MmfLaunch L = {dd, didx, count, n, st};
        ok = ok && mmf_launch_hetrd(L, dA, dV, dW, dD, dE, dtau, 1, tc, dst) == cudaSuccess &&
             cudaStreamSynchronize(st) == cudaSuccess;
        std::vector<float2> hR((size_t)mat * count);
        ok = ok && cudaMemcpy(hR.data(), dA, sizeof(float2) * mat * count, cudaMemcpyDeviceToHost) == cudaSuccess &&
             cudaMemcpy(hD.data(), dD, sizeof(double) * n * count, cudaMemcpyDeviceToHost) == cudaSuccess &&
             cudaMemcpy(hE.data(), dE, sizeof(double) * n * count, cudaMemcpyDeviceToHost) == cudaSuccess &&
             cudaMemcpy(htau.data(), dtau, sizeof(float2) * n * count, cudaMemcpyDeviceToHost) == cudaSuccess &&
             cudaMemcpy(hst.data(), dst, sizeof(int) * count, cudaMemcpyDeviceToHost) == cudaSuccess;
        if (ok) {
            for (int s = 0; s < count; ++s)
                if (hst[s] != 0) rc = 1;
            double err = 0.0, ref = 0.0;
            std::vector<double2> B((size_t)n * n), v(n), y(n);
            for (int s = 0; s < std::min(count, 2); ++s) {
                const float2* A0 = hA.data() + s * mat;
                const float2* R = hR.data() + s * mat;
                for (int c = 0; c < n; ++c)
                    for (int r = 0; r < n; ++r) {
                        const float2 a = A0[r + (int64_t)c * ld];
                        B[r + (size_t)c * n] = make_double2(a.x, a.y);
                        ref = std::max(ref, std::hypot((double)a.x, (double)a.y));
                    }
                for (int k = 0; k + 1 < n; ++k) {  // B <- P_k^H B P_k, P_k = I - tau v v^H
                    const float2 tf = htau[(size_t)s * n + k];
                    const double tr = tf.x, ti = tf.y;
                    for (int r = 0; r < n; ++r) {
                        if (r <= k) v[r] = make_double2(0.0, 0.0);
                        else if (r == k + 1) v[r] = make_double2(1.0, 0.0);
                        else v[r] = make_double2(R[r + (int64_t)k * ld].x, R[r + (int64_t)k * ld].y);
                    }
                    // B <- B P = B - tau (B v) v^H
                    for (int r = 0; r < n; ++r) {
                        double yr = 0.0, yi = 0.0;
                        for (int c = k + 1; c < n; ++c) {
                            const double2 b = B[r + (size_t)c * n];
                            yr += b.x * v[c].x - b.y * v[c].y;
                            yi += b.x * v[c].y + b.y * v[c].x;
                        }
                        const double ur = tr * yr - ti * yi, ui = tr * yi + ti * yr;  // tau (B v)_r
                        for (int c = k + 1; c < n; ++c) {  // - u conj(v_c)
                            double2& b = B[r + (size_t)c * n];
                            b.x -= ur * v[c].x + ui * v[c].y;
                            b.y -= ui * v[c].x - ur * v[c].y;
                        }
                    }
                    // B <- P^H B = B - conj(tau) v (v^H B)
                    for (int c = 0; c < n; ++c) {
                        double yr = 0.0, yi = 0.0;
                        for (int r = k + 1; r < n; ++r) {
                            const double2 b = B[r + (size_t)c * n];
                            yr += v[r].x * b.x + v[r].y * b.y;
                            yi += v[r].x * b.y - v[r].y * b.x;
                        }
                        const double ur = tr * yr + ti * yi, ui = tr * yi - ti * yr;  // conj(tau) (v^H B)_c
                        for (int r = k + 1; r < n; ++r) {
                            double2& b = B[r + (size_t)c * n];
                            b.x -= v[r].x * ur - v[r].y * ui;
                            b.y -= v[r].x * ui + v[r].y * ur;
                        }
                    }
                }
                for (int c = 0; c < n; ++c)
                    for (int r = 0; r < n; ++r) {
                        double2 t = make_double2(0.0, 0.0);
                        if (r == c) t.x = hD[(size_t)s * n + r];
                        else if (r == c + 1) t.x = hE[(size_t)s * n + c];
                        else if (c == r + 1) t.x = hE[(size_t)s * n + r];
                        const double2 b = B[r + (size_t)c * n];
                        err = std::max(err, std::hypot(b.x - t.x, b.y - t.y));
                    }
            }
            *max_err = err;
            *max_ref = ref;
        }
    }
    if (!ok) rc = -4;
    cudaFree(dd);
    cudaFree(didx);
    cudaFree(dst);
    cudaFree(dA);
    cudaFree(dV);
    cudaFree(dW);
    cudaFree(dtau);
    cudaFree(dD);
    cudaFree(dE);
    cudaStreamDestroy(st);
    return rc;
}
