// k_hetrd_large.cu -- S2 for one large system: the blocked Householder reduction of k_hetrd.cu
// (same reflectors, same deferred panel updates, same outputs) spread over the whole GPU.
//
// Only the lower triangle is kept (as on the one-CTA path): y = A22 v is a Hermitian product in
// which each lower entry serves its row and (conjugated) its column; a grid of CTAs each owns a
// 128 x 128 block on or below the diagonal and adds its row and column sums into y with atomics.
// Per column k (panel position i) the host enqueues four launches: (1) the grid finishes the previous
// column's w, applies the pending panel updates to column k and sums |A(r, k)|^2 below the
// subdiagonal, and the last CTA to finish forms the reflector; (2) the grid scales the column into v,
// clears y and sums the short products W^H v, V^H v; (3) the grid forms y = A22 v; (4) the grid
// applies the panel corrections, w = tau y and the partial sums of w^H v.  The column's steps are
// spread over the grid because they read the panel (m x 2i entries): one CTA streamed it at a few tens
// of GB/s, as long as the gemv over the whole trailing matrix.  A column is bound by its launches until
// m is several thousand (n = 5832: 48 us a column, of which the lower triangle's reads at the copy rate
// take 13; with six launches and a row per thread 286 ms, with four and four threads a row 167), so there
// are as few as the dependences allow, and each is launched with programmatic
// stream serialisation: its CTAs are set up while the previous kernel drains and wait for it at their
// start.  After each panel a grid-wide
// update A -= V W^H + W V^H touches the lower triangle of the trailing matrix.  It stays on the
// FP32 / FP64 units: tens of thousands of small CTAs hide its HBM latency, which a tensor-core version
// with one CTA per SM and one tile in flight did not (7.2 against 5.4 ms per panel at n = 17576).
#include "mmf_internal.h"

#define LG_B 256      // threads per CTA
#define LG_R 64       // rows per CTA of the column kernels, LG_G threads to a row: with a thread per row its
#define LG_G (LG_B / LG_R)  // up to 64 panel loads went by in four L2 latencies and 15 CTAs (15 us a kernel)
#define LG_TILE 64    // trailing-update tile

struct LgScalars {     // per-column scalars shared between the launches (device memory)
    double2 tau;       // reflector scalar (in the working precision, widened)
    double2 dot;       // accumulated w^H v
    double2 scale;     // 1 / (alpha - beta): multiplies the column into v
    double xn2;        // accumulated |A(r, k)|^2 over r >= k + 2 (cleared with the reflector)
    unsigned int done;  // CTAs of the column update that have finished (cleared with the reflector)
    unsigned int pad;
};

// Programmatic stream serialisation: a kernel may be started before its predecessor on the stream has
// finished; lg_wait returns once it has (all of its writes visible), lg_go lets the successor start.
// What a kernel reads is thus written while it already runs, up to its lg_wait: no pointer here may be
// declared __restrict__ (data unchanged for the kernel's whole life, which allows read-only loads and loads
// ahead of the wait).
__device__ __forceinline__ void lg_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void lg_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
static_assert(sizeof(LgScalars) <= 8 * sizeof(double), "the scalars fit the system's 8-double auxiliary slot");

template <class R>
__device__ __forceinline__ R cta_sum(R v, R* red) {
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        R s = (threadIdx.x < (int)(blockDim.x >> 5)) ? red[threadIdx.x] : R(0);
        s = warp_sum(s);
        if (threadIdx.x == 0) red[32] = s;
    }
    __syncthreads();
    R r = red[32];
    __syncthreads();
    return r;
}

__device__ __forceinline__ void atomic_add_cx(double2* p, double2 v) {
    atomicAdd(&p->x, v.x);
    atomicAdd(&p->y, v.y);
}
__device__ __forceinline__ void atomic_add_cx(float2* p, float2 v) {
    atomicAdd(&p->x, v.x);
    atomicAdd(&p->y, v.y);
}

// alpha2 = -(1/2) tau (w^H v) of the previous column: w += alpha2 v completes it
template <class C, class R>
__device__ __forceinline__ C lg_alpha2(const LgScalars* sc) {
    const C tk = from_c128<C>(sc->tau);
    return R(-0.5) * (tk * from_c128<C>(sc->dot));
}

// (1) column k = j0 + i over the grid: the last correction of W(:, i - 1) on this CTA's rows, the
// pending panel updates of rows k .., and the sum of |A(r, k)|^2 over r >= k + 2 into sc->xn2; the last
// CTA forms the reflector (one thread) and clears the sums of the column's later steps.  vbuf still
// holds the previous column's v (from row k on).
template <class R>
__global__ void __launch_bounds__(LG_B) k_lg_colupd(typename Cx<R>::T* A, int n, int ld, int k, int i,
                                                    const typename Cx<R>::T* V,
                                                    typename Cx<R>::T* W,
                                                    const typename Cx<R>::T* vbuf,
                                                    typename Cx<R>::T* xbuf, LgScalars* sc,
                                                    double* dd, double* ee,
                                                    typename Cx<R>::T* tau) {
    typedef typename Cx<R>::T C;
    __shared__ C wk[MMF_NB], vk[MMF_NB], ps[LG_G - 1][LG_R];
    __shared__ R red[33];
    __shared__ bool last;
    const int tid = threadIdx.x;
    lg_wait();
    lg_go();
    const C a2 = i > 0 ? lg_alpha2<C, R>(sc) : czero<C>();
    if (tid < i) {
        const C v = V[k + (int64_t)tid * ld];
        // (row k of W(:, i - 1) is corrected by the first CTA of this launch: from its uncorrected copy)
        const C w = tid == i - 1 ? xbuf[2 * MMF_NB] + a2 * v : W[k + (int64_t)tid * ld];
        wk[tid] = conj(w);
        vk[tid] = conj(v);
    }
    __syncthreads();
    // thread (row, g): columns g, g + LG_G, ... of the panel, all of them loaded before the one store
    const int rl = tid & (LG_R - 1), g = tid / LG_R, r = k + blockIdx.x * LG_R + rl;
    C acc = czero<C>(), acc2 = czero<C>(), x = czero<C>();
    if (r < n) {
        constexpr int NU = MMF_NB / LG_G;
        C w[NU], v[NU], vp = czero<C>();
        if (g == 0) x = A[(int64_t)k * ld + r];
        if (i > 0) vp = vbuf[r - k];
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            const int c = g + u * LG_G;
            w[u] = c < i ? W[r + (int64_t)c * ld] : czero<C>();
            v[u] = c < i ? V[r + (int64_t)c * ld] : czero<C>();
        }
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            const int c = g + u * LG_G;
            if (c < i) {
                if (c == i - 1) {
                    w[u] = w[u] + a2 * vp;
                    W[r + (int64_t)c * ld] = w[u];
                }
                acc = cmac(acc, v[u], wk[c]);
                acc2 = cmac(acc2, w[u], vk[c]);
            }
        }
    }
    if (g > 0) ps[g - 1][rl] = acc + acc2;
    __syncthreads();
    R part = 0;
    if (g == 0 && r < n) {
        acc = acc + acc2;
#pragma unroll
        for (int q = 0; q < LG_G - 1; ++q) acc = acc + ps[q][rl];
        if (i > 0) {
            x = x - acc;
            A[(int64_t)k * ld + r] = x;
        }
        if (r >= k + 2) part = abs2(x);
    }
    const R sum = cta_sum(part, red);
    if (tid == 0) {
        if (sum != R(0)) atomicAdd(&sc->xn2, (double)sum);
        __threadfence();
        last = atomicAdd(&sc->done, 1u) + 1u == gridDim.x;
    }
    __syncthreads();
    if (!last) return;
    if (tid < 2 * MMF_NB) xbuf[tid] = czero<C>();
    if (tid != 0) return;
    __threadfence();
    const C* col = A + (int64_t)k * ld;
    dd[k] = (double)__ldcg(col + k).x;
    const R xn2 = (R)__ldcg(&sc->xn2);
    sc->xn2 = 0.0;
    sc->done = 0u;
    if (k == n - 1) return;
    const C alpha = __ldcg(col + k + 1);
    C t, s;
    R beta;
    if (xn2 == R(0) && alpha.y == R(0)) {
        t = czero<C>();
        s = czero<C>();
        beta = alpha.x;
    } else {
        beta = -copysign(sqrt(alpha.x * alpha.x + alpha.y * alpha.y + xn2), alpha.x);
        t = mk((beta - alpha.x) / beta, -alpha.y / beta);
        const C den = mk(alpha.x - beta, alpha.y);
        const R dn = abs2(den);
        s = mk(den.x / dn, -den.y / dn);
    }
    ee[k] = (double)beta;
    tau[k] = t;
    sc->tau = to_c128(t);
    sc->scale = to_c128(s);
    sc->dot = make_double2(0.0, 0.0);
}

// (2) v from column k over the grid (rows of this CTA): A(r, k) <- v_r below the subdiagonal,
// V(:, i), vbuf, y = 0; then the CTA's parts of x_w = W^H v and x_v = V^H v (warp per product)
template <class R>
__global__ void __launch_bounds__(LG_B) k_lg_vscale(typename Cx<R>::T* A, int n, int ld, int k, int i,
                                                    typename Cx<R>::T* V,
                                                    const typename Cx<R>::T* W,
                                                    typename Cx<R>::T* vbuf,
                                                    typename Cx<R>::T* ybuf,
                                                    typename Cx<R>::T* xbuf, const LgScalars* sc) {
    typedef typename Cx<R>::T C;
    __shared__ C vs[LG_R];
    const int tid = threadIdx.x, r0 = blockIdx.x * LG_R, r = r0 + tid;
    lg_wait();
    lg_go();
    const C scale = from_c128<C>(sc->scale);
    if (tid < LG_R) {
        C v = czero<C>();
        if (r < n) {
            if (r == k + 1) {
                v = mk(R(1), R(0));
            } else if (r > k + 1) {
                C* pc = A + (int64_t)k * ld + r;
                v = *pc * scale;
                *pc = v;
            }
            if (r > k) {
                vbuf[r - k - 1] = v;
                ybuf[r - k - 1] = czero<C>();
            }
            V[r + (int64_t)i * ld] = v;
        }
        vs[tid] = v;  // zero at and above row k, and past n
    }
    __syncthreads();
    if (r0 + LG_R <= k + 1) return;  // no row of this CTA lies below row k
    // a warp's up to eight products together, so that all of their loads are in flight
    const int lane = tid & 31, warp = tid >> 5;
    constexpr int NW = LG_B / 32, NQ = 2 * MMF_NB / NW;
    C acc[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) acc[q] = czero<C>();
#pragma unroll
    for (int u = 0; u < LG_R / 32; ++u) {
        const int rr = r0 + lane + 32 * u;
        const C v = vs[lane + 32 * u];
        if (rr > k && rr < n) {
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const int task = warp + NW * q;
                const C* P = (task & 1) ? V : W;
                if (task < 2 * i) acc[q] = cmacc(acc[q], P[rr + (int64_t)(task >> 1) * ld], v);
            }
        }
    }
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        const int task = warp + NW * q;
        if (task >= 2 * i) break;
        acc[q].x = warp_sum(acc[q].x);
        acc[q].y = warp_sum(acc[q].y);
        if (lane == 0) atomic_add_cx(&xbuf[task], acc[q]);  // xbuf[2c] = (W^H v)_c, xbuf[2c+1] = (V^H v)_c
    }
}

// (3) y += A22 v from the lower triangle of A22 = A(k+1:, k+1:): one CTA per 128 x 128 block
// (I, J) with I >= J, numbered along block rows (block b: I = floor((sqrt(8 b + 1) - 1) / 2),
// J = b - I (I + 1) / 2).  Thread (row r, column half h) reads its 64 entries A(r, c) once and
// adds a(r, c) v_c to its row's sum and conj(a(r, c)) v_r to column c's sum (strictly below the
// diagonal; the diagonal entry once, as a real number).  Column sums: a butterfly reduce-scatter
// of 8 columns at a time over the 32 rows of a warp (16 shuffles for 16 values), then shared
// memory over the block's four warps of that half.
#define LG_HB 128
template <class R>
__global__ void __launch_bounds__(256) k_lg_hemv(const typename Cx<R>::T* A, int n, int ld, int k,
                                                 const typename Cx<R>::T* vbuf,
                                                 typename Cx<R>::T* ybuf) {
    typedef typename Cx<R>::T C;
    __shared__ C vr_s[LG_HB], vc_s[LG_HB];
    __shared__ C colsum[4][LG_HB];  // [warp within the half][column]
    const int m = n - k - 1;
    const int bI = (int)((sqrt(8.0 * blockIdx.x + 1.0) - 1.0) * 0.5);
    int I = bI, J = (int)blockIdx.x - bI * (bI + 1) / 2;
    if (J > I) {  // rounding of the square root: the next block row
        J -= I + 1;
        ++I;
    } else if (J < 0) {  // or the previous one
        --I;
        J += I + 1;
    }
    const int r0 = I * LG_HB, c0 = J * LG_HB;
    if (r0 >= m) return;
    const int tid = threadIdx.x;
    lg_wait();
    lg_go();
    if (tid < LG_HB) {
        vr_s[tid] = (r0 + tid < m) ? vbuf[r0 + tid] : czero<C>();
        vc_s[tid] = (c0 + tid < m) ? vbuf[c0 + tid] : czero<C>();
    }
    __syncthreads();
    const int rl = tid & (LG_HB - 1), h = tid >> 7, lane = tid & 31, wq = (tid >> 5) & 3;
    const int r = r0 + rl;
    const bool rok = r < m;
    const C vr = vr_s[rl];
    const C* a = A + (k + 1 + (rok ? r : 0)) + (int64_t)(k + 1 + c0 + 64 * h) * ld;
    C acc = czero<C>();
    auto load = [&](int q0, C* av) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int cl = 64 * h + q0 + u, c = c0 + cl;
            const bool ok = rok && c < m && (I > J || c <= r);
            av[u] = ok ? a[(int64_t)(q0 + u) * ld] : czero<C>();
        }
    };
    C av[8];
    load(0, av);
#pragma unroll 2
    for (int q0 = 0; q0 < 64; q0 += 8) {
        C nx[8] = {};  // the next 8 columns, loading while these are multiplied
        if (q0 + 8 < 64) load(q0 + 8, nx);
        R cv[16];  // column parts of the 8 columns (Re, Im), strictly below the diagonal
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int cl = 64 * h + q0 + u, c = c0 + cl;
            const bool diag = (I == J) && c == r;
            const C aa = diag ? mk(av[u].x, R(0)) : av[u];
            acc = cmac(acc, aa, vc_s[cl]);
            const C cp = diag ? czero<C>() : cmulc(av[u], vr);
            cv[2 * u] = cp.x;
            cv[2 * u + 1] = cp.y;
        }
        // the 16 sums over the warp's 32 rows by a butterfly reduce-scatter: after the rounds
        // with lane offsets 16, 8, 4, 2 lane L holds value (L >> 1) & 15 summed over 16 lanes,
        // and the last round adds its partner's
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            const bool hi = lane & 16;
            const R keep = hi ? cv[t + 8] : cv[t], send = hi ? cv[t] : cv[t + 8];
            cv[t] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
        }
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const bool hi = lane & 8;
            const R keep = hi ? cv[t + 4] : cv[t], send = hi ? cv[t] : cv[t + 4];
            cv[t] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
        }
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const bool hi = lane & 4;
            const R keep = hi ? cv[t + 2] : cv[t], send = hi ? cv[t] : cv[t + 2];
            cv[t] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
        }
        {
            const bool hi = lane & 2;
            const R keep = hi ? cv[1] : cv[0], send = hi ? cv[0] : cv[1];
            cv[0] = keep + __shfl_xor_sync(0xffffffffu, send, 2);
        }
        cv[0] += __shfl_xor_sync(0xffffffffu, cv[0], 1);
        if ((lane & 1) == 0) {
            const int idx = (lane >> 1) & 15;  // column q0 + idx / 2, Re (idx even) or Im
            reinterpret_cast<R*>(&colsum[wq][64 * h + q0 + (idx >> 1)])[idx & 1] = cv[0];
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) av[u] = nx[u];
    }
    if (rok) atomic_add_cx(&ybuf[r], acc);
    __syncthreads();
    if (tid < LG_HB) {
        const int c = c0 + tid;
        if (c < m) {
            // the four warps of the column's half: rows 0..127 of the block
            C s = colsum[0][tid];
            for (int w = 1; w < 4; ++w) s = s + colsum[w][tid];
            atomic_add_cx(&ybuf[c], s);
        }
    }
}

// (4) y -= V x_w + W x_v;  w = tau y (into W(:, i));  dot += w^H v;  w at row k + 1 also into
// xbuf[2 NB], where the next column's CTAs read it while its owner corrects W
template <class R>
__global__ void __launch_bounds__(LG_B) k_lg_w(int n, int ld, int k, int i,
                                               const typename Cx<R>::T* V,
                                               typename Cx<R>::T* W,
                                               const typename Cx<R>::T* vbuf,
                                               const typename Cx<R>::T* ybuf,
                                               typename Cx<R>::T* xbuf, LgScalars* sc) {
    typedef typename Cx<R>::T C;
    __shared__ C xs[2 * MMF_NB], ps[LG_G - 1][LG_R];
    __shared__ R red[33];
    const int m = n - k - 1;
    lg_wait();
    lg_go();
    if (threadIdx.x < 2 * i) xs[threadIdx.x] = xbuf[threadIdx.x];
    __syncthreads();
    const C tk = from_c128<C>(sc->tau);
    const int rl = threadIdx.x & (LG_R - 1), g = threadIdx.x / LG_R, rp = blockIdx.x * LG_R + rl;
    C acc = czero<C>(), acc2 = czero<C>(), y = czero<C>();
    if (rp < m) {
        if (g == 0) y = ybuf[rp];
#pragma unroll
        for (int u = 0; u < MMF_NB / LG_G; ++u) {
            const int c = g + u * LG_G;
            if (c < i) {
                acc = cmac(acc, V[(k + 1 + rp) + (int64_t)c * ld], xs[2 * c]);
                acc2 = cmac(acc2, W[(k + 1 + rp) + (int64_t)c * ld], xs[2 * c + 1]);
            }
        }
    }
    if (g > 0) ps[g - 1][rl] = acc + acc2;
    __syncthreads();
    C dpart = czero<C>();
    if (g == 0 && rp < m) {
        acc = acc + acc2;
#pragma unroll
        for (int q = 0; q < LG_G - 1; ++q) acc = acc + ps[q][rl];
        const C w = tk * (y - acc);
        W[(k + 1 + rp) + (int64_t)i * ld] = w;
        if (rp == 0) xbuf[2 * MMF_NB] = w;
        dpart = cmulc(w, vbuf[rp]);
    }
    const R dx = cta_sum(dpart.x, red), dy = cta_sum(dpart.y, red);
    if (threadIdx.x == 0) atomic_add_cx(&sc->dot, make_double2((double)dx, (double)dy));
}

// the last correction of a panel's last column, W(:, i) += alpha2 v below row k
template <class R>
__global__ void __launch_bounds__(LG_B) k_lg_w2(int n, int ld, int k, int i, typename Cx<R>::T* W,
                                                const typename Cx<R>::T* vbuf, const LgScalars* sc) {
    typedef typename Cx<R>::T C;
    lg_wait();
    lg_go();
    const int r = k + 1 + blockIdx.x * LG_B + threadIdx.x;
    if (r < n) W[r + (int64_t)i * ld] = W[r + (int64_t)i * ld] + lg_alpha2<C, R>(sc) * vbuf[r - k - 1];
}

// trailing update of the lower triangle: A(c0:, c0:) -= V W^H + W V^H, 64 x 64 tiles on and below
// the diagonal (the diagonal tiles masked to r >= c), the panel's columns staged 8 at a time
#define LG_KC 8
template <class R>
__global__ void __launch_bounds__(256) k_lg_her2k(typename Cx<R>::T* A, int n, int ld, int c0, int nb,
                                                  const typename Cx<R>::T* V,
                                                  const typename Cx<R>::T* W) {
    typedef typename Cx<R>::T C;
    __shared__ C tVr[LG_KC][LG_TILE], tWr[LG_KC][LG_TILE], tVc[LG_KC][LG_TILE], tWc[LG_KC][LG_TILE];
    const int rbase = c0 + blockIdx.x * LG_TILE, cbase = c0 + blockIdx.y * LG_TILE;
    lg_wait();
    lg_go();
    if (rbase >= n || cbase >= n || blockIdx.x < blockIdx.y) return;
    const int rr = threadIdx.x & 63, cg = threadIdx.x >> 6;  // 4 column groups, 16 columns each
    C acc[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) acc[q] = czero<C>();
    for (int p0 = 0; p0 < nb; p0 += LG_KC) {
        __syncthreads();
        for (int e = threadIdx.x; e < LG_KC * LG_TILE; e += 256) {
            const int p = e / LG_TILE, q = e - p * LG_TILE;
            const int r = rbase + q, c = cbase + q;
            const bool pv = p0 + p < nb;
            tVr[p][q] = (pv && r < n) ? V[r + (int64_t)(p0 + p) * ld] : czero<C>();
            tWr[p][q] = (pv && r < n) ? W[r + (int64_t)(p0 + p) * ld] : czero<C>();
            tVc[p][q] = (pv && c < n) ? conj(V[c + (int64_t)(p0 + p) * ld]) : czero<C>();
            tWc[p][q] = (pv && c < n) ? conj(W[c + (int64_t)(p0 + p) * ld]) : czero<C>();
        }
        __syncthreads();
#pragma unroll
        for (int p = 0; p < LG_KC; ++p) {
            const C a = tVr[p][rr], b = tWr[p][rr];
#pragma unroll
            for (int q = 0; q < 16; ++q) {
                const int cc = cg + 4 * q;
                acc[q] = cmac(cmac(acc[q], a, tWc[p][cc]), b, tVc[p][cc]);
            }
        }
    }
    const int r = rbase + rr;
    if (r < n)
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            const int c = cbase + cg + 4 * q;
            if (c < n && r >= c) {
                C* pa = A + r + (int64_t)c * ld;
                *pa = *pa - acc[q];
            }
        }
}

// a launch with programmatic stream serialisation (see lg_wait)
template <class... P, class... X>
static cudaError_t lg_launch(void (*kern)(P...), dim3 grid, cudaStream_t st, X... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, P(args)...);
}
static_assert(LG_B == 256, "every kernel of the reduction has 256 threads");

template <class R>
static cudaError_t run_large(typename Cx<R>::T* A, int n, int ld, typename Cx<R>::T* V, typename Cx<R>::T* W,
                             typename Cx<R>::T* work, LgScalars* sc, double* dd, double* ee,
                             typename Cx<R>::T* tau, cudaStream_t st) {
    typedef typename Cx<R>::T C;
    C* vbuf = work;
    C* ybuf = work + n;
    C* xbuf = work + 2 * (size_t)n;  // 2 NB sums, then w at row k + 1
    cudaError_t e = cudaMemsetAsync(sc, 0, sizeof(LgScalars), st);
    for (int j0 = 0; j0 < n && e == cudaSuccess; j0 += MMF_NB) {
        const int nb = min(MMF_NB, n - j0);
        for (int i = 0; i < nb && e == cudaSuccess; ++i) {
            const int k = j0 + i, m = n - k - 1;
            e = lg_launch(k_lg_colupd<R>, dim3((n - k + LG_R - 1) / LG_R), st, A, n, ld, k, i, V, W, vbuf, xbuf, sc, dd,
                          ee, tau);
            if (k == n - 1) break;
            const int g = (m + LG_B - 1) / LG_B, gb = (m + LG_HB - 1) / LG_HB;
            if (e == cudaSuccess)
                e = lg_launch(k_lg_vscale<R>, dim3((n + LG_R - 1) / LG_R), st, A, n, ld, k, i, V, W, vbuf, ybuf, xbuf, sc);
            if (e == cudaSuccess) e = lg_launch(k_lg_hemv<R>, dim3(gb * (gb + 1) / 2), st, A, n, ld, k, vbuf, ybuf);
            if (e == cudaSuccess) e = lg_launch(k_lg_w<R>, dim3((m + LG_R - 1) / LG_R), st, n, ld, k, i, V, W, vbuf, ybuf, xbuf, sc);
            if (e == cudaSuccess && i == nb - 1) e = lg_launch(k_lg_w2<R>, dim3(g), st, n, ld, k, i, W, vbuf, sc);
        }
        const int c0 = j0 + nb;
        if (c0 < n && e == cudaSuccess) {
            const int g = (n - c0 + LG_TILE - 1) / LG_TILE;
            e = lg_launch(k_lg_her2k<R>, dim3(g, g), st, A, n, ld, c0, nb, V, W);
        }
    }
    return e == cudaSuccess ? cudaGetLastError() : e;
}

// One large system (host-side descriptor copy `d`, device pointers into the batch pools).
// work: 2 n + 2 NB + 1 complex elements of the working precision, aligned to one; sc: one LgScalars.
cudaError_t mmf_launch_hetrd_large(const MmfDesc& d, void* H, void* Vp, void* Wp, double* dvec, double* evec,
                                   void* tau, void* work, void* sc, int fp32, cudaStream_t st) {
    if (fp32)
        return run_large<float>((float2*)H + d.mat_off, d.n, d.ld, (float2*)Vp + d.pan_off, (float2*)Wp + d.pan_off,
                                (float2*)work, (LgScalars*)sc, dvec + d.vec_off, evec + d.vec_off,
                                (float2*)tau + d.vec_off, st);
    return run_large<double>((double2*)H + d.mat_off, d.n, d.ld, (double2*)Vp + d.pan_off, (double2*)Wp + d.pan_off,
                             (double2*)work, (LgScalars*)sc, dvec + d.vec_off, evec + d.vec_off,
                             (double2*)tau + d.vec_off, st);
}
