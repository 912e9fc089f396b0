// k_hetrd_small.cu -- S2 for small systems: complex Householder reduction of H_F to real tridiagonal
// form with the whole matrix in one CTA's shared memory.
//
// The reflectors and conventions are those of k_hetrd.cu (P_k^H A(k+1:, k) = beta_k e_1 with beta_k
// real; d, e, tau, and v[k+2:] stored in A(k+2:, k)), the update is unblocked: per column
//   x = A(k+1:, k) -> v, tau, beta;  y = A22 v;  w = tau y - (1/2) |tau|^2 (v^H y) v;
//   A22 <- A22 - v w^H - w v^H.
// The lower triangle is kept packed by columns (n (n + 1) / 2 entries), so several CTAs share an SM.
//
// Why a kernel of its own: at n = 82 the panel form of k_hetrd spends a column's 50 microseconds in
// barriers, L2 latencies and short dot products over the panel.  Here the FP64 units are what a column
// waits for most (one warp-wide FP64 instruction per 64 cycles and scheduler, 19 cycles over the SM's four:
// one system keeps its SM's at 61 %, the rest is barriers and shared memory's latency): the O(m^2)
// steps run on all warps (the update over the packed triangle's entries in line, so that no lane idles
// at a column's end), the O(m) ones a row per thread, and the scalars in one warp.  Measured in FP64
// at n = 82: one system 1.0 ms (k_hetrd 4.3), 200 systems 1.5 ms (k_hetrd 8.4).
#include "mmf_internal.h"

#define HS_THREADS 512
#define HS_WARPS (HS_THREADS / 32)
#define HS_ROWS 160   // at least the largest n

// entry (r, c), r >= c, of the packed lower triangle
__device__ __forceinline__ int hs_at(int n, int r, int c) { return c * n - c * (c - 1) / 2 + r - c; }

template <class R>
__host__ __device__ constexpr size_t hs_bytes(int n) {
    // triangle, v, w, partial sums of y
    return sizeof(typename Cx<R>::T) * ((size_t)n * (n + 1) / 2 + (2 + HS_WARPS) * (size_t)n);
}

template <class R>
__global__ void __launch_bounds__(HS_THREADS)
k_hetrd_small(const MmfDesc* __restrict__ descs, const int* __restrict__ idx, typename Cx<R>::T* __restrict__ H,
              double* __restrict__ dvec, double* __restrict__ evec, typename Cx<R>::T* __restrict__ taupool) {
    typedef typename Cx<R>::T C;
    extern __shared__ __align__(16) unsigned char hs_smem[];
    __shared__ C s_tau, s_scale, s_dot[HS_ROWS / 32];
    const MmfDesc d = descs[idx[blockIdx.x]];
    const int n = d.n, ld = d.ld;
    C* A = H + d.mat_off;
    double* dd = dvec + d.vec_off;
    double* ee = evec + d.vec_off;
    C* tau = taupool + d.vec_off;
    C* L = reinterpret_cast<C*>(hs_smem);
    C* v = L + (size_t)n * (n + 1) / 2;
    C* w = v + n;
    C* part = w + n;  // HS_WARPS x n
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    for (int c = warp; c < n; c += HS_WARPS)
        for (int r = c + lane; r < n; r += 32) L[hs_at(n, r, c)] = A[r + (int64_t)c * ld];
    __syncthreads();
    for (int k = 0; k < n - 1; ++k) {
        const int m = n - k - 1, k1 = k + 1;
        const C* x = L + hs_at(n, k1, k);  // column k below the diagonal
        if (warp == 0) {
            R s = R(0);
            for (int e = 1 + lane; e < m; e += 32) s += abs2(x[e]);
            s = warp_sum(s);
            C t, scale;
            R beta;
            warp_reflector<R, C>(x[0], s, lane, t, beta, scale);
            if (lane == 0) {
                dd[k] = (double)L[hs_at(n, k, k)].x;
                ee[k] = (double)beta;
                tau[k] = t;
                s_tau = t;
                s_scale = scale;
            }
        }
        __syncthreads();
        if (tid < m) {
            const C ve = tid == 0 ? mk(R(1), R(0)) : x[tid] * s_scale;
            v[tid] = ve;
            if (tid > 0) A[k1 + tid + (int64_t)k * ld] = ve;  // for the back-transform
        }
        __syncthreads();
        // y = A22 v: the warps split into groups of rows (32 each) and, within them, of columns
        const int nrb = (m + 31) / 32;
        const int np = HS_WARPS / nrb;  // warps per row block
        if (warp < nrb * np) {
            const int rb = warp / np, p = warp - rb * np;
            const int i = rb * 32 + lane;  // row k1 + i
            if (i < m) {
                // entry (i, c): from the lower triangle along the lanes (c <= i), or the conjugate of
                // (c, i) from the lane's own column
                C a0 = czero<C>(), a1 = czero<C>();
                auto entry = [&](int c) {
                    C a = L[c <= i ? hs_at(n, k1 + i, k1 + c) : hs_at(n, k1 + c, k1 + i)];
                    a.y = c < i ? a.y : c == i ? R(0) : -a.y;
                    return a;
                };
                int c = p;
                for (; c + np < m; c += 2 * np) {  // two independent chains
                    a0 = cmac(a0, entry(c), v[c]);
                    a1 = cmac(a1, entry(c + np), v[c + np]);
                }
                if (c < m) a0 = cmac(a0, entry(c), v[c]);
                part[p * n + i] = a0 + a1;
            }
        }
        __syncthreads();
        C u = czero<C>();
        if (warp < nrb) {
            C dot = czero<C>();
            if (tid < m) {
                C y = part[tid], y1 = czero<C>();
                for (int p = 1; p < np; p += 2) {
                    y1 = y1 + part[p * n + tid];
                    if (p + 1 < np) y = y + part[(p + 1) * n + tid];
                }
                u = s_tau * (y + y1);
                dot = cmulc(u, v[tid]);
            }
            dot.x = warp_sum(dot.x);
            dot.y = warp_sum(dot.y);
            if (lane == 0) s_dot[warp] = dot;
        }
        __syncthreads();
        if (tid < m) {
            C dot = s_dot[0];
            for (int q = 1; q < nrb; ++q) dot = dot + s_dot[q];
            w[tid] = u + (R(-0.5) * (s_tau * dot)) * v[tid];
        }
        __syncthreads();
        // A22 <- A22 - v w^H - w v^H over the packed triangle from (k1, k1) on
        C* tri = L + hs_at(n, k1, k1);
        const int ne = m * (m + 1) / 2;
        for (int e = tid; e < ne; e += HS_THREADS) {
            // column c of entry e: the triangle from its end, u = ne - 1 - e, has rows of 1, 2, ... entries
            const int uu = ne - 1 - e;
            int q = (int)((sqrtf(8.0f * (float)uu + 1.0f) - 1.0f) * 0.5f);
            if ((q + 1) * (q + 2) / 2 <= uu) ++q;
            if (q * (q + 1) / 2 > uu) --q;
            const int c = m - 1 - q, i = m - 1 - (uu - q * (q + 1) / 2);
            // v_i conj(w_c) + w_i conj(v_c)
            tri[e] = cmsubc(cmsubc(tri[e], w[c], v[i]), v[c], w[i]);
        }
        __syncthreads();
    }
    if (tid == 0) dd[n - 1] = (double)L[hs_at(n, n - 1, n - 1)].x;
}

// Back-transform Z = P_0 P_1 ... P_{n-2} Y of the same systems (S5): a CTA takes HS_BT_NC columns of
// Z in shared memory and applies the reflectors one by one, last first, each column's rows dealt over
// HS_BT_RG threads.  Bound by the FP64 units (8 n^3 / 2 real flops a system; 93 % of their rate with 200
// systems), with two barriers a reflector, where the blocked form's T factors and 64-row tiles cost more
// than they save at these sizes: n = 82 in FP64, one system 0.2 ms (k_larft and k_backtransform 1.27), 200
// systems 1.2 ms (4.65).
#define HS_BT_NC 16
#define HS_BT_THREADS 128
#define HS_BT_RG (HS_BT_THREADS / HS_BT_NC)

template <class R>
__global__ void __launch_bounds__(HS_BT_THREADS)
k_bt_small(const MmfDesc* __restrict__ descs, const int* __restrict__ idx, const typename Cx<R>::T* __restrict__ H,
           const typename Cx<R>::T* __restrict__ taupool, const double* __restrict__ Yg,
           typename Cx<R>::T* __restrict__ Zout) {
    typedef typename Cx<R>::T C;
    extern __shared__ __align__(16) unsigned char hs_smem[];
    __shared__ C vs[2][HS_ROWS], red[HS_BT_THREADS / 32][HS_BT_NC];
    C(*z)[HS_BT_NC] = reinterpret_cast<C(*)[HS_BT_NC]>(hs_smem);  // n x HS_BT_NC
    const MmfDesc d = descs[idx[blockIdx.y]];
    const int n = d.n, ld = d.ld;
    const int c0 = blockIdx.x * HS_BT_NC;
    if (c0 >= n) return;
    const C* A = H + d.mat_off;
    const C* tau = taupool + d.vec_off;
    const double* Y = Yg + d.sq_off;
    C* Z = Zout + d.mat_off;
    const int tx = threadIdx.x, cl = tx % HS_BT_NC, g = tx / HS_BT_NC, warp = tx >> 5;
    for (int r = g; r < n; r += HS_BT_RG)
        z[r][cl] = mk(c0 + cl < n ? (R)Y[(int64_t)r * n + c0 + cl] : R(0), R(0));
    // v of reflector k on rows k + 1 .. n - 1: 1, then A(k + 2 .., k)
    if (tx == 0) vs[0][0] = mk(R(1), R(0));
    C t = tau[n - 2];
    __syncthreads();
    int buf = 0;
    for (int k = n - 2; k >= 0; --k) {
        const int m = n - k - 1;
        C v0 = czero<C>(), v1 = v0, tn = v0;  // the next reflector, loading meanwhile
        if (k > 0) {
            const C* a = A + (k + 1) + (int64_t)(k - 1) * ld;  // entry e of v, e >= 1, at a[e - 1]
            if (tx < m) v0 = a[tx];
            if (tx + HS_BT_THREADS < m) v1 = a[tx + HS_BT_THREADS];
            tn = tau[k - 1];
        }
        const C* v = vs[buf];
        C w = czero<C>(), w1 = w;
        int i = g;
        for (; i + HS_BT_RG < m; i += 2 * HS_BT_RG) {
            w = cmacc(w, v[i], z[k + 1 + i][cl]);
            w1 = cmacc(w1, v[i + HS_BT_RG], z[k + 1 + i + HS_BT_RG][cl]);
        }
        if (i < m) w = cmacc(w, v[i], z[k + 1 + i][cl]);
        w = w + w1;
#pragma unroll
        for (int o = HS_BT_NC; o < 32; o <<= 1) {
            w.x += __shfl_xor_sync(0xffffffffu, w.x, o);
            w.y += __shfl_xor_sync(0xffffffffu, w.y, o);
        }
        if ((tx & 31) < HS_BT_NC) red[warp][cl] = w;
        __syncthreads();
        w = red[0][cl];
#pragma unroll
        for (int q = 1; q < HS_BT_THREADS / 32; ++q) w = w + red[q][cl];
        const C tw = t * w;
        for (int q = g; q < m; q += HS_BT_RG) z[k + 1 + q][cl] = cmsub(z[k + 1 + q][cl], tw, v[q]);
        if (k > 0) {
            C* vn = vs[buf ^ 1];
            if (tx == 0) vn[0] = mk(R(1), R(0));
            if (tx < m) vn[tx + 1] = v0;
            if (tx + HS_BT_THREADS < m) vn[tx + HS_BT_THREADS + 1] = v1;
            t = tn;
        }
        __syncthreads();
        buf ^= 1;
    }
    const int nc = min(HS_BT_NC, n - c0);
    for (int e = tx; e < nc * n; e += HS_BT_THREADS) {
        const int c = e / n, r = e - c * n;
        Z[r + (int64_t)(c0 + c) * ld] = z[r][c];
    }
}

template <class R>
static cudaError_t launch_bt_small(const MmfLaunch& L, const void* H, const void* tau, const double* Y, void* Z) {
    typedef typename Cx<R>::T C;
    const size_t sm = sizeof(C) * HS_BT_NC * (size_t)L.nmax;
    cudaError_t e = cudaFuncSetAttribute(k_bt_small<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    k_bt_small<R><<<dim3((L.nmax + HS_BT_NC - 1) / HS_BT_NC, L.count), HS_BT_THREADS, sm, L.stream>>>(
        L.desc, L.idx, (const C*)H, (const C*)tau, Y, (C*)Z);
    return cudaGetLastError();
}

template <class R>
static cudaError_t launch_small(const MmfLaunch& L, void* H, double* dvec, double* evec, void* tau) {
    typedef typename Cx<R>::T C;
    const size_t sm = hs_bytes<R>(L.nmax);
    cudaError_t e = cudaFuncSetAttribute(k_hetrd_small<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    k_hetrd_small<R><<<L.count, HS_THREADS, sm, L.stream>>>(L.desc, L.idx, (C*)H, dvec, evec, (C*)tau);
    return cudaGetLastError();
}

// Largest n of the one-CTA reduction: the triangle has to leave room for a second CTA on the SM
// (113 KB each) up to n = 103 in FP64 and n = 152 in FP32.  Above that one SM's FP64 lanes are the
// limit (n^3), and k_hetrd's cluster takes over.
int mmf_hetrd_small_n(int fp32) { return fp32 ? 152 : 103; }

cudaError_t mmf_launch_hetrd_small(const MmfLaunch& L, void* H, double* dvec, double* evec, void* tau, int fp32) {
    if (L.count <= 0) return cudaSuccess;
    if (L.nmax > mmf_hetrd_small_n(fp32)) return cudaErrorInvalidValue;
    return fp32 ? launch_small<float>(L, H, dvec, evec, tau) : launch_small<double>(L, H, dvec, evec, tau);
}

cudaError_t mmf_launch_bt_small(const MmfLaunch& L, const void* H, const void* tau, const double* Y, void* Z, int fp32) {
    if (L.count <= 0) return cudaSuccess;
    if (L.nmax > mmf_hetrd_small_n(fp32)) return cudaErrorInvalidValue;
    return fp32 ? launch_bt_small<float>(L, H, tau, Y, Z) : launch_bt_small<double>(L, H, tau, Y, Z);
}
