// ibf_viscous.cu -- sm_103a kernels of the factored implicit viscous solve
// (Section "Fluid Mechanics", Eq. nstime_discr with the viscous terms advanced by
// Crank-Nicolson; Section "Fluid domain", provisional-step paragraph: the implicit
// operator split into one tridiagonal solve per direction, Thomas' algorithm, with a
// Sherman-Morrison perturbation on the periodic lines):
//
//   out = (I - beta Lz)^-1 (I - beta Ly)^-1 (I - beta Lx)^-1 rhs,  beta = alpha dt / (2 Re)
//
// for each velocity component.  On the periodic, uniform x and y lines (I - beta L)
// is circulant: its inverse -- the result the cyclic Thomas solve with the
// Sherman-Morrison correction returns -- divides Fourier coefficient m by
// 1 + beta (4/h^2) sin^2(pi m / n).  The x and y factors are therefore applied in
// the spectrum the projection's transforms already produce, and only z keeps a
// tridiagonal solve.  One component is four launches:
//   k_xfwd<XM_COPY>  x-FFT of the field (ibf_kernels.cu), spectrum in column blocks
//   k_yhelm          y-FFT, division by both factors, inverse y-FFT, in place (ibf_planes.cu)
//   k_xinv STORE     inverse x-FFT into the plan's per-cell workspace (ibf_kernels.cu)
//   k_zhelm_tile     Thomas along z for every (i, j) column, held in shared memory, fp64
//                    output (k_zhelm, which streams, for tall columns).
// The z operator is the second difference of the component's own grid: cell centres
// with no-slip walls (mirror ghosts) for u and v, interior faces for w (its wall faces
// stay zero).
#include "ibf_common.cuh"
#include "ibf_viscous.h"

namespace ibf {

// Per grid (one block each): thread 0 builds the Thomas pivots of (I - beta Lz) for the
// cell-centre operator (u, v), thread 1 those of the interior-face operator (w), the
// other threads the x and y factors of k_yhelm.  Per grid and operator, at
// tab + 6 z_off + 3 op (nz+1): the sub-diagonal a_r, the pivot inverse inv_r and the
// normalised super-diagonal cp_r (nz+1 entries each), so that the forward sweep is
// y_r = (f_r - a_r y_{r-1}) inv_r and the back substitution x_r = y_r - cp_r x_{r+1}.
// fp64, with fp32 copies at the same offsets in tabf (and fxyf).
__global__ void k_helm_table(Work w, double beta, double *tab, float *tabf, const long long *fxy_off, double *fxy,
                             float *fxyf) {
    const int g = blockIdx.x, op = threadIdx.x;
    const GridDev &G = w.grids[g];
    if (op >= 2) {
        // the x and y factors 1 / (1 + beta (4/h^2) sin^2(pi m / n)) of the x-modes m < nxh
        // and the y-modes n < ny, at fxy + fxy_off[g] (nxh + ny entries)
        double *f = fxy + fxy_off[g];
        float *ff = fxyf + fxy_off[g];
        for (int t = op - 2; t < G.nxh + G.ny; t += blockDim.x - 2) {
            const bool isx = t < G.nxh;
            const int m = isx ? t : t - G.nxh;
            const double s = sinpi((double)m / (double)(isx ? G.nx : G.ny));
            const double r = isx ? G.rdx : G.rdy;
            const double v = 1.0 / (1.0 + beta * 4.0 * r * r * s * s);
            f[t] = v;
            ff[t] = (float)v;
        }
        return;
    }
    const int nz = G.nz, zo = G.z_off;
    const double *rhz = w.z.rhz + zo, *rgzf = w.z.rgzf + zo;  // 1/hz_k; 1/(zc_k - zc_{k-1}) on interior faces
    const size_t base = 6 * (size_t)zo + 3 * (size_t)op * (size_t)(nz + 1), len = (size_t)(nz + 1);
    double *a = tab + base, *inv = a + len, *cp = inv + len;
    float *af = tabf + base, *invf = af + len, *cpf = invf + len;
    const int n = op == 0 ? nz : nz - 1;
    double cprev = 0.0;
    for (int r = 0; r < n; ++r) {
        double lo, up, extra = 0.0;
        if (op == 0) {
            // centre r: neighbours across faces r and r+1; at a wall the mirror ghost
            // (minus the value) sits hz away, adding its coupling to the diagonal
            lo = r > 0 ? rhz[r] * rgzf[r] : rhz[0] * rhz[0];
            up = r < nz - 1 ? rhz[r] * rgzf[r + 1] : rhz[nz - 1] * rhz[nz - 1];
            if (r == 0) extra += lo;
            if (r == nz - 1) extra += up;
        } else {
            // interior face k = r + 1, between the centres k-1 and k
            const int k = r + 1;
            lo = rhz[k - 1] * rgzf[k];
            up = rhz[k] * rgzf[k];
        }
        const double sub = r > 0 ? -beta * lo : 0.0;
        const double sup = r < n - 1 ? -beta * up : 0.0;
        const double diag = 1.0 + beta * (lo + up + extra);
        const double iv = 1.0 / (diag - sub * cprev);
        cprev = sup * iv;
        a[r] = sub;
        inv[r] = iv;
        cp[r] = cprev;
        af[r] = (float)sub;
        invf[r] = (float)iv;
        cpf[r] = (float)cprev;
    }
}

// Thomas along z of every (i, j) column of grid g.  Input: the x/y-solved field in the
// plan's per-cell workspace (fp32 phi_hi on the mixed path, fp64 phi_ws on the fp64
// path), planes r < n; the forward sweep overwrites it with y_r, the back substitution
// writes out (fp64).  zshift = 1: w, whose n = nz - 1 unknowns are the interior faces
// (out planes 1..nz-1; the wall faces 0 and nz are set to zero); zshift = 0: u or v.
template <typename T> struct HelmTab;
template <> struct HelmTab<float> {
    __device__ __forceinline__ static const float *get(const double *, const float *f) { return f; }
    __device__ __forceinline__ static float *ws(const Work &w) { return w.phi_hi; }
};
template <> struct HelmTab<double> {
    __device__ __forceinline__ static const double *get(const double *d, const float *) { return d; }
    __device__ __forceinline__ static double *ws(const Work &w) { return w.phi_ws; }
};

template <typename T>
__global__ void __launch_bounds__(kZHelmThreads) k_zhelm(Work w, int g, int zshift, const double *tab,
                                                         const float *tabf, double *out) {
    const GridDev &G = w.grids[g];
    const long long plane = (long long)G.nx * G.ny;
    const long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= plane) return;
    const int nz = G.nz, n = nz - zshift;
    const size_t base = 6 * (size_t)G.z_off + 3 * (size_t)zshift * (size_t)(nz + 1), len = (size_t)(nz + 1);
    const T *a = HelmTab<T>::get(tab, tabf) + base, *inv = a + len, *cp = inv + len;
    T *f = HelmTab<T>::ws(w) + G.cell_off + c;
    T y = (T)0;
#pragma unroll 4
    for (int r = 0; r < n; ++r) {
        y = (f[r * plane] - a[r] * y) * inv[r];
        f[r * plane] = y;
    }
    T x = (T)0;
#pragma unroll 4
    for (int r = n - 1; r >= 0; --r) {
        x = f[r * plane] - cp[r] * x;
        out[(r + zshift) * plane + c] = (double)x;
    }
    if (zshift) {
        out[c] = 0.0;
        out[nz * plane + c] = 0.0;
    }
}

// (double)x by integer operations for normal numbers (a conversion runs at the fp64 pipe's
// rate: one a cell takes as long as k_zhelm_tile's memory traffic)
__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ double widen(float x) {
    const unsigned b = __float_as_uint(x), e = b & 0x7F800000u;
    if (e == 0u || e == 0x7F800000u) return (double)x;  // zero, subnormal, inf, nan
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + 0x38000000u)), (int)(b << 29));
}

// The same solve with kZHelmCols columns held in shared memory between the two sweeps, one
// warp a CTA: the workspace is read once and never written (12 B a cell in fp32 instead of
// 20, three trips to L2 or HBM down to two).  All of a tile's copies are issued at once
// (cp.async, in four groups of levels), and eight levels' values are in registers before the
// chain that uses them.  384x384x192 mixed 213 -> 94 us (12 B a cell at HBM rate: 50),
// 192x144x101 fp64 48 -> 27 us.
// Shared memory: values [np][32], then a, inv and cp [np] each, np the levels in whole batches of 8.
template <typename T>
__global__ void __launch_bounds__(kZHelmCols) k_zhelm_tile(Work w, int g, int zshift, const double *tab,
                                                           const float *tabf, double *out) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int C = kZHelmCols, NG = 4, B = 8;
    const GridDev &G = w.grids[g];
    const long long plane = (long long)G.nx * G.ny, c0 = (long long)blockIdx.x * C;
    const int nz = G.nz, n = nz - zshift, lane = threadIdx.x, nc = (int)min((long long)C, plane - c0);
    const size_t base = 6 * (size_t)G.z_off + 3 * (size_t)zshift * (size_t)(nz + 1), len = (size_t)(nz + 1);
    const T *a = HelmTab<T>::get(tab, tabf) + base, *inv = a + len, *cp = inv + len;
    const T *f = HelmTab<T>::ws(w) + G.cell_off + c0;
    const int np = (n + B - 1) & ~(B - 1);  // whole batches: the pad is read, never used
    T *xs = reinterpret_cast<T *>(smem_raw), *sa = xs + (size_t)np * C, *si = sa + np, *sc = si + np;
    const int per = ((n + NG - 1) / NG + B - 1) & ~(B - 1);
    constexpr int V = 16 / (int)sizeof(T), LV = C / V, ST = 32 / LV;  // values a copy, lanes and levels a turn
    const bool vec = (plane & (V - 1)) == 0 && (G.cell_off & (V - 1)) == 0;
    const T *gx = f + (long long)(lane / LV) * plane + (lane % LV) * V;
    T *dx = xs + (lane / LV) * C + (lane % LV) * V;
    const bool in = (lane % LV) * V < nc;
#pragma unroll
    for (int q = 0; q < NG; ++q) {
        const int k0 = q * per, k1 = min(n, k0 + per);
        if (vec) {
#pragma unroll 4
            for (int k = k0 + lane / LV; k < k1; k += ST) {
                if (in) cp_async<16>(dx, gx);
                gx += ST * plane;
                dx += ST * C;
            }
        } else {
            for (int k = k0; k < k1; ++k)
                if (lane < nc) cp_async<sizeof(T)>(xs + k * C + lane, f + (long long)k * plane + lane);
        }
        cp_async_commit();
    }
    for (int k = lane; k < n; k += 32) {
        sa[k] = a[k];
        si[k] = inv[k];
        sc[k] = cp[k];
    }
    // one batch of levels: values and a sweep's coefficients (16-byte broadcast reads)
    struct Batch {
        T r[B], e[B], v[B];
    };
    auto coef = [](const T *c, T (&d)[B]) {
        constexpr int Q = 16 / (int)sizeof(T);
        struct alignas(16) Vec {
            T x[Q];
        };
#pragma unroll
        for (int q = 0; q < B / Q; ++q) {
            const Vec t = *reinterpret_cast<const Vec *>(c + q * Q);
#pragma unroll
            for (int u = 0; u < Q; ++u) d[q * Q + u] = t.x[u];
        }
    };
    auto fetch_up = [&](int kb, Batch &t) {
#pragma unroll
        for (int u = 0; u < B; ++u) t.r[u] = xs[(kb + u) * C + lane];
        coef(sa + kb, t.e);
        coef(si + kb, t.v);
    };
    auto fetch_down = [&](int kb, Batch &t) {
#pragma unroll
        for (int u = 0; u < B; ++u) t.r[u] = xs[(kb + u) * C + lane];
        coef(sc + kb, t.e);
    };
    Batch t0, t1;
    T y = (T)0;
    auto up = [&](int kb, const Batch &t) {
#pragma unroll
        for (int u = 0; u < B; ++u) {
            y = (t.r[u] - t.e[u] * y) * t.v[u];  // levels past n - 1 write the pad
            xs[(kb + u) * C + lane] = y;
        }
    };
    auto sweep_up = [&](int k0, int k1) {  // two batches a turn, the next one's loads before the stores
        if (k0 >= k1) return;
        fetch_up(k0, t0);
        for (int kb = k0; kb < k1; kb += 2 * B) {
            if (kb + B < k1) fetch_up(kb + B, t1);
            up(kb, t0);
            if (kb + B >= k1) break;
            if (kb + 2 * B < k1) fetch_up(kb + 2 * B, t0);
            up(kb + B, t1);
        }
    };
    cp_async_wait<3>();
    __syncwarp();
    sweep_up(0, min(n, per));
    cp_async_wait<2>();
    __syncwarp();
    sweep_up(per, min(n, 2 * per));
    cp_async_wait<1>();
    __syncwarp();
    sweep_up(2 * per, min(n, 3 * per));
    cp_async_wait<0>();
    __syncwarp();
    sweep_up(3 * per, n);
    const bool live = lane < nc;
    double *o = out + c0 + (long long)(n - 1 + zshift) * plane;  // (warp-uniform)
    T x = (T)0;
    auto down = [&](int cnt, const Batch &t) {
#pragma unroll
        for (int u = B - 1; u >= 0; --u) {
            if (u < cnt) {
                x = t.r[u] - t.e[u] * x;
                if (live) o[lane] = widen(x);
                o -= plane;
            }
        }
    };
    const int kl = np - B;  // the last batch, n - kl levels
    if (n > 0) {
        fetch_down(kl, t0);
        if (kl > 0) fetch_down(kl - B, t1);
        down(n - kl, t0);
        for (int kb = kl - B; kb >= 0; kb -= 2 * B) {
            if (kb >= B) fetch_down(kb - B, t0);
            down(B, t1);
            if (kb < B) break;
            if (kb >= 2 * B) fetch_down(kb - 2 * B, t1);
            down(B, t0);
        }
    }
    if (zshift && live) {
        out[c0 + lane] = 0.0;
        out[nz * plane + c0 + lane] = 0.0;
    }
}

cudaError_t launch_helm_table(const Work &w, int ngrids, double beta, double *tab, float *tabf,
                              const long long *fxy_off, double *fxy, float *fxyf, cudaStream_t st) {
    if (ngrids <= 0) return cudaSuccess;
    k_helm_table<<<ngrids, 128, 0, st>>>(w, beta, tab, tabf, fxy_off, fxy, fxyf);
    return cudaGetLastError();
}

cudaError_t launch_zhelm(int mixed, const Work &w, int g, long long ncol, int nz, int zshift, const double *tab,
                         const float *tabf, double *out, cudaStream_t st) {
    if (ncol <= 0) return cudaSuccess;
    const size_t tile = zhelm_tile_smem(mixed, nz);
    // beyond four CTAs an SM only where the plane is small: on wide grids k_zhelm streams at the HBM
    // rate (1024x1024x512 mixed: tile 2.69 ms, k_zhelm 2.57; 256x256x512: 189 us against 285)
    if (2 * tile <= kZHelmTileMost || (tile <= kZHelmTileMost && ncol < (1ll << 18))) {
        const unsigned nt = (unsigned)((ncol + kZHelmCols - 1) / kZHelmCols);
        if (mixed) k_zhelm_tile<float><<<nt, kZHelmCols, tile, st>>>(w, g, zshift, tab, tabf, out);
        else k_zhelm_tile<double><<<nt, kZHelmCols, tile, st>>>(w, g, zshift, tab, tabf, out);
        return cudaGetLastError();
    }
    const unsigned nb = (unsigned)((ncol + kZHelmThreads - 1) / kZHelmThreads);
    if (mixed) k_zhelm<float><<<nb, kZHelmThreads, 0, st>>>(w, g, zshift, tab, tabf, out);
    else k_zhelm<double><<<nb, kZHelmThreads, 0, st>>>(w, g, zshift, tab, tabf, out);
    return cudaGetLastError();
}

cudaError_t set_smem_limits_visc(int mixed) {
    return set_smem_cap(mixed ? (const void *)k_zhelm_tile<float> : (const void *)k_zhelm_tile<double>);
}

}  // namespace ibf
