// ibf_yz.cuh -- device code shared by the streaming / slab y/z kernels (ibf_yz.cu) and the
// plane-parallel ones (ibf_planes.cu): DCT passes around an FFT, block-wide scans, the
// (0,0) mode.
#pragma once
#include "ibf_common.cuh"

namespace ibf {

template <typename T> __device__ __forceinline__ const T *zarr(const double *d, const float *f);
template <> __device__ __forceinline__ const double *zarr<double>(const double *d, const float *) { return d; }
template <> __device__ __forceinline__ const float *zarr<float>(const double *, const float *f) { return f; }

// Rotations of the DCT twiddles, w a and conj(w) a with w = exp(-i pi n/(2N)), n <= N/2, whose
// cosine is the larger part: only the product with the sine is rounded by itself.  Written out
// because the compiler is free to round either one: the plane-parallel kernels' form of
// these lines came out with the larger product rounded, half a unit in the last place of the
// mode itself (phi after one sweep, walls in y, median error over 24 fields: 3x512x5 3.7e-9
// against 2.9e-9, 4x1024x5 3.8e-8 against 2.3e-8, 96x288x40 9.4e-11 against 7.2e-11).
template <typename T> __device__ __forceinline__ cx<T> dct_rot(const cx<T> &w, const cx<T> &a) {
    return {fma(w.x, a.x, -(w.y * a.y)), fma(w.x, a.y, w.y * a.x)};
}
template <typename T> __device__ __forceinline__ cx<T> dct_rotc(const cx<T> &w, const cx<T> &a) {
    return {fma(w.x, a.x, w.y * a.y), fma(w.x, a.y, -(w.y * a.x))};
}

// DCT-II post-twiddle of the FFT V (in place, FFT output order) of every Makhoul-
// reordered sequence of a column block: with P = W^n V_n, Q = conj(W^n) V_{N-n},
// W = exp(-i pi/(2N)), the coefficients are X_n = (P + Q)/2 and X_{N-n} = i (P - Q)/2
// (complex-linear, so it holds for complex columns); X_0 = V_0.  Ends synchronised.
template <typename T>
__device__ __forceinline__ void dct_post(cx<T> *buf, int nseq, int sstride, int N, int N1, int N2,
                                         const FDiv &fN1, const cx<T> *W) {
    const int half = N >> 1;
    for (int t = threadIdx.x; t < nseq * half; t += blockDim.x) {
        const int sq = t / half, n = t - sq * half + 1;
        cx<T> *seq = buf + sq * sstride;
        const int pa = pos_tr(n, N1, N2, fN1), pb = pos_tr(N - n, N1, N2, fN1);
        const cx<T> a = seq[pa], b = seq[pb], w = W[n];
        const cx<T> P = dct_rot(w, a), Q = dct_rotc(w, b);
        if (pa == pb) {  // n = N/2
            seq[pa] = {(P.x + Q.x) * (T)0.5, (P.y + Q.y) * (T)0.5};
        } else {
            seq[pa] = {(P.x + Q.x) * (T)0.5, (P.y + Q.y) * (T)0.5};
            seq[pb] = {(Q.y - P.y) * (T)0.5, (P.x - Q.x) * (T)0.5};
        }
    }
    __syncthreads();
}

// Inverse of dct_post (DCT-III input stage, in place): V_n = conj(W^n)(X_n - i X_{N-n}),
// V_{N-n} = W^n (X_n + i X_{N-n}); V_0 = X_0.  An unscaled inverse FFT of V followed by
// the un-reordering returns the sequence whose DCT-II divided by N was X.  Ends synchronised.
template <typename T>
__device__ __forceinline__ void dct_pre(cx<T> *buf, int nseq, int sstride, int N, int N1, int N2,
                                        const FDiv &fN1, const cx<T> *W) {
    const int half = N >> 1;
    for (int t = threadIdx.x; t < nseq * half; t += blockDim.x) {
        const int sq = t / half, n = t - sq * half + 1;
        cx<T> *seq = buf + sq * sstride;
        const int pa = pos_tr(n, N1, N2, fN1), pb = pos_tr(N - n, N1, N2, fN1);
        const cx<T> a = seq[pa], b = seq[pb], w = W[n];
        const cx<T> d = {a.x + b.y, a.y - b.x};  // X_n - i X_{N-n}
        const cx<T> e = {a.x - b.y, a.y + b.x};  // X_n + i X_{N-n}
        seq[pa] = dct_rotc(w, d);
        if (pa != pb) seq[pb] = dct_rot(w, e);
    }
    __syncthreads();
}

// In-place inclusive prefix sums of a[0..n) in fp64 (rev: suffix sums, a[i] = sum over
// j >= i), all threads of the block: each thread scans a contiguous chunk, the chunk totals
// are scanned by warp shuffles and across warps through wsum[blockDim / 32]; a fixed order.
static __device__ void block_scan_fp64(double *a, int n, bool rev, double *wsum) {
    const int T = blockDim.x, t = threadIdx.x, lane = t & 31, wid = t >> 5, nw = T >> 5;
    const int per = (n + T - 1) / T, b0 = min(n, t * per), b1 = min(n, b0 + per);
    auto at = [&](int i) -> double & { return a[rev ? n - 1 - i : i]; };
    double loc = 0.0;
    for (int i = b0; i < b1; ++i) {
        loc += at(i);
        at(i) = loc;
    }
    double x = loc;  // inclusive scan of the chunk totals within the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    double ex = __shfl_up_sync(0xffffffffu, x, 1);  // exclusive: the chunks before this one
    if (lane == 0) ex = 0.0;
    if (lane == 31) wsum[wid] = x;
    __syncthreads();
    if (wid == 0) {
        double v = lane < nw ? wsum[lane] : 0.0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double y = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v += y;
        }
        if (lane < nw) wsum[lane] = v;
    }
    __syncthreads();
    const double off = wid > 0 ? ex + wsum[wid - 1] : ex;
    for (int i = b0; i < b1; ++i) at(i) += off;
    __syncthreads();
}

// The sums of one plane of the right-hand side (and, in a refinement pass, of phi) by one
// warp: the forward x kernels leave one slot per row block (two with the half-block CTAs),
// added lane-strided then by a butterfly of shuffles (a fixed order) into the plane's first
// slot, the only one that the (0,0) solve reads.
__device__ __forceinline__ void plane_sums(const Work &w, const GridDev &G, int k, int first_solve) {
    const int lane = threadIdx.x & 31, np = G.nrb * (w.xfwd_split ? 2 : 1);
    double *pk = w.partial + G.part_off + (size_t)k * np, *qk = w.partial_phi + G.part_off + (size_t)k * np;
    double S = 0.0, P = 0.0;
    for (int r = lane; r < np; r += 32) {
        S += pk[r];
        if (!first_solve) P += qk[r];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        S += __shfl_xor_sync(0xffffffffu, S, o);
        if (!first_solve) P += __shfl_xor_sync(0xffffffffu, P, o);
    }
    // every lane's loads are done (the shuffles consumed them) and only lane 0 read slot 0
    if (lane == 0) {
        pk[0] = S;
        if (!first_solve) qk[0] = P;
    }
}

// ================================================================ the (0,0) mode (fp64, one CTA of k_00 per grid)
// Shared memory (sh00_bytes): right-hand side, hz, the flux terms / running sums, the
// increments of phi, the centre distances gz (their divisions overlap the first loads).
// Every plane's sums lie in the plane's first slot (plane_sums).  to_spec: the solution also
// goes to the (0,0) slot of the spectrum's planes (spectral z).
template <typename T>
__device__ __forceinline__ void mode00_solve(const Work &w, int g, int first_solve, bool to_spec, double *sh00) {
    __shared__ double red[8];
    const GridDev &G = w.grids[g];
    const int nz = G.nz, nrb = G.nrb, zo = G.z_off;
    const int L = nz + 1;
    double *rhs = sh00, *hz = rhs + L, *S = hz + L, *inc = S + L, *gz = inc + L;
    const double *part = w.partial + G.part_off, *partp = w.partial_phi + G.part_off;
    double loc = 0.0, locp = 0.0;
    bool bad = false;
    const int np = nrb * (w.xfwd_split ? 2 : 1);
    double lmax = 0.0;
    // kLv levels of a thread at a time, every load before the first use: with more levels than
    // threads the loads' latency is what this solve waits for
    constexpr int kLv = 8;
    for (int k0 = threadIdx.x; k0 < nz; k0 += kLv * blockDim.x) {
        double sb[kLv], sp[kLv], h[kLv], rg[kLv];
#pragma unroll
        for (int u = 0; u < kLv; ++u) {
            const int k = k0 + u * blockDim.x;
            const bool in = k < nz;
            sb[u] = in ? __ldcg(part + (size_t)k * np) : 0.0;
            sp[u] = in && !first_solve ? __ldcg(partp + (size_t)k * np) : 0.0;
            h[u] = in ? __ldg(w.z.hz + zo + k) : 0.0;
            rg[u] = k + 1 < nz ? __ldg(w.z.rgzf + zo + k + 1) : 1.0;
        }
#pragma unroll
        for (int u = 0; u < kLv; ++u) {
            const int k = k0 + u * blockDim.x;
            if (k >= nz) break;
            const double m = sb[u] * G.inv_nxy;  // plane mean of b (first solve) or of the residual
            if (!isfinite(m)) bad = true;
            rhs[k] = m;
            hz[k] = h[u];
            gz[k] = 1.0 / rg[u];  // gz_{k+1}
            lmax = fmax(lmax, fabs(m));
            loc += h[u] * m;
            if (!first_solve) locp += h[u] * (sp[u] * G.inv_nxy);
        }
    }
    if (bad) atomicOr(w.err, 1u << 6);  // IBF_ERR_NONFINITE
    // In a refinement pass rhs[k] is already the plane mean of the residual
    // b - <b> - L phi (summed from its per-cell values, which are small once phi is
    // close): forming it instead from the plane means of b and of phi would carry the
    // rounding of phi's plane means, amplified by the z part of L (up to 1/(hz gz) next
    // to a stretched wall), into the correction.
    const double tot = Red<F64Arith>::sum(loc, red);
    // weighted mean of the phi being refined: the correction also removes it, so that
    // phi + delta keeps a zero weighted mean (L cannot see a constant)
    const double totp = first_solve ? 0.0 : Red<F64Arith>::sum(locp, red);
    // a Dirichlet outlet makes the (0,0) system regular: nothing to remove
    if (threadIdx.x == 0) red[0] = G.dir_top ? 0.0 : tot / G.sum_hz;
    __syncthreads();
    const double mean = red[0];
    if (first_solve) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) lmax = fmax(lmax, __shfl_xor_sync(0xffffffffu, lmax, o));
        __syncthreads();  // red[0] (the mean) has been read by every thread
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = lmax;
        __syncthreads();
        if (threadIdx.x == 0) {
            w.mean_b[g] = mean;
            double scale = 0.0;
            for (int i = 0; i < (int)(blockDim.x >> 5); ++i) scale = fmax(scale, red[i]);
            // compatibility defect large compared with the plane means -> warning
            if (fabs(mean) > 1e-8 * scale && fabs(mean) > 0.0) atomicOr(w.err, 1u << 7);
        }
        __syncthreads();
    }
    // The (0,0) system in flux form.  Row k of L along z, times hz_k, is a difference of
    // face fluxes, hz_k (L phi)_k = F_{k+1/2} - F_{k-1/2} with F_{k+1/2} =
    // (phi_{k+1} - phi_k) / gz_{k+1} and F_{-1/2} = 0 at the bottom wall, so
    //   F_{k+1/2} = S_k = sum_{j <= k} hz_j d_j,      d = right-hand side less its mean,
    //   phi_k     = phi_{k+1} - gz_{k+1} S_k          (integrated down from level nz-1).
    // Neumann top: the top flux is zero (S_{nz-1} = 0 up to rounding, since d has zero
    // weighted mean), phi_{nz-1} is pinned to 0 and the weighted mean removed below.
    // Dirichlet outlet: the top flux is -hz_{nz-1} ez_top phi_{nz-1} = S_{nz-1}, which
    // fixes phi_{nz-1}.  The two running sums are the exact solve of the system; unlike
    // an elimination on the rows a_k, -(a_k + c_k), c_k (whose reduced diagonals cancel
    // by orders of magnitude on a stretched grid) they leave a residual at the rounding
    // of the fluxes.  The running sums are block-wide scans (a fixed order).
    for (int k = threadIdx.x; k < nz; k += blockDim.x) S[k] = hz[k] * (rhs[k] - mean);
    __syncthreads();
    block_scan_fp64(S, nz, false, red);  // S_k, in place
    for (int k = threadIdx.x; k + 1 < nz; k += blockDim.x) inc[k] = S[k] * gz[k];
    __syncthreads();
    block_scan_fp64(inc, nz - 1, true, red);  // inc[k] = sum_{j = k}^{nz-2} gz_{j+1} S_j
    const double ph_top = G.dir_top ? -S[nz - 1] / (hz[nz - 1] * G.ez_top) : 0.0;
    double lsv = 0.0;
    for (int k = threadIdx.x; k < nz; k += blockDim.x) {
        const double ph = k + 1 < nz ? ph_top - inc[k] : ph_top;
        rhs[k] = ph;
        lsv += hz[k] * ph;
    }
    __syncthreads();
    const double sv = Red<F64Arith>::sum(lsv, red);
    if (threadIdx.x == 0) rhs[nz] = G.dir_top ? 0.0 : (sv + totp) / G.sum_hz;  // weighted mean to remove
    __syncthreads();
    const double mphi = rhs[nz];
    cx<T> *spec = reinterpret_cast<cx<T> *>(w.spec) + G.spec_off;
    const size_t stride = (size_t)G.ncb * G.ny * G.mb;
    for (int k = threadIdx.x; k < nz; k += blockDim.x) {
        const double v = rhs[k] - mphi;
        if (to_spec) spec[(size_t)k * stride] = {(T)v, (T)0};
        w.sol00[zo + k] = v;
    }
}

// The same solve by one warp without a block barrier, for the z-solve launch's extra CTAs,
// where small grids wait for it: every lane takes a contiguous run of levels, the running sums
// are lane sums and one shuffle scan, sums that are needed together reduce together.  96x72x45
// mixed: the z-solve launch 12.8 -> 12.3 us; 64x64x512 34.9 -> 29.9.  Of mode00_solve's five
// arrays in shared memory it uses three: the right-hand side (then phi), hz and gz.
template <typename T>
__device__ __forceinline__ void mode00_warp(const Work &w, int g, int first_solve, double *sh00) {
    const GridDev &G = w.grids[g];
    const int nz = G.nz, zo = G.z_off, lane = threadIdx.x & 31, L = nz + 1;
    double *rhs = sh00, *hz = rhs + L, *gz = hz + L;
    const int np = G.nrb * (w.xfwd_split ? 2 : 1);
    const double *part = w.partial + G.part_off, *partp = w.partial_phi + G.part_off;
    const int per = (nz + 31) / 32, k0 = min(nz, lane * per), k1 = min(nz, k0 + per);
    double loc = 0.0, locp = 0.0, lmax = 0.0;
    bool bad = false;
    constexpr int kLv = 4;  // levels whose loads go together
    for (int kb = k0; kb < k1; kb += kLv) {
        double sb[kLv], sp[kLv], h[kLv], rg[kLv];
#pragma unroll
        for (int u = 0; u < kLv; ++u) {
            const int k = kb + u;
            const bool in = k < k1;
            sb[u] = in ? __ldcg(part + (size_t)k * np) : 0.0;
            sp[u] = in && !first_solve ? __ldcg(partp + (size_t)k * np) : 0.0;
            h[u] = in ? __ldg(w.z.hz + zo + k) : 0.0;
            rg[u] = in && k + 1 < nz ? __ldg(w.z.rgzf + zo + k + 1) : 1.0;
        }
#pragma unroll
        for (int u = 0; u < kLv; ++u) {
            if (kb + u >= k1) break;
            const double m = sb[u] * G.inv_nxy;  // plane mean of b (first solve) or of the residual
            bad |= !isfinite(m);
            rhs[kb + u] = m;
            hz[kb + u] = h[u];
            gz[kb + u] = 1.0 / rg[u];  // gz_{k+1}
            lmax = fmax(lmax, fabs(m));
            loc += h[u] * m;
            locp += h[u] * (sp[u] * G.inv_nxy);
        }
    }
    if (bad) atomicOr(w.err, 1u << 6);  // IBF_ERR_NONFINITE
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        loc += __shfl_xor_sync(0xffffffffu, loc, o);
        locp += __shfl_xor_sync(0xffffffffu, locp, o);
        lmax = fmax(lmax, __shfl_xor_sync(0xffffffffu, lmax, o));
    }
    const double mean = G.dir_top ? 0.0 : loc / G.sum_hz;  // a Dirichlet outlet: nothing to remove
    if (first_solve && lane == 0) {
        w.mean_b[g] = mean;
        // compatibility defect large compared with the plane means -> warning
        if (fabs(mean) > 1e-8 * lmax && fabs(mean) > 0.0) atomicOr(w.err, 1u << 7);
    }
    auto scan = [&](double x, bool up) {  // sum over the lanes before (up: after) this one
        double in = x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double y = up ? __shfl_down_sync(0xffffffffu, in, o) : __shfl_up_sync(0xffffffffu, in, o);
            if (up ? lane + o < 32 : lane >= o) in += y;
        }
        const double ex = up ? __shfl_down_sync(0xffffffffu, in, 1) : __shfl_up_sync(0xffffffffu, in, 1);
        return (up ? lane == 31 : lane == 0) ? 0.0 : ex;
    };
    // fluxes S_k = sum_{j <= k} hz_j (rhs_j - mean), then phi_k = phi_top - sum_{j >= k} gz_{j+1} S_j
    double run = 0.0;
    for (int k = k0; k < k1; ++k) run += hz[k] * (rhs[k] - mean);
    double S = scan(run, false);
    for (int k = k0; k < k1; ++k) {
        S += hz[k] * (rhs[k] - mean);
        rhs[k] = k + 1 < nz ? S * gz[k] : 0.0;
    }
    const double Stop = __shfl_sync(0xffffffffu, S, (nz - 1) / per);  // S_{nz-1}
    run = 0.0;
    for (int k = k0; k < k1; ++k) run += rhs[k];
    double inc = scan(run, true);
    const double ph_top = G.dir_top ? -Stop / (w.z.hz[zo + nz - 1] * G.ez_top) : 0.0;
    double sv = 0.0;
    for (int k = k1 - 1; k >= k0; --k) {
        inc += rhs[k];
        rhs[k] = ph_top - inc;
        sv += hz[k] * rhs[k];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sv += __shfl_xor_sync(0xffffffffu, sv, o);
    const double mphi = G.dir_top ? 0.0 : (sv + (first_solve ? 0.0 : locp)) / G.sum_hz;  // weighted mean to remove
    cx<T> *spec = reinterpret_cast<cx<T> *>(w.spec) + G.spec_off;
    const size_t stride = (size_t)G.ncb * G.ny * G.mb;
    __syncwarp();
    for (int k = lane; k < nz; k += 32) {
        const double v = rhs[k] - mphi;
        spec[(size_t)k * stride] = {(T)v, (T)0};
        w.sol00[zo + k] = v;
    }
}

}  // namespace ibf
