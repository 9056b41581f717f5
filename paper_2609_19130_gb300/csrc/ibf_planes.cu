// ibf_planes.cu -- sm_103a kernels of the plane-parallel y/z path: the y transforms of all
// planes at once (k_yfft), then the z systems of all modes (k_zsolve); and the viscous solve's
// y step (k_yhelm), made of the same transform passes.  Compiled twice:
// IBF_PART 0 the fp32 kernels, 1 the fp64 ones.
#include "ibf_viscous.h"
#include "ibf_yz.cuh"

#include <type_traits>

namespace ibf {

// ================================================================ plane-parallel y/z path
// Streaming walks the planes of a column block one after the other, so it needs several
// hundred column blocks to fill the GPU (one CTA each) and pays the latency of a plane's
// transform nz times in a row.  Here the y transforms of all planes run at once (k_yfft)
// and the z systems of all modes after them (k_zsolve, one thread per mode, or k_zsolve_tile).
// The spectrum is read and written three times instead of twice (four times with k_zsolve,
// whose two sweeps each cross it), mostly inside L2 at the sizes that take this path.  The
// y-modes of a column block lie in natural order (slot n of sequence mm: n mb + mm).
//
// y transform of gb consecutive column blocks (sequences) of one plane.  Periodic y: the
// first pass of the two-level FFT reads its inputs from global memory straight into
// registers (lanes over columns: runs of N2 values, 16 and more loads in flight per
// thread), the second writes its outputs straight back (natural order: lanes over q1, runs
// of N1 values), so a value crosses shared memory once and the block waits once.  A
// wall-bounded y (ydct_col_pass, ydct_pairs) needs two more crossings for its DCT twiddles:
// 256x192x129, forward 64 -> 40 us, inverse 53 -> 45.
// MAXP: the largest register DFT of the launch's grids.  The 16-point DFT and smaller ones
// fit 64 registers in fp32, which keeps eight CTAs per SM resident instead of four.
// sums (forward; 1 the projection's first solve, 2 a refinement's, 0 none): the first CTA of
// each plane also adds the plane's sums for the (0,0) mode, which the next launch solves.
template <typename T, int P, int DIR>
__device__ __forceinline__ void yfft_first_pass(cx<T> *buf, int sstride, const cx<T> *pl, int nslot, int mb, int N1,
                                                int N2, const FDiv &fmb, const FDiv &fn, int nseq, int nvalid,
                                                const cx<T> *tw) {
    // forward: columns c (P = N1 rows of stride N2); inverse: rows q1 (P = N2 modes of stride N1)
    const int nt = DIR < 0 ? N2 : N1, ntask = nseq * nt;
    for (int t = threadIdx.x; t < ntask; t += blockDim.x) {
        const int rest = (int)fdiv((unsigned)t, fmb), mm = t - rest * mb;
        const int q = (int)fdiv((unsigned)rest, fn), c = rest - q * nt;
        const int sq = q * mb + mm;
        if (sq >= nvalid) continue;
        const cx<T> *src = pl + (size_t)q * nslot + c * mb + mm;
        cx<T> x[P];
#pragma unroll
        for (int r = 0; r < P; ++r) x[r] = src[r * nt * mb];
        IPDFT<T, P, P, 0, 1, DIR>::run(x);
        cx<T> *seq = buf + sq * sstride;
        if (DIR < 0) {
            if (c > 0) ip_store<T, P, 0, true, false>(x, seq + c, N2 + 1, tw + c, N2);
            else ip_store<T, P, 0, false, false>(x, seq + c, N2 + 1, tw, 0);
        } else {
            cx<T> *row = seq + c * (N2 + 1);
            if (c > 0) ip_store<T, P, 0, true, true>(x, row, 1, tw + N1 * N2 + c, N1);
            else ip_store<T, P, 0, false, false>(x, row, 1, tw, 0);
        }
    }
}
template <typename T, int P, int DIR>
__device__ __forceinline__ void yfft_second_pass(const cx<T> *buf, int sstride, cx<T> *pl, int nslot, int mb, int N1,
                                                 int N2, const FDiv &fmb, const FDiv &fn, int nseq, int nvalid) {
    // forward: rows q1 (P = N2), outputs n = q1 + N1 p; inverse: columns c (P = N1), outputs r N2 + c
    const int nt = DIR < 0 ? N1 : N2, ntask = nseq * nt;
    for (int t = threadIdx.x; t < ntask; t += blockDim.x) {
        const int rest = (int)fdiv((unsigned)t, fmb), mm = t - rest * mb;
        const int q = (int)fdiv((unsigned)rest, fn), c = rest - q * nt;
        const int sq = q * mb + mm;
        if (sq >= nvalid) continue;
        const cx<T> *seq = buf + sq * sstride + (DIR < 0 ? c * (N2 + 1) : c);
        const int ld = DIR < 0 ? 1 : N2 + 1;
        cx<T> x[P];
#pragma unroll
        for (int r = 0; r < P; ++r) x[r] = seq[r * ld];
        IPDFT<T, P, P, 0, 1, DIR>::run(x);
        ip_store<T, P, 0, false, false>(x, pl + (size_t)q * nslot + c * mb + mm, nt * mb, nullptr, 0);
    }
}

// DCT-II along a wall-bounded y through an FFT (Makhoul): the same two register passes with
// the sample order i(p) of FFT input p folded into the global accesses (the inverse of
// dct_perm), and the pairwise post (forward) or pre (inverse) twiddles of modes n and N - n
// between shared and global memory: three crossings of shared memory, not five.
__device__ __forceinline__ int dct_sample(int p, int n) { return 2 * p < n ? 2 * p : 2 * (n - p) - 1; }

template <typename T, int P, int DIR>
__device__ __forceinline__ void ydct_col_pass(cx<T> *buf, int sstride, cx<T> *pl, int nslot, int mb, int ny, int N2,
                                              const FDiv &fmb, const FDiv &fN2, int nseq, int nvalid, const cx<T> *tw) {
    const int ntask = nseq * N2;
    for (int t = threadIdx.x; t < ntask; t += blockDim.x) {
        const int rest = (int)fdiv((unsigned)t, fmb), mm = t - rest * mb;
        const int q = (int)fdiv((unsigned)rest, fN2), c = rest - q * N2;
        const int sq = q * mb + mm;
        if (sq >= nvalid) continue;
        cx<T> *g = pl + (size_t)q * nslot + mm, *seq = buf + sq * sstride + c;
        cx<T> x[P];
        if (DIR < 0) {
#pragma unroll
            for (int r = 0; r < P; ++r) x[r] = g[dct_sample(r * N2 + c, ny) * mb];
            IPDFT<T, P, P, 0, 1, DIR>::run(x);
            if (c > 0) ip_store<T, P, 0, true, false>(x, seq, N2 + 1, tw + c, N2);
            else ip_store<T, P, 0, false, false>(x, seq, N2 + 1, tw, 0);
        } else {
#pragma unroll
            for (int r = 0; r < P; ++r) x[r] = seq[r * (N2 + 1)];
            IPDFT<T, P, P, 0, 1, DIR>::run(x);
            cx<T> z[P];
            ip_store<T, P, 0, false, false>(x, z, 1, tw, 0);
#pragma unroll
            for (int r = 0; r < P; ++r) g[dct_sample(r * N2 + c, ny) * mb] = z[r];
        }
    }
}

// forward: X_n = (P + Q)/2, X_{N-n} = i (P - Q)/2 with P = W^n V_n, Q = conj(W^n) V_{N-n}, from the
// FFT in shared memory to global; inverse: V_n = conj(W^n)(X_n - i X_{N-n}), V_{N-n} = W^n (X_n +
// i X_{N-n}), from global to shared memory; X_0 = V_0 (dct_post and dct_pre, whose arithmetic
// this is).
template <typename T, int DIR>
__device__ __forceinline__ void ydct_pairs(cx<T> *buf, int sstride, cx<T> *pl, int nslot, int mb, int N, int N1, int N2,
                                           const FDiv &fmb, const FDiv &fN1, int nseq, int nvalid, const cx<T> *W) {
    const int np = (N >> 1) + 1;
    for (int t = threadIdx.x; t < nseq * np; t += blockDim.x) {
        const int rest = (int)fdiv((unsigned)t, fmb), mm = t - rest * mb, q = rest / np, n = rest - q * np;
        const int sq = q * mb + mm;
        if (sq >= nvalid) continue;
        cx<T> *seq = buf + sq * sstride, *g = pl + (size_t)q * nslot + mm;
        const int m = n == 0 ? 0 : N - n;
        cx<T> &sa = seq[pos_tr(n, N1, N2, fN1)], &sb = seq[pos_tr(m, N1, N2, fN1)];
        const cx<T> w = W[n];
        if (DIR < 0) {
            const cx<T> a = sa, b = sb;
            const cx<T> P = dct_rot(w, a), Q = dct_rotc(w, b);
            g[n * mb] = n == 0 ? a : cx<T>{(P.x + Q.x) * (T)0.5, (P.y + Q.y) * (T)0.5};
            if (m != n) g[m * mb] = {(Q.y - P.y) * (T)0.5, (P.x - Q.x) * (T)0.5};
        } else {
            const cx<T> a = g[n * mb], b = g[m * mb];
            const cx<T> d = {a.x + b.y, a.y - b.x};  // X_n - i X_{N-n}
            const cx<T> e = {a.x - b.y, a.y + b.x};  // X_n + i X_{N-n}
            sa = n == 0 ? a : dct_rotc(w, d);
            if (m != n) sb = dct_rot(w, e);
        }
    }
}

template <typename T, int DIR, bool W, int MAXP>
__global__ void __launch_bounds__(kYZThreads, sizeof(T) == 4 ? (MAXP <= 16 ? 8 : 4) : (MAXP <= 16 ? 4 : 2))
    k_yfft(Work w, int sums) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int b = blockIdx.x;
    const int g = find_grid(w.yfft_start, w.ngrids, b);
    const GridDev &G = w.grids[g];
    const int lb = b - __ldg(w.yfft_start + g);
    const int ncb = G.ncb, gb = G.yf_gb, ngrp = G.yf_ngrp, k = lb / ngrp, cb0 = (lb - k * ngrp) * gb;
    const int ny = G.ny, mb = G.mb, nxh = G.nxh;
    const int N1 = G.ny1, N2 = G.ny2, sstride = fft_seq_len(N1, N2) + 1;
    const FDiv fN1 = G.fny1, fN2 = G.fny2, fmb = G.fmb;
    const int nslot = ny * mb;
    const int nb = min(gb, ncb - cb0), nseq = nb * mb;
    const int nvalid = min(nseq, nxh - cb0 * mb);
    const cx<T> *twy = reinterpret_cast<const cx<T> *>(w.twy) + G.twy_off;
    cx<T> *buf = reinterpret_cast<cx<T> *>(smem_raw);
    cx<T> *pl = reinterpret_cast<cx<T> *>(w.spec) + G.spec_off + ((size_t)k * ncb + cb0) * nslot;
    if (DIR < 0 && sums && cb0 == 0 && threadIdx.x >= kYZThreads - 32) plane_sums(w, G, k, sums == 1);
    if constexpr (W) {
        if (G.wall_y) {
            const cx<T> *dcty = reinterpret_cast<const cx<T> *>(w.twy) + G.dcty_off;
            auto cols = [&]() {
                switch (N1) {
#define IBF_CASE(P)                                                                                                   \
    case P:                                                                                                           \
        if constexpr (P <= MAXP)                                                                                      \
            ydct_col_pass<T, P, DIR>(buf, sstride, pl, nslot, mb, ny, N2, fmb, fN2, nseq, nvalid, twy);               \
        break;
                    IBF_FFT_SIZES(IBF_CASE)
#undef IBF_CASE
                    default: break;
                }
            };
            if (DIR < 0) {
                cols();
            } else {
                ydct_pairs<T, DIR>(buf, sstride, pl, nslot, mb, ny, N1, N2, fmb, fN1, nseq, nvalid, dcty);
            }
            __syncthreads();
            fft_row_pass<T, DIR, MAXP>(buf, nvalid, sstride, N1, N2, fN1, twy, threadIdx.x, blockDim.x);
            __syncthreads();
            if (DIR < 0) {
                ydct_pairs<T, DIR>(buf, sstride, pl, nslot, mb, ny, N1, N2, fmb, fN1, nseq, nvalid, dcty);
            } else {
                cols();
            }
            return;
        }
    }
    switch (DIR < 0 ? N1 : N2) {
#define IBF_CASE(P)                                                                                                 \
    case P:                                                                                                         \
        if constexpr (P <= MAXP)                                                                                    \
            yfft_first_pass<T, P, DIR>(buf, sstride, pl, nslot, mb, N1, N2, fmb, DIR < 0 ? fN2 : fN1, nseq, nvalid, \
                                       twy);                                                                        \
        break;
        IBF_FFT_SIZES(IBF_CASE)
#undef IBF_CASE
        default: break;
    }
    __syncthreads();
    switch (DIR < 0 ? N2 : N1) {
#define IBF_CASE(P)                                                                                                   \
    case P:                                                                                                           \
        if constexpr (P <= MAXP)                                                                                      \
            yfft_second_pass<T, P, DIR>(buf, sstride, pl, nslot, mb, N1, N2, fmb, DIR < 0 ? fN1 : fN2, nseq, nvalid); \
        break;
        IBF_FFT_SIZES(IBF_CASE)
#undef IBF_CASE
        default: break;
    }
}

// The viscous solve's y step: y-FFT, multiplication by fx_m fy_n, fx_m = 1/(1 + beta (4/dx^2)
// sin^2(pi m/nx)) and fy_n likewise (tables of k_helm_table), inverse y-FFT, of gb column
// blocks of one plane of grid g's x-spectrum, in place (row order in and out).  The x-FFT
// scaled by 1/(nx ny), so the unnormalised inverse returns the field.  The forward row pass
// leaves a thread with the very modes that the inverse row pass takes, so the factors and the
// inverse follow in its registers: two crossings of shared memory instead of six.
// 384x384x192 mixed 177 -> 71 us, 192x144x101 fp64 249 -> 181 us.
template <typename T, int P, int K>
__device__ __forceinline__ void helm_scale(const cx<T> (&x)[P], cx<T> (&z)[P], T fx, const T *fy, int N1) {
    if constexpr (K < P) {
        const T f = fx * fy[N1 * K];
        const cx<T> v = x[ip_rev(P, K)];
        z[K] = {v.x * f, v.y * f};
        helm_scale<T, P, K + 1>(x, z, fx, fy, N1);
    }
}
template <typename T, int P>
__device__ __forceinline__ void yhelm_row_pass(cx<T> *buf, int sstride, int mb, int N1, const FDiv &fmb, const FDiv &fN1,
                                               int nseq, int nvalid, const T *fx, const T *fy, const cx<T> *tw) {
    const int ntask = nseq * N1;
    for (int t = threadIdx.x; t < ntask; t += blockDim.x) {
        const int rest = (int)fdiv((unsigned)t, fmb), mm = t - rest * mb;
        const int q = (int)fdiv((unsigned)rest, fN1), q1 = rest - q * N1;
        const int sq = q * mb + mm;
        if (sq >= nvalid) continue;
        cx<T> *row = buf + sq * sstride + q1 * (P + 1);
        cx<T> x[P], z[P];
#pragma unroll
        for (int r = 0; r < P; ++r) x[r] = row[r];
        IPDFT<T, P, P, 0, 1, -1>::run(x);
        helm_scale<T, P, 0>(x, z, fx[sq], fy + q1, N1);
        IPDFT<T, P, P, 0, 1, 1>::run(z);
        if (q1 > 0) ip_store<T, P, 0, true, true>(z, row, 1, tw + N1 * P + q1, N1);
        else ip_store<T, P, 0, false, false>(z, row, 1, tw, 0);
    }
}
template <typename T, int MAXP>
__global__ void __launch_bounds__(kYZThreads, sizeof(T) == 4 ? (MAXP <= 16 ? 8 : 4) : (MAXP <= 16 ? 4 : 2))
    k_yhelm(Work w, int g, const T *fxy) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const GridDev &G = w.grids[g];
    const int ncb = G.ncb, gb = G.yf_gb, ngrp = G.yf_ngrp, k = blockIdx.x / ngrp, cb0 = (blockIdx.x - k * ngrp) * gb;
    const int ny = G.ny, mb = G.mb, nxh = G.nxh;
    const int N1 = G.ny1, N2 = G.ny2, sstride = fft_seq_len(N1, N2) + 1;
    const FDiv fN1 = G.fny1, fN2 = G.fny2, fmb = G.fmb;
    const int nslot = ny * mb, nseq = min(gb, ncb - cb0) * mb, nvalid = min(nseq, nxh - cb0 * mb);
    const cx<T> *twy = reinterpret_cast<const cx<T> *>(w.twy) + G.twy_off;
    cx<T> *buf = reinterpret_cast<cx<T> *>(smem_raw);
    cx<T> *pl = reinterpret_cast<cx<T> *>(w.spec) + G.spec_off + ((size_t)k * ncb + cb0) * nslot;
    const T *fx = fxy + cb0 * mb, *fy = fxy + nxh;
    switch (N1) {
#define IBF_CASE(P)                                                                                                     \
    case P:                                                                                                             \
        if constexpr (P <= MAXP)                                                                                        \
            yfft_first_pass<T, P, -1>(buf, sstride, pl, nslot, mb, N1, N2, fmb, fN2, nseq, nvalid, twy);                \
        break;
        IBF_FFT_SIZES(IBF_CASE)
#undef IBF_CASE
        default: break;
    }
    __syncthreads();
    switch (N2) {
#define IBF_CASE(P)                                                                                                     \
    case P:                                                                                                             \
        if constexpr (P <= MAXP)                                                                                        \
            yhelm_row_pass<T, P>(buf, sstride, mb, N1, fmb, fN1, nseq, nvalid, fx, fy, twy);                            \
        break;
        IBF_FFT_SIZES(IBF_CASE)
#undef IBF_CASE
        default: break;
    }
    __syncthreads();
    switch (N1) {
#define IBF_CASE(P)                                                                                                     \
    case P:                                                                                                             \
        if constexpr (P <= MAXP)                                                                                        \
            yfft_second_pass<T, P, 1>(buf, sstride, pl, nslot, mb, N1, N2, fmb, fN2, nseq, nvalid);                     \
        break;
        IBF_FFT_SIZES(IBF_CASE)
#undef IBF_CASE
        default: break;
    }
}

// Thomas along z of every mode, one thread per mode of a grid (slot gs of the flattened
// [column block][slot] index, so plane k of the spectrum is one contiguous run of ncb*nslot
// modes), pivots from the plan's table: forward elimination (d' overwrites the spectrum),
// then back substitution (phi_hat).  The (0,0) modes of grids 0..n00-1 are solved by the
// first n00 blocks, beside the others at no time of their own; with n00 = 0 they come from
// sol00 (k_00).  A level's arithmetic waits
// for the level before it but its loads do not: they are issued kZBatch levels ahead into
// registers, before the stores of the levels in hand (which the compiler may not move them
// across), so that a thread keeps up to two batches of loads in flight.
constexpr int kZBatch = 8;
// the (0,0) solve out of line: inlined, its registers and code slow the sweeps' loops
template <typename T>
__device__ __noinline__ void mode00_call(const Work &w, int g, int first_solve, double *sh) {
    if (threadIdx.x < 32) mode00_warp<T>(w, g, first_solve, sh);
}
template <typename T>
__global__ void __launch_bounds__(kZSolveThreads) k_zsolve(Work w, int n00, int first_solve) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if ((int)blockIdx.x < n00) {
        mode00_call<T>(w, blockIdx.x, first_solve, reinterpret_cast<double *>(smem_raw));
        return;
    }
    const int b = blockIdx.x - n00, g = find_grid(w.zsolve_start, w.ngrids, b);
    const GridDev &G = w.grids[g];
    const int gs = (b - __ldg(w.zsolve_start + g)) * kZSolveThreads + threadIdx.x;
    const int nslot = G.ny * G.mb, M = G.ncb * nslot, nz = G.nz;
    if (gs >= M || (gs == 0 && n00 > 0)) return;
    const bool singular = gs == 0;
    cx<T> *sp = reinterpret_cast<cx<T> *>(w.spec) + G.spec_off + gs;
    const T *tb = reinterpret_cast<const T *>(w.tab) + G.tab_off + gs;
    const T *a = zarr<T>(w.z.az, w.z.azf) + G.z_off;
    const T *c = zarr<T>(w.z.cz, w.z.czf) + G.z_off;
    const double *s00 = w.sol00 + G.z_off;
    cx<T> r[kZBatch], rn[kZBatch];
    T v[kZBatch], vn[kZBatch];
    auto load = [&](int k0, cx<T> (&x)[kZBatch], T (&y)[kZBatch], bool up) {
#pragma unroll
        for (int u = 0; u < kZBatch; ++u) {
            const int k = up ? k0 + u : nz - 1 - (k0 + u);
            if (k0 + u < nz) {
                x[u] = sp[(size_t)k * M];
                y[u] = __ldg(tb + (size_t)k * M);
            }
        }
    };
    cx<T> s = {(T)0, (T)0};
    load(0, rn, vn, true);
    for (int k0 = 0; k0 < nz; k0 += kZBatch) {
#pragma unroll
        for (int u = 0; u < kZBatch; ++u) { r[u] = rn[u]; v[u] = vn[u]; }
        if (k0 + kZBatch < nz) load(k0 + kZBatch, rn, vn, true);
#pragma unroll
        for (int u = 0; u < kZBatch; ++u) {
            const int k = k0 + u;
            if (k >= nz) break;
            const T ak = __ldg(a + k);
            s = {(r[u].x - ak * s.x) * v[u], (r[u].y - ak * s.y) * v[u]};
            sp[(size_t)k * M] = s;
        }
    }
    s = {(T)0, (T)0};
    load(0, rn, vn, false);
    for (int k0 = 0; k0 < nz; k0 += kZBatch) {
#pragma unroll
        for (int u = 0; u < kZBatch; ++u) { r[u] = rn[u]; v[u] = vn[u]; }
        if (k0 + kZBatch < nz) load(k0 + kZBatch, rn, vn, false);
#pragma unroll
        for (int u = 0; u < kZBatch; ++u) {
            const int k = nz - 1 - (k0 + u);
            if (k < 0) break;
            const T cp = __ldg(c + k) * v[u];
            s = {r[u].x - cp * s.x, r[u].y - cp * s.y};
            if (singular) s = {(T)s00[k], (T)0};
            sp[(size_t)k * M] = s;
        }
    }
}

#if IBF_PART == 0
// The same solve with the column of every mode held in shared memory between the two sweeps
// (fp32, up to kZTileMaxNz levels): the spectrum is read and written once instead of twice,
// and the pivots read once (20 B per mode and level instead of 40).  One warp per CTA takes
// kZTile = 16 modes, two lanes a mode: the real and the imaginary part obey the same real
// recurrence.  All of the tile's copies are issued at once (cp.async, in four groups of
// levels), so the forward sweep starts on the first quarter while the rest is on its way and
// 100 KB and more per SM are in flight; the other CTAs of the SM load or store meanwhile.
// 512x512x256: 181 us against k_zsolve's 264 (3.7 TB/s of its 20 B: an SM's columns wait on
// one warp's dependent chain per scheduler, two sweeps of 256 levels); 256^3 50 against 78.
// Taller columns leave fewer warps per SM, so from kZTileMaxNz levels on k_zsolve, which
// streams at the HBM rate, is faster unless the grid has few modes (512 levels, us, tile /
// k_zsolve: 1024x1024 2166 / 1607, 512x512 600 / 533, 64x64 30 / 114).
// Shared memory: spectrum tile [nz][16] complex, pivots [nz][16], a [nz], c [nz].
__global__ void __launch_bounds__(32) k_zsolve_tile(Work w, int n00, int first_solve) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if ((int)blockIdx.x < n00) {
        mode00_call<float>(w, blockIdx.x, first_solve, reinterpret_cast<double *>(smem_raw));
        return;
    }
    const int b = blockIdx.x - n00, g = find_grid(w.zsolve_start, w.ngrids, b);
    const GridDev &G = w.grids[g];
    const int gs0 = (b - __ldg(w.zsolve_start + g)) * kZTile;
    const int M = G.ncb * G.ny * G.mb, nz = G.nz, lane = threadIdx.x;
    const int nm = min(kZTile, M - gs0);  // modes of this tile
    cx<float> *sp = reinterpret_cast<cx<float> *>(w.spec) + G.spec_off + gs0;
    const float *tb = reinterpret_cast<const float *>(w.tab) + G.tab_off + gs0;
    float *xs = reinterpret_cast<float *>(smem_raw);   // [k][2 kZTile]
    const int nzp = (nz + kZBatch - 1) & ~(kZBatch - 1);  // whole batches: the pad is read, never used
    float *ts = xs + (size_t)nzp * (2 * kZTile);          // [k][kZTile]
    float *sa = ts + (size_t)nzp * kZTile, *sc = sa + nzp;
    constexpr int NG = 4;
    const int per = ((nz + NG - 1) / NG + kZBatch - 1) & ~(kZBatch - 1);  // levels per group, whole batches (of 8)
    // 16-byte copies need every plane's run of modes aligned: an even number of modes per
    // plane for the spectrum, a multiple of four for the pivots (offsets alike)
    const bool v2 = ((M | (int)G.spec_off) & 1) == 0, v4 = ((M | (int)G.tab_off) & 3) == 0;
    const bool aligned = v2 && v4;
    // aligned: eight lanes a level of the spectrum (four levels a turn), four lanes a level of
    // the pivots (eight a turn); the addresses only advance
    const size_t bM = (size_t)M;
    const cx<float> *gx = sp + (size_t)(lane >> 3) * bM + (lane & 7) * 2;
    const float *gt = tb + (size_t)(lane >> 2) * bM + (lane & 3) * 4;
    float *dx = xs + (lane >> 3) * 32 + (lane & 7) * 4, *dt = ts + (lane >> 2) * 16 + (lane & 3) * 4;
    const bool inx = (lane & 7) * 2 < nm, intb = (lane & 3) * 4 < nm;
#pragma unroll
    for (int q = 0; q < NG; ++q) {
        const int k0 = q * per, k1 = min(nz, k0 + per);
        if (aligned) {
#pragma unroll 4
            for (int k = k0 + (lane >> 3); k < k1; k += 4) {
                if (inx) cp_async<16>(dx, gx);
                gx += 4 * bM;
                dx += 4 * 32;
            }
#pragma unroll 4
            for (int k = k0 + (lane >> 2); k < k1; k += 8) {
                if (intb) cp_async<16>(dt, gt);
                gt += 8 * bM;
                dt += 8 * 16;
            }
        } else {
            for (int t = k0 * 16 + lane; t < k1 * 16; t += 32) {
                const int k = t >> 4, c = t & 15;
                if (c < nm) {
                    cp_async<8>(xs + k * 32 + 2 * c, sp + (size_t)k * M + c);
                    cp_async<4>(ts + k * 16 + c, tb + (size_t)k * M + c);
                }
            }
        }
        cp_async_commit();
    }
    for (int k = lane; k < nz; k += 32) {
        sa[k] = __ldg(w.z.azf + G.z_off + k);
        sc[k] = __ldg(w.z.czf + G.z_off + k);
    }
    const int mode = lane >> 1;
    const bool live = mode < nm && !(n00 > 0 && gs0 + mode == 0);
    // one batch of levels from kb on into registers
    float s = 0.f;
    auto fetch = [&](int kb, const float *coef, float (&r)[kZBatch], float (&v)[kZBatch], float (&e)[kZBatch]) {
        const float *x = xs + kb * 32 + lane, *t = ts + kb * 16 + mode;
        const float4 e0 = *reinterpret_cast<const float4 *>(coef + kb), e1 = *reinterpret_cast<const float4 *>(coef + kb + 4);
#pragma unroll
        for (int u = 0; u < kZBatch; ++u) {
            r[u] = x[u * 32];
            v[u] = t[u * 16];
        }
        e[0] = e0.x; e[1] = e0.y; e[2] = e0.z; e[3] = e0.w;
        e[4] = e1.x; e[5] = e1.y; e[6] = e1.z; e[7] = e1.w;
    };
    float r[2][kZBatch], v[2][kZBatch], e[2][kZBatch];
    auto up = [&](int kb, const float (&rr)[kZBatch], const float (&vv)[kZBatch], const float (&ee)[kZBatch]) {
        float *x = xs + kb * 32 + lane;
#pragma unroll
        for (int u = 0; u < kZBatch; ++u) {
            s = (rr[u] - ee[u] * s) * vv[u];  // levels past nz - 1 write the pad
            x[u * 32] = s;
        }
    };
    auto sweep_up = [&](int k0, int k1) {  // two batches a turn, the second's loads before the first's stores
        if (k0 >= k1) return;
        fetch(k0, sa, r[0], v[0], e[0]);
        for (int kb = k0; kb < k1; kb += 2 * kZBatch) {
            if (kb + kZBatch < k1) fetch(kb + kZBatch, sa, r[1], v[1], e[1]);
            up(kb, r[0], v[0], e[0]);
            if (kb + kZBatch >= k1) break;
            if (kb + 2 * kZBatch < k1) fetch(kb + 2 * kZBatch, sa, r[0], v[0], e[0]);
            up(kb + kZBatch, r[1], v[1], e[1]);
        }
    };
    cp_async_wait<3>();
    __syncwarp();
    sweep_up(0, min(nz, per));
    cp_async_wait<2>();
    __syncwarp();
    sweep_up(per, min(nz, 2 * per));
    cp_async_wait<1>();
    __syncwarp();
    sweep_up(2 * per, min(nz, 3 * per));
    cp_async_wait<0>();
    __syncwarp();
    sweep_up(3 * per, nz);
    s = 0.f;
    const size_t lvl = 2 * (size_t)M;  // floats per plane
    float *out = reinterpret_cast<float *>(sp), *po = out + (size_t)(nz - 1) * lvl;  // (warp-uniform)
    auto down = [&](int n, const float (&rr)[kZBatch], const float (&vv)[kZBatch], const float (&ee)[kZBatch]) {
#pragma unroll
        for (int u = kZBatch - 1; u >= 0; --u) {
            if (u < n) {
                const float cp = ee[u] * vv[u];
                s = rr[u] - cp * s;
                if (live) po[lane] = s;
                po -= lvl;
            }
        }
    };
    const int kl = nzp - kZBatch;  // the last batch, nz - kl levels
    fetch(kl, sc, r[0], v[0], e[0]);
    if (kl > 0) fetch(kl - kZBatch, sc, r[1], v[1], e[1]);
    down(nz - kl, r[0], v[0], e[0]);
    for (int kb = kl - kZBatch; kb >= 0; kb -= 2 * kZBatch) {
        if (kb >= kZBatch) fetch(kb - kZBatch, sc, r[0], v[0], e[0]);
        down(kZBatch, r[1], v[1], e[1]);
        if (kb < kZBatch) break;
        if (kb >= 2 * kZBatch) fetch(kb - 2 * kZBatch, sc, r[1], v[1], e[1]);
        down(kZBatch, r[0], v[0], e[0]);
    }
    if (gs0 == 0 && n00 == 0) {  // the (0,0) mode: its fp64 solution instead
        __syncwarp();
        for (int k = lane; k < nz; k += 32) sp[(size_t)k * M] = {(float)w.sol00[G.z_off + k], 0.f};
    }
}

#endif

// ================================================================ launchers
#if IBF_PART == 0
typedef float PartT;
#define IBF_PART_NAME(x) x##_f32
#else
typedef double PartT;
#define IBF_PART_NAME(x) x##_f64
#endif

cudaError_t IBF_PART_NAME(launch_yfft)(int inverse, const Work &w, int nblk, int maxp, int sums, size_t smem,
                                       cudaStream_t st) {
    if (nblk <= 0) return cudaSuccess;
    const dim3 gr = grid1(nblk);
    auto go = [&](auto dtag) {
        constexpr int DIR = decltype(dtag)::value;
        if (w.walls && maxp <= 16) k_yfft<PartT, DIR, true, 16><<<gr, kYZThreads, smem, st>>>(w, sums);
        else if (w.walls) k_yfft<PartT, DIR, true, 32><<<gr, kYZThreads, smem, st>>>(w, sums);
        else if (maxp <= 16) k_yfft<PartT, DIR, false, 16><<<gr, kYZThreads, smem, st>>>(w, sums);
        else k_yfft<PartT, DIR, false, 32><<<gr, kYZThreads, smem, st>>>(w, sums);
    };
    if (inverse) go(std::integral_constant<int, 1>{});
    else go(std::integral_constant<int, -1>{});
    return cudaGetLastError();
}

cudaError_t IBF_PART_NAME(launch_yhelm)(const Work &w, int g, int nblk, int maxp, const PartT *fxy, size_t smem,
                                        cudaStream_t st) {
    if (nblk <= 0) return cudaSuccess;
    if (maxp <= 16) k_yhelm<PartT, 16><<<grid1(nblk), kYZThreads, smem, st>>>(w, g, fxy);
    else k_yhelm<PartT, 32><<<grid1(nblk), kYZThreads, smem, st>>>(w, g, fxy);
    return cudaGetLastError();
}

// tilesmem: shared memory of k_zsolve_tile, 0 for k_zsolve
cudaError_t IBF_PART_NAME(launch_zsolve)(const Work &w, int nblk, int n00, int first, int maxnz, size_t tilesmem,
                                         cudaStream_t st) {
    if (nblk <= 0) return cudaSuccess;
    const size_t smem00 = n00 > 0 ? sh00_bytes(maxnz) : 0;
#if IBF_PART == 0
    if (tilesmem > 0) {
        k_zsolve_tile<<<grid1(nblk + n00), 32, tilesmem > smem00 ? tilesmem : smem00, st>>>(w, n00, first);
        return cudaGetLastError();
    }
#endif
    k_zsolve<PartT><<<grid1(nblk + n00), kZSolveThreads, smem00, st>>>(w, n00, first);
    return cudaGetLastError();
}

cudaError_t IBF_PART_NAME(set_smem_limits_planes)(const Work &w) {
    const void *per[] = {(const void *)k_yfft<PartT, -1, false, 16>, (const void *)k_yfft<PartT, 1, false, 16>,
                         (const void *)k_yfft<PartT, -1, false, 32>, (const void *)k_yfft<PartT, 1, false, 32>},
               *wall[] = {(const void *)k_yfft<PartT, -1, true, 16>, (const void *)k_yfft<PartT, 1, true, 16>,
                          (const void *)k_yfft<PartT, -1, true, 32>, (const void *)k_yfft<PartT, 1, true, 32>},
               *any[] = {(const void *)k_yhelm<PartT, 16>, (const void *)k_yhelm<PartT, 32>,
#if IBF_PART == 0
                         (const void *)k_zsolve_tile,
#endif
               };
    cudaError_t e = cudaSuccess;
    for (const void *fn : w.walls ? wall : per)
        if (e == cudaSuccess) e = set_smem_cap(fn);
    for (const void *fn : any)
        if (e == cudaSuccess) e = set_smem_cap(fn);
    return e;
}

}  // namespace ibf
