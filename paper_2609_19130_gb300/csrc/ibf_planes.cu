// ibf_planes.cu -- sm_103a kernels of the plane-parallel y/z path: the y transforms of all
// planes at once (k_yfft), then the z systems of all modes (k_zsolve).  Compiled twice:
// IBF_PART 0 the fp32 kernels, 1 the fp64 ones.
#include "ibf_yz.cuh"

#include <type_traits>

namespace ibf {

// ================================================================ plane-parallel y/z path
// Streaming walks the planes of a column block one after the other, so it needs several
// hundred column blocks to fill the GPU (one CTA each) and pays the latency of a plane's
// transform nz times in a row.  Here the y transforms of all planes run at once (k_yfft)
// and the z systems of all modes after them (k_zsolve, one thread per mode).  The spectrum
// crosses memory three times instead of twice, mostly inside L2 at the sizes that take
// this path.  The y-modes of a column block lie in natural order (slot n of sequence mm:
// n mb + mm).
//
// y transform of gb consecutive column blocks (sequences) of one plane.  Periodic y: the
// first pass of the two-level FFT reads its inputs from global memory straight into
// registers (lanes over columns: runs of N2 values, 16 and more loads in flight per
// thread), the second writes its outputs straight back (natural order: lanes over q1, runs
// of N1 values), so a value crosses shared memory once and the block waits once.  Plans
// with a wall-bounded direction (W) stage every pass through shared memory, where the DCT's
// pre / post pass of a wall-bounded y works.
// MAXP: the largest register DFT of the launch's grids.  The 16-point DFT and smaller ones
// fit 64 registers in fp32, which keeps eight CTAs per SM resident instead of four.
// The first n00 blocks each solve one grid's (0,0) mode (forward only), which needs nothing
// from the transforms: beside them it costs no time of its own.
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

template <typename T, int DIR, bool W, int MAXP>
__global__ void __launch_bounds__(kYZThreads, sizeof(T) == 4 ? (MAXP <= 16 ? 8 : 4) : (MAXP <= 16 ? 4 : 2))
    k_yfft(Work w, int n00, int first_solve) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (DIR < 0 && (int)blockIdx.x < n00) {
        mode00_solve<T, true>(w, blockIdx.x, first_solve, reinterpret_cast<double *>(smem_raw));
        return;
    }
    const int b = blockIdx.x - n00;
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
    if constexpr (!W) {
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
    } else {
        const int wall_y = G.wall_y;
        const cx<T> *dcty = reinterpret_cast<const cx<T> *>(w.twy) + G.dcty_off;
        const int tid = threadIdx.x, nthr = blockDim.x, ntot = nb * nslot;
        for (int t = tid; t < ntot; t += nthr) {
            const int q = t / nslot, ts = t - q * nslot;
            const int r = (int)fdiv((unsigned)ts, fmb), sq = q * mb + (ts - r * mb);
            // forward: row r of the x-spectrum; inverse: y-mode r
            const int pos = DIR < 0 ? pos_nat(wall_y ? dct_perm(r, ny) : r, fN2) : pos_tr(r, N1, N2, fN1);
            buf[sq * sstride + pos] = sq < nvalid ? pl[t] : cx<T>{(T)0, (T)0};
        }
        __syncthreads();
        if (DIR > 0 && wall_y) dct_pre<T>(buf, nseq, sstride, ny, N1, N2, fN1, dcty);
        fft_batch<T, DIR>(buf, nseq, sstride, N1, N2, fN1, fN2, twy);
        if (DIR < 0 && wall_y) dct_post<T>(buf, nseq, sstride, ny, N1, N2, fN1, dcty);
        for (int t = tid; t < ntot; t += nthr) {
            const int q = t / nslot, ts = t - q * nslot;
            const int r = (int)fdiv((unsigned)ts, fmb), sq = q * mb + (ts - r * mb);
            const int pos = DIR < 0 ? pos_tr(r, N1, N2, fN1) : pos_nat(wall_y ? dct_perm(r, ny) : r, fN2);
            if (sq < nvalid) pl[t] = buf[sq * sstride + pos];
        }
    }
}

// Thomas along z of every mode, one thread per mode of a grid (slot gs of the flattened
// [column block][slot] index, so plane k of the spectrum is one contiguous run of ncb*nslot
// modes), pivots from the plan's table: forward elimination (d' overwrites the spectrum),
// then back substitution (phi_hat), the (0,0) mode from sol00.  A level's arithmetic waits
// for the level before it but its loads do not: they are issued kZBatch levels ahead into
// registers, before the stores of the levels in hand (which the compiler may not move them
// across), so that a thread keeps up to two batches of loads in flight.
constexpr int kZBatch = 8;
template <typename T>
__global__ void __launch_bounds__(kZSolveThreads) k_zsolve(Work w) {
    const int g = find_grid(w.zsolve_start, w.ngrids, blockIdx.x);
    const GridDev &G = w.grids[g];
    const int gs = (blockIdx.x - __ldg(w.zsolve_start + g)) * kZSolveThreads + threadIdx.x;
    const int nslot = G.ny * G.mb, M = G.ncb * nslot, nz = G.nz;
    if (gs >= M) return;
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

// ================================================================ launchers
#if IBF_PART == 0
typedef float PartT;
#define IBF_PART_NAME(x) x##_f32
#else
typedef double PartT;
#define IBF_PART_NAME(x) x##_f64
#endif

cudaError_t IBF_PART_NAME(launch_yfft)(int inverse, const Work &w, int nblk, int maxp, int n00, int first, size_t smem,
                                       cudaStream_t st) {
    if (nblk <= 0) return cudaSuccess;
    const int ne = inverse ? 0 : n00;
    const dim3 gr = grid1(nblk + ne);
    auto go = [&](auto dtag) {
        constexpr int DIR = decltype(dtag)::value;
        if (w.walls) k_yfft<PartT, DIR, true, 32><<<gr, kYZThreads, smem, st>>>(w, ne, first);
        else if (maxp <= 16) k_yfft<PartT, DIR, false, 16><<<gr, kYZThreads, smem, st>>>(w, ne, first);
        else k_yfft<PartT, DIR, false, 32><<<gr, kYZThreads, smem, st>>>(w, ne, first);
    };
    if (inverse) go(std::integral_constant<int, 1>{});
    else go(std::integral_constant<int, -1>{});
    return cudaGetLastError();
}

cudaError_t IBF_PART_NAME(launch_zsolve)(const Work &w, int nblk, cudaStream_t st) {
    if (nblk <= 0) return cudaSuccess;
    k_zsolve<PartT><<<grid1(nblk), kZSolveThreads, 0, st>>>(w);
    return cudaGetLastError();
}

cudaError_t IBF_PART_NAME(set_smem_limits_planes)() {
    const void *fns[] = {(const void *)k_yfft<PartT, -1, false, 16>, (const void *)k_yfft<PartT, 1, false, 16>,
                         (const void *)k_yfft<PartT, -1, false, 32>, (const void *)k_yfft<PartT, 1, false, 32>,
                         (const void *)k_yfft<PartT, -1, true, 32>,  (const void *)k_yfft<PartT, 1, true, 32>};
    cudaError_t e = cudaSuccess;
    for (const void *fn : fns)
        if (e == cudaSuccess) e = set_smem_cap(fn);
    return e;
}

}  // namespace ibf
