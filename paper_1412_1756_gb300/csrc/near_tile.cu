// Near field (Section III-B, Eq. (ZI), first sum): y_i = sum_j Z_ij x_j over
// the stored blocks of each leaf box and its neighbours, as one small matrix
// product per leaf box: [rows of the box] x [strip columns] times
// [strip columns] x [right-hand sides].
//
// One CTA per (leaf box, column chunk, row split), 256 threads.  A thread
// keeps 4 rows x CT columns in registers, so one strip value feeds 2 CT
// multiply-adds and one x value eight; the threads left over after
// (rows / 4) x (columns / CT) tiles split the strip columns among
// themselves, which keeps the CTA full from two right-hand sides (36 ways on
// a 26-row box) to 64 (2 ways).  Chunks of KC strip columns - their values,
// contiguous in the column-major strip, and the gathered x rows - are staged
// in shared memory by cp.async one chunk ahead.  The partial sums are added
// in a fixed order through shared memory at the end.
//
// Bound: instruction issue (69 % active at 64 columns); with two columns the
// bytes of the strips.  Measured, one row per thread and chunks of 16 columns
// before -> this (FP32, us): 30,720-unknown sphere 2 columns 44 -> 36, 10
// columns 120 -> 67, 40 columns 245 -> 132; 122,880 unknowns, 34 columns 765
// -> 400; 115,200-unknown cube, 64 columns 313 -> 293.  One column is left to
// the kernel of one row per thread (28 against 30 us on 28,800 unknowns).
// FP64 is bound by its arithmetic (two multiply-adds per SM and cycle): the
// tiles win only where row splits spread few boxes over the GPU (1,920
// unknowns, 8 columns 105 -> 73) and lose elsewhere (28,800 unknowns, 4
// columns 134 -> 185).
#include "device.h"

#include <algorithm>

namespace mlfma {

namespace {

template <class R> struct Cplx;
template <> struct Cplx<float> { using T = float2; };
template <> struct Cplx<double> { using T = double2; };

template <int BYTES>
__device__ __forceinline__ void cp_n(void *smem, const void *gmem)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    if constexpr (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(s), "l"(gmem), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_commit_n() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait_n() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

constexpr int kNT = 256;   // threads
constexpr int kRT = 4;     // rows per thread

// xu: bytes of one cp.async piece of an x row (16, 8 or 4: what B, the chunk
// and the element size allow); lsh: a power of two of lanes copies one row.
template <class R, int CT>
__global__ void __launch_bounds__(kNT, sizeof(R) == 4 ? 3 : 2) k_near_tile(DevNear nr, const typename Cplx<R>::T *__restrict__ val,
                                                   const R *__restrict__ xp, typename Cplx<R>::T *__restrict__ yp, int B,
                                                   int NBC, int KC, int zcap, int xcap, int xu, int lsh)
{
    using C = typename Cplx<R>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    // [2][zcap] strip values, [2][xcap] x rows, the strip's column indices; the partial sums reuse the first two at the end
    C *zs = reinterpret_cast<C *>(smem_raw);
    R *xs = reinterpret_cast<R *>(zs + 2 * (size_t)zcap);
    int *s_col = reinterpret_cast<int *>(xs + 2 * (size_t)xcap);
    const int nch = (B + NBC - 1) / NBC, box = blockIdx.x / nch, b0 = (blockIdx.x - box * nch) * NBC;
    const int nb = min(NBC, B - b0), ncg = (nb + CT - 1) / CT, XP = ncg * CT;
    const int R0 = nr.box_ptr[box], nrow = nr.box_ptr[box + 1] - R0;
    const int c0 = nr.col_ptr[box], ncol = nr.col_ptr[box + 1] - c0;
    const int64_t off = nr.strip_off[box];
    // this CTA's rows, a multiple of kRT per split
    const int per = ((nrow + kRT - 1) / kRT + gridDim.y - 1) / gridDim.y * kRT;
    const int ra = blockIdx.y * per, rb = min(nrow, ra + per);
    if (ra >= rb) return;
    const int nchunk = (ncol + KC - 1) / KC, t = threadIdx.x;
    for (int c = t; c < ncol; c += kNT) s_col[c] = nr.strip_col[c0 + c];
    for (int e = t; e < 2 * xcap; e += kNT) xs[e] = R(0);   // columns past the last stay zero
    __syncthreads();
    const int pass = min(rb - ra, kNT / ncg * kRT);   // rows per pass (ncg <= kNT)
    for (int rp = ra; rp < rb; rp += pass) {
        const int rows = min(pass, rb - rp), nrg = (rows + kRT - 1) / kRT, tiles = nrg * ncg;
        const int KS = kNT / tiles, ks = t / tiles, tile = t - ks * tiles, rg = tile / ncg, cg = tile - rg * ncg;
        const bool whole = rows == nrow;   // the strip's columns are staged as they lie, else rows [rp, rp + rows)
        auto stage = [&](int k) {
            const int cb = k * KC, cn = min(KC, ncol - cb);
            char *xd = reinterpret_cast<char *>(xs + (size_t)(k & 1) * xcap);
            const int units = nb * (int)sizeof(R) / xu, rowb = XP * (int)sizeof(R);
            for (int cc = t >> lsh; cc < cn; cc += kNT >> lsh) {
                const char *src = reinterpret_cast<const char *>(xp + (int64_t)s_col[cb + cc] * B + b0);
                for (int p = t & ((1 << lsh) - 1); p < units; p += 1 << lsh) {
                    if (xu == 16) cp_n<16>(xd + cc * rowb + 16 * p, src + 16 * p);
                    else if (xu == 8) cp_n<8>(xd + cc * rowb + 8 * p, src + 8 * p);
                    else cp_n<4>(xd + cc * rowb + 4 * p, src + 4 * p);
                }
            }
            C *zd = zs + (size_t)(k & 1) * zcap;
            if (whole) {
                const int64_t first = off + (int64_t)cb * nrow;
                const int lead = sizeof(C) == 8 ? (int)(first & 1) : 0;   // 16-byte pieces start at an even element
                const C *src = val + first - lead;
                const int n = cn * nrow + lead;
                constexpr int E = 16 / (int)sizeof(C);
                for (int e = t * E; e < n; e += kNT * E) {
                    if (e + E <= n) cp_n<16>(zd + e, src + e);
                    else cp_n<(int)sizeof(C)>(zd + e, src + e);
                }
            } else {
                const C *src = val + off + (int64_t)cb * nrow + rp;
                for (int e = t; e < cn * rows; e += kNT) {
                    const int cc = e / rows, r = e - cc * rows;
                    cp_n<(int)sizeof(C)>(zd + e, src + (int64_t)cc * nrow + r);
                }
            }
            cp_commit_n();
        };
        // a thread's rows are rg, rg + nrg, ...: neighbouring row groups read neighbouring strip values
        C acc[kRT][CT];
#pragma unroll
        for (int i = 0; i < kRT; ++i)
#pragma unroll
            for (int j = 0; j < CT; ++j) acc[i][j] = C{0, 0};
        stage(0);
        for (int k = 0; k < nchunk; ++k) {
            if (k + 1 < nchunk) {
                stage(k + 1);
                cp_wait_n<1>();
            } else {
                cp_wait_n<0>();
            }
            __syncthreads();
            if (ks < KS) {
                const int cb = k * KC, cn = min(KC, ncol - cb);
                const int lead = whole && sizeof(C) == 8 ? (int)((off + (int64_t)cb * nrow) & 1) : 0;
                const C *z = zs + (size_t)(k & 1) * zcap + lead + rg;   // rows past the last are read and dropped
                const R *x = xs + (size_t)(k & 1) * xcap + cg * CT;
#pragma unroll 2
                for (int cc = ks; cc < cn; cc += KS) {
                    R xv[CT];
                    if constexpr (CT == 4 && sizeof(R) == 4) {
                        const float4 v = *reinterpret_cast<const float4 *>(x + cc * XP);
                        xv[0] = v.x; xv[1] = v.y; xv[2] = v.z; xv[3] = v.w;
                    } else {
#pragma unroll
                        for (int j = 0; j < CT; ++j) xv[j] = x[cc * XP + j];
                    }
                    const C *zc = z + cc * rows;
#pragma unroll
                    for (int i = 0; i < kRT; ++i) {
                        const C zi = zc[i * nrg];
#pragma unroll
                        for (int j = 0; j < CT; ++j) {
                            acc[i][j].x = fma(zi.x, xv[j], acc[i][j].x);
                            acc[i][j].y = fma(zi.y, xv[j], acc[i][j].y);
                        }
                    }
                }
            }
            __syncthreads();
        }
        auto put = [&](int r, int b, C s) {
            if (r < rows && b < nb) yp[(int64_t)(R0 + rp + r) * B + b0 + b] = s;
        };
        if (KS == 1) {
            if (ks == 0)
#pragma unroll
                for (int i = 0; i < kRT; ++i)
#pragma unroll
                    for (int j = 0; j < CT; ++j) put(rg + i * nrg, cg * CT + j, acc[i][j]);
        } else {   // the column splits' partial sums, one output per thread
            C *part = reinterpret_cast<C *>(smem_raw);   // [KS][kRT][CT][tiles]
            const int outs = kRT * CT * tiles;
            if (ks < KS)
#pragma unroll
                for (int i = 0; i < kRT; ++i)
#pragma unroll
                    for (int j = 0; j < CT; ++j) part[ks * outs + (i * CT + j) * tiles + tile] = acc[i][j];   // KS > 1 only in the last pass
            __syncthreads();
            for (int e = t; e < outs; e += kNT) {
                const int n = min(KS, KC);   // the others had no column
                C p[4] = {};                 // in four chains: one of n terms rounds more often
#pragma unroll 2
                for (int g = 0; g + 3 < n; g += 4)
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const C w = part[(g + j) * outs + e];
                        p[j].x += w.x;
                        p[j].y += w.y;
                    }
#pragma unroll
                for (int j = 0; j < 3; ++j)
                    if (j < (n & 3)) {
                        const C w = part[((n & ~3) + j) * outs + e];
                        p[j].x += w.x;
                        p[j].y += w.y;
                    }
                const C s{(p[0].x + p[1].x) + (p[2].x + p[3].x), (p[0].y + p[1].y) + (p[2].y + p[3].y)};
                const int ij = e / tiles, te = e - ij * tiles, i = ij / CT, j = ij - i * CT, r = te / ncg;
                put(r + i * nrg, (te - r * ncg) * CT + j, s);
            }
        }
        __syncthreads();
    }
}

template <class R, int CT>
cudaError_t go(const ProductArgs<R> &a, int most, cudaStream_t s)
{
    using C = typename Cplx<R>::T;
    // a small remainder is shared out, 65 columns as 36 + 29 (30,720 unknowns: 245 us as 64 + 1, 228 so; 96 columns 245 as
    // 64 + 32, 257 as 48 + 48)
    const int chunks = (a.B + most - 1) / most, rest = a.B % most;
    const int nbc = rest > 0 && 2 * rest < most ? ((a.B + chunks - 1) / chunks + CT - 1) / CT * CT : most;
    const int nch = (a.B + nbc - 1) / nbc, ncg = (std::min(a.B, nbc) + CT - 1) / CT, XP = ncg * CT;
    // few columns: the strips stream past, so larger chunks keep more bytes in flight; large boxes take what fits (boxes of
    // 175 rows, FP64, 4 columns: 482 us with chunks of 32, 986 by the kernel of one row per thread; where 64 fit, 32 for
    // the sake of more CTAs per SM lose, 120 against 105 us at 4 FP32 columns)
    int KC = ncg <= 2 ? 64 : 32;
    auto need = [&](int kc) {
        const size_t z = (size_t)(kc * a.nr.max_rows + 8) / 2 * 2, x = (size_t)(kc * XP + 3) / 4 * 4;
        // the column indices follow the staging buffers; the partial sums may run over them (they are used up by then)
        return std::max(2 * z * sizeof(C) + 2 * x * sizeof(R) + (size_t)a.nr.max_cols * sizeof(int), (size_t)kNT * kRT * CT * sizeof(C));
    };
    while (KC > 16 && need(KC) > (size_t)kNearTileSmem) KC /= 2;
    const int zcap = (KC * a.nr.max_rows + 8) / 2 * 2;   // even, so the second buffer stays 16-byte aligned
    const int xcap = (KC * XP + 3) / 4 * 4;
    const size_t smem = need(KC);
    if (smem > (size_t)kNearTileSmem) return cudaErrorInvalidConfiguration;
    // pieces of an x row: as wide as B, the chunk and the buffer's address allow
    const int chunk = std::min(a.B, nbc);
    const uintptr_t align = reinterpret_cast<uintptr_t>(a.xp) | ((uintptr_t)a.B * sizeof(R)) | ((uintptr_t)chunk * sizeof(R)) |
                            ((uintptr_t)(a.B % chunk) * sizeof(R)) | ((uintptr_t)XP * sizeof(R));
    const int xu = (align & 15) == 0 ? 16 : (align & 7) == 0 ? 8 : 4;
    if (xu < (int)sizeof(R) || (reinterpret_cast<uintptr_t>(a.near_val) & 15) != 0) return cudaErrorInvalidConfiguration;
    int lsh = 0;
    while (lsh < 5 && (1 << lsh) < chunk * (int)sizeof(R) / xu) ++lsh;
    const int64_t ctas = (int64_t)a.nr.nleaf * nch;
    int rs = 1;   // row splits: fill the GPU when the tree has few leaf boxes
    while (ctas * rs < 2 * 152 && 4 * rs * kRT <= a.nr.max_rows) rs *= 2;
    k_near_tile<R, CT><<<dim3((unsigned)ctas, rs), kNT, smem, s>>>(a.nr, reinterpret_cast<const C *>(a.near_val), a.xp,
                                                                   reinterpret_cast<C *>(a.yp), a.B, nbc, KC, zcap, xcap, xu, lsh);
    return cudaGetLastError();
}

}  // namespace

template <class R>
cudaError_t launch_near_tile(const ProductArgs<R> &a, cudaStream_t s)
{
    if (a.B < 2 || a.nr.nleaf < 1) return cudaErrorInvalidConfiguration;
    if constexpr (sizeof(R) == 4) return a.B == 2 ? go<R, 2>(a, 2, s) : go<R, 4>(a, 64, s);
    else return go<R, 2>(a, 16, s);
}

template <class R>
cudaError_t prime_near_tile()
{
    cudaError_t e;
#define ALLOW(k) do { if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kNearTileSmem)) != cudaSuccess) return e; } while (0)
    ALLOW((k_near_tile<R, 2>));
    if constexpr (sizeof(R) == 4) ALLOW((k_near_tile<R, 4>));
#undef ALLOW
    return cudaSuccess;
}

template cudaError_t launch_near_tile<float>(const ProductArgs<float> &, cudaStream_t);
template cudaError_t launch_near_tile<double>(const ProductArgs<double> &, cudaStream_t);
template cudaError_t prime_near_tile<float>();
template cudaError_t prime_near_tile<double>();

}  // namespace mlfma
