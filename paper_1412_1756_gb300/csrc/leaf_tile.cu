// Radiation and reception at the leaf level (Section III: the aggregation
// S_m(q) = sum_j V_j(q) x_j over the unknowns j of leaf box m, and the
// disaggregation y_j += sum_q w_q conj(V_j(q)) . G_m(q) over the samples q,
// both tangential components; w_q carries the quadrature weight and the far
// constant), as small matrix products with register tiles whose thread grid
// follows the box and the number of columns.
//
// Radiation: one CTA per (leaf box, column chunk, sample split); a thread
// keeps 2 samples x CC columns x both components; per unknown one x load (CC
// columns) and two pattern loads feed 8 CC multiply-adds.  The box's x rows
// are staged once, the patterns stream through shared memory by cp.async one
// step (RR unknowns x the CTA's samples) ahead, one barrier per step.
//
// Measured, the kernels of fixed column chunks before -> this (FP32, us):
// 30,720-unknown sphere 2 columns 38 -> 29, 10 columns 117 -> 52, 40 columns
// 115 -> 92; 115,200-unknown cube, five digits, 6 columns 309 -> 199, 80
// columns 1,107 -> 955.  Whole chunks of 64 columns stay with
// k_radiate_quads (618 against 675 on the 115,200-unknown cube), one column
// with k_radiate (7 against 8 on 480 unknowns).  FP64 is bound by its
// arithmetic: the tiles win where sample splits spread few boxes over the GPU
// (1,920 unknowns, 8 columns 77 -> 42) and lose elsewhere (28,800 unknowns, 4
// columns 300 -> 500).
//
// Reception: one CTA per (leaf box, column chunk, row split); a thread keeps
// 4 rows x 2 or 4 columns (the second pair half the chunk away, so that
// neighbouring threads read neighbouring 16 bytes); per sample two or four
// field loads and four pattern loads feed 64 or 128 multiply-adds.  With few
// columns (below 16) the threads left over after the tiles split the samples
// (KS ways) and the partial sums are added in a fixed order; otherwise every
// sum runs over the samples in order.  In FP32 the samples of a tile (two
// samples from 17 to 31 columns) are added up first and then join the running
// sum: chained into it, four roundings per sample are of the running sum's
// size, and five digits magnify them 700-fold (30,720-unknown sphere, error
// against FP64 4.7e-5 at 8 columns, 6.8e-5 at 15, 4.5e-5 at 17; so 3.6e-5,
// 3.9e-5, 3.5e-5, where k_receive_tiled with one rounding per sample has
// 3.6e-5; reception takes 0-8 % longer).  From 32 columns up the sum is
// chained as in k_receive_pairs, which these widths may take as well: any
// other order would move five-digit products by 1e-4.
// The field tile is requested one tile
// ahead and scaled by w_q on its way to shared memory, the patterns arrive
// by cp.async one tile ahead.  Bound: instruction issue.  Measured, before ->
// this (FP32, us): 30,720-unknown sphere 2 columns 47 -> 35, 10 columns 117
// -> 63, 40 columns 250 -> 193; 122,880 unknowns, 34 columns 818 -> 537;
// 115,200-unknown cube, 64 columns 1,307 -> 1,230.  FP64: 1,920 unknowns, 8
// columns 186 -> 80, 32 columns 328 -> 213; 28,800 unknowns, five digits, 32
// columns 5,244 -> 4,640.  Which widths and trees keep other kernels stands at
// the rules (launch_receive, launch_receive_tile).
#include "device.h"

#include <algorithm>
#include <type_traits>

namespace mlfma {

namespace {

template <class R> struct Cplx;
template <> struct Cplx<float> { using T = float2; };
template <> struct Cplx<double> { using T = double2; };

// both tangential components of a pattern sample, or two complex columns
template <class R> struct alignas(16) Four { R x, y, z, w; };

__device__ __forceinline__ void cp16l(void *smem, const void *gmem)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem) : "memory");
}
template <class T>
__device__ __forceinline__ void cp_elem(T *smem, const T *gmem)
{
#pragma unroll
    for (int k = 0; k < (int)(sizeof(T) / 16); ++k)
        cp16l(reinterpret_cast<char *>(smem) + 16 * k, reinterpret_cast<const char *>(gmem) + 16 * k);
}
__device__ __forceinline__ void commit_l() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void wait_all_l() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// ----------------------------------------------------------- radiation ---
// ncq column groups of CC, SL sample slots (a thread's samples are sl and
// sl + SL of the CTA's tile of 2 SL), RR unknowns per step.
template <class R, int CC>
__global__ void __launch_bounds__(256) k_radiate_tile(const int32_t *__restrict__ box_ptr, const Four<R> *__restrict__ V4,
                                                      const R *__restrict__ xp, typename Cplx<R>::T *__restrict__ S, int K,
                                                      int B, int Bs, int ncq, int SL, int RR)
{
    using C = typename Cplx<R>::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int NB = CC * ncq, QT = 2 * SL;
    Four<R> *Vs = reinterpret_cast<Four<R> *>(smem_raw);      // [2][RR][QT]
    R *xs = reinterpret_cast<R *>(Vs + 2 * RR * QT);          // [unknowns][NB]
    const int nch = (B + NB - 1) / NB, box = blockIdx.x / nch, b0 = (blockIdx.x - box * nch) * NB;
    const int nb = min(NB, B - b0);
    const int sl = threadIdx.x / ncq, cq = threadIdx.x - sl * ncq;   // sl >= SL: no tile (staging only)
    const int cols = max(0, min(CC, nb - CC * cq));
    const int j0 = box_ptr[box], nj = box_ptr[box + 1] - j0;
    const bool vec = (B % CC) == 0 && (Bs % 2) == 0 &&
                     ((reinterpret_cast<uintptr_t>(xp) | reinterpret_cast<uintptr_t>(S)) & 15) == 0;
    for (int e = threadIdx.x; e < nj * ncq; e += blockDim.x) {   // x rows of the box, zero past the chunk's columns
        const int j = e / ncq, d = e - j * ncq, c = max(0, min(CC, nb - CC * d));
        const R *src = xp + (int64_t)(j0 + j) * B + b0 + CC * d;
        R *dst = xs + (size_t)j * NB + CC * d;
        if (CC == 4 && sizeof(R) == 4 && c == 4 && vec) {
            *reinterpret_cast<float4 *>(dst) = *reinterpret_cast<const float4 *>(src);
        } else {
#pragma unroll
            for (int k = 0; k < CC; ++k) dst[k] = k < c ? src[k] : R(0);
        }
    }
    // this CTA's sample tiles
    const int ntile = (K + QT - 1) / QT, tper = (ntile + gridDim.y - 1) / gridDim.y;
    const int ta = blockIdx.y * tper, tb = min(ntile, ta + tper);
    if (ta >= tb) return;
    const int nchk = max(1, (nj + RR - 1) / RR), s0 = ta * nchk, s1 = tb * nchk;
    // (row, sample) of this thread's first pattern element of a step, and the step to its next
    const int wr0 = threadIdx.x / QT, wq0 = threadIdx.x - wr0 * QT, dr = blockDim.x / QT, dq = blockDim.x - dr * QT;
    auto stage = [&](int step) {
        const int tile = step / nchk, chk = step - tile * nchk;
        const int q0 = tile * QT, r0 = chk * RR, nr = min(RR, nj - r0), nq = K - q0;
        Four<R> *d = Vs + (step & 1) * RR * QT;
        const Four<R> *src = V4 + (int64_t)(j0 + r0) * K + q0;
        int r = wr0, qx = wq0;
        for (int e = threadIdx.x; e < nr * QT; e += blockDim.x) {
            if (qx < nq) cp_elem(d + e, src + (int64_t)r * K + qx);   // samples past the last: stale values, dropped
            r += dr;
            qx += dq;
            if (qx >= QT) {
                qx -= QT;
                ++r;
            }
        }
        commit_l();
    };
    R acc[2][2][CC][2];   // [sample][component][column][re, im]
    auto zero = [&]() {
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int m = 0; m < 2; ++m)
#pragma unroll
                for (int c = 0; c < CC; ++c) acc[a][m][c][0] = acc[a][m][c][1] = R(0);
    };
    zero();
    stage(s0);
    for (int step = s0; step < s1; ++step) {
        wait_all_l();
        __syncthreads();   // the step's patterns are in; everyone is done with the other buffer
        if (step + 1 < s1) stage(step + 1);
        if (sl >= SL) continue;
        const int tile = step / nchk, chk = step - tile * nchk;
        const int r0 = chk * RR, nr = min(RR, nj - r0);
        const Four<R> *vs = Vs + (step & 1) * RR * QT + sl;
        const R *xr = xs + (size_t)r0 * NB + CC * cq;
#pragma unroll 4
        for (int r = 0; r < nr; ++r) {
            R xv[CC];
            if constexpr (CC == 4 && sizeof(R) == 4) {
                const float4 x = *reinterpret_cast<const float4 *>(xr + r * NB);
                xv[0] = x.x; xv[1] = x.y; xv[2] = x.z; xv[3] = x.w;
            } else {
#pragma unroll
                for (int c = 0; c < CC; ++c) xv[c] = xr[r * NB + c];
            }
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                const Four<R> v = vs[r * QT + a * SL];   // (theta re, im, phi re, im) of the unknown at this sample
#pragma unroll
                for (int c = 0; c < CC; ++c) {
                    acc[a][0][c][0] = fma(v.x, xv[c], acc[a][0][c][0]);
                    acc[a][0][c][1] = fma(v.y, xv[c], acc[a][0][c][1]);
                    acc[a][1][c][0] = fma(v.z, xv[c], acc[a][1][c][0]);
                    acc[a][1][c][1] = fma(v.w, xv[c], acc[a][1][c][1]);
                }
            }
        }
        if (chk == nchk - 1) {   // the tile's sums are complete: store and restart
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                const int q = tile * QT + sl + a * SL;
                if (q < K && cols) {
#pragma unroll
                    for (int m = 0; m < 2; ++m) {
                        C *o = S + (((int64_t)box * 2 + m) * K + q) * Bs + b0 + CC * cq;
                        if (CC == 4 && sizeof(R) == 4 && cols == 4 && vec) {
                            float4 *o4 = reinterpret_cast<float4 *>(o);
                            o4[0] = make_float4(acc[a][m][0][0], acc[a][m][0][1], acc[a][m][CC / 4][0], acc[a][m][CC / 4][1]);
                            o4[1] = make_float4(acc[a][m][CC / 2][0], acc[a][m][CC / 2][1], acc[a][m][CC - 1][0], acc[a][m][CC - 1][1]);
                        } else {
#pragma unroll
                            for (int c = 0; c < CC; ++c)
                                if (c < cols) o[c] = C{acc[a][m][c][0], acc[a][m][c][1]};
                        }
                    }
                }
            }
            zero();
        }
    }
}

// ----------------------------------------------------------- reception ---
constexpr int kRows = 4;   // rows per thread

// acc += conj(v) * g
template <class R>
__device__ __forceinline__ void cmacc(R (&acc)[2], R vx, R vy, R gx, R gy)
{
    acc[0] = fma(vx, gx, fma(vy, gy, acc[0]));
    acc[1] = fma(vx, gy, fma(-vy, gx, acc[1]));
}

// acc += the sum over NS samples of both components' conj(v) * g
template <class R, int NS>
__device__ __forceinline__ void samples_acc(R (&acc)[2], const Four<R> (&v)[NS], const R (&g0)[NS][2], const R (&g1)[NS][2])
{
    R t[2] = {R(0), R(0)};
#pragma unroll
    for (int n = 0; n < NS; ++n) {
        cmacc(t, v[n].x, v[n].y, g0[n][0], g0[n][1]);
        cmacc(t, v[n].z, v[n].w, g1[n][0], g1[n][1]);
    }
    acc[0] += t[0];
    acc[1] += t[1];
}

// CW columns of the field per thread
template <class R, int CW> struct alignas(CW * 2 * sizeof(R) >= 16 ? 16 : CW * 2 * sizeof(R)) Cols { R v[2 * CW]; };

// ncp column groups (CW columns each) per CTA, CPT of them per thread (group
// cp, cp + ncp / CPT, ...), tiles of QT samples, RP rows per pass at most;
// NE: field elements a thread stages per tile.
template <class R, int CW, int QT, int NE, int CPT, bool SUM>
__global__ void __launch_bounds__(256, sizeof(R) == 4 && CPT == 1 ? 3 : (sizeof(R) == 4 ? 2 : 1)) k_receive_tile(const int32_t *__restrict__ box_ptr, const Four<R> *__restrict__ V4,
                                                      DevLevel<R> lf, typename Cplx<R>::T *__restrict__ yp, int B, int Bs,
                                                      int ncp, int RP)
{
    using C = typename Cplx<R>::T;
    using G1 = Cols<R, CW>;
    // acc is one tile's sum, tot the running sum
    constexpr bool TS = SUM && CPT == 1;
    constexpr int VP = QT + 1;   // pitch of a staged pattern row: the rows a warp reads fall in different banks
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int GT = 2 * QT * ncp;                            // field tile: [component][sample][column group]
    Four<R> *Vs = reinterpret_cast<Four<R> *>(smem_raw);    // [2][RP][VP]
    G1 *Gs = reinterpret_cast<G1 *>(Vs + 2 * RP * VP);      // [2][GT]
    const int K = lf.K, NB = CW * ncp, t = threadIdx.x, nt = blockDim.x;
    const int nch = (B + NB - 1) / NB, box = blockIdx.x / nch, b0 = (blockIdx.x - box * nch) * NB;
    const int nb = min(NB, B - b0);
    const int i0 = box_ptr[box], nrow = box_ptr[box + 1] - i0;
    const int per = ((nrow + kRows - 1) / kRows + gridDim.y - 1) / gridDim.y * kRows;
    const int ra = blockIdx.y * per, rz = min(nrow, ra + per);
    const C *G = reinterpret_cast<const C *>(lf.G) + (int64_t)box * 2 * K * Bs + b0;
    const bool vec = (Bs % CW) == 0 && (b0 % CW) == 0 && (reinterpret_cast<uintptr_t>(lf.G) & 15) == 0;
    const int ntile = (K + QT - 1) / QT;
    // this thread's field elements of a tile: (sample, offset from the tile's first sample, columns)
    int gq[NE], gc[NE];
    int go[NE];
#pragma unroll
    for (int i = 0; i < NE; ++i) {
        const int e = t + i * nt, mq = e / ncp, p = e - mq * ncp, m = mq / QT;
        gq[i] = mq - m * QT;
        gc[i] = e < GT ? max(0, min(CW, nb - CW * p)) : -1;   // -1: no element
        go[i] = (m * K + gq[i]) * Bs + CW * p;
    }
    // the loads are consumed (scaled and stored) after the tile in hand is done
    auto load_g = [&](int tile, G1 (&g)[NE], R (&w)[NE]) {
#pragma unroll
        for (int i = 0; i < NE; ++i) {
            const int q = tile * QT + gq[i];
            w[i] = R(0);
#pragma unroll
            for (int k = 0; k < 2 * CW; ++k) g[i].v[k] = R(0);
            if (gc[i] > 0 && q < K) {
                const C *src = G + go[i] + (int64_t)tile * QT * Bs;
                if (vec && gc[i] == CW) {
                    g[i] = *reinterpret_cast<const G1 *>(src);
                } else {
#pragma unroll
                    for (int k = 0; k < CW; ++k)
                        if (k < gc[i]) { g[i].v[2 * k] = src[k].x; g[i].v[2 * k + 1] = src[k].y; }
                }
                w[i] = lf.wq[q];
            }
        }
    };
    auto store_g = [&](int buf, G1 (&g)[NE], const R (&w)[NE]) {
#pragma unroll
        for (int i = 0; i < NE; ++i) {
#pragma unroll
            for (int k = 0; k < 2 * CW; ++k) g[i].v[k] *= w[i];
            if (gc[i] >= 0) Gs[buf * GT + t + i * nt] = g[i];
        }
    };
    for (int rp = ra; rp < rz; rp += RP) {
        const int rows = min(RP, rz - rp), nrg = (rows + kRows - 1) / kRows, nct = ncp / CPT, tiles = nrg * nct;
        const int KS = CPT == 1 ? max(1, nt / tiles) : 1;
        const int ks = t / tiles, tile_id = t - ks * tiles, rg = tile_id / nct, cp = tile_id - rg * nct;
        auto stage_v = [&](int tile, int buf) {
            const int q0 = tile * QT, nq = K - q0;
            Four<R> *vd = Vs + (size_t)buf * RP * VP;
            const Four<R> *src = V4 + (int64_t)(i0 + rp) * K + q0;
            const int qx = t % QT;
            if (qx < nq)
                for (int r = t / QT; r < rows; r += nt / QT) cp_elem(vd + r * VP + qx, src + (int64_t)r * K + qx);
            commit_l();
        };
        R acc[CPT][kRows][CW][2];   // rows rg, rg + nrg, ...: [column group][row][column][re, im]
#pragma unroll
        for (int u = 0; u < CPT; ++u)
#pragma unroll
            for (int k = 0; k < kRows; ++k)
#pragma unroll
                for (int c = 0; c < CW; ++c) acc[u][k][c][0] = acc[u][k][c][1] = R(0);
        R tot[TS ? kRows : 1][CW][2] = {};
        {
            G1 g[NE];
            R w[NE];
            stage_v(0, 0);
            load_g(0, g, w);
            store_g(0, g, w);
            wait_all_l();
            __syncthreads();
        }
        for (int tile = 0; tile < ntile; ++tile) {
            const int buf = tile & 1, nq = min(QT, K - tile * QT);
            G1 g[NE];
            R w[NE];
            if (tile + 1 < ntile) {
                stage_v(tile + 1, buf ^ 1);
                load_g(tile + 1, g, w);
            }
            if (ks < KS) {
                const G1 *gs = Gs + (size_t)buf * GT + cp, *gs2 = gs + QT * ncp;
                const Four<R> *vs = Vs + (size_t)buf * RP * VP + rg * VP;   // rows past the last: stale values, dropped
                if constexpr (CPT == 1 || !SUM) {
#pragma unroll 2
                    for (int qx = ks; qx < nq; qx += KS) {
                        G1 g0[CPT], g1[CPT];
#pragma unroll
                        for (int u = 0; u < CPT; ++u) {
                            g0[u] = gs[qx * ncp + u * nct];
                            g1[u] = gs2[qx * ncp + u * nct];
                        }
#pragma unroll
                        for (int k = 0; k < kRows; ++k) {
                            const Four<R> v = vs[k * nrg * VP + qx];
#pragma unroll
                            for (int u = 0; u < CPT; ++u) {
#pragma unroll
                                for (int c = 0; c < CW; ++c) cmacc(acc[u][k][c], v.x, v.y, g0[u].v[2 * c], g0[u].v[2 * c + 1]);
#pragma unroll
                                for (int c = 0; c < CW; ++c) cmacc(acc[u][k][c], v.z, v.w, g1[u].v[2 * c], g1[u].v[2 * c + 1]);
                            }
                        }
                    }
                    if (TS) {
#pragma unroll
                        for (int k = 0; k < kRows; ++k)
#pragma unroll
                            for (int c = 0; c < CW; ++c)
#pragma unroll
                                for (int h = 0; h < 2; ++h) {
                                    tot[k][c][h] += acc[0][k][c][h];
                                    acc[0][k][c][h] = R(0);
                                }
                    }
                } else {
                    auto step = [&](int qx, auto ns) {
                        constexpr int NS = decltype(ns)::value;
                        G1 g0[NS][CPT], g1[NS][CPT];
#pragma unroll
                        for (int n = 0; n < NS; ++n)
#pragma unroll
                            for (int u = 0; u < CPT; ++u) {
                                g0[n][u] = gs[(qx + n) * ncp + u * nct];
                                g1[n][u] = gs2[(qx + n) * ncp + u * nct];
                            }
#pragma unroll
                        for (int k = 0; k < kRows; ++k) {
                            Four<R> v[NS];
#pragma unroll
                            for (int n = 0; n < NS; ++n) v[n] = vs[k * nrg * VP + qx + n];
#pragma unroll
                            for (int u = 0; u < CPT; ++u)
#pragma unroll
                                for (int c = 0; c < CW; ++c) {
                                    R a0[NS][2], a1[NS][2];
#pragma unroll
                                    for (int n = 0; n < NS; ++n)
#pragma unroll
                                        for (int h = 0; h < 2; ++h) {
                                            a0[n][h] = g0[n][u].v[2 * c + h];
                                            a1[n][h] = g1[n][u].v[2 * c + h];
                                        }
                                    samples_acc<R, NS>(acc[u][k][c], v, a0, a1);
                                }
                        }
                    };
                    int qx = 0;   // KS = 1
                    for (; qx + 1 < nq; qx += 2) step(qx, std::integral_constant<int, 2>{});
                    if (qx < nq) step(qx, std::integral_constant<int, 1>{});
                }
            }
            if (tile + 1 < ntile) store_g(buf ^ 1, g, w);
            wait_all_l();
            __syncthreads();   // the next tile is in; everyone is done with this one
        }
        if (TS)
#pragma unroll
            for (int k = 0; k < kRows; ++k)
#pragma unroll
                for (int c = 0; c < CW; ++c)
#pragma unroll
                    for (int h = 0; h < 2; ++h) acc[0][k][c][h] = tot[k][c][h];
        auto add = [&](int r, int b, C s) {
            if (r < rows && b < nb) {
                C *y = yp + (int64_t)(i0 + rp + r) * B + b0 + b;
                *y = C{y->x + s.x, y->y + s.y};
            }
        };
        if (KS == 1) {
            if (ks == 0)
#pragma unroll
                for (int u = 0; u < CPT; ++u)
#pragma unroll
                    for (int k = 0; k < kRows; ++k)
#pragma unroll
                        for (int c = 0; c < CW; ++c)
                            add(rg + k * nrg, CW * (cp + u * nct) + c, C{acc[u][k][c][0], acc[u][k][c][1]});
        } else if constexpr (CPT == 1) {   // the sample splits' partial sums, one output per thread
            C *part = reinterpret_cast<C *>(smem_raw);   // [KS][kRows][CW][tiles]
            const int outs = kRows * CW * tiles;
            if (ks < KS)
#pragma unroll
                for (int k = 0; k < kRows; ++k)
#pragma unroll
                    for (int c = 0; c < CW; ++c) part[ks * outs + (k * CW + c) * tiles + tile_id] = C{acc[0][k][c][0], acc[0][k][c][1]};
            __syncthreads();
            for (int e = t; e < outs; e += nt) {
                const int n = min(KS, QT);   // the others had no sample
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
                const int kc = e / tiles, te = e - kc * tiles, k = kc / CW, c = kc - k * CW, r = te / ncp;
                add(r + k * nrg, (te - r * ncp) * CW + c, s);
            }
            __syncthreads();
        }
    }
}

constexpr int kLeafSmem = 200 * 1024;

}  // namespace

namespace {

template <class R, int CC>
cudaError_t radiate_go(const ProductArgs<R> &a, int Bs, cudaStream_t s)
{
    const DevLevel<R> &Lf = a.lv[a.leaf];
    // column chunks and sample tiles of even size: 65 columns as 36 + 29 and not 64 + 1, 288 samples as 144 + 144 and not
    // 256 + 32, whose last CTA or step leaves most threads idle
    const int groups = (a.B + CC - 1) / CC, most = sizeof(R) == 4 ? 16 : 8, nch = (groups + most - 1) / most;
    const int ncq = (groups + nch - 1) / nch;
    const int64_t ctas = (int64_t)Lf.nbox * ((a.B + CC * ncq - 1) / (CC * ncq));
    int SL = std::max(1, std::min(256 / ncq, (Lf.K + 1) / 2));   // a thread's two samples are one slot
    // few leaf boxes: shorter sample tiles, so that their splits fill the GPU
    while (SL * ncq > 32 && ctas * ((Lf.K + 2 * SL - 1) / (2 * SL)) < 2 * 152) SL = (SL + 1) / 2;
    SL = std::min((SL * ncq + 31) / 32 * 32 / ncq, (Lf.K + 1) / 2);   // the last warp's threads
    const int ntile = (Lf.K + 2 * SL - 1) / (2 * SL);
    SL = (Lf.K + 2 * ntile - 1) / (2 * ntile);
    const int threads = (SL * ncq + 31) / 32 * 32, QT = 2 * SL, RR = std::max(1, 1024 / QT);
    const size_t smem = (size_t)2 * RR * QT * sizeof(Four<R>) + (size_t)a.nr.max_rows * ncq * CC * sizeof(R);
    if (smem > (size_t)kLeafSmem) return cudaErrorInvalidConfiguration;
    int qs = 1;
    while (ctas * qs < 2 * 152 && qs < ntile) ++qs;
    k_radiate_tile<R, CC><<<dim3((unsigned)ctas, qs), threads, smem, s>>>(
        a.nr.box_ptr, reinterpret_cast<const Four<R> *>(a.V), a.xp, reinterpret_cast<typename Cplx<R>::T *>(Lf.S), Lf.K, a.B,
        Bs, ncq, SL, RR);
    return cudaGetLastError();
}

// Row groups of the usual leaf box, a quarter above the mean; larger boxes take more passes.
template <class R>
int usual_groups(const ProductArgs<R> &a, int nbox)
{
    const int mean = (int)(a.n / std::max(1, nbox)) + 1;
    return (mean + mean / 4 + kRows - 1) / kRows;
}

template <class R, int CW, int QT, int NE, int CPT = 1, bool SUM = sizeof(R) == 4>
cudaError_t receive_go(const ProductArgs<R> &a, int Bs, int ncp, cudaStream_t s)
{
    const DevLevel<R> &Lf = a.lv[a.leaf];
    constexpr bool split = CPT == 1;   // the samples are split over the threads left over
    const int nct = ncp / CPT;
    const int64_t ctas = (int64_t)Lf.nbox * ((a.B + CW * ncp - 1) / (CW * ncp));
    const int all = (a.nr.max_rows + kRows - 1) / kRows;   // row groups of the largest box
    int rs = 1;   // row splits: fill the GPU when the tree has few leaf boxes
    while (ctas * rs < 2 * 152 && 4 * rs * kRows <= a.nr.max_rows) rs *= 2;
    const int least = std::max((2 * QT * ncp + NE - 1) / NE, 64);   // NE field elements per thread and tile
    int threads = split ? 256 : std::min(256, (std::max(nct * usual_groups(a, Lf.nbox), least) + 31) / 32 * 32);
    // a split needs fewer than the whole box: down to what runs in one wave (128 registers a thread)
    while (!split && rs > 1 && ctas * rs > 152 * (512 / threads) && threads - 32 >= std::max(least, nct * ((all + rs - 1) / rs)))
        threads -= 32;
    const int RP = std::min(all, threads / nct) * kRows;
    if (2 * QT * ncp > NE * threads || (int64_t)2 * Lf.K * Bs > INT32_MAX) return cudaErrorInvalidConfiguration;   // 32-bit field offsets
    const size_t stage = (size_t)4 * QT * ncp * sizeof(Cols<R, CW>) + (size_t)2 * RP * (QT + 1) * sizeof(Four<R>);
    const size_t part = split ? (size_t)256 * kRows * CW * 2 * sizeof(R) : 0;
    const size_t smem = std::max(stage, part);
    if (smem > (size_t)kLeafSmem) return cudaErrorInvalidConfiguration;
    k_receive_tile<R, CW, QT, NE, CPT, SUM><<<dim3((unsigned)ctas, rs), threads, smem, s>>>(
        a.nr.box_ptr, reinterpret_cast<const Four<R> *>(a.V), Lf, reinterpret_cast<typename Cplx<R>::T *>(a.yp), a.B, Bs, ncp, RP);
    return cudaGetLastError();
}

}  // namespace

template <class R>
cudaError_t launch_radiate_tile(const ProductArgs<R> &a, int Bs, cudaStream_t s)
{
    if (a.B < 2) return cudaErrorInvalidConfiguration;
    if constexpr (sizeof(R) == 4) return a.B == 2 ? radiate_go<R, 2>(a, Bs, s) : radiate_go<R, 4>(a, Bs, s);
    else return radiate_go<R, 2>(a, Bs, s);
}

template <class R>
cudaError_t launch_receive_tile(const ProductArgs<R> &a, int Bs, cudaStream_t s)
{
    if (a.B < 2) return cudaErrorInvalidConfiguration;
    const int ncp = (a.B + 1) / 2;
    if constexpr (sizeof(R) == 4) {
        if (ncp <= 4) return receive_go<R, 2, 32, 1>(a, Bs, ncp, s);
        if (ncp <= 8) return receive_go<R, 2, 16, 1>(a, Bs, ncp, s);
        // From 17 columns up, k_receive_pairs (32 columns a CTA) where the tile's chunks of 64 leave a third of their
        // columns empty (a remainder of 1-32, but for boxes of 96 rows and more), and where no column is empty in
        // either (32, or a remainder of 61-64 on fewer than 4,096 boxes) but the tile's threads take the larger boxes
        // in two passes.  Pairs / tile, us: 80 columns of 30,720 unknowns 350 / 459, of 7,680 139 / 217; 32
        // columns of 30,720 145 / 174, of 115,200 708 / 804, of 42,960 (plate, one pass) 255 / 220; 64 columns of
        // 28,800 391 / 422, of 115,200 1,302 / 1,277; 96 columns on boxes of 175 rows 406 / 270.
        const int nct = std::min((ncp + 1) / 2, 16), rest = a.B % 64;
        const bool passes = (a.nr.max_rows + kRows - 1) / kRows > std::max(64, (nct * usual_groups(a, a.lv[a.leaf].nbox) + 31) / 32 * 32) / nct;
        const bool full = a.B == 32 || ((rest == 0 || rest > 60) && a.lv[a.leaf].nbox < 4096);
        if ((a.B > 64 && rest > 0 && rest <= 32 && a.nr.max_rows < 96) || (full && passes)) return launch_receive_pairs(a, Bs, 32, s);
        const int pairs = std::min((ncp + 1) / 2 * 2, 32);
        return a.B < 32 ? receive_go<R, 2, 8, 4, 2, true>(a, Bs, pairs, s) : receive_go<R, 2, 8, 4, 2, false>(a, Bs, pairs, s);
    } else {
        return receive_go<R, 2, 16, 1>(a, Bs, std::min(ncp, 8), s);
    }
}

template <class R>
cudaError_t prime_leaf_tile()
{
    cudaError_t e;
#define ALLOW(k) do { if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kLeafSmem)) != cudaSuccess) return e; } while (0)
    ALLOW((k_radiate_tile<R, 2>));
    ALLOW((k_receive_tile<R, 2, 16, 1, 1, sizeof(R) == 4>));
    if constexpr (sizeof(R) == 4) {
        ALLOW((k_radiate_tile<R, 4>));
        ALLOW((k_receive_tile<R, 2, 32, 1, 1, true>)); ALLOW((k_receive_tile<R, 2, 8, 4, 2, true>)); ALLOW((k_receive_tile<R, 2, 8, 4, 2, false>));
    }
#undef ALLOW
    return cudaSuccess;
}

template cudaError_t launch_radiate_tile<float>(const ProductArgs<float> &, int, cudaStream_t);
template cudaError_t launch_radiate_tile<double>(const ProductArgs<double> &, int, cudaStream_t);
template cudaError_t launch_receive_tile<float>(const ProductArgs<float> &, int, cudaStream_t);
template cudaError_t launch_receive_tile<double>(const ProductArgs<double> &, int, cudaStream_t);
template cudaError_t prime_leaf_tile<float>();
template cudaError_t prime_leaf_tile<double>();

}  // namespace mlfma
