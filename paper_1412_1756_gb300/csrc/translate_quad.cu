// Translation of FP32 fields (Section III-A, Eq. (8): the incoming field of
// a box is the sum over its interaction list of the diagonal translation
// function times the source box's outgoing field, sample by sample), grouped
// by parent as the plan lists it: one entry names a source box and, for each
// child of the parent, the translation type it needs or none.
//
// A CTA takes one parent's children at 128 consecutive (sample, column quad)
// items, one item per thread.  A thread loads a source value once per entry
// (both components of its four columns) and applies it to four children at a
// time from accumulators in registers; a parent with more than four children
// takes a second pass over its entries.  The coefficients of the parent's
// types at the CTA's samples are staged in shared memory.
//
// Bound: the latency of the source rows from L2 at five CTAs per SM (94
// registers, 64 of them accumulators), issue slots 60 % active; FP32 pipe a
// third.  The items are numbered over (sample, quad) without gaps, so that a
// column count that is no multiple of 16 leaves no thread idle; fixed chunks
// of 32 columns had cost (30,720-unknown sphere, leaf level) 384 us at 40
// columns against 240, and (122,880 unknowns) 1,440 us at 34 against 942.
// Where every quad is whole and aligned, five CTAs without prefetch measured
// faster (64 columns, 115,200-unknown cube: 1,889 against 1,942 us with the
// next entry's sources requested ahead in four CTAs); where columns are
// missing, the loads are longer and requesting ahead wins (34 columns: 942
// against 1,020).  Tried and slower: packed fma.rn.f32x2 (1,960 to 2,400 us,
// it takes twice the FP32 pipe's cycles and more registers), the sources
// streamed through a shared-memory ring by cp.async.bulk and mbarriers
// (3,280 us).
#include "device.h"

#include <algorithm>

namespace mlfma {

namespace {

constexpr int kThreads = 128;
constexpr int kMaxEntries = 216;   // entries of one parent (the plan's bound)
constexpr int kCh = 4;             // children per pass
constexpr unsigned kNone = 0xffffu;   // (entry, child) slot without a translation

// A thread's four columns are two pairs: where every quad is whole, pairs qd
// and qd + nqd of the row, so that neighbouring threads read neighbouring 16
// bytes (as four adjacent columns, each 16-byte load of a warp touched twice
// the lines: 1,936 against 1,889 us, 64 columns of the 115,200-unknown cube);
// else adjacent ones.
// One pair of a field row: one 16-byte load when both columns exist and are
// aligned, else the existing ones (zero past the end).
__device__ __forceinline__ float4 ld_pair(const float2 *p, int cols, bool a16)
{
    if (cols == 2 && a16) return *reinterpret_cast<const float4 *>(p);
    const float2 u = cols > 0 ? p[0] : make_float2(0.f, 0.f), v = cols > 1 ? p[1] : make_float2(0.f, 0.f);
    return make_float4(u.x, u.y, v.x, v.y);
}

__device__ __forceinline__ void st_pair(float2 *p, int cols, bool a16, float4 v, int accumulate)
{
    if (cols == 2 && a16) {
        float4 *q = reinterpret_cast<float4 *>(p);
        if (accumulate) {
            const float4 o = *q;
            v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w;
        }
        *q = v;
        return;
    }
    const float2 w[2] = {make_float2(v.x, v.y), make_float2(v.z, v.w)};
#pragma unroll
    for (int k = 0; k < 2; ++k)
        if (k < cols) {
            float2 y = w[k];
            if (accumulate) {
                const float2 o = p[k];
                y.x += o.x;
                y.y += o.y;
            }
            p[k] = y;
        }
}

// acc (two complex columns) += a * s
__device__ __forceinline__ void cmac2(float4 &acc, float2 a, float4 s)
{
    acc.x = fmaf(a.x, s.x, fmaf(-a.y, s.y, acc.x));
    acc.y = fmaf(a.x, s.y, fmaf(a.y, s.x, acc.y));
    acc.z = fmaf(a.x, s.z, fmaf(-a.y, s.w, acc.z));
    acc.w = fmaf(a.x, s.w, fmaf(a.y, s.z, acc.w));
}

// FULL: every item's four columns exist and are 16-byte aligned (B a
// multiple of four, even row stride, aligned fields), so the loads and
// stores take the two-vector path without a run-time test.  PRE: the next
// entry's sources are requested before the current one is used.
template <bool FULL, bool PRE, int MINB>
__global__ void __launch_bounds__(kThreads, MINB) k_translate_q4(DevLevel<float> lv, int B, int Bs, int accumulate, int nqd, int QS)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int64_t s_off[kMaxEntries];                  // offset of each entry's source field
    __shared__ __align__(16) uint16_t s_ty[kMaxEntries * 8];   // per (entry, child): its row of the coefficients, or kNone
    const int K = lv.K;
    const int64_t KB = (int64_t)K * Bs;
    const int P = blockIdx.x, i0 = (blockIdx.z * gridDim.y + blockIdx.y) * kThreads;
    if (i0 >= K * nqd) return;   // of the last z slice
    const int q0 = i0 / nqd, nq = min(K, (i0 + kThreads - 1) / nqd + 1) - q0;   // nq <= QS
    const int e0 = lv.grp_ptr[P], ne = lv.grp_ptr[P + 1] - e0;
    const int m0 = lv.pchild_ptr[P], nc = lv.pchild_ptr[P + 1] - m0;
    const int l0 = lv.lty_ptr[P], nl = lv.lty_ptr[P + 1] - l0;
    const bool a16 = FULL || ((Bs % 2) == 0 && ((reinterpret_cast<uintptr_t>(lv.S) | reinterpret_cast<uintptr_t>(lv.G)) & 15) == 0);
    const float2 *al = reinterpret_cast<const float2 *>(lv.alpha);
    float2 *s_al = reinterpret_cast<float2 *>(smem_raw);   // [local type][QS]
    for (int i = threadIdx.x; i < nl * QS; i += kThreads) {
        const int lt = i / QS, qq = i - lt * QS;
        s_al[i] = qq < nq ? al[(int64_t)lv.lty[l0 + lt] * K + q0 + qq] : make_float2(0.f, 0.f);
    }
    for (int e = threadIdx.x; e < ne; e += kThreads) s_off[e] = (int64_t)lv.grp_src[e0 + e] * 2 * KB;
    for (int e = threadIdx.x; e < ne * 8; e += kThreads) {
        const int t = lv.grp_lty[(int64_t)e0 * 8 + e];
        s_ty[e] = (uint16_t)(t < 0 ? kNone : (unsigned)(t * QS));   // t * QS < 2^16 - 1 (checked by the launcher)
    }
    __syncthreads();
    const int q = (i0 + threadIdx.x) / nqd, qd = i0 + threadIdx.x - q * nqd;
    if (q >= K) return;
    const int b = FULL ? 2 * qd : 4 * qd, hi = FULL ? 2 * nqd : 2;   // the first pair, and from it to the second
    const int cl = FULL ? 2 : min(2, B - b), ch = FULL ? 2 : max(0, min(2, B - b - hi));   // their columns
    const float2 *S = reinterpret_cast<const float2 *>(lv.S) + (int64_t)q * Bs + b;
    const float2 *alq = s_al + (q - q0);
    auto load = [&](int e, float4 (&s)[2][2]) {
        const float2 *src = S + s_off[e];
        if (FULL) {
            s[0][0] = *reinterpret_cast<const float4 *>(src);
            s[0][1] = *reinterpret_cast<const float4 *>(src + hi);
            s[1][0] = *reinterpret_cast<const float4 *>(src + KB);
            s[1][1] = *reinterpret_cast<const float4 *>(src + KB + hi);
        } else {
            s[0][0] = ld_pair(src, cl, a16);
            s[0][1] = ld_pair(src + hi, ch, a16);
            s[1][0] = ld_pair(src + KB, cl, a16);
            s[1][1] = ld_pair(src + KB + hi, ch, a16);
        }
    };
    for (int c0 = 0; c0 < nc; c0 += kCh) {
        float4 acc[kCh][2][2];   // [child][component][column pair]
#pragma unroll
        for (int c = 0; c < kCh; ++c)
#pragma unroll
            for (int m = 0; m < 2; ++m) acc[c][m][0] = acc[c][m][1] = make_float4(0.f, 0.f, 0.f, 0.f);
        const int nch = min(kCh, nc - c0);
        float4 nx[2][2];
        if (PRE && ne > 0) load(0, nx);
#pragma unroll 2
        for (int e = 0; e < ne; ++e) {
            float4 s[2][2];
            if (PRE) {
#pragma unroll
                for (int m = 0; m < 2; ++m) { s[m][0] = nx[m][0]; s[m][1] = nx[m][1]; }
                if (e + 1 < ne) load(e + 1, nx);
            } else {
                load(e, s);
            }
            // the four children's coefficient rows (16-bit each) of this pass
            const uint2 tyv = *reinterpret_cast<const uint2 *>(&s_ty[e * 8 + c0]);
            const unsigned tw[2] = {tyv.x, tyv.y};
#pragma unroll
            for (int c = 0; c < kCh; ++c) {
                if (c >= nch) break;
                const unsigned off = (tw[c >> 1] >> (16 * (c & 1))) & 0xffffu;
                if (off != kNone) {
                    const float2 a = alq[off];
#pragma unroll
                    for (int m = 0; m < 2; ++m) {
                        cmac2(acc[c][m][0], a, s[m][0]);
                        cmac2(acc[c][m][1], a, s[m][1]);
                    }
                }
            }
        }
        float2 *G = reinterpret_cast<float2 *>(lv.G) + (int64_t)q * Bs + b;
#pragma unroll
        for (int c = 0; c < kCh; ++c) {
            if (c >= nch) break;
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                float2 *o = G + ((int64_t)(m0 + c0 + c) * 2 + m) * KB;
                st_pair(o, cl, a16, acc[c][m][0], accumulate);
                st_pair(o + hi, ch, a16, acc[c][m][1], accumulate);
            }
        }
    }
}

template <bool FULL, bool PRE, int MINB>
cudaError_t go(const DevLevel<float> &lv, int B, int Bs, int acc, int nqd, int QS, size_t smem, cudaStream_t s)
{
    // a level of 8,192 samples (a body of 19 wavelengths) at 4,096 columns has 65,536 chunks of items, one more than
    // grid.y takes: slices of equal size in z
    const int64_t chunks = ((int64_t)lv.K * nqd + kThreads - 1) / kThreads, nz = (chunks + 65534) / 65535;
    if (lv.K > (1 << 30) / nqd) return cudaErrorInvalidConfiguration;   // 32-bit item numbers (nz <= 129)
    const dim3 grid(lv.nparent, (unsigned)((chunks + nz - 1) / nz), (unsigned)nz);
    k_translate_q4<FULL, PRE, MINB><<<grid, kThreads, smem, s>>>(lv, B, Bs, acc, nqd, QS);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_translate_quad(const DevLevel<float> &lv, int B, int Bs, int acc, int variant, cudaStream_t s)
{
    if (B < 1 || !lv.lty || !lv.grp_lty || lv.max_grp > kMaxEntries) return cudaErrorInvalidConfiguration;
    const int nqd = (B + 3) / 4;
    const int QS = std::min(lv.K, (kThreads - 2 + nqd) / nqd + 1);   // samples a CTA's items touch, at most
    const size_t smem = (size_t)lv.max_lty * QS * sizeof(float2);
    if (smem > (size_t)(96 * 1024) || (int64_t)lv.max_lty * QS >= (int64_t)kNone) return cudaErrorInvalidConfiguration;
    const bool full = B % 4 == 0 && Bs % 2 == 0 &&
                      ((reinterpret_cast<uintptr_t>(lv.S) | reinterpret_cast<uintptr_t>(lv.G)) & 15) == 0;
    const bool pre = variant == 32 || (variant != 16 && !full);   // the built-in choice as measured (figures above)
    if (full) return pre ? go<true, true, 4>(lv, B, Bs, acc, nqd, QS, smem, s) : go<true, false, 5>(lv, B, Bs, acc, nqd, QS, smem, s);
    return pre ? go<false, true, 4>(lv, B, Bs, acc, nqd, QS, smem, s) : go<false, false, 4>(lv, B, Bs, acc, nqd, QS, smem, s);
}

cudaError_t prime_translate_quad()
{
    cudaError_t e;
#define ALLOW(k) do { if ((e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024)) != cudaSuccess) return e; } while (0)
    ALLOW((k_translate_q4<false, false, 4>)); ALLOW((k_translate_q4<false, true, 4>));
    ALLOW((k_translate_q4<true, true, 4>)); ALLOW((k_translate_q4<true, false, 5>));
#undef ALLOW
    return cudaSuccess;
}

}  // namespace mlfma
