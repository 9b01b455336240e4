// update_fx.cu -- trailing (Schur) update of FP64 fronts on the FP16 tensor cores, by integer digits.
//
// C[i][j] -= sum_t L21[i][t] W21[j][t] on the lower triangle of the trailing block (the dense contraction of the
// multifrontal LDL^T), K = panel width (<= 64), in the digit products of fixed_digits.cuh.  W21 = L21 D, so
// column t of both is first scaled by a power of two near sqrt|d_t| (L21 up, W21 down: a small pivot makes a
// whole column of L21 large); then every row of each is one block of digits with its own scale.  The panel's
// trsm (factor.cu) writes the digits.
//
// Digit blocks: 64 rows x 16 k of one operand, 8 KB, the k blocks of a 64-row block one after another for
// each 16 rows: [16-row group][k block][digit pair][lane][16 bytes].  Lane 4 g + t holds, of digits 2 u and
// 2 u + 1, rows g and g + 8 at k = 2 t, 2 t + 1, 2 t + 8, 2 t + 9: the A fragment of 16 rows, and the B
// fragments of two groups of 8 rows.
//
// CTA: 4 warps, 64 rows x 32 columns of C, 32 x 16 a warp (9 digit sums x 16 accumulators a lane).  Bound by
// the FP16 products (43 of 16 x 8 x 16 for each 2048 FP64 FMAs): 294 us a launch at L = 18 on average, where the
// same update in FP64 FMAs at 95% of their rate took 1550.
#include "factor.h"
#include "fixed_digits.cuh"
#include "solve_tile.cuh"

namespace mbl {

namespace {

constexpr int UF_THREADS = 128;
constexpr int UF_GROUP = 4 * 32 * 4;  // words of 16 rows x 16 k
constexpr size_t UF_SMEM = (size_t)(4 + 2) * (NB / 16) * UF_GROUP * 4;

__device__ __forceinline__ int find_update_desc(const PanelDesc *d, int nd, int64_t b) {
    int lo = 0, hi = nd - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (d[mid].off3 <= b) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__global__ void __launch_bounds__(UF_THREADS, 2)
    k_fx_update(const PanelDesc *descs, int nd, const int64_t *fo, const int32_t *fsz, double *arena,
                const uint32_t *Ld, const uint32_t *Wd, const int32_t *eL, const int32_t *eW) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const int64_t t64 = blockIdx.x >> 1;
    const int half = blockIdx.x & 1;
    const PanelDesc d = descs[find_update_desc(descs, nd, t64)];
    const int s = d.front, f = fsz[s], w = d.w;
    const int64_t t = t64 - d.off3;
    int bi = (int)((sqrt(8.0 * (double)t + 1.0) - 1.0) * 0.5);
    while ((int64_t)(bi + 1) * (bi + 2) / 2 <= t) ++bi;
    while ((int64_t)bi * (bi + 1) / 2 > t) --bi;
    const int bj = (int)(t - (int64_t)bi * (bi + 1) / 2);
    const int base = d.k0 + w, i0 = base + bi * TB, j0 = base + bj * TB + 32 * half;
    if (j0 >= f) return;
    const int nk = (w + 15) / 16, nwords = nk * UF_GROUP;  // words of a 16-row group
    uint4 *A = reinterpret_cast<uint4 *>(smraw), *Bs = A + 4 * (NB / 16) * (UF_GROUP / 4);
    {
        const uint4 *la = reinterpret_cast<const uint4 *>(Ld + (d.xd + (int64_t)bi * nk) * 4 * UF_GROUP);
        const uint4 *wb = reinterpret_cast<const uint4 *>(Wd + (d.xd + (int64_t)bj * nk) * 4 * UF_GROUP + (int64_t)2 * half * nwords);
        for (int u = threadIdx.x; u < nwords; u += UF_THREADS) cp_async16(A + u, la + u);
        for (int u = threadIdx.x; u < nwords / 2; u += UF_THREADS) cp_async16(Bs + u, wb + u);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, wm = wp & 1, wn = wp >> 1, g = lane >> 2, tt = lane & 3;
    float acc[2][2][FX_NL][4];  // [16-row group][8-column group][digit sum][fragment]
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int l = 0; l < FX_NL; ++l)
#pragma unroll
                for (int k = 0; k < 4; ++k) acc[a][b][l][k] = 0.f;
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    for (int kb = 0; kb < nk; ++kb) {
        uint32_t b[2][FX_ND][2];
#pragma unroll
        for (int u = 0; u < FX_ND / 2; ++u) {
            const uint4 q = Bs[(wn * nk + kb) * (UF_GROUP / 4) + u * 32 + lane];
            const uint32_t wd[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int n = 0; n < 2; ++n) {
                    b[n][2 * u + e][0] = fx_half2(wd[2 * e + n], 0x4140);
                    b[n][2 * u + e][1] = fx_half2(wd[2 * e + n], 0x4342);
                }
        }
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int u = 0; u < FX_ND / 2; ++u) {
                const uint4 q = A[((2 * wm + m) * nk + kb) * (UF_GROUP / 4) + u * 32 + lane];
                const uint32_t wd[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int i = 2 * u + e;
                    const uint32_t a[4] = {fx_half2(wd[2 * e], 0x4140), fx_half2(wd[2 * e + 1], 0x4140),
                                           fx_half2(wd[2 * e], 0x4342), fx_half2(wd[2 * e + 1], 0x4342)};
#pragma unroll
                    for (int j = 0; j < FX_ND && i + j < FX_NL; ++j)
#pragma unroll
                        for (int n = 0; n < 2; ++n) fx_mma(acc[m][n][i + j], a, b[n][j][0], b[n][j][1]);
                }
            }
    }
    double *F = arena + fo[s];
    const int32_t *el = eL + (d.off2 + bi) * RB, *ew = eW + (d.off2 + bj) * RB + 32 * half;
#pragma unroll
    for (int n = 0; n < 2; ++n) {
        double c[2][4];
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int gi = i0 + 16 * (2 * wm + m) + g + 8 * (k >> 1), gj = j0 + 16 * wn + 8 * n + 2 * tt + (k & 1);
                c[m][k] = gi < f && gj <= gi ? F[(int64_t)gj * f + gi] : 0.0;
            }
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int ri = 16 * (2 * wm + m) + g + 8 * (k >> 1), rj = 16 * wn + 8 * n + 2 * tt + (k & 1);
                const int gi = i0 + ri, gj = j0 + rj;
                if (gi >= f || gj > gi) continue;
                int64_t hi, lo;
                fx_collect<false>(acc[m][n], k, hi, lo);
                F[(int64_t)gj * f + gi] = c[m][k] - fx_value(hi, lo, el[ri], ew[rj]);
            }
    }
}

}  // namespace

void fx_update(const PanelStep &stp, const PanelDesc *dd, const Plan &p, double *arena, const void *digits,
               const int32_t *scales, cudaStream_t st) {
    smem_limit((const void *)k_fx_update, UF_SMEM);
    const uint32_t *Ld = static_cast<const uint32_t *>(digits), *Wd = Ld + p.max_step_xd * 4 * UF_GROUP;
    k_fx_update<<<(unsigned)(2 * stp.n3), UF_THREADS, UF_SMEM, st>>>(dd, stp.nd, p.d_sn_fo.data(), p.d_sn_f.data(), arena, Ld,
                                                                     Wd, scales, scales + p.max_step_n2 * RB);
    MBL_LAUNCH_CHECK();
}

}  // namespace mbl
