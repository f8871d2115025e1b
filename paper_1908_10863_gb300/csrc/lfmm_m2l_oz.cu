// lfmm_m2l_oz.cu -- free-space M2L (eq. metole) of the FP64 form on the tcgen05
// tensor cores, by digit products.  The idea, to split the operands of a matrix
// product into pieces whose products a fast unit adds without rounding, is
// K. Ozaki, T. Ogita, S. Oishi, S. M. Rump, "Error-free transformations of
// matrix multiplication by using fast routines of matrix multiplication and its
// applications", Numer. Algorithms 59 (2012), 95-118.
//
// The same tiles, offset classes and operators A_o as the float32 tensor-core
// M2L (lfmm_m2l_tc.cu), in FP64 accuracy.  Operands are scaled by powers of
// two (2^e per coefficient takes the factorials out, one power per level puts
// its largest multipole into [1/4, 1/2); operators are below 1/2) and written
// in seven signed digits of nine bits, t = sum_i d_i 2^{-9 i}, |d_i| <= 256:
// small integers, exact in float16.  An MMA of two digit matrices is then an
// integer contraction, exact in the float32 accumulator while its sums stay
// below 2^24 in magnitude, and
//   A X = sum_d 2^{-9 d} sum_{i + j = d} A_i X_j,
// of which the diagonals d = 2 .. 8 are kept (28 products).  What is dropped is
// at most 2^-62.4 per term (six products of up to 2^16, weight 2^-81), 2^-65.3
// in the mean square of random operands: the relative error of an offset's
// contribution measures 7e-17 against 3.5e-16 for FP64 multiply-adds.  That is
// relative to the level's largest multipole: boxes within 2^-10 of it are finer
// than in FP64, smaller ones coarser.  A target sees the large boxes too, so
// what it loses stays below its own rounding unless their charges cancel.
// Measured, superposition in the worst of 512 cells, 20,000 charges of size 1
// and a few large ones: a lone charge of 1e9 2.5e-15 (FP64 multiply-adds
// 3.0e-15), a pair of +-1e9 8.9e-13 (9.1e-14), a quadrupole of them 2.2e-10
// (1.4e-10).  Seven accumulators, one per diagonal, 64 columns each, take 448 of
// the 512 tensor-memory columns.
//   Size of the sums: the leading digits follow the operands' own magnitudes
// (row sums of |A| below about 3, so d = 2 stays near 2^19).  A full diagonal of
// trailing digits over a window of OZ_WIN offsets could reach
// 4 (p+1)^2 7 2^16 = 2^27.7, four bits past exact; its standard deviation, digits
// being as good as uniform, is below 2^20.5, so that 2^24 is eleven deviations
// away.  Exact is therefore a matter of probability, not of a bound: operands
// whose digits line up in sign over hundreds of terms with those of an
// operator's row would be rounded.  Equal multipoles in every box and charges
// of repeating digits do not come near (the results of 1, 1/3, 1/511 and 255/511
// on a lattice agree to rounding).
// Every window the accumulators are read back, converted to integers and added
// with their weights into two 64-bit integers per output (units 2^-36, 2^-72);
// the sum of all a CTA's offsets becomes one FP64 number and one atomic.
//
// Bound: L2 -> shared memory, 344 KB per 64 targets and offset at p = 10 (the
// operators' digits are two thirds of it), then the MMAs' operand reads.
// Measured, N = 65,536, p = 10: 2.19 ms against 51.3 ms for the FP64
// multiply-adds of k_m2l_gemm, whose pipe (2 per clock and SM) was full; 1,000
// charges: 2.58 -> 0.20 ms.
//
// One CTA (one per SM) = (tile of 64 targets, group of offsets, 128-row half of
// the outputs where (p+1)^2 > 128):
//   warps 0..7  gather the digits of the sources of a (offset, K chunk of 32)
//               stage by 16-byte cp.async, thread 0 starts the bulk copy of
//               the operator's digits; at the end of a window they read the
//               accumulators back;
//   warp 8      one thread issues the MMAs.
// Offsets at which no target of the tile has a source are skipped.  Waits are
// bounded as in lfmm_m2l_tc.cu.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "lfmm_ctx.h"
#include "lfmm_tc.cuh"

#define LF_CHECK(call)                                    \
    do {                                                  \
        cudaError_t e_ = (call);                          \
        if (e_ != cudaSuccess) return lf_cuda(e_, #call); \
    } while (0)
#define LF_TRY(expr)                \
    do {                            \
        LfErr r_ = (expr);          \
        if (!r_.empty()) return r_; \
    } while (0)

#define OZ_N LFMM_OZ_TILE                 // targets per tile (MMA N)
#define OZ_NOFF 189
#define OZ_NALL 343
#define OZ_WARPS 8
#define OZ_THREADS (32 * OZ_WARPS + 32)
#define OZ_X_BYTES (OZ_N * TC_ROWB)       // one multipole digit of a stage
#define OZ_STAGE (OZ_S * (OZ_A_BYTES + OZ_X_BYTES))
#define OZ_NST 2
#define OZ_SMEM (OZ_NST * OZ_STAGE + 1024)
#define OZ_MAXG 27                        // offsets per CTA at most
#define OZ_WIN 4                          // offsets per window at p <= 10 (2 above)

struct OzArgs {
    const int4* tiles;       // level, class, start, count; level < 0: merged tile
    const int* sorted;
    const int* slots;
    const int* cls;
    const double* levelh;
    const int4* mseg;
    const unsigned char* A;  // [343][half][chunk][digit][8 KB], pre-swizzled
    const __half* Ms;        // digits [box][OZ_S][mrow]
    const double* cscale;    // 2^e per packed coefficient
    const unsigned long long* gmax;  // largest scaled coefficient (double bits), [16] per right-hand side
    double* L;
    int nc, nk, nkc, nh, mrow, groups, win;
    size_t ms_stride, l_stride;
    int* err;
};

// the OZ_S digits of t, |t| < 1/2, as float16 integers, leading digit first
__device__ __forceinline__ void oz_digits(double t, __half d[OZ_S])
{
    long long v = __double2ll_rn(t * 9223372036854775808.0);  // 2^63
#pragma unroll
    for (int i = OZ_S - 1; i > 0; --i) {
        const int r = ((int)(v + 256) & 511) - 256;
        d[i] = __int2half_rn(r);
        v = (v - r) >> OZ_B;
    }
    d[0] = __int2half_rn((int)v);
}

__device__ __forceinline__ int oz_target(const OzArgs& g, const int4& tile, int t, int& level)
{
    level = 0;
    if (t >= tile.w) return -1;
    if (tile.x >= 0) {
        level = tile.x;
        return g.sorted[tile.z + t];
    }
    const int4* sg = g.mseg + (size_t)(-1 - tile.x) * LFMM_TC_MSEG;
    for (int k = 0; k < tile.z; ++k) {
        const int4 r = sg[k];
        if (t < r.z) {
            level = r.x;
            return g.sorted[r.y + t];
        }
        t -= r.z;
    }
    return -1;
}

__global__ void __launch_bounds__(OZ_THREADS, 1) k_m2l_oz(OzArgs g)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                         ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t full_bar[OZ_NST], empty_bar[OZ_NST], accf_bar, acce_bar;
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    __shared__ unsigned s_mask;
    __shared__ int s_tb[OZ_N];
    __shared__ double s_ih[OZ_N];
    __shared__ int s_src[OZ_MAXG][OZ_N];
    __shared__ int s_act[OZ_MAXG];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int item = blockIdx.x;
    const int half = item % g.nh;
    item /= g.nh;
    const int4 tile = g.tiles[item / g.groups];
    const int grp = item % g.groups, goff = OZ_NOFF / g.groups;
    const int cl = tile.y, cnt = tile.w, nc = g.nc, nkc = g.nkc;
    if (tid == 0) s_mask = 0u;
    __syncthreads();
    if (tid < OZ_N) {
        int level;
        const int tb = oz_target(g, tile, tid, level);
        s_tb[tid] = tb;
        // operators carry 1/2; 1/h of the scaled expansions
        s_ih[tid] = tb >= 0 ? 2.0 / (oz_scale(g.gmax[(size_t)blockIdx.y * 16 + level]) * g.levelh[level]) : 0.0;
        unsigned any = 0;
        const int* src = g.slots + (size_t)(tb >= 0 ? tb : 0) * OZ_NOFF + grp * goff;
        for (int o = 0; o < goff; ++o) {
            const int s = tb >= 0 ? src[o] : -1;
            s_src[o][tid] = s;
            any |= s >= 0 ? 1u << o : 0u;
        }
        any = __reduce_or_sync(0xffffffffu, any);
        if (lane == 0 && any) atomicOr(&s_mask, any);
    }
    __syncthreads();
    const unsigned mask = s_mask;
    const int nact = __popc(mask);
    if (nact == 0) return;  // block-uniform, before anything is allocated
    if (tid < goff && ((mask >> tid) & 1u)) s_act[__popc(mask & ((1u << tid) - 1u))] = tid;
    const int nstage = nact * nkc, wst = g.win * nkc;  // stages, stages per window
    if (tid == 0) {
        for (int s = 0; s < OZ_NST; ++s) {
            mbar_init(&full_bar[s], OZ_WARPS + 1);
            mbar_init(&empty_bar[s], 1);
        }
        mbar_init(&accf_bar, 1);
        mbar_init(&acce_bar, OZ_WARPS);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == OZ_WARPS) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;

    if (warp < OZ_WARPS) {
        long long hi[32], lo[32];  // sums of this thread's row and 32 columns, units 2^-36 and 2^-72
#pragma unroll
        for (int i = 0; i < 32; ++i) hi[i] = lo[i] = 0;
        const int q4 = warp & 3, ch = warp >> 2;
        const int rot = (item / g.groups) % nact;
        const __half* Ms = g.Ms + (size_t)blockIdx.y * g.ms_stride;
        int armed = 0;
        bool ok = true;
        for (int it = 0; it <= nstage; ++it) {
            if (it < nstage && ok) {
                const int s = it % OZ_NST;
                const int ol = s_act[(it / nkc + rot) % nact], kc = it % nkc;
                if (it >= OZ_NST && !mbar_wait(&empty_bar[s], (it / OZ_NST - 1) & 1)) atomicExch(&s_abort, 1);
                if (__any_sync(0xffffffffu, *(volatile int*)&s_abort)) {
                    ok = false;
                } else {
                    unsigned char* st = sm + (size_t)s * OZ_STAGE;
                    if (tid == 0) {
                        const int o = g.cls[cl * OZ_NOFF + grp * goff + ol];
                        mbar_arrive_tx(&full_bar[s], OZ_S * OZ_A_BYTES);
                        bulk_g2s(st, g.A + (((size_t)o * g.nh + half) * nkc + kc) * (OZ_S * OZ_A_BYTES),
                                 OZ_S * OZ_A_BYTES, &full_bar[s]);
                        armed = it + 1;
                    }
                    unsigned char* xs = st + OZ_S * OZ_A_BYTES;
                    const uint32_t xbase = smem_u32(xs);
                    // row tid / 4, 16-byte quarter tid % 4, every digit
                    const int row = tid >> 2, chunk = tid & 3;
                    const int src = s_src[ol][row];
                    const uint32_t off = swz16(row, chunk * 8);
                    const __half* gs = Ms + (size_t)(src >= 0 ? src : 0) * (OZ_S * g.mrow) + kc * TH_KC + chunk * 8;
#pragma unroll
                    for (int i = 0; i < OZ_S; ++i) {
                        if (src >= 0)
                            cp_async16(xbase + i * OZ_X_BYTES + off, gs + (size_t)i * g.mrow);
                        else
                            *reinterpret_cast<float4*>(xs + i * OZ_X_BYTES + off) = make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                }
            }
            cp_async_commit();
            if (it == 0) continue;
            // hand the previous stage over
            cp_async_wait<1>();
            fence_async_smem();
            __syncwarp();
            if (!ok) break;
            if (lane == 0) mbar_arrive(&full_bar[(it - 1) % OZ_NST]);
            // ... and at the end of a window read the accumulators back
            if (it % wst == 0 || it == nstage) {
                const int w = (it - 1) / wst;
                const bool got = mbar_wait(&accf_bar, w & 1);
                tc_fence_after();
                if (!__all_sync(0xffffffffu, got && !*(volatile int*)&s_abort)) {
                    atomicExch(&s_abort, 1);
                    ok = false;
                    break;
                }
                const uint32_t ta = tmem + ((uint32_t)(32 * q4) << 16) + (uint32_t)(32 * ch);
#pragma unroll
                for (int dh = 0; dh < 2 * OZ_S; ++dh) {
                    const int d = dh >> 1, c0 = 16 * (dh & 1);
                    float v[16];
                    tc_ld16(ta + (uint32_t)(d * OZ_N + c0), v);
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const int n = __float2int_rn(v[i]);
                        if (d < 3)
                            hi[c0 + i] += (long long)n * (1ll << (OZ_B * (2 - d)));
                        else
                            lo[c0 + i] += (long long)n * (1ll << (OZ_B * (6 - d)));
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&acce_bar);
            }
        }
        cp_async_wait<0>();
        if (tid == 0 && *(volatile int*)&s_abort)  // drain: the bulk copies this thread issued
            for (int j = (armed > OZ_NST ? armed - OZ_NST : 0); j < armed; ++j)
                mbar_wait(&full_bar[j % OZ_NST], (j / OZ_NST) & 1);
        if (ok) {
            const int row = 128 * half + 32 * q4 + lane;
            if (row < nc) {
                const double rs = g.cscale[row];
                double* L = g.L + (size_t)blockIdx.y * g.l_stride + row;
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    const int j = 32 * ch + i;
                    if (j < cnt) {
                        const double v = (double)hi[i] * 0x1p-36 + (double)lo[i] * 0x1p-72;
                        atomicAdd(L + (size_t)s_tb[j] * nc, v * (s_ih[j] * rs));
                    }
                }
            }
        } else if (lane == 0) {
            atomicAdd(g.err, 1);
        }
    } else {
        // ---------------- MMA issuer ----------------
        if (lane == 0) {
            const uint32_t idesc = tc_idesc_f16(128, OZ_N);
            bool ok = true;
            for (int it = 0; it < nstage && ok; ++it) {
                const int s = it % OZ_NST, iw = it % wst;
                if (iw == 0 && it > 0) {  // the accumulators of the last window have been read
                    if (!mbar_wait(&acce_bar, (it / wst - 1) & 1)) ok = false;
                    tc_fence_after();
                }
                if (!ok || !mbar_wait(&full_bar[s], (it / OZ_NST) & 1)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t ab = smem_u32(sm + (size_t)s * OZ_STAGE), xb = ab + OZ_S * OZ_A_BYTES;
                const int nks = (g.nk - (it % nkc) * TH_KC) > 16 ? 2 : 1;
                for (int ks = 0; ks < nks; ++ks)
#pragma unroll
                    for (int i = 0; i < OZ_S; ++i)
#pragma unroll
                        for (int j = 0; j < OZ_S - i; ++j)
                            tc_mma_f16(tmem + (uint32_t)((i + j) * OZ_N), smem_desc(ab + i * OZ_A_BYTES + 32 * ks),
                                       smem_desc(xb + j * OZ_X_BYTES + 32 * ks), idesc,
                                       (iw == 0 && ks == 0 && i == 0) ? 0u : 1u);
                tc_commit(&empty_bar[s]);
                if (iw == wst - 1 || it == nstage - 1) tc_commit(&accf_bar);
            }
            if (!ok) atomicExch(&s_abort, 1);
        }
        __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == OZ_WARPS) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// ---------------------------------------------------------------------------
// Operands.
// ---------------------------------------------------------------------------
// FP64 operators A [343][KP in][RP out] -> digits, one block per (offset, half,
// chunk); rows r of the half, K elements k of the chunk (inputs in the order of
// lf_coef_order).  Entries scaled by
// 2^{-e_in - e_out} / 2 stay below 1/2; a larger one is counted in bad.
__global__ void __launch_bounds__(256) k_oz_blob(const double* __restrict__ A, int KP, int RP, int nc, int nk, int nh,
                                                 int nkc, const int* __restrict__ perm, const double* __restrict__ cs, unsigned char* __restrict__ blob, int* __restrict__ bad)
{
    const int kc = blockIdx.x % nkc, half = (blockIdx.x / nkc) % nh, o = blockIdx.x / (nkc * nh);
    unsigned char* p0 = blob + (size_t)blockIdx.x * (OZ_S * OZ_A_BYTES);
    for (int i = threadIdx.x; i < TH_KC * 128; i += 256) {
        const int k = i / 128, r = i - k * 128, kp = kc * TH_KC + k, row = 128 * half + r;
        const int kin = kp < nk ? perm[kp] : -1;
        double v = 0.0;
        if (kin >= 0 && row < nc) {
            v = A[((size_t)o * KP + kin) * RP + row] / cs[kin] / cs[row] * 0.5;
            if (!(fabs(v) < 0.5)) atomicAdd(bad, 1);
        }
        __half d[OZ_S];
        oz_digits(v, d);
#pragma unroll
        for (int q = 0; q < OZ_S; ++q) *reinterpret_cast<__half*>(p0 + (size_t)q * OZ_A_BYTES + swz16(r, k)) = d[q];
    }
}

struct OzLevels {
    int depth;
    int off[17];
};
__device__ __forceinline__ int oz_level(const OzLevels& lv, int b)
{
    int l = lv.depth;
    while (l > 0 && b >= lv.off[l - 1]) --l;
    return l;
}

// largest scaled multipole |M_k| 2^{e_k} of each level, as double bits in
// gmax[16 rhs + level] (zeroed when the charges were sorted); one block per 32
// boxes, met in shared memory
__global__ void __launch_bounds__(256) k_oz_max(const double* __restrict__ M, int nbox, int nc,
                                                const double* __restrict__ cs, const __grid_constant__ OzLevels lv,
                                                unsigned long long* __restrict__ gmax)
{
    __shared__ unsigned long long s_max[16];
    if (threadIdx.x < 16) s_max[threadIdx.x] = 0ull;
    __syncthreads();
    M += (size_t)blockIdx.y * nbox * nc;
    const int lane = threadIdx.x & 31, i0 = blockIdx.x * 32 + (threadIdx.x >> 5) * 4;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        const int b = i0 + u;
        if (b >= nbox) break;
        unsigned long long m = 0;
        for (int k = lane; k < nc; k += 32) {
            const unsigned long long v = (unsigned long long)__double_as_longlong(fabs(M[(size_t)b * nc + k] * cs[k]));
            m = v > m ? v : m;
        }
        const unsigned h = __reduce_max_sync(0xffffffffu, (unsigned)(m >> 32));
        const unsigned lw = __reduce_max_sync(0xffffffffu, (unsigned)(m >> 32) == h ? (unsigned)m : 0u);
        if (lane == 0) atomicMax(&s_max[oz_level(lv, b)], ((unsigned long long)h << 32) | lw);
    }
    __syncthreads();
    if (threadIdx.x < 16 && s_max[threadIdx.x] != 0ull) {
        unsigned long long* g = gmax + (size_t)blockIdx.y * 16 + threadIdx.x;
        if (s_max[threadIdx.x] > *(volatile unsigned long long*)g) atomicMax(g, s_max[threadIdx.x]);
    }
}

// multipoles [box][nc] -> digits [box][OZ_S][mrow] in the K order (zero padded),
// one thread per pair of coefficients
__global__ void __launch_bounds__(256) k_oz_split(const double* __restrict__ M, int nbox, int nc, int nk,
                                                  int mrow, const int* __restrict__ perm,
                                                  const double* __restrict__ cs,
                                                  const __grid_constant__ OzLevels lv,
                                                  const unsigned long long* __restrict__ gmax,
                                                  __half* __restrict__ Ms)
{
    const int per = mrow / 2;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)nbox * per) return;
    M += (size_t)blockIdx.y * nbox * nc;
    Ms += (size_t)blockIdx.y * nbox * OZ_S * mrow;
    const int b = (int)(i / per), k = (int)(i % per) * 2;
    const double s = oz_scale(gmax[(size_t)blockIdx.y * 16 + oz_level(lv, b)]);
    __half d0[OZ_S], d1[OZ_S];
    const int j0 = k < nk ? perm[k] : -1, j1 = k + 1 < nk ? perm[k + 1] : -1;
    oz_digits(j0 >= 0 ? M[(size_t)b * nc + j0] * cs[j0] * s : 0.0, d0);
    oz_digits(j1 >= 0 ? M[(size_t)b * nc + j1] * cs[j1] * s : 0.0, d1);
    __half* out = Ms + (size_t)b * OZ_S * mrow + k;
#pragma unroll
    for (int q = 0; q < OZ_S; ++q) *reinterpret_cast<__half2*>(out + (size_t)q * mrow) = __halves2half2(d0[q], d1[q]);
}

// ---------------------------------------------------------------------------
// Host.
// ---------------------------------------------------------------------------
bool lf_m2l_oz_ok(const lfmm_ctx* ctx) { return ctx->m2l_rm > 0 && lf_nc(ctx->p) <= 256; }

// operator digits, coefficient scales and order, once per context: at the end of
// the first build of the FP64 form that has M2L pairs, or when a built context
// takes that form.  It reads the range check back, so no evaluation may be the
// first to come here (lfmm_evaluate_device does not wait for the device).
LfErr lf_oz_prepare(lfmm_ctx* ctx, cudaStream_t st)
{
    if (ctx->oz_ready || ctx->precision || !lf_m2l_oz_ok(ctx)) return LfErr();
    if (!(ctx->m2l_ntiles > 0 && ctx->oz_ntiles > 0) && ctx->m2r_nbatch == 0) return LfErr();
    const int p = ctx->p, nc = lf_nc(p), nh = (nc + 127) / 128, RP = ctx->m2l_rp;
    std::vector<int> perm, e;
    lf_coef_order(p, perm);
    lf_coef_exponents(p, e);
    const int nk = (int)perm.size(), nkc = (nk + TH_KC - 1) / TH_KC;
    std::vector<double> cs(nc);
    for (int j = 0; j < nc; ++j) cs[j] = std::ldexp(1.0, e[j]);
    LF_TRY(lf_reserve(ctx->oz_cscale, nc * sizeof(double)));
    LF_TRY(lf_reserve(ctx->oz_perm, nk * sizeof(int)));
    LF_TRY(lf_reserve(ctx->oz_A, (size_t)OZ_NALL * nh * nkc * OZ_S * OZ_A_BYTES));
    LF_CHECK(cudaMemcpyAsync(ctx->oz_cscale.ptr, cs.data(), nc * sizeof(double), cudaMemcpyHostToDevice, st));
    LF_CHECK(cudaMemcpyAsync(ctx->oz_perm.ptr, perm.data(), nk * sizeof(int), cudaMemcpyHostToDevice, st));
    int* bad = reinterpret_cast<int*>(ctx->counts.as<char>() + LFMM_OZ_BAD_OFF);
    LF_CHECK(cudaMemsetAsync(bad, 0, sizeof(int), st));
    LF_CHECK(cudaFuncSetAttribute(k_m2l_oz, cudaFuncAttributeMaxDynamicSharedMemorySize, OZ_SMEM));
    ++ctx->launches, k_oz_blob<<<OZ_NALL * nh * nkc, 256, 0, st>>>(ctx->m2l_A64.as<double>(), RP, RP, nc, nk, nh, nkc,
                                                                   ctx->oz_perm.as<int>(), ctx->oz_cscale.as<double>(),
                                                                   ctx->oz_A.as<unsigned char>(), bad);
    LF_TRY(lf_cuda(cudaGetLastError(), "operator digits"));
    int n = 0;
    LF_CHECK(lf_d2h(&n, bad, sizeof(int), st));
    if (n) return "internal: free M2L operator out of the digit range";
    ctx->oz_nk = nk;
    ctx->oz_ready = 1;
    return LfErr();
}

// the multipoles of every box as digits, for the free M2L and the keyed
// reaction M2L of this evaluation
LfErr lf_oz_split(lfmm_ctx* ctx, cudaStream_t st)
{
    LF_TRY(lf_oz_prepare(ctx, st));  // (done already, unless that failed)
    const int nb = ctx->nbox_total, nr = ctx->nrhs_b, nc = lf_nc(ctx->p), nk = ctx->oz_nk;
    const int mrow = (nk + TH_KC - 1) / TH_KC * TH_KC;
    LF_TRY(lf_reserve(ctx->oz_Ms, (size_t)nb * OZ_S * mrow * sizeof(__half) * nr));
    unsigned long long* gm = reinterpret_cast<unsigned long long*>(ctx->counts.as<char>() + LFMM_TCMAX_OFF);
    OzLevels lv;
    lv.depth = ctx->depth;
    for (int l = 0; l < 17; ++l) lv.off[l] = l <= ctx->depth ? ctx->levels[l].off : 0;
    const double* M = ctx->Mexp.as<double>();
    ++ctx->launches, k_oz_max<<<dim3((nb + 31) / 32, nr), 256, 0, st>>>(M, nb, nc, ctx->oz_cscale.as<double>(), lv, gm);
    const int64_t tot = (int64_t)nb * (mrow / 2);
    ++ctx->launches, k_oz_split<<<dim3((unsigned)((tot + 255) / 256), nr), 256, 0, st>>>(
        M, nb, nc, nk, mrow, ctx->oz_perm.as<int>(), ctx->oz_cscale.as<double>(), lv, gm, ctx->oz_Ms.as<__half>());
    return lf_cuda(cudaGetLastError(), "multipole digits");
}

LfErr lf_m2l_oz(lfmm_ctx* ctx, cudaStream_t st)
{
    if (ctx->oz_ntiles == 0) return LfErr();
    const int nb = ctx->nbox_total, nr = ctx->nrhs_b, nc = lf_nc(ctx->p);
    OzArgs g;
    g.nc = nc;
    g.nk = ctx->oz_nk;
    g.nh = (nc + 127) / 128;
    g.nkc = (g.nk + TH_KC - 1) / TH_KC;
    g.mrow = g.nkc * TH_KC;
    g.win = nc <= 128 ? OZ_WIN : OZ_WIN / 2;
    g.tiles = ctx->oz_tiles.as<int4>();
    g.sorted = ctx->m2l_sorted.as<int>();
    g.slots = ctx->m2l_slots.as<int>();
    g.cls = ctx->m2l_cls.as<int>();
    g.levelh = ctx->m2l_levelh.as<double>();
    g.mseg = ctx->oz_mseg.as<int4>();
    g.A = ctx->oz_A.as<unsigned char>();
    g.Ms = ctx->oz_Ms.as<__half>();
    g.cscale = ctx->oz_cscale.as<double>();
    g.gmax = reinterpret_cast<unsigned long long*>(ctx->counts.as<char>() + LFMM_TCMAX_OFF);
    g.L = ctx->Lexp.as<double>();
    // 27 offsets per CTA amortise its read-back and FP64 atomics; 9 or 3 where
    // the tiles are too few to give every SM several CTAs
    const int64_t units = (int64_t)ctx->oz_ntiles * g.nh * nr;
    g.groups = units * 7 >= 4 * 152 ? 7 : (units * 21 >= 2 * 152 ? 21 : 63);
    g.ms_stride = (size_t)nb * OZ_S * g.mrow;
    g.l_stride = (size_t)nb * nc;
    g.err = reinterpret_cast<int*>(ctx->counts.as<char>() + LFMM_TIMEOUT_OFF);
    ++ctx->launches, k_m2l_oz<<<dim3(ctx->oz_ntiles * g.groups * g.nh, nr), OZ_THREADS, OZ_SMEM, st>>>(g);
    return lf_cuda(cudaGetLastError(), "m2l digit products");
}
