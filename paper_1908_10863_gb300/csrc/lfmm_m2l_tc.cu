// lfmm_m2l_tc.cu -- free-space M2L (eq. metole) on the tcgen05 tensor cores.
//
// The same per-offset real-linear maps A_o as the CUDA-core GEMM in
// lfmm_m2l.cu, evaluated as D[r][j] = sum_o sum_k A_o[r][k] X_o[j][k] with
//   r = output coefficient (M = 128 rows, expansions with (p+1)^2 <= 128),
//   j = target box of the tile (N = 256 columns, one level and octant class),
//   k = input coefficient of the source at offset o (K = 128 in chunks of
//       TH_KC, only the chunks that hold the (p+1)^2 inputs),
// accumulated in tensor memory (128 lanes x 256 float32 columns).  The wide
// form takes 128 < (p+1)^2 <= 256 (p = 11 .. 14): two 128-row halves of r,
// K = 256, tiles of 128 targets (see k_m2l_tc<true>).
//
// Precision: float32 operands as sums of two float16 pieces (11 + 11 bits, the
// significand of two TF32 pieces), the operator (a1 + a2, from its FP64
// values) and the multipoles (x1 + x2, split once per evaluation), with the
// three products a1 x1 + a1 x2 + a2 x1 (~2^-21 of |a||x| per product).  Float16
// has half the bytes of TF32 in L2, shared memory and the MMAs' operand reads,
// and twice the multiply rate; its five exponent bits are no limit after
// scaling by powers of two:
//   - coefficient (n, m) carries 2^e, e = log2 sqrt((n - m)! (n + m)!) rounded
//     (M scaled up by it, L down), which takes the factorials out of the
//     expansions and of the operators (entries below 2);
//   - each level's multipoles are scaled by one power of two that puts the
//     largest scaled coefficient into [2^13, 2^14) (k_tc_max), so the pieces
//     lose nothing above 2^-39 of that largest coefficient.
// What limits the result is the tensor core's float32 accumulation: its error
// grows with the number of MMAs added to an accumulator that is already large.
// So the input coefficients run from the highest degree to the lowest (K is
// ordered by degree, and a unit takes K chunk by K chunk, each for all its
// offsets): the small contributions of the high degrees meet in a small
// accumulator, and only the last chunk, degrees 0 to 4, adds at full size.
// Each CTA takes only some of the 189 offsets, and the CTAs of a tile are
// joined by float atomics.
//
// Measured (config-2 geometry, M2L alone; Err2(phi) of the float32 form
// against the FP64 form), TF32 pieces in offset order -> float16 pieces in
// degree order: N = 1M, p = 10: 2.25 ms, 2.1e-6 -> 1.33 ms, 0.66e-6; N = 262,144,
// p = 6: 0.208 -> 0.137 ms, 1.5e-6 -> 0.6e-6; the wide form, N = 65,536, p = 14:
// 1.29 ms, 6.8e-7 -> 0.93 ms, 3.1e-7, the error of the compensated CUDA-core sums
// (7.9 ms), so the wide form is the default.  Float16 pieces in offset order: 1.45
// ms, 1.26e-6 at N = 1M.  Bound: L2 -> shared memory, 192 KB per tile and
// offset (8.8 GB at N = 1M, 6.6 TB/s); the MMAs alone would take 0.6 ms.
//
// One CTA = (tile of 256 targets, 9 of its 189 offsets):
//   warps 0..7  gather the 256 pre-split source multipoles of a (K chunk,
//               offset) stage with 16-byte cp.async into the swizzled
//               K-major layout (zeros where a target has no source there), ahead
//               of the tensor cores; thread 0 also starts the bulk
//               copy of the matching operator chunk (stored pre-split and
//               pre-swizzled in HBM);
//   warp 8      one thread issues the MMAs of a stage (3 products x 2 K steps of 16) and commits them to
//               the stage's "empty" barrier;
//   epilogue    warps 0..7 read the accumulator (tcgen05.ld), scale by 1/h and the inverse
//               operand scales and add into the local expansions (float atomics: the CTAs of a
//               tile's offset groups meet there).
// Two stages of 48 KB (K chunks of 32, 64-byte swizzle) per CTA buffer the
// operands, handed to the tensor cores one stage after their copies start;
// two CTAs share an SM, so four stages are in flight per SM.
// Tiles of one octant class share their offset list; each tile walks it from a different starting offset so
// that concurrent CTAs read different operator chunks.  Every barrier wait is
// bounded; on a timeout the CTA records an error, stops issuing work, waits
// (bounded) for its copies in flight and frees its tensor memory.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <cstring>
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

#define TC_N 256                     // targets per tile (MMA N)
#define TC_M 128                     // output coefficients (MMA M)
#define TC_NKC (128 / TH_KC)         // K chunks (K = 128)
#define TC_RCH (TC_ROWB / 16)        // 16-byte chunks per row
#define TC_NOFF 189                  // offsets per octant class
#define TC_NALL 343
#define TC_PROD_WARPS 8
#define TC_THREADS (32 * TC_PROD_WARPS + 32)
#define TC_A_BYTES (TC_M * TC_ROWB)  // one operator piece of a stage
#define TC_X_BYTES (TC_N * TC_ROWB)  // one multipole piece of a stage
#define TC_AP 2                      // operator pieces
#define TC_XP 2                      // multipole pieces
#define TC_STAGE_BYTES (TC_AP * TC_A_BYTES + TC_XP * TC_X_BYTES)
#define TC_MROW 128                  // halves per multipole piece row in the split copy (256 B)
// Two CTAs per SM (97 KB of shared memory and 256 tensor-memory columns
// each), two 48 KB stages apiece: one CTA's prologue, gathers and atomic
// epilogue overlap the other's MMAs.
#ifndef TC_STAGES
#define TC_STAGES 2
#endif
#ifndef TC_LAG
#define TC_LAG (TC_STAGES / 2)           // stages between a stage's copies and its hand-over
#endif
#ifndef TC_MINB
#define TC_MINB 2                        // resident CTAs per SM
#endif
#define TC_SMEM (TC_STAGES * TC_STAGE_BYTES + 1024)
#define TC_TMEM_COLS 256
#define TC_WIDE_STAGES 4             // wide form: one CTA per SM
#define TC_WIDE_SMEM (TC_WIDE_STAGES * TC_STAGE_BYTES + 1024)
#define TC_MSEG LFMM_TC_MSEG
// offsets per CTA whose source boxes are kept in shared memory: every K chunk
// walks the offsets again, and a load from the slot table (one 32-byte sector
// per target) at each stage cost 0.2 ms at N = 1M.  Larger groups read the table.
#define TC_SRC 9

struct TcArgs {
    const int4* tiles;      // level, class, start, count
    const int* sorted;      // target boxes grouped by (level, class)
    const int* slots;       // [box][noff] source box at each offset of the class, or -1
    const int* cls;         // [class][noff] operator index of each class position
    int noff;               // offsets per class: 189 (M2L), 1 (L2L: parent)
    int unit_scale;         // 1: add D as it is (L2L); 0: add D / h_level (M2L)
    const double* levelh;   // box size per level
    const int4* mseg;       // merged tiles' runs [merged tile][TC_MSEG]: (level, start, count, 0)
    const unsigned char* A; // [343][4 chunks][2 pieces x 8 KB], pre-swizzled
    const __half* Ms;       // split, scaled expansions [box][2 pieces][128]
    const float* cscale;    // 2^e of every coefficient (output rows)
    float unscale;          // inverse of the operators' common scale
    const unsigned* gmax;   // largest scaled coefficients of the sources, [32] per right-hand side
    int gslot;              // slot of the source level: the target's level + gslot
    float* L;               // locals [box][nc]
    int nc;
    int nk, nkc;            // K positions in use, and chunks of TH_KC that hold them
    size_t ms_stride;       // per right-hand side (blockIdx.y): split multipoles, in halves
    size_t l_stride;        // per right-hand side: local expansions, in floats
    int groups;             // CTAs per tile (offset groups; divides noff)
    int* err;               // [0]: timeouts
};

// Target t of a tile (a box id, or -1 past the tile's count) and its output
// scale (1 for L2L, 1/h of the target's level for M2L).  A tile with
// level < 0 is a merged tile: the leftover runs (fewer targets than a tile)
// of one octant class on several levels, listed at mseg[-1 - level] with
// tile.z runs; its columns take the runs in order, each with its level's
// scale (the operators depend only on the class and the offset).
__device__ __forceinline__ float tc_out_scale(const TcArgs& g, int level)
{
    // 1/h, and the inverse of the sources' and the operators' scales
    const float s = g.unscale / tc_scale(g.gmax[(size_t)blockIdx.y * 32 + level + g.gslot]);
    return g.unit_scale ? s : s * (1.f / (float)g.levelh[level]);
}
__device__ __forceinline__ int tc_tile_target(const TcArgs& g, const int4& tile, int t, float& ih)
{
    ih = 0.f;
    if (t >= tile.w) return -1;
    if (tile.x >= 0) {
        ih = tc_out_scale(g, tile.x);
        return g.sorted[tile.z + t];
    }
    const int4* sg = g.mseg + (size_t)(-1 - tile.x) * TC_MSEG;
    for (int k = 0; k < tile.z; ++k) {
        const int4 r = sg[k];
        if (t < r.z) {
            ih = tc_out_scale(g, r.x);
            return g.sorted[r.y + t];
        }
        t -= r.z;
    }
    return -1;
}

// WIDE: expansions with 128 < (p+1)^2 <= 256 (p <= 15): the output rows are
// two 128-row halves (two MMAs per K step), K runs over 16 chunks, and a tile
// holds 128 targets, so a stage keeps its 48 KB.  With twice the MMAs per
// offset, the large product a1 x1 gets an accumulator of its own (256
// columns) and the two correction products share a second one: the float32
// accumulation drift of the tensor cores grows with the MMAs summed into
// one accumulator, and the corrections are 2^-11 of the large product.  The
// 512 columns allow one CTA per SM, which then runs four stages.
template <bool WIDE>
__global__ void __launch_bounds__(TC_THREADS, WIDE ? 1 : TC_MINB) k_m2l_tc(TcArgs g)
{
    constexpr int TN = WIDE ? 128 : TC_N;       // targets per tile (MMA N)
    constexpr int MH = WIDE ? 2 : 1;            // 128-row halves of the output (MMA M = 128 each)
    constexpr int NKC = WIDE ? 2 * TC_NKC : TC_NKC;      // K chunks per operator in the blob
    constexpr int MROW = WIDE ? 2 * TC_MROW : TC_MROW;  // halves per multipole piece row
    constexpr int ABYTES = MH * TC_A_BYTES;     // one operator piece of a stage
    constexpr int XBYTES = TN * TC_ROWB;        // one multipole piece of a stage
    constexpr int NST = WIDE ? TC_WIDE_STAGES : TC_STAGES;
    constexpr int LAG = WIDE ? TC_WIDE_STAGES / 2 : TC_LAG;
    constexpr uint32_t COLS = WIDE ? 2 * TC_TMEM_COLS : TC_TMEM_COLS;
    constexpr uint32_t SMALL = WIDE ? TC_TMEM_COLS : 0;  // accumulator of the correction products
    static_assert(TC_AP * ABYTES + TC_XP * XBYTES == TC_STAGE_BYTES, "stage size");
    extern __shared__ unsigned char smem_raw[];
    unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                         ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t full_bar[NST], empty_bar[NST], done_bar;
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    __shared__ int s_tb[TC_N];
    __shared__ float s_ih[TC_N];  // output scale of each target column
    __shared__ int s_src[TC_SRC][TN];
    __shared__ unsigned s_mask;     // offsets with a source (groups of at most TC_SRC offsets)
    __shared__ int s_act[TC_SRC];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int item = blockIdx.x;
    const int4 tile = g.tiles[item / g.groups];
    const int grp = item % g.groups;
    const int goff = g.noff / g.groups;
    const int cl = tile.y, cnt = tile.w;
    const int nc = g.nc;
    const int nkc = g.nkc;  // K chunks that hold coefficients (the rest are zero)
    const bool listed = goff <= TC_SRC;

    if (tid == 0) s_mask = 0u;
    __syncthreads();
    if (tid < TN) {
        float ih;
        const int tb = tc_tile_target(g, tile, tid, ih);
        s_tb[tid] = tb;
        s_ih[tid] = ih;
        if (listed) {
            const int* src = g.slots + (size_t)(tb >= 0 ? tb : 0) * g.noff + grp * goff;
            unsigned any = 0;
#pragma unroll
            for (int o = 0; o < TC_SRC; ++o)
                if (o < goff) {
                    const int s = tb >= 0 ? src[o] : -1;
                    s_src[o][tid] = s;
                    any |= s >= 0 ? 1u << o : 0u;
                }
            any = __reduce_or_sync(0xffffffffu, any);
            if (lane == 0 && any) atomicOr(&s_mask, any);
        }
    }
    __syncthreads();
    // offsets at which some target of the tile has a source; the others (thin
    // layers, small trees) are skipped
    const unsigned mask = s_mask;
    const int nact = listed ? __popc(mask) : goff;
    if (nact == 0) return;  // block-uniform, before anything is allocated
    if (listed && tid < goff && ((mask >> tid) & 1u)) s_act[__popc(mask & ((1u << tid) - 1u))] = tid;
    const int nstage = nact * nkc;
    if (tid == 0) {
        for (int s = 0; s < NST; ++s) {
            mbar_init(&full_bar[s], TC_PROD_WARPS + 1);  // one arrival per producer warp + the bulk copy's
            mbar_init(&empty_bar[s], 1);
        }
        mbar_init(&done_bar, 1);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == TC_PROD_WARPS) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;

    if (warp < TC_PROD_WARPS) {
        // ---------------- producers ----------------
        // stage it is filled at iteration it and handed to the tensor cores at
        // iteration it + TC_LAG, once its copies have landed
        const int ptid = tid;  // 0 .. 255
        const int rot = (item / g.groups) % nact;
        int armed = 0;         // stages with a bulk copy issued by this thread, for the bounded drain
        const int my_row = (WIDE ? (warp & 3) : warp) * 32 + lane;
        const int* my_slots = g.slots + (size_t)max(s_tb[my_row], 0) * g.noff + grp * goff;
        int it = 0;
        for (; it < nstage; ++it) {
            const int s = it % NST, round = it / NST;
            const int oa = (it + rot) % nact, ol = listed ? s_act[oa] : oa;
            const int oi = grp * goff + ol, kc = nkc - 1 - it / nact;
            // source of this thread's row at the stage's offset
            const int my_src = listed ? s_src[ol][my_row] : (s_tb[my_row] >= 0 ? my_slots[ol] : -1);
            if (it >= NST) {
                if (!mbar_wait(&empty_bar[s], (round - 1) & 1)) atomicExch(&s_abort, 1);
            }
            if (__any_sync(0xffffffffu, *(volatile int*)&s_abort)) break;  // warp-uniform
            unsigned char* st = sm + (size_t)s * TC_STAGE_BYTES;
            if (ptid == 0) {
                const int o = g.cls[cl * g.noff + oi];
                mbar_arrive_tx(&full_bar[s], TC_AP * ABYTES);
                bulk_g2s(st, g.A + ((size_t)o * NKC + kc) * (TC_AP * ABYTES), TC_AP * ABYTES, &full_bar[s]);
                armed = it + 1;
            }
            unsigned char* xs = st + TC_AP * ABYTES;
            const uint32_t xbase = smem_u32(xs);
            // 32 rows x TC_RCH chunks of 16 B per warp and piece: both pieces
            // per warp (256 rows), or warps 4..7 the second piece (128 rows)
            constexpr int NI = WIDE ? TC_RCH : 2 * TC_RCH;
#pragma unroll
            for (int i = 0; i < NI; ++i) {
                const int piece = WIDE ? (warp >> 2) : i / TC_RCH;
                const int flat = (WIDE ? i : i % TC_RCH) * 32 + lane;  // chunk-major over the warp's 32 rows
                const int rl = flat / TC_RCH, chunk = flat % TC_RCH;
                const int src = __shfl_sync(0xffffffffu, my_src, rl);
                const int row = (WIDE ? (warp & 3) : warp) * 32 + rl;
                const uint32_t off = piece * XBYTES + swz16(row, chunk * 8);
                if (src >= 0) {
                    const __half* gsrc = g.Ms + (size_t)blockIdx.y * g.ms_stride +
                                         ((size_t)src * TC_XP + piece) * MROW + kc * TH_KC + chunk * 8;
                    cp_async16(xbase + off, gsrc);
                } else {
                    *reinterpret_cast<float4*>(xs + off) = make_float4(0.f, 0.f, 0.f, 0.f);
                }
            }
            cp_async_commit();
            if (it >= LAG) {
                cp_async_wait<LAG>();
                fence_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&full_bar[(it - LAG) % NST]);
            }
        }
        cp_async_wait<0>();
        fence_async_smem();
        __syncwarp();
        if (lane == 0)
            for (int j = (it > LAG ? it - LAG : 0); j < it; ++j) mbar_arrive(&full_bar[j % NST]);
        // drain: the bulk copies this thread issued complete on their full barriers
        if (ptid == 0 && *(volatile int*)&s_abort) {
            for (int j = (armed > NST ? armed - NST : 0); j < armed; ++j)
                mbar_wait(&full_bar[j % NST], (j / NST) & 1);
        }
        // ---------------- epilogue ----------------
        const bool ok = mbar_wait(&done_bar, 0);
        tc_fence_after();
        if (ok && !*(volatile int*)&s_abort) {
            const int q = warp & 3, half = warp >> 2;
            // narrow: half = target half of the 256 columns; wide: half = the
            // 128-row half of the outputs, whose accumulator starts at column half * TN
            const int row = (WIDE ? 128 * half : 0) + 32 * q + lane;
            const float rs = row < nc ? g.cscale[row] : 0.f;
#pragma unroll 1
            for (int ch = 0; ch < 4; ++ch) {
                const int col0 = (WIDE ? 0 : half * 128) + ch * 32;  // first target of the chunk
                float v[32];
                const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)((WIDE ? half * TN : 0) + col0);
                tc_ld32(ta, v);
                if (WIDE) {
                    float w[32];
                    tc_ld32(ta + SMALL, w);
#pragma unroll
                    for (int i = 0; i < 32; ++i) v[i] += w[i];
                }
                if (row < nc) {
#pragma unroll
                    for (int i = 0; i < 32; ++i) {
                        const int j = col0 + i;
                        if (j < cnt) atomicAdd(g.L + (size_t)blockIdx.y * g.l_stride + (size_t)s_tb[j] * nc + row, v[i] * s_ih[j] * rs);
                    }
                }
            }
        } else if (lane == 0) {
            atomicAdd(g.err, 1);
        }
    } else {
        // ---------------- MMA issuer ----------------
        if (lane == 0) {
            const uint32_t idesc = tc_idesc_f16(TC_M, TN);
            bool ok = true;
            for (int it = 0; it < nstage && ok; ++it) {
                const int s = it % NST, round = it / NST;
                if (!mbar_wait(&full_bar[s], round & 1)) {
                    ok = false;
                    atomicExch(&s_abort, 1);
                    break;
                }
                tc_fence_after();
                const uint32_t base = smem_u32(sm + (size_t)s * TC_STAGE_BYTES);
                const uint32_t xb = base + TC_AP * ABYTES;
                // the small products first: a2 x1, a1 x2, a1 x1
                const int pa[3] = {1, 0, 0}, px[3] = {0, 1, 0};
                // K steps of 16 that hold coefficients (both but in an operator's last chunk)
                const int nks = (g.nk - (nkc - 1 - it / nact) * TH_KC) > 16 ? 2 : 1;
#pragma unroll
                for (int prod = 0; prod < 3; ++prod) {
                    const uint32_t a = base + pa[prod] * ABYTES;
                    const uint32_t b = xb + px[prod] * XBYTES;
                    // narrow: one accumulator; wide: a1 x1 alone, the corrections in the second
                    const uint32_t acc = (WIDE && prod < 2) ? SMALL : 0u;
                    const bool starts = prod == 0 || (WIDE && prod == 2);  // may start its accumulator
#pragma unroll
                    for (int ks = 1; ks >= 0; --ks) {
                        if (ks >= nks) continue;
#pragma unroll
                        for (int h = 0; h < MH; ++h)
                            tc_mma_f16(tmem + acc + (uint32_t)(h * TN), smem_desc(a + h * TC_A_BYTES + 32 * ks),
                                       smem_desc(b + 32 * ks), idesc,
                                       (it == 0 && starts && ks == nks - 1) ? 0u : 1u);
                    }
                }
                tc_commit(&empty_bar[s]);
            }
            tc_commit(&done_bar);
        }
        __syncwarp();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == TC_PROD_WARPS) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(COLS)
                     : "memory");
    }
}

// ---------------------------------------------------------------------------
// Persistent form of the free M2L (one CTA per SM).
//
// The work units are the (tile, offset group) pairs of k_m2l_tc; each CTA
// walks units u = blockIdx.x, blockIdx.x + gridDim.x, ... with one pipeline
// that never drains between units:
//   warps 0..7   producers: operator chunk by bulk copy, multipole rows by
//                16-byte cp.async gathers, TCP_STAGES stages of 48 KB, each
//                handed to the tensor cores TCP_LAG stages after its copies
//                start (stage counter global over the CTA's units);
//   warp 8       one thread issues the MMAs of a unit into one of two
//                256-column tensor-memory accumulators (unit parity), and
//                commits the unit to that accumulator's "full" barrier;
//   warps 9..12  epilogue: read the finished accumulator (tcgen05.ld; warp w
//                reads lanes 32 (w mod 4) .. + 31), scale by 1/h and add into
//                the local expansions, then release the accumulator, while
//                the tensor cores already work on the next unit.
// Same arithmetic, offset groups and error behaviour as k_m2l_tc; every
// barrier wait is bounded as there.
// ---------------------------------------------------------------------------
#ifndef TCP_STAGES
#define TCP_STAGES 4
#endif
#ifndef TCP_LAG
#define TCP_LAG 2
#endif
#define TCP_EPI_WARPS 4
#define TCP_THREADS (32 * (TC_PROD_WARPS + 1 + TCP_EPI_WARPS))
#define TCP_SMEM (TCP_STAGES * TC_STAGE_BYTES + 1024)
#define TCP_TMEM_COLS 512

__global__ void __launch_bounds__(TCP_THREADS, 1) k_m2l_tcp(TcArgs g, int nunits)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                         ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t full_bar[TCP_STAGES], empty_bar[TCP_STAGES], accf_bar[2], acce_bar[2];
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int goff = g.noff / g.groups;
    const int nstage = goff * g.nkc;  // stages per unit
    const int nc = g.nc;

    if (tid == 0) {
        for (int s = 0; s < TCP_STAGES; ++s) {
            mbar_init(&full_bar[s], TC_PROD_WARPS + 1);  // one arrival per producer warp + the bulk copy's
            mbar_init(&empty_bar[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&accf_bar[b], 1);              // the MMA thread's commit
            mbar_init(&acce_bar[b], TCP_EPI_WARPS);  // one arrival per epilogue warp
        }
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == TC_PROD_WARPS) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(TCP_TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;

    if (warp < TC_PROD_WARPS) {
        // ---------------- producers ----------------
        const int row = warp * 32 + lane;  // this thread's target row of every tile
        int armed = 0;                     // stages with a bulk copy issued by this thread
        int it = 0;                        // global stage counter
        bool stop = false;
        for (int u = blockIdx.x; u < nunits && !stop; u += gridDim.x) {
            const int4 tile = g.tiles[u / g.groups];
            const int grp = u % g.groups;
            const int cl = tile.y;
            float ih_unused;
            const int my_tb = tc_tile_target(g, tile, row, ih_unused);
            const int rot = (u / g.groups) % goff;
            int my_src = -1;
            // the next stage's source is loaded one stage ahead
            int nxt_src = (my_tb >= 0) ? g.slots[(size_t)my_tb * g.noff + grp * goff + rot % goff] : -1;
            for (int j = 0; j < nstage; ++j, ++it) {
                const int s = it % TCP_STAGES, round = it / TCP_STAGES;
                const int oi = grp * goff + (j + rot) % goff, kc = g.nkc - 1 - j / goff;
                if (it >= TCP_STAGES) {
                    if (!mbar_wait(&empty_bar[s], (round - 1) & 1)) atomicExch(&s_abort, 1);
                }
                if (__any_sync(0xffffffffu, *(volatile int*)&s_abort)) {  // warp-uniform
                    stop = true;
                    break;
                }
                unsigned char* st = sm + (size_t)s * TC_STAGE_BYTES;
                if (row == 0) {
                    const int o = g.cls[cl * g.noff + oi];
                    mbar_arrive_tx(&full_bar[s], TC_AP * TC_A_BYTES);
                    bulk_g2s(st, g.A + ((size_t)o * TC_NKC + kc) * (TC_AP * TC_A_BYTES), TC_AP * TC_A_BYTES,
                             &full_bar[s]);
                    armed = it + 1;
                }
                my_src = nxt_src;
                if (my_tb >= 0) nxt_src = g.slots[(size_t)my_tb * g.noff + grp * goff + (j + 1 + rot) % goff];
                unsigned char* xs = st + TC_AP * TC_A_BYTES;
                const uint32_t xbase = smem_u32(xs);
#pragma unroll
                for (int i = 0; i < 2 * TC_RCH; ++i) {
                    const int piece = i / TC_RCH;
                    const int flat = (i % TC_RCH) * 32 + lane;  // chunk-major over the warp's 32 rows
                    const int rl = flat / TC_RCH, chunk = flat % TC_RCH;
                    const int src = __shfl_sync(0xffffffffu, my_src, rl);
                    const int r = warp * 32 + rl;
                    const uint32_t off = piece * TC_X_BYTES + swz16(r, chunk * 8);
                    if (src >= 0) {
                        const __half* gsrc = g.Ms + (size_t)blockIdx.y * g.ms_stride +
                                             ((size_t)src * TC_XP + piece) * TC_MROW + kc * TH_KC + chunk * 8;
                        cp_async16(xbase + off, gsrc);
                    } else {
                        *reinterpret_cast<float4*>(xs + off) = make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                }
                cp_async_commit();
                if (it >= TCP_LAG) {
                    cp_async_wait<TCP_LAG>();
                    fence_async_smem();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&full_bar[(it - TCP_LAG) % TCP_STAGES]);
                }
            }
        }
        cp_async_wait<0>();
        fence_async_smem();
        __syncwarp();
        if (lane == 0)
            for (int j = (it > TCP_LAG ? it - TCP_LAG : 0); j < it; ++j) mbar_arrive(&full_bar[j % TCP_STAGES]);
        // drain: the bulk copies this thread issued complete on their full barriers
        if (row == 0 && *(volatile int*)&s_abort) {
            for (int j = (armed > TCP_STAGES ? armed - TCP_STAGES : 0); j < armed; ++j)
                mbar_wait(&full_bar[j % TCP_STAGES], (j / TCP_STAGES) & 1);
        }
    } else if (warp == TC_PROD_WARPS) {
        // ---------------- MMA issuer ----------------
        if (lane == 0) {
            const uint32_t idesc = tc_idesc_f16(TC_M, TC_N);
            int it = 0, ul = 0;
            bool ok = true;
            for (int u = blockIdx.x; u < nunits && ok; u += gridDim.x, ++ul) {
                const int b = ul & 1;
                if (ul >= 2 && !mbar_wait(&acce_bar[b], ((ul >> 1) - 1) & 1)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t acc = tmem + (uint32_t)(b * TC_N);
                for (int j = 0; j < nstage; ++j, ++it) {
                    const int s = it % TCP_STAGES, round = it / TCP_STAGES;
                    if (!mbar_wait(&full_bar[s], round & 1)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t base = smem_u32(sm + (size_t)s * TC_STAGE_BYTES);
                    const uint32_t xb = base + TC_AP * TC_A_BYTES;
                    const int pa[3] = {1, 0, 0}, px[3] = {0, 1, 0};  // a2 x1, a1 x2, a1 x1
                    const int nks = (g.nk - (g.nkc - 1 - j / goff) * TH_KC) > 16 ? 2 : 1;
#pragma unroll
                    for (int prod = 0; prod < 3; ++prod) {
                        const uint32_t a = base + pa[prod] * TC_A_BYTES;
                        const uint32_t bb = xb + px[prod] * TC_X_BYTES;
#pragma unroll
                        for (int ks = 1; ks >= 0; --ks)
                            if (ks < nks)
                                tc_mma_f16(acc, smem_desc(a + 32 * ks), smem_desc(bb + 32 * ks), idesc,
                                           (j == 0 && prod == 0 && ks == nks - 1) ? 0u : 1u);
                    }
                    tc_commit(&empty_bar[s]);
                }
                if (!ok) break;
                tc_commit(&accf_bar[b]);
            }
            if (!ok) atomicExch(&s_abort, 1);
        }
        __syncwarp();
    } else {
        // ---------------- epilogue ----------------
        // (no barrier between the epilogue warps: each decides on its own,
        // so a warp that gives up on a timed-out wait cannot strand another)
        const int q = warp & 3;  // tensor-memory lanes 32 q .. 32 q + 31
        const int r = 32 * q + lane;
        const float rs = r < nc ? g.cscale[r] : 0.f;
        int ul = 0;
        for (int u = blockIdx.x; u < nunits; u += gridDim.x, ++ul) {
            const int b = ul & 1;
            const int4 tile = g.tiles[u / g.groups];
            const int cnt = tile.w;
            const bool ok = mbar_wait(&accf_bar[b], (ul >> 1) & 1);
            tc_fence_after();
            if (!ok || *(volatile int*)&s_abort) {
                if (lane == 0) atomicAdd(g.err, 1);
                atomicExch(&s_abort, 1);
                break;
            }
            float* Lb = g.L + (size_t)blockIdx.y * g.l_stride;
#pragma unroll 1
            for (int ch = 0; ch < TC_N / 32; ++ch) {
                const int col0 = ch * 32;
                if (col0 >= cnt) break;  // warp-uniform
                // target box of column col0 + lane, handed to every lane by shuffles
                const int jl = col0 + lane;
                float ihl;
                const int tbl = tc_tile_target(g, tile, jl, ihl);
                float v[32];
                tc_ld32(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(b * TC_N + col0), v);
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    const int tb = __shfl_sync(0xffffffffu, tbl, i);
                    const float ih = __shfl_sync(0xffffffffu, ihl, i);
                    if (r < nc && tb >= 0) atomicAdd(Lb + (size_t)tb * nc + r, v[i] * ih * rs);
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&acce_bar[b]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == TC_PROD_WARPS) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TCP_TMEM_COLS)
                     : "memory");
    }
}

// ---------------------------------------------------------------------------
// Host: operator blob and launch.
// ---------------------------------------------------------------------------
// Packed index of the K-th input coefficient, by degree, in pairs at even
// positions: Re and Im of (n, m) for m >= 1, and the real (n, 0) of two
// successive degrees (-1: no coefficient).  The reaction M2L forms its operators
// pair by pair (lfmm_m2r.cu).
void lf_coef_order(int p, std::vector<int>& perm)
{
    perm.clear();
    for (int n = 0; n <= p; ++n) {
        if (n & 1) {
            perm.push_back(lf_re(n - 1, 0));
            perm.push_back(lf_re(n, 0));
        }
        // (the pair of singles goes before the larger of its two degrees)
        for (int m = 1; m <= n; ++m) {
            perm.push_back(lf_re(n, m));
            perm.push_back(lf_im(p, n, m));
        }
    }
    if (!(p & 1)) {
        perm.push_back(lf_re(p, 0));
        perm.push_back(-1);
    }
}

// binary exponent of each packed coefficient's scale: log2 sqrt((n-m)! (n+m)!), rounded
void lf_coef_exponents(int p, std::vector<int>& e)
{
    const int nc = lf_nc(p);
    e.assign(nc, 0);
    for (int j = 0; j < nc; ++j) {
        int n, m, im;
        lf_decode(p, j, n, m, im);
        e[j] = (int)std::lround(0.5 * (std::lgamma(n - m + 1.0) + std::lgamma(n + m + 1.0)) / std::log(2.0));
    }
}

// Device operators A [nops][KP in][RP out] (FP64) -> the tensor-core operator
// blob: per operator nkc K chunks of two float16 pieces, each piece mh 128-row
// halves (mh = 2 for the wide form), pre-swizzled.  Entries are scaled by
// 2^{sin e_in - e_out} (sin = -1: multipoles in, +1: locals in) and by
// 2^TC_ASHIFT.  Scaled by the exponents they stay below 2 for every order (the
// factorials leave binomial coefficients of N over 2^{N+1} or less), so the
// pieces stay below 2^13; an entry beyond float16's range is counted in bad.
// One block per (operator, K chunk).
#define TC_ASHIFT 12
__global__ void __launch_bounds__(256) k_tc_blob(const double* __restrict__ A, int KP, int RP, int nc, int nk,
                                                 const int* __restrict__ perm, const float* __restrict__ cs, int sin,
                                                 int mh, unsigned char* __restrict__ blob, int* __restrict__ bad)
{
    const int nkc = mh * TC_NKC, o = blockIdx.x / nkc, kc = blockIdx.x % nkc;
    unsigned char* p0 = blob + (size_t)blockIdx.x * TC_AP * mh * TC_A_BYTES;
    for (int i = threadIdx.x; i < TH_KC * mh * TC_M; i += 256) {
        const int k = i / (mh * TC_M), r = i - k * (mh * TC_M), kk = kc * TH_KC + k;
        double v = 0.0;
        if (kk < nk && r < nc && perm[kk] >= 0) {
            const int kin = perm[kk];
            const double si = sin < 0 ? 1.0 / (double)cs[kin] : (double)cs[kin];
            v = A[((size_t)o * KP + kin) * RP + r] * si / (double)cs[r] * (double)(1 << TC_ASHIFT);
            if (!(fabs(v) < 60000.0)) atomicAdd(bad, 1);
        }
#pragma unroll
        for (int piece = 0; piece < TC_AP; ++piece) {
            const __half h = __float2half_rn((float)v);
            *reinterpret_cast<__half*>(p0 + ((size_t)piece * mh + r / TC_M) * TC_A_BYTES + swz16(r % TC_M, k)) = h;
            v -= (double)__half2float(h);
        }
    }
}

static LfErr tc_blob(lfmm_ctx* ctx, const DevBuf& A64, int nops, int KP, int RP, int sin, bool wide, DevBuf& out)
{
    const int mh = wide ? 2 : 1, nkc = mh * TC_NKC;
    LF_TRY(lf_reserve(out, (size_t)nops * nkc * TC_AP * mh * TC_A_BYTES));
    LF_TRY(lf_reserve(ctx->counts, 65536));
    int* bad = reinterpret_cast<int*>(ctx->counts.as<char>() + LFMM_TIMEOUT_OFF);
    LF_CHECK(cudaMemsetAsync(bad, 0, sizeof(int), ctx->s_main));
    ++ctx->launches, k_tc_blob<<<nops * nkc, 256, 0, ctx->s_main>>>(
        A64.as<double>(), KP, RP, lf_nc(ctx->p), ctx->tc_nk, ctx->tc_perm.as<int>(), ctx->tc_cscale.as<float>(), sin, mh,
        out.as<unsigned char>(), bad);
    LF_TRY(lf_cuda(cudaGetLastError(), "tensor-core operators"));
    int n = 0;
    LF_CHECK(lf_d2h(&n, bad, sizeof(int), ctx->s_main));
    return n ? LfErr("internal: tensor-core operator out of range") : LfErr();
}

// from the context's device operators m2l_A64 [343][KP][RP] and l2l_A64 [8][KP][RP]
LfErr lf_setup_m2l_tc(lfmm_ctx* ctx, int KP, int RP)
{
    const int nc = lf_nc(ctx->p);
    ctx->m2l_tc_ok = 0;
    ctx->m2l_tc_wide = 0;
    if (nc > 2 * TC_M || KP < nc || RP < nc) return LfErr();
    const bool wide = nc > TC_M;
    std::vector<int> e;
    lf_coef_exponents(ctx->p, e);
    std::vector<int> perm;
    lf_coef_order(ctx->p, perm);
    std::vector<float> cs(nc);
    for (int k = 0; k < nc; ++k) cs[k] = std::ldexp(1.f, e[k]);
    LF_TRY(lf_reserve(ctx->tc_cscale, nc * sizeof(float)));
    LF_CHECK(cudaMemcpy(ctx->tc_cscale.ptr, cs.data(), nc * sizeof(float), cudaMemcpyHostToDevice));
    // for every (N, mu) the smallest exponent its reaction table value is scaled
    // with: terms T(n + k, l + m) and T(n + k, |l - m|) of inputs (n, m), outputs (k, l)
    const int p = ctx->p, TS = 2 * p + 1;
    std::vector<int> emin((size_t)TS * TS, 1000);
    for (int n = 0; n <= p; ++n)
        for (int m = 0; m <= n; ++m)
            for (int k = 0; k <= p; ++k)
                for (int l = 0; l <= k; ++l) {
                    const int x = e[lf_re(n, m)] + e[lf_re(k, l)];
                    int& a = emin[(size_t)(n + k) * TS + l + m];
                    int& b = emin[(size_t)(n + k) * TS + std::abs(l - m)];
                    a = std::min(a, x);
                    b = std::min(b, x);
                }
    LF_TRY(lf_reserve(ctx->m2r_emin, emin.size() * sizeof(int)));
    LF_CHECK(cudaMemcpy(ctx->m2r_emin.ptr, emin.data(), emin.size() * sizeof(int), cudaMemcpyHostToDevice));
    ctx->tc_nk = (int)perm.size();
    LF_TRY(lf_reserve(ctx->tc_perm, perm.size() * sizeof(int)));
    LF_CHECK(cudaMemcpy(ctx->tc_perm.ptr, perm.data(), perm.size() * sizeof(int), cudaMemcpyHostToDevice));
    // the wide form serves the free M2L only; L2L stays on the CUDA cores
    // (the uploads above ran on the legacy stream, which s_main does not wait for)
    LF_CHECK(cudaDeviceSynchronize());
    LF_TRY(tc_blob(ctx, ctx->m2l_A64, TC_NALL, KP, RP, -1, wide, ctx->m2l_Atc));
    if (!wide) LF_TRY(tc_blob(ctx, ctx->l2l_A64, 8, KP, RP, 1, false, ctx->l2l_Atc));
    LF_CHECK(cudaFuncSetAttribute(k_m2l_tc<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM));
    LF_CHECK(cudaFuncSetAttribute(k_m2l_tc<false>, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
    LF_CHECK(cudaFuncSetAttribute(k_m2l_tc<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_WIDE_SMEM));
    LF_CHECK(cudaFuncSetAttribute(k_m2l_tc<true>, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
    LF_CHECK(cudaFuncSetAttribute(k_m2l_tcp, cudaFuncAttributeMaxDynamicSharedMemorySize, TCP_SMEM));
    LF_CHECK(cudaFuncSetAttribute(k_m2l_tcp, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
    int nsm = 0;
    LF_CHECK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device));
    ctx->num_sms = nsm > 0 ? nsm : 152;
    ctx->m2l_tc_wide = wide ? 1 : 0;
    ctx->m2l_tc_ok = 1;
    return LfErr();
}

// level of a global box id (levels are stored finest first)
struct TcLevels {
    int depth;
    int off[17];
};
__device__ __forceinline__ int tc_level(const TcLevels& lv, int b)
{
    int l = lv.depth;
    while (l > 0 && b >= lv.off[l - 1]) --l;
    return l;
}

// largest scaled magnitude |X_k| 2^{+-e_k} of the boxes b0 .. b0 + count - 1,
// per level, as float bits in gmax[32 rhs + slot0 + level] (zeroed when the
// charges were sorted); one warp per box, the block's boxes met in shared
// memory (one global atomic per box, or eight boxes per warp one after the
// other, took 10 to 15 us on any tree).
__global__ void __launch_bounds__(256) k_tc_max(const float* __restrict__ X, int nbox, int nc, int b0, int count,
                                                const float* __restrict__ cs, int inv,
                                                const __grid_constant__ TcLevels lv, int slot0,
                                                unsigned* __restrict__ gmax)
{
    __shared__ unsigned s_max[8];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, i = blockIdx.x * 8 + w;
    unsigned m = 0u;
    if (i < count) {
        const float* Xb = X + ((size_t)blockIdx.y * nbox + b0 + i) * nc;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int k = lane + 32 * q;
            if (k < nc) {
                const float c = cs[k];
                m = max(m, __float_as_uint(fabsf(Xb[k] * (inv ? 1.f / c : c))));
            }
        }
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) s_max[w] = m;
    __syncthreads();
    // the first warp of each level in the block takes the level's maximum on
    if (lane == 0 && i < count) {
        const int l = tc_level(lv, b0 + i);
        if (w > 0 && tc_level(lv, b0 + i - 1) == l) return;
        for (int v = w + 1; v < 8 && i + v - w < count && tc_level(lv, b0 + i + v - w) == l; ++v) m = max(m, s_max[v]);
        unsigned* g = gmax + (size_t)blockIdx.y * 32 + slot0 + l;
        if (m > *(volatile unsigned*)g) atomicMax(g, m);
    }
}

// expansions [box][nc] -> two scaled float16 pieces per box, rows padded to
// mrow halves (128, or 256 for the wide form) in K order, for the boxes b0 ..
// b0 + count - 1 (the arrays hold nbox boxes per right-hand side, blockIdx.y); one thread
// per 8 coefficients
__global__ void __launch_bounds__(256) k_split_m(const float* __restrict__ M, int nbox, int nc, int nk, int mrow, int b0,
                                                 int count, const float* __restrict__ cs, int inv,
                                                 const __grid_constant__ TcLevels lv,
                                                 int slot0, const unsigned* __restrict__ gmax,
                                                 const int* __restrict__ perm, __half* __restrict__ Ms)
{
    const int per = mrow / 8;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)count * per) return;
    M += (size_t)blockIdx.y * nbox * nc;
    Ms += (size_t)blockIdx.y * nbox * TC_XP * mrow;
    const int b = b0 + (int)(i / per), k0 = (int)(i % per) * 8;
    const float s = tc_scale(gmax[(size_t)blockIdx.y * 32 + slot0 + tc_level(lv, b)]);
    __align__(16) __half hi[8], lo[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
        const int k = k0 + u;
        float x = 0.f;
        const int j = k < nk ? perm[k] : -1;
        if (j >= 0) {
            x = M[(size_t)b * nc + j] * (inv ? 1.f / cs[j] : cs[j]) * s;
        }
        hi[u] = __float2half_rn(x);
        lo[u] = __float2half_rn(x - __half2float(hi[u]));
    }
    __half* out = Ms + (size_t)b * TC_XP * mrow + k0;
    *reinterpret_cast<uint4*>(out) = *reinterpret_cast<const uint4*>(hi);
    *reinterpret_cast<uint4*>(out + mrow) = *reinterpret_cast<const uint4*>(lo);
}

static int ms_row(const lfmm_ctx* ctx) { return ctx->m2l_tc_wide ? 2 * TC_MROW : TC_MROW; }
static unsigned* tc_gmax(lfmm_ctx* ctx) { return reinterpret_cast<unsigned*>(ctx->counts.as<char>() + LFMM_TCMAX_OFF); }

// scale and split the expansions of the boxes b0 .. b0 + count - 1: multipoles
// (locals = 0) or locals (1)
static LfErr split_boxes(lfmm_ctx* ctx, const float* src, int b0, int count, int locals, cudaStream_t st)
{
    if (count <= 0) return LfErr();
    static_assert(LFMM_TCMAX_OFF + LFMM_RHS_BATCH * 32 * 4 <= 65536, "counter buffer");
    const int nb = ctx->nbox_total, nr = ctx->nrhs_b, mrow = ms_row(ctx), nc = lf_nc(ctx->p);
    LF_TRY(lf_reserve(ctx->m2l_Ms, (size_t)nb * TC_XP * mrow * sizeof(__half) * nr));
    TcLevels lv;
    lv.depth = ctx->depth;
    for (int l = 0; l < 17; ++l) lv.off[l] = l <= ctx->depth ? ctx->levels[l].off : 0;
    unsigned* gm = tc_gmax(ctx);
    ++ctx->launches, k_tc_max<<<dim3((count + 7) / 8, nr), 256, 0, st>>>(
        src, nb, nc, b0, count, ctx->tc_cscale.as<float>(), locals, lv, 16 * locals, gm);
    const int64_t tot = (int64_t)count * (mrow / 8);
    ++ctx->launches, k_split_m<<<dim3((unsigned)((tot + 255) / 256), nr), 256, 0, st>>>(
        src, nb, nc, ctx->tc_nk, mrow, b0, count, ctx->tc_cscale.as<float>(), locals, lv, 16 * locals, gm,
        ctx->tc_perm.as<int>(), ctx->m2l_Ms.as<__half>());
    return lf_cuda(cudaGetLastError(), "split");
}

static TcArgs tc_args(lfmm_ctx* ctx)
{
    const int nb = ctx->nbox_total;
    TcArgs g;
    g.levelh = ctx->m2l_levelh.as<double>();
    g.mseg = ctx->tc_mseg.as<int4>();
    g.Ms = ctx->m2l_Ms.as<__half>();
    g.cscale = ctx->tc_cscale.as<float>();
    g.gmax = tc_gmax(ctx);
    g.ms_stride = (size_t)nb * TC_XP * ms_row(ctx);
    g.l_stride = (size_t)nb * lf_nc(ctx->p);
    g.nc = lf_nc(ctx->p);
    g.nk = ctx->tc_nk;
    g.nkc = (g.nk + TH_KC - 1) / TH_KC;
    g.err = reinterpret_cast<int*>(ctx->counts.as<char>() + LFMM_TIMEOUT_OFF);
    return g;
}

// the multipoles of every box as float16 pieces, for the free M2L and the
// keyed reaction M2L of this evaluation
LfErr lf_tc_split(lfmm_ctx* ctx, cudaStream_t st)
{
    return split_boxes(ctx, ctx->Mexp.as<float>(), 0, ctx->nbox_total, 0, st);
}

LfErr lf_m2l_tc(lfmm_ctx* ctx, cudaStream_t st)
{
    if (ctx->m2l_tc_ntiles == 0) return LfErr();
    const int nr = ctx->nrhs_b;
    TcArgs g = tc_args(ctx);
    g.gslot = 0;
    g.unscale = 1.f / (float)(1 << TC_ASHIFT);
    g.tiles = ctx->m2l_tc_tiles.as<int4>();
    g.sorted = ctx->m2l_sorted.as<int>();
    g.slots = ctx->m2l_slots.as<int>();
    g.cls = ctx->m2l_cls.as<int>();
    g.noff = TC_NOFF;
    g.unit_scale = 0;
    g.A = ctx->m2l_Atc.as<unsigned char>();
    g.L = ctx->Lexp.as<float>();
    // automatic: 9 offsets per accumulator, 3 in the wide form
    g.groups = ctx->tc_groups > 0 ? ctx->tc_groups : (ctx->m2l_tc_wide ? 63 : 21);
    const int nunits = ctx->m2l_tc_ntiles * g.groups;
    // the persistent form pays off when every SM walks many units; a small
    // tree (or one of many problems sharing the GPU in a batch) keeps one
    // CTA per unit, two of which share an SM
    if (ctx->m2l_tc_wide) {
        ++ctx->launches, k_m2l_tc<true><<<dim3(nunits, nr), TC_THREADS, TC_WIDE_SMEM, st>>>(g);
    } else if (ctx->tc_persistent && nunits * nr >= 4 * ctx->num_sms) {
        // one CTA per SM (shared memory and the 512 tensor-memory columns allow
        // no second); all right-hand sides share the SMs
        int per = std::max(1, ctx->num_sms / std::max(1, nr));
        per = std::min(per, nunits);
        ++ctx->launches, k_m2l_tcp<<<dim3(per, nr), TCP_THREADS, TCP_SMEM, st>>>(g, nunits);
    } else {
        ++ctx->launches, k_m2l_tc<false><<<dim3(nunits, nr), TC_THREADS, TC_SMEM, st>>>(g);
    }
    return lf_cuda(cudaGetLastError(), "m2l tensor-core gemm");
}

// L2L into the boxes at `level` (from their parents) on the tensor cores: the
// parents' locals are scaled and split first, the products added atomically
// onto the M2L results.
LfErr lf_l2l_tc(lfmm_ctx* ctx, int level, cudaStream_t st)
{
    const int t0 = ctx->tc_l2l_first[level], t1 = ctx->tc_l2l_first[level + 1];
    if (t1 <= t0) return LfErr();
    if (ctx->m2l_tc_wide) return LfErr("internal: tensor-core L2L needs (p+1)^2 <= 128");
    const LfmmLevel& src = ctx->levels[level - 1];
    LF_TRY(split_boxes(ctx, ctx->Lexp.as<float>(), src.off, src.nbox, 1, st));
    TcArgs g = tc_args(ctx);
    g.sorted = ctx->m2l_sorted.as<int>();
    g.slots = ctx->box_parent.as<int>();
    g.noff = 1;
    g.A = ctx->l2l_Atc.as<unsigned char>();
    g.L = ctx->Lexp.as<float>();
    g.groups = 1;
    g.gslot = 16 - 1;  // the parents' level
    g.unscale = 1.f / (float)(1 << TC_ASHIFT);
    g.tiles = ctx->tc_shift_tiles.as<int4>() + t0;
    g.cls = ctx->shift_cls.as<int>();
    g.unit_scale = 1;
    ++ctx->launches, k_m2l_tc<false><<<dim3((t1 - t0) * g.groups, ctx->nrhs_b), TC_THREADS, TC_SMEM, st>>>(g);
    return lf_cuda(cudaGetLastError(), "l2l tensor-core gemm");
}

// Self-check of the bounded-wait path: one thread waits on a barrier that
// expects two arrivals and gets one, so the wait must run out after `limit`
// cycles and count a timeout, exactly as a stalled pipeline stage would.
__global__ void k_wait_probe(long long limit, int* err)
{
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x != 0) return;
    mbar_init(&bar, 2);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_arrive(&bar);
    if (!mbar_wait_for(&bar, 0, limit)) atomicAdd(err, 1);
}

LfErr lf_wait_probe(lfmm_ctx* ctx, double limit_ms, int* timed_out)
{
    int khz = 0;  // SM clock; the GB300's maximum (2.07 GHz) if the runtime does not report it
    if (cudaDeviceGetAttribute(&khz, cudaDevAttrClockRate, ctx->device) != cudaSuccess) {
        (void)cudaGetLastError();
        khz = 0;
    }
    if (khz <= 0) khz = 2070000;
    const long long limit = (long long)(limit_ms * (double)khz);
    int* err = reinterpret_cast<int*>(ctx->counts.as<char>() + LFMM_TIMEOUT_OFF);
    LF_CHECK(cudaMemsetAsync(err, 0, sizeof(int), ctx->s_main));
    ++ctx->launches, k_wait_probe<<<1, 32, 0, ctx->s_main>>>(limit, err);
    LF_TRY(lf_cuda(cudaGetLastError(), "wait probe"));
    LF_CHECK(lf_d2h(timed_out, err, sizeof(int), ctx->s_main));
    LF_CHECK(cudaMemsetAsync(err, 0, sizeof(int), ctx->s_main));
    return LfErr();
}

int lf_m2l_tc_tile(const lfmm_ctx* ctx) { return ctx->m2l_tc_wide ? 128 : TC_N; }
