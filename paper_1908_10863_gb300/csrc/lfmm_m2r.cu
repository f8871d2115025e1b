// lfmm_m2r.cu -- reaction-component M2L (eqs. metoleimage1, coefintable)
// grouped by geometry key.
//
// The offset o = (t - P(s))/h of a reaction M2L pair, P the polarization map
// of the source box, is an integer vector up to a vertical fraction fixed per
// (component, level).  The translation then depends only on the key
// (component, level, offset): the Sommerfeld table of the pair (leading image
// in closed form + Gauss-Laguerre remainder, all (N, mu)) is computed once per
// (component, level, rho^2, oz) after a build, and at evaluation time the pairs
// of one key are applied together (Y = A_key X, X the gathered source
// multipoles), added atomically into the targets' local expansions.  The
// reflection sign (-1)^{n+m} of the multipole (s = -1 maps) and the
// (-1)^{N+mu} of an a = 2 component belong to A_key.
// The float32 form applies the keys on the tensor cores (k_m2r_tc), the FP64 form with p <= 15 by digit products there (k_m2r_oz),
// every other case in the rotated frame (k_m2r_rot).  A level with
// an entry outside the key range, and the coarser ones, keep the per-pair kernel.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
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

static inline int lf_blocks(int64_t n, int t) { return (int)((n + t - 1) / t); }

#define R_TB 64   // pairs per batch
#define R_T 256   // threads per block of the rotated form
#define RR_CB 16  // columns it stages at a time above p = 10
#define RT_PMAX 14  // largest order of the float32 form
#define KEY_NONE 0xffffffffu


// key = level (4 bits) | comp (7 bits) | offset index (12 bits, offsets in
// [-7, 7]^3): sorted keys group a level's keys together, so the keys of the
// levels left to the per-pair kernel are a prefix.  The offset index is oz, then
// the rank of (ox, oy) by rho^2, so the keys that share a table (one oz and
// rho^2) are neighbours.
#define R_OR 7
#define R_OW (2 * R_OR + 1)
#define R_LAT (R_OW * R_OW)
struct LatRank {
    unsigned char rank[R_LAT], lat[R_LAT];  // (ox + 7) 15 + (oy + 7) to rank, and back
    constexpr LatRank() : rank(), lat()
    {
        int n = 0;
        for (int r2 = 0; r2 <= 2 * R_OR * R_OR; ++r2)
            for (int i = 0; i < R_LAT; ++i) {
                const int x = i / R_OW - R_OR, y = i % R_OW - R_OR;
                if (x * x + y * y == r2) {
                    rank[i] = (unsigned char)n;
                    lat[n++] = (unsigned char)i;
                }
            }
    }
};
static constexpr LatRank h_lat = LatRank();
static __device__ const LatRank d_lat = LatRank();
__host__ __device__ __forceinline__ const LatRank& r_lat()
{
#ifdef __CUDA_ARCH__
    return d_lat;
#else
    return h_lat;
#endif
}
__host__ __device__ __forceinline__ uint32_t rkey(int c, int l, int ox, int oy, int oz)
{
    return ((uint32_t)l << 19) | ((uint32_t)c << 12) |
           (uint32_t)((oz + R_OR) * R_LAT + r_lat().rank[(ox + R_OR) * R_OW + (oy + R_OR)]);
}
__host__ __device__ __forceinline__ void rkey_decode(uint32_t key, int& c, int& l, int& ox, int& oy, int& oz)
{
    c = (int)((key >> 12) & 127u);
    l = (int)(key >> 19);
    int oi = (int)(key & 4095u);
    const int la = r_lat().lat[oi % R_LAT];
    ox = la / R_OW - R_OR;
    oy = la % R_OW - R_OR;
    oz = oi / R_LAT - R_OR;
}

// Keys of the reaction M2L entries of one level, from the boxes' grid cells.
// Lateral offsets are exact integers.  The vertical offset of the source's
// polarization image, in box units, (iz_t + 1/2) - s (iz_s + 1/2) - K, is
// n + f with the integer n = iz_t - s iz_s + base and the fraction f fixed per
// (component, level) (0 on levels where the interfaces are grid planes); the
// key holds n, the table is taken at n + f.  An entry outside the key's
// offset range counts in bad[level] (its level then stays per pair).
struct RkLevels {
    int depth;
    int off[17];  // first box of each level (finest first)
};
__global__ void k_m2r_keys(const LfmmComp* __restrict__ comps, int nb, const __grid_constant__ RkLevels lv,
                           const int4* __restrict__ grid, const int* __restrict__ zbase,
                           const int* __restrict__ rbeg, const int* __restrict__ rend,
                           const uint32_t* __restrict__ rent, uint32_t* __restrict__ keys,
                           uint32_t* __restrict__ vals, int* __restrict__ tgt, int* __restrict__ bad)
{
    // one warp per target box of the keyed levels, lanes over its entries
    const int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (t >= nb) return;
    int level = lv.depth;
    while (level > 0 && t >= lv.off[level - 1]) --level;
    const int4 gt = grid[t];
    for (int e = rbeg[t] + (threadIdx.x & 31); e < rend[t]; e += 32) {
        uint32_t v = rent[e];
        int c = (int)(v >> LFMM_ENT_SHIFT);
        int s = (int)(v & LFMM_ENT_MASK);
        const LfmmComp& cp = comps[c];
        const int4 gs = grid[s];
        const int sz = cp.s > 0.0 ? 1 : -1;
        const int ox = gt.x - gs.x, oy = gt.y - gs.y, oz = gt.z - sz * gs.z + zbase[c * 16 + level];
        const bool ok = ox >= -R_OR && ox <= R_OR && oy >= -R_OR && oy <= R_OR && oz >= -R_OR && oz <= R_OR;
        if (!ok) atomicAdd(bad + level, 1);
        keys[e] = ok ? rkey(c, level, ox, oy, oz) : KEY_NONE;
        vals[e] = (uint32_t)e;
        tgt[e] = t;
    }
}

__global__ void k_key_flags(const uint32_t* __restrict__ keys, int n, int* __restrict__ f)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    f[i] = (i == 0 || keys[i] != keys[i - 1]) ? 1 : 0;
}

__global__ void k_key_starts(const uint32_t* __restrict__ keys, int n, const int* __restrict__ f,
                             const int* __restrict__ idx, int* __restrict__ kstart, uint32_t* __restrict__ kval)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || !f[i]) return;
    kstart[idx[i]] = i;
    kval[idx[i]] = keys[i];
}

// Remainder values at the quadrature nodes: they depend on (component, level,
// oz) only, not on the lateral distance, so about 15 tables share them.  In
// media of four and five layers each is a solve of the interface problem and
// a coupling series, which took most of the tables' time (four layers, 2,808
// tables: 0.744 -> 0.331 + 0.080 ms).
template <bool GEN>
__global__ void __launch_bounds__(128) k_m2r_nodes(const LfmmComp* __restrict__ comps, const int4* __restrict__ ndesc,
                                                   int nnode, const double* __restrict__ levelh,
                                                   const double* __restrict__ zfrac, const double* __restrict__ gt,
                                                   int Q, double* __restrict__ out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nnode * Q) return;
    const int4 d = ndesc[i / Q];
    const int c = d.x, l = d.y, q = i % Q;
    const LfmmComp& cp = comps[c];
    if (!cp.has_rem) return;
    const double vz = (double)d.z + zfrac[c * 16 + l], zz = (cp.a == 1) ? vz : -vz;
    const double S = levelh[l];
    out[i] = lf_sigma_rem<GEN>(cp, gt[q] / (zz + cp.zeta_r / S) / S);
}

// One block per table: the box-unit table (lead + remainder) with the a = 2 sign.
// One Sommerfeld table per (component, level, rho^2, oz): the table depends on
// the lateral distance only; the azimuth enters through the phases applied
// when the operator is formed.  tdesc: component | level << 8, node set, rho^2, oz.
// tscale (p <= 15): the exponent s for which no entry of an operator made of the
// table, two values at most with their scales 2^{-e} (emin), reaches 2^{15 - s};
// tabf (p <= 14): the table times 2^s in float32, which k_m2r_tc reads (half the
// bytes, and no conversions on the FP64 pipe: applying s there instead cost it 1%).
__global__ void __launch_bounds__(128) k_m2r_tables(const LfmmComp* __restrict__ comps, const int4* __restrict__ tdesc,
                                                    int ntab, const double* __restrict__ levelh,
                                                    const double* __restrict__ zfrac, int P,
                                                    const double* __restrict__ gt, const double* __restrict__ gw, int Q,
                                                    const double* __restrict__ nodes, double* __restrict__ tables,
                                                    const int* __restrict__ emin, int* __restrict__ tscale,
                                                    float* __restrict__ tabf)
{
    __shared__ int s_exp;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int TS = 2 * P + 1, TT = TS * TS;
    double* sT = reinterpret_cast<double*>(smem_raw);
    double* sJ = sT + TT;
    double* sA = sJ + Q * TS;
    const int k = blockIdx.x;
    const int4 d = tdesc[k];
    const int c = d.x & 255, l = d.x >> 8, oz = d.w;
    const LfmmComp& cp = comps[c];
    const double rho = sqrt((double)d.z);
    const double vz = (double)oz + zfrac[c * 16 + l];  // image offset n + f in box units
    const double zz = (cp.a == 1) ? vz : -vz;
    for (int j = threadIdx.x; j < TT; j += blockDim.x) sT[j] = 0.0;
    if (threadIdx.x == 0) s_exp = -4096;
    __syncthreads();
    lf_sommerfeld_table_block<false>(cp, rho, zz, levelh[l], 2 * P, sT, TS, Q, gt, gw, sJ, sA,
                                     nodes + (size_t)d.y * Q);
    double* out = tables + (size_t)k * TT;
    int ex = -4096;  // largest binary exponent of a scaled value
    for (int j = threadIdx.x; j < TT; j += blockDim.x) {
        int N = j / TS, mu = j - N * TS;
        double v = (mu <= N) ? sT[j] : 0.0;
        if (cp.a == 2 && ((N + mu) & 1)) v = -v;
        out[j] = v;
        if (emin && mu <= N && v != 0.0)
            ex = max(ex, (int)(((unsigned)__double2hiint(v) >> 20) & 0x7ffu) - 1023 - emin[j]);
    }
    if (!emin) return;
    ex = __reduce_max_sync(0xffffffffu, ex);
    if ((threadIdx.x & 31) == 0) atomicMax(&s_exp, ex);
    __syncthreads();
    const int ts = max(-100, min(100, 13 - s_exp));  // (float32 powers of two)
    if (threadIdx.x == 0) tscale[k] = ts;
    if (!tabf) return;
    const double s = __hiloint2double((1023 + ts) << 20, 0);
    for (int j = threadIdx.x; j < TT; j += blockDim.x) {
        const int N = j / TS, mu = j - N * TS;
        const double v = (mu <= N) ? sT[j] * s : 0.0;
        tabf[(size_t)k * TT + j] = (float)((cp.a == 2 && ((N + mu) & 1)) ? -v : v);
    }
}

// ---------------------------------------------------------------------------
// Build-time preparation.
// ---------------------------------------------------------------------------
LfErr lf_prepare_m2r(lfmm_ctx* ctx, cudaStream_t st)
{
    ctx->m2r_nkeys = 0;
    ctx->m2r_nbatch = 0;
    ctx->m2r_ntab = 0;
    ctx->m2r_dev_pending = 0;
    ctx->stats[LFMM_STAT_REACTION_KEYS] = 0;
    ctx->stats[LFMM_STAT_REACTION_TABLES] = 0;
    ctx->m2r_keyed_from = ctx->depth + 1;
    ctx->m2r_pending_ne = 0;
    ctx->m2r_nent = 0;
    if (ctx->m2r_total == 0) return LfErr();
    // every level with reaction entries is keyed; a level some of whose
    // entries fall outside the key's offset range stays per pair (found at
    // lf_prepare_m2r_finish)
    int la = ctx->depth + 1;
    for (int l = 0; l <= ctx->depth; ++l)
        if (ctx->levels[l].m2r_count > 0) {
            la = l;
            break;
        }
    if (la > ctx->depth) return LfErr();
    ctx->m2r_la = la;
    // per (component, level): the image's vertical offset in box units is
    // iz_t - s iz_s + g with g = (1 - s)/2 - K, K = (o + (s - 1) z0)/h; split
    // as an integer base (for the keys) and a fraction in [0, 1) (for the tables)
    {
        static_assert(LFMM_PIN_M2R + LFMM_MAXCOMP * 16 * (sizeof(double) + sizeof(int)) <= LFMM_PIN_BYTES,
                      "pinned regions");
        double* zf = lf_pin<double>(ctx, LFMM_PIN_M2R);
        int* zb = lf_pin<int>(ctx, LFMM_PIN_M2R + LFMM_MAXCOMP * 16 * sizeof(double));
        for (int c = 0; c < LFMM_MAXCOMP; ++c)
            for (int l = 0; l < 16; ++l) {
                double g = 0.0;
                if (c < ctx->ncomp && l <= ctx->depth) {
                    const LfmmComp& cp = ctx->comp[c];
                    const double K = (cp.o + (cp.s - 1.0) * ctx->origin[2]) / ctx->levels[l].h;
                    g = 0.5 * (1.0 - cp.s) - K;
                }
                const double b = std::floor(g + 1e-9);
                zb[c * 16 + l] = (int)b;
                zf[c * 16 + l] = std::max(0.0, g - b);
            }
        LF_TRY(lf_reserve(ctx->m2r_zfrac, LFMM_MAXCOMP * 16 * sizeof(double)));
        LF_TRY(lf_reserve(ctx->m2r_zbase, LFMM_MAXCOMP * 16 * sizeof(int)));
        LF_CHECK(cudaMemcpyAsync(ctx->m2r_zfrac.ptr, zf, LFMM_MAXCOMP * 16 * sizeof(double), cudaMemcpyHostToDevice, st));
        LF_CHECK(cudaMemcpyAsync(ctx->m2r_zbase.ptr, zb, LFMM_MAXCOMP * 16 * sizeof(int), cudaMemcpyHostToDevice, st));
    }
    int64_t first = -1, last = -1;
    for (int l = la; l <= ctx->depth; ++l) {
        const LfmmLevel& lv = ctx->levels[l];
        if (lv.m2r_count == 0) continue;
        if (first < 0) first = lv.m2r_base;
        last = lv.m2r_base + lv.m2r_count;
    }
    if (first < 0) return LfErr();
    const int ne = (int)(last - first);
    LF_TRY(lf_reserve(ctx->m2r_keys, (size_t)ne * 4 + 16));
    LF_TRY(lf_reserve(ctx->m2r_order, (size_t)ne * 4 + 16));
    LF_TRY(lf_reserve(ctx->m2r_tgt, (size_t)ctx->m2r_total * 4 + 16));
    int* bad = reinterpret_cast<int*>(ctx->counts.as<char>() + 32768);  // [16 levels]
    LF_CHECK(cudaMemsetAsync(bad, 0, 16 * sizeof(int), st));
    // entries of levels la .. depth are contiguous: index them relative to `first`
    uint32_t* keys = ctx->m2r_keys.as<uint32_t>();
    uint32_t* vals = ctx->m2r_order.as<uint32_t>();
    {
        // levels la .. depth hold the box ids [0, end of la), finest first
        RkLevels lv;
        lv.depth = ctx->depth;
        for (int l = 0; l < 17; ++l) lv.off[l] = l <= ctx->depth ? ctx->levels[l].off : 0;
        const int nb = ctx->levels[la].off + ctx->levels[la].nbox;
        ++ctx->launches, k_m2r_keys<<<lf_blocks(nb, 4), 128, 0, st>>>(
            ctx->comp_dev.as<LfmmComp>(), nb, lv, ctx->box_grid.as<int4>(), ctx->m2r_zbase.as<int>(),
            ctx->m2r_off.as<int>(), ctx->m2r_off.as<int>() + ctx->nbox_total, ctx->m2r_ent.as<uint32_t>(),
            keys - first, vals - first, ctx->m2r_tgt.as<int>(), bad);
    }
    LF_TRY(lf_cuda(cudaGetLastError(), "m2r keys"));
    // vals hold absolute entry indices (e), keys sorted ascending
    // keys use bits 0..22 (level << 19 | component << 12 | offset): three digits
    LF_TRY(lf_radix_sort(ctx, keys, vals, ne, st, 0, 3, 1));
    LF_TRY(lf_reserve(ctx->flags, (size_t)ne * 4 + 16));
    LF_TRY(lf_reserve(ctx->idx, (size_t)ne * 4 + 16));
    int* fl = ctx->flags.as<int>();
    int* ix = ctx->idx.as<int>();
    ++ctx->launches, k_key_flags<<<lf_blocks(ne, 256), 256, 0, st>>>(keys, ne, fl);
    // the key count comes back with the last flag and scan value (pinned, no
    // wait here): the key arrays are sized for one key per entry
    int* klast = lf_pin<int>(ctx, LFMM_PIN_SCAN + 8);
    LF_CHECK(cudaMemcpyAsync(klast, fl + ne - 1, sizeof(int), cudaMemcpyDeviceToHost, st));
    LF_TRY(lf_scan_i32(ctx, fl, ix, ne, nullptr, st, 1));
    LF_CHECK(cudaMemcpyAsync(klast + 1, ix + ne - 1, sizeof(int), cudaMemcpyDeviceToHost, st));
    LF_TRY(lf_reserve(ctx->m2r_kstart, (size_t)(ne + 1) * 4));
    LF_TRY(lf_reserve(ctx->m2r_kval, (size_t)(ne + 1) * 4));
    ++ctx->launches, k_key_starts<<<lf_blocks(ne, 256), 256, 0, st>>>(keys, ne, fl, ix, ctx->m2r_kstart.as<int>(),
                                                                       ctx->m2r_kval.as<uint32_t>());
    LF_TRY(lf_cuda(cudaGetLastError(), "m2r key starts"));
    ctx->m2r_pending_ne = ne;  // the rest (key count, tables, batches) in lf_prepare_m2r_finish
    return LfErr();
}

// After lf_prepare_m2r: wait for its device part on st, read the keys back
// and set up the tables and batches.
LfErr lf_prepare_m2r_finish(lfmm_ctx* ctx, cudaStream_t st)
{
    const int ne = ctx->m2r_pending_ne;
    ctx->m2r_nent = ne;
    if (ne <= 0) return LfErr();
    ctx->m2r_pending_ne = 0;
    LF_CHECK(cudaStreamSynchronize(st));
    const int* klast = lf_pin<int>(ctx, LFMM_PIN_SCAN + 8);
    const int64_t nk = (int64_t)klast[0] + klast[1];
    int* bad = reinterpret_cast<int*>(ctx->counts.as<char>() + 32768);
    // key starts, key values and the per-level range counts come back into
    // the pinned buffer when they fit (one synchronisation), else into host
    // vectors (the pinned region's staged uploads are complete by now)
    const size_t pin_need = sizeof(int) * (2 * (size_t)nk + 17);
    const bool pinned = LFMM_PIN_M2R + pin_need <= LFMM_PIN_BYTES;
    std::vector<int>& kst_h = ctx->m2r_kstart_h;
    std::vector<uint32_t>& kv_h = ctx->m2r_kval_h;
    if (!pinned) {
        kst_h.resize(nk + 1);
        kv_h.resize(nk);
    }
    int* kstart = pinned ? lf_pin<int>(ctx, LFMM_PIN_M2R) : kst_h.data();
    uint32_t* kv = pinned ? lf_pin<uint32_t>(ctx, LFMM_PIN_M2R + sizeof(int) * (nk + 1)) : kv_h.data();
    int* hbad = pinned ? lf_pin<int>(ctx, LFMM_PIN_M2R + sizeof(int) * (2 * (size_t)nk + 1))
                       : lf_pin<int>(ctx, LFMM_PIN_SCAN + 16);
    LF_CHECK(cudaMemcpyAsync(kstart, ctx->m2r_kstart.ptr, sizeof(int) * nk, cudaMemcpyDeviceToHost, st));
    LF_CHECK(cudaMemcpyAsync(kv, ctx->m2r_kval.ptr, sizeof(uint32_t) * nk, cudaMemcpyDeviceToHost, st));
    LF_CHECK(cudaMemcpyAsync(hbad, bad, 16 * sizeof(int), cudaMemcpyDeviceToHost, st));
    LF_CHECK(cudaStreamSynchronize(st));
    kstart[nk] = ne;
    // levels from keyed_from on are keyed: below it, a level with an entry
    // outside the key range (and every coarser one) stays per pair.  Their
    // keys (sorted by level first) are a prefix, and the out-of-range ones
    // (KEY_NONE) the suffix
    int keyed_from = ctx->m2r_la;
    for (int l = ctx->m2r_la; l <= ctx->depth && l < 16; ++l)
        if (hbad[l] > 0) keyed_from = l + 1;
    ctx->m2r_keyed_from = keyed_from;
    int64_t k0 = 0, k1 = nk;
    while (k0 < nk && (int)(kv[k0] >> 19) < keyed_from) ++k0;  // (KEY_NONE >> 19 exceeds every level)
    while (k1 > k0 && kv[k1 - 1] == KEY_NONE) --k1;
    const int64_t nku = k1 - k0;
    ctx->m2r_kfirst = (int)k0;
    if (nku <= 0) return LfErr();
    // tables, one per distinct (component, level, rho^2, oz)
    std::vector<int4>& tdesc = ctx->m2r_tdesc_h;
    std::vector<int>& ktab = ctx->m2r_ktab_h;
    std::vector<int4>& ndesc = ctx->m2r_ndesc_h;
    tdesc.clear();
    ndesc.clear();
    ktab.assign(nku, 0);
    {
        // keys arrive sorted by (component, level, offset): within one
        // (component, level) run a table is identified by (rho^2, oz), looked
        // up in a direct-indexed slot array (a generation stamp instead of
        // clearing it per run); tables are numbered in order of first use
        constexpr int NR2 = 2 * R_OR * R_OR + 1;
        std::vector<int>& slot = ctx->m2r_slot_h;
        std::vector<uint32_t>& stamp = ctx->m2r_stamp_h;
        slot.assign((size_t)NR2 * R_OW, 0);
        stamp.assign((size_t)NR2 * R_OW, 0u);
        uint32_t gen = 0, run = ~0u;
        int node_of[R_OW];  // node set of each oz in the current (component, level) run
        for (int64_t k = k0; k < k1; ++k) {
            int c, l, ox, oy, oz;
            rkey_decode(kv[k], c, l, ox, oy, oz);
            if ((kv[k] >> 12) != run) {
                run = kv[k] >> 12;
                ++gen;
                std::fill(node_of, node_of + R_OW, -1);
            }
            const int r2 = ox * ox + oy * oy;
            const size_t i = (size_t)r2 * R_OW + (oz + R_OR);
            if (stamp[i] != gen) {
                stamp[i] = gen;
                slot[i] = (int)tdesc.size();
                int& node = node_of[oz + R_OR];
                if (node < 0) {
                    node = (int)ndesc.size();
                    ndesc.push_back(make_int4(c, l, oz, 0));
                }
                tdesc.push_back(make_int4(c | l << 8, node, r2, oz));
            }
            ktab[k - k0] = slot[i];
        }
    }
    const int ntab = (int)tdesc.size();
    const int P = ctx->p, TS = 2 * P + 1, TT = TS * TS;
    LF_TRY(lf_reserve(ctx->m2r_tables, (size_t)ntab * TT * 8 + 16));
    LF_TRY(lf_reserve(ctx->m2r_tdesc, (size_t)ntab * sizeof(int4) + 16));
    LF_TRY(lf_reserve(ctx->m2r_tscale, (size_t)ntab * sizeof(int) + 16));
    if (P <= RT_PMAX) LF_TRY(lf_reserve(ctx->m2r_tabf, (size_t)ntab * TT * sizeof(float) + 16));
    LF_TRY(lf_reserve(ctx->m2r_ndesc, ndesc.size() * sizeof(int4) + 16));
    LF_CHECK(cudaMemcpyAsync(ctx->m2r_tdesc.ptr, tdesc.data(), ntab * sizeof(int4), cudaMemcpyHostToDevice, st));
    LF_CHECK(cudaMemcpyAsync(ctx->m2r_ndesc.ptr, ndesc.data(), ndesc.size() * sizeof(int4), cudaMemcpyHostToDevice, st));
    double* hl = ctx->m2r_levelh_h;
    for (int l = 0; l < 16; ++l) hl[l] = (l <= ctx->depth) ? ctx->levels[l].h : 0.0;
    LF_TRY(lf_reserve(ctx->m2r_levelh, sizeof(double) * 16));
    LF_CHECK(cudaMemcpyAsync(ctx->m2r_levelh.ptr, hl, sizeof(double) * 16, cudaMemcpyHostToDevice, st));
    ctx->m2r_ntab = ntab;
    // batches of R_TB pairs of one key: key index, first sorted entry, count | key << 8, table
    std::vector<int4>& batches = ctx->m2r_batches_h;
    batches.clear();
    // (above p = 15, where only k_m2r_rot applies them: pairs of one table, as
    // many as it stages at a time, so that no block outlasts the others)
    const int most = P > 15 ? RR_CB : R_TB;
    for (int64_t k = k0, k2; k < k1; k = k2) {
        k2 = k + 1;
        while (P > 15 && k2 < k1 && ktab[k2 - k0] == ktab[k - k0]) ++k2;
        for (int s = kstart[k]; s < kstart[k2]; s += most)
            batches.push_back(make_int4((int)(k - k0), s, std::min(most, kstart[k2] - s) | (int)(kv[k] << 8),
                                        ktab[k - k0]));
    }
    ctx->m2r_nkeys = (int)nku;
    ctx->m2r_nbatch = (int)batches.size();
    LF_TRY(lf_reserve(ctx->m2r_batches, batches.size() * sizeof(int4) + 16));
    LF_CHECK(cudaMemcpyAsync(ctx->m2r_batches.ptr, batches.data(), batches.size() * sizeof(int4),
                             cudaMemcpyHostToDevice, st));
    // (the host staging vectors live in the context; the build synchronises at its end)
    ctx->stats[LFMM_STAT_REACTION_KEYS] = nku;
    ctx->stats[LFMM_STAT_REACTION_TABLES] = ntab;
    // the tables themselves are device work of the first
    // evaluation after this build (lf_m2r_device), beside its upward pass
    ctx->m2r_dev_pending = 1;
    return LfErr();
}

// Sommerfeld tables of the keys (FP64) and the keys' (source, target) pairs,
// enqueued on `st` (the first evaluation after a build
// runs this on the near-field stream, so it overlaps the far field's upward
// pass and free M2L; the reaction M2L waits for it).
// (source box, target box) of every reaction M2L entry in key order
__global__ void k_m2r_pairs(const uint32_t* __restrict__ order, const uint32_t* __restrict__ ent,
                            const int* __restrict__ tgt, int ne, int2* __restrict__ out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ne) return;
    const uint32_t e = order[i];
    out[i] = make_int2((int)(ent[e] & LFMM_ENT_MASK), tgt[e]);
}

LfErr lf_m2r_device(lfmm_ctx* ctx, cudaStream_t st)
{
    if (ctx->m2r_nbatch == 0 || ctx->m2r_ntab == 0) {
        ctx->m2r_dev_pending = 0;
        return LfErr();
    }
    const int ntab = ctx->m2r_ntab;
    const int P = ctx->p, TS = 2 * P + 1, TT = TS * TS, Q = ctx->gl_q_m2l;
    const size_t sm = sizeof(double) * ((size_t)TT + 2 * (size_t)Q * TS);
    constexpr int MS = 2 * LFMM_PMAX + 1;
    const int nnode = (int)ctx->m2r_ndesc_h.size();
    // (sized here: LFMM_OPT_QUAD_NODES may have changed Q since the build)
    LF_TRY(lf_reserve(ctx->m2r_nodes, (size_t)nnode * Q * sizeof(double) + 16));
    auto nodk = (ctx->L >= 3) ? k_m2r_nodes<true> : k_m2r_nodes<false>;
    ++ctx->launches, nodk<<<lf_blocks((int64_t)nnode * Q, 128), 128, 0, st>>>(
        ctx->comp_dev.as<LfmmComp>(), ctx->m2r_ndesc.as<int4>(), nnode, ctx->m2r_levelh.as<double>(),
        ctx->m2r_zfrac.as<double>(), ctx->gl_t_m2l.as<double>(), Q, ctx->m2r_nodes.as<double>());
    LF_TRY(lf_smem_limit(k_m2r_tables, sizeof(double) * (MS * MS + 2 * LFMM_QMAX * MS)));
    ++ctx->launches, k_m2r_tables<<<ntab, 128, sm, st>>>(
        ctx->comp_dev.as<LfmmComp>(), ctx->m2r_tdesc.as<int4>(), ntab, ctx->m2r_levelh.as<double>(),
        ctx->m2r_zfrac.as<double>(), P, ctx->gl_t_m2l.as<double>(), ctx->gl_w_m2l.as<double>(), Q,
        ctx->m2r_nodes.as<double>(), ctx->m2r_tables.as<double>(), ctx->m2r_emin.as<int>(),
        ctx->m2r_tscale.as<int>(), P <= RT_PMAX ? ctx->m2r_tabf.as<float>() : nullptr);
    LF_TRY(lf_cuda(cudaGetLastError(), "m2r tables"));
    if (ctx->m2r_nent > 0) {
        LF_TRY(lf_reserve(ctx->m2r_pairs, (size_t)ctx->m2r_nent * sizeof(int2) + 16));
        ++ctx->launches, k_m2r_pairs<<<lf_blocks(ctx->m2r_nent, 256), 256, 0, st>>>(
            ctx->m2r_order.as<uint32_t>(), ctx->m2r_ent.as<uint32_t>(), ctx->m2r_tgt.as<int>(), ctx->m2r_nent,
            ctx->m2r_pairs.as<int2>());
        LF_TRY(lf_cuda(cudaGetLastError(), "m2r pairs"));
    }
    ctx->m2r_dev_pending = 0;  // only once both are enqueued
    return LfErr();
}

// ---------------------------------------------------------------------------
// Evaluation in the rotated frame (FP64, and float32 off the tensor cores).
//
// Turned about z by the key's azimuth phi (M' = M e^{i m phi}, a diagonal),
// the coefficients of eq. coefintable are the real table T(N, |mu|), so the
// real parts of the locals see only real parts and the imaginary ones only
// imaginary parts:
//   Re L'(k, l) = (-1)^k sum_n [ T(n+k, l) Re M'(n, 0) + sum_m (T(n+k, m+l) + s T(n+k, |l-m|)) Re M'(n, m) ]
//   Im L'(k, l) = (-1)^k sum_n             sum_m (T(n+k, m+l) - s T(n+k, |l-m|)) Im M'(n, m)
// with s = (-1)^m for m <= l, (-1)^l beyond.  That is half the multiply-adds of
// the dense (p+1)^2 x (p+1)^2 operator, and the two entries come from two table
// values, so no operator is stored: the table (a few KB) stays in shared
// memory, and a pair of additions serves C columns.  The azimuth enters only
// with the columns, so pairs of every key that shares the table can be columns
// of one batch (above p = 15 they are).  One block per batch (and part of the rows); an item is one (k, l) for C columns,
// C the width in {2, 4, 8} that pads the batch least.
// FP64 (2 multiply-adds per clock and SM) bounds it.  Orders above 15 integrated a
// table per pair before: 2,848 charges, 6,910 pairs, p = 20: 27.0 ms -> 3.08 with
// batches of one key (4.6 pairs) and one block each, 2.53 with the rows in eight
// shares, 1.98 with the pairs of a table in batches of up to 16 and four shares.
// Float32, p = 14, 65,536 charges: 1.78 (stored operators and a GEMM) -> 0.83 ms.
// ---------------------------------------------------------------------------
#define RR_PH 32  // orders m <= 2p of p <= 15 (k_m2r_oz), m <= p of every other

struct RRotArgs {
    int p, nc, cb;          // order, coefficients, columns staged at a time
    const int4* batches;    // key index, first sorted entry, count | key << 8, table
    const double* tables;   // [table][TS][TS]
    const LfmmComp* comps;
    const double* phase;    // [225 lateral offsets][cos | sin][RR_PH]
    const uint32_t* keys;   // key of each sorted entry
    const int2* pairs;      // (source box, target box) per sorted entry
    const double* levelh;
    const void* M;
    void* L;
    size_t stride;          // expansions per right-hand side, in elements
    int nr;
};

// e^{i m phi}, m < RR_PH, of every lateral key offset, FP64
__global__ void k_m2r_phase64(double* out)
{
    const int b = blockIdx.x, m = threadIdx.x;
    const int ox = b / R_OW - R_OR, oy = b % R_OW - R_OR;
    const double phi = (ox == 0 && oy == 0) ? 0.0 : atan2((double)oy, (double)ox);
    double sn, cs;
    sincos(m * phi, &sn, &cs);
    out[(size_t)b * 2 * RR_PH + m] = cs;
    out[(size_t)b * 2 * RR_PH + RR_PH + m] = sn;
}

// columns [0, cnt) of the staged chunk, rows part of nparts
template <typename R, int C>
__device__ __forceinline__ void rr_apply(int p, int nc, const R* sT, const R* sXr, const R* sXi, int cb, int cnt,
                                         const int* s_tgt, const double* __restrict__ phase, const int* s_lat, R ih,
                                         R* __restrict__ L, int part, int nparts)
{
    const int nre = lf_nre(p), TS = 2 * p + 1;
    const int ng = (cnt + C - 1) / C, items = nre * ng;
    // an equal share of the items; which warps hold them turns with the block
    // (warps 0 and 1 of every block would share two of the SM's four FP64 units)
    const int i0 = items * part / nparts, i1 = items * (part + 1) / nparts;
    for (int it = i0 + (int)((threadIdx.x + 32 * blockIdx.x) & (R_T - 1)); it < i1; it += R_T) {
        const int row = it / ng, c0 = (it - row * ng) * C;
        int k, l, dummy;
        lf_decode(p, row, k, l, dummy);
        R ar[C], ai[C];
#pragma unroll
        for (int c = 0; c < C; ++c) ar[c] = ai[c] = R(0);
        const R* xr = sXr + c0;
        const R* xi = sXi + c0;
        for (int n = 0; n <= p; ++n) {
            const R* Tr = sT + (n + k) * TS;
            {
                const R e = Tr[l];
#pragma unroll
                for (int c = 0; c < C; ++c) ar[c] += e * xr[c];
                xr += cb;
                xi += cb;
            }
#pragma unroll 2
            for (int m = 1; m <= n; ++m) {
                const int d = l - m;
                const R t1 = Tr[m + l];
                R t2 = Tr[d < 0 ? -d : d];
                if ((d < 0 ? l : m) & 1) t2 = -t2;
                const R er = t1 + t2, ei = t1 - t2;
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    ar[c] += er * xr[c];
                    ai[c] += ei * xi[c];
                }
                xr += cb;
                xi += cb;
            }
        }
        const R sg = (k & 1) ? -ih : ih;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            if (c0 + c >= cnt) break;
            R* Lt = L + (size_t)s_tgt[c0 + c] * nc;
            const double* ph = phase + (size_t)s_lat[c0 + c] * 2 * RR_PH + l;
            const R cr = sg * (R)ph[0], sr = sg * (R)ph[RR_PH];
            atomicAdd(Lt + row, cr * ar[c] - sr * ai[c]);
            if (l > 0) atomicAdd(Lt + lf_im(p, k, l), sr * ar[c] + cr * ai[c]);
        }
    }
}

template <typename R>
__global__ void __launch_bounds__(R_T) k_m2r_rot(RRotArgs g)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_src[R_TB], s_tgt[R_TB], s_lat[R_TB];
    const int p = g.p, nc = g.nc, nre = lf_nre(p), TS = 2 * p + 1, cb = g.cb, tid = threadIdx.x;
    R* sXr = reinterpret_cast<R*>(smem_raw);  // [(n, m)][cb]
    R* sXi = sXr + nre * cb;
    R* sT = sXi + nre * cb;  // [TS][TS]
    const int4 b = g.batches[blockIdx.x];
    const int start = b.y, cnt = b.z & 255;
    int c, lev, ox, oy, oz;
    rkey_decode((uint32_t)b.z >> 8, c, lev, ox, oy, oz);
    const bool refl = g.comps[c].refl != 0;
    const R ih = (R)(1.0 / g.levelh[lev]);
    if (tid < R_TB) {
        const int2 pr = (tid < cnt) ? g.pairs[start + tid] : make_int2(-1, -1);
        s_src[tid] = pr.x;
        s_tgt[tid] = pr.y;
        int c1, l1;
        rkey_decode(g.keys[start + min(tid, cnt - 1)], c1, l1, ox, oy, oz);
        s_lat[tid] = (ox + R_OR) * R_OW + (oy + R_OR);
    }
    const double* Tk = g.tables + (size_t)b.w * TS * TS;
    for (int j = tid; j < TS * TS; j += R_T) sT[j] = (R)Tk[j];
    for (int r = 0; r < g.nr; ++r) {
        const R* M = reinterpret_cast<const R*>(g.M) + (size_t)r * g.stride;
        R* L = reinterpret_cast<R*>(g.L) + (size_t)r * g.stride;
        for (int q0 = 0; q0 < cnt; q0 += cb) {
            const int nq = min(cb, cnt - q0);
            __syncthreads();  // the tables are in shared memory; the previous chunk has been read
            // rotated (and for reflections sign-flipped) multipoles; columns past the batch: zeros
            for (int i = tid; i < nre * cb; i += R_T) {
                const int j = i / nre, x = i - j * nre;  // column, (n, m)
                R vr = R(0), vi = R(0);
                if (j < nq) {
                    int n, m, dummy;
                    lf_decode(p, x, n, m, dummy);
                    const R* Ms = M + (size_t)s_src[q0 + j] * nc;
                    const R mr = Ms[x], mi = m > 0 ? Ms[lf_im(p, n, m)] : R(0);
                    const double* ph = g.phase + (size_t)s_lat[q0 + j] * 2 * RR_PH + m;
                    const R cm = (R)ph[0], sm = (R)ph[RR_PH];
                    vr = mr * cm - mi * sm;
                    vi = mr * sm + mi * cm;
                    if (refl && ((n + m) & 1)) {
                        vr = -vr;
                        vi = -vi;
                    }
                }
                sXr[x * cb + j] = vr;
                sXi[x * cb + j] = vi;
            }
            __syncthreads();
            // padded cost of each width: two additions and 2 C multiply-adds per (n, m)
            const int w2 = ((nq + 1) / 2) * 6, w4 = ((nq + 3) / 4) * 10, w8 = ((nq + 7) / 8) * 18;
            if (w8 <= w4 && w8 <= w2)
                rr_apply<R, 8>(p, nc, sT, sXr, sXi, cb, nq, s_tgt + q0, g.phase, s_lat + q0, ih, L, blockIdx.y,
                               gridDim.y);
            else if (w4 <= w2)
                rr_apply<R, 4>(p, nc, sT, sXr, sXi, cb, nq, s_tgt + q0, g.phase, s_lat + q0, ih, L, blockIdx.y,
                               gridDim.y);
            else
                rr_apply<R, 2>(p, nc, sT, sXr, sXi, cb, nq, s_tgt + q0, g.phase, s_lat + q0, ih, L, blockIdx.y,
                               gridDim.y);
        }
    }
}

// ---------------------------------------------------------------------------
// Tensor-core form (float32, p <= 14): one CTA per batch of up to R_TB pairs
// of one key, and per 128-row part of the outputs where (p+1)^2 > 128 (the wide
// form: one vector at a time, the two correction products in an accumulator of
// their own, as in the free M2L's).  The key's operator is never stored: the CTA forms
// it in shared memory from the key's Sommerfeld table and the lateral phases,
// directly as two float16 pieces a1 + a2 in the 64-byte-swizzled K-major layout
// of the MMA's A operand (M = 128 output coefficients, K = the input
// coefficients by falling degree in chunks of 32), scaled like the free M2L's
// operators (lfmm_m2l_tc.cu: 2^{-e} per coefficient, folded into the signs
// below) and by a power of two of the table's own (tscale): the image series of
// a thin layer of high permittivity adds up to thousands, weak reflections to
// little, and float16 has five exponent bits.  The source multipoles (B operand) are the scaled float16 pieces
// which that M2L split once per evaluation, gathered by 16-byte cp.async;
// products a2 x1 + a1 x2 + a1 x1.  Operator entries come from a table W of the
// complex reaction coefficient extended to negative orders.  They are formed in
// blocks of two rows (Re and Im of an output (k, l)) by two columns (Re and Im
// of an input (n, m)): the four entries are sums and differences of the parts
// of W(n+k, l+m) and W(n+k, l-m), so a block costs two 8-byte loads (one entry
// at a time took two 4-byte loads and two of offsets and signs each, and the
// shared-memory pipe bounded the kernel).  Orders m = 0 have one part only; two
// of them share a row or column pair.  While the tensor cores take one chunk
// the threads form the next.
//   V = 1: one vector, A and X of a chunk in two buffers (48 KB), three CTAs
// per SM, which leaves room for the near field beside it.
//   V = 2: several vectors; the whole operator (64 KB) is formed once and kept,
// and the vectors stream past it two at a time, two CTAs per SM.
// The eight warps read the accumulator back (warp w: lanes 32 (w mod 4) ..,
// every second 32-column block), scale it by 1/h and the inverse operand
// scales and add it into the targets' local expansions.  Every wait is
// bounded: on a timeout the CTA counts it in err and skips its read-backs.
// Measured, p = 10, float16 pieces against TF32 pieces with the operator formed
// again for every vector: 64 vectors of 262,144 charges 13.8 -> 4.95 ms.  One
// vector, N = 1M: 0.258 ms with entries formed one at a time, 0.17 to 0.19 in blocks.
// The wide form, 65,536 charges, p = 14: 0.825 ms (k_m2r_rot) -> 0.52 ms, the
// evaluation's difference from the FP64 form unchanged (3.2e-7).
// ---------------------------------------------------------------------------
#define RT_THREADS 256
#define RT_PH 32                        // stride of the phase table (orders m <= 2p <= 28)
#define RT_NKC 4                        // K chunks at most where the operator is kept
#define RT_A_CHUNK (128 * TC_ROWB)      // one K chunk of one operator piece: 128 rows x 64 B
#define RT_X_CHUNK (R_TB * TC_ROWB)     // one K chunk of one multipole piece and vector: 64 rows x 64 B
template <int V, bool WIDE>
struct RtShape {
    static constexpr int P = WIDE ? RT_PMAX : 10;                   // largest order
    static constexpr int W = (2 * P + 1) * (4 * P + 1);        // entries of the table W
    static constexpr int CP = WIDE ? 128 : 64;                 // column pairs
    static constexpr int MROW = WIDE ? 256 : 128;              // halves per box and multipole piece
    static constexpr bool KEEP = V > 1;                        // operator kept for all vectors
    static constexpr int NA = KEEP ? RT_NKC : 2;               // operator chunks in shared memory
    static constexpr int XB = 2 * V * RT_X_CHUNK;              // multipole bytes of a chunk: two pieces
    static constexpr int SMEM = NA * 2 * RT_A_CHUNK + 2 * XB + 512;
    static constexpr int MINB = KEEP ? 2 : 3;                  // resident CTAs per SM
    static constexpr uint32_t COLS = WIDE ? 128 : 64 * V;      // tensor-memory columns
};

struct RTcArgs {
    int p, nc, nk, nkc;     // order, coefficients, K positions, chunks of 32 that hold them
    int parts;              // 128-row parts of the outputs
    const int4* batches;    // key index, first sorted entry, count | key << 8, table
    const float* tables;    // [table][TS][TS], times 2^tscale (k_m2r_tables)
    const int* tscale;      // per table
    const LfmmComp* comps;
    const float* phase;     // [225 lateral offsets][cos | sin][RT_PH] (k_m2r_phase)
    const int2* pairs;      // (source box, target box) per sorted entry (k_m2r_pairs)
    const double* levelh;
    const __half* Ms;       // split multipoles [box][2 pieces][MROW]
    const float* cscale;    // 2^e per packed coefficient
    const int* perm;        // packed index of each K position (and row), -1: none
    const unsigned* gmax;   // largest scaled multipole per level (float bits), [32] per right-hand side
    float* L;
    size_t ms_stride, stride;  // per right-hand side: halves of Ms, floats of L
    int nr;
    int* err;               // [0]: timeouts
};

// e^{i m phi} of every lateral key offset (ox, oy) in [-7, 7]^2, m <= 2p:
// FP64 sincos rounded to float32, [offset][cos | sin][RT_PH]
__global__ void k_m2r_phase(int p, float* out)
{
    const int b = blockIdx.x, m = threadIdx.x;
    if (m > 2 * p) return;
    const int ox = b / R_OW - R_OR, oy = b % R_OW - R_OR;
    const double phi = (ox == 0 && oy == 0) ? 0.0 : atan2((double)oy, (double)ox);
    double sn, cs;
    sincos(m * phi, &sn, &cs);
    out[(size_t)b * 2 * RT_PH + m] = (float)cs;
    out[(size_t)b * 2 * RT_PH + RT_PH + m] = (float)sn;
}

__device__ __forceinline__ float rt_pow2(int e) { return __int_as_float((e + 127) << 23); }  // |e| <= 126

template <int V, bool WIDE>
__global__ void __launch_bounds__(RT_THREADS, RtShape<V, WIDE>::MINB) k_m2r_tc(RTcArgs g)
{
    typedef RtShape<V, WIDE> S;
    extern __shared__ unsigned char smem_raw[];
    // 512-byte alignment: the period of the 64-byte swizzle
    unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 511) &
                                                         ~(uintptr_t)511);
    unsigned char* smx = sm + S::NA * 2 * RT_A_CHUNK;
    // W(N, mu) = 2^tscale T(N, |mu|) e^{i mu phi} for mu in [-2p, 2p], extended to
    // negative orders by W(N, -mu) = (-1)^mu conj W(N, mu); [N][mu + 2p], rows of 4p + 1
    __shared__ float2 sW[S::W];
    __shared__ float sPh[2 * RT_PH];
    // column pairs: offsets of the two W terms from the row's, their signs and
    // scales; y < 0: two real inputs (n, 0), -1 - offset of the second
    __shared__ int2 s_co[S::CP];
    __shared__ float2 s_cf[S::CP];
    // row pairs (rows t and 64 + t): packed rows (-1: none), offsets; z == w: Re and Im of one (k, l)
    __shared__ int4 s_row[64];
    __shared__ float2 s_rk[64];  // (-1)^k with the rows' scales
    __shared__ int s_prow[128];
    __shared__ int s_src[R_TB], s_tgt[R_TB];
    __shared__ __align__(8) uint64_t bar[2];
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    __shared__ float s_as;  // 2^-tscale
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int p = g.p, nc = g.nc, nkc = g.nkc, TS = 2 * p + 1, WS = 4 * p + 1, TSZ = TS * WS;
    const int part = WIDE ? blockIdx.x % g.parts : 0;
    const int4 b = g.batches[WIDE ? blockIdx.x / g.parts : blockIdx.x];
    // the batch carries its key and table: one dependent load to everything else
    const int start = b.y, cnt = b.z & 255, tab = b.w;
    if (cnt <= 0 || cnt > R_TB) return;
    const int Np = (cnt + 15) & ~15;  // columns per vector
    int c, lev, ox, oy, oz;
    rkey_decode((uint32_t)b.z >> 8, c, lev, ox, oy, oz);
    const bool refl = g.comps[c].refl != 0;

    if (tid < 64) {
        // row pair of this part: Re and Im of a (k, l), or two (k, 0)
        const int i = 128 * part + 2 * tid;
        int4 r = make_int4(-1, -1, 0, 0);
        float2 sk = make_float2(0.f, 0.f);
        if (i < g.nk) {
            r.x = g.perm[i];
            r.y = g.perm[i + 1];
            int k, l, im;
            lf_decode(p, r.x, k, l, im);
            r.z = r.w = k * WS + l + 2 * p;
            sk.x = sk.y = ((k & 1) ? -1.f : 1.f) / g.cscale[r.x];
            if (l == 0) {
                r.w = -1;  // (not an Re / Im pair)
                sk.y = 0.f;
                if (r.y >= 0) {
                    lf_decode(p, r.y, k, l, im);
                    r.w = k * WS + l + 2 * p;
                    sk.y = ((k & 1) ? -1.f : 1.f) / g.cscale[r.y];
                }
            }
        }
        s_row[tid] = r;
        s_rk[tid] = sk;
        s_prow[tid] = r.x;
        s_prow[64 + tid] = r.y;
    } else if (tid >= RT_THREADS - S::CP) {
        // column pair: K positions 2c and 2c + 1
        const int cc = tid - (RT_THREADS - S::CP), c2 = 2 * cc;
        int2 o = make_int2(0, 0);
        float2 f = make_float2(0.f, 0.f);
        if (c2 < g.nk) {
            const int j0 = g.perm[c2], j1 = g.perm[c2 + 1];
            int n, m, im;
            lf_decode(p, j0, n, m, im);
            // the multipole's reflection sign (-1)^{n+m} for s = -1 maps, and (-1)^m of the second term
            const float c = (refl && ((n + m) & 1) ? -1.f : 1.f) / g.cscale[j0];
            if (m > 0) {
                o = make_int2(n * WS + m, n * WS - m);
                f = make_float2(c, (m & 1) ? -c : c);
            } else {
                o.x = n * WS;
                f.x = c;
                o.y = -1;
                if (j1 >= 0) {
                    int n1;
                    lf_decode(p, j1, n1, m, im);
                    o.y = -1 - n1 * WS;
                    f.y = (refl && (n1 & 1) ? -1.f : 1.f) / g.cscale[j1];
                }
            }
        }
        s_co[cc] = o;
        s_cf[cc] = f;
    }
    if (tid < R_TB) {
        const int2 pr = (tid < cnt) ? g.pairs[start + tid] : make_int2(-1, -1);
        s_src[tid] = pr.x;
        s_tgt[tid] = pr.y;
    }
    else if (tid < R_TB + 2 * RT_PH)
        sPh[tid - R_TB] = g.phase[(size_t)((ox + R_OR) * R_OW + (oy + R_OR)) * 2 * RT_PH + (tid - R_TB)];
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(S::COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        s_abort = 0;
        s_as = rt_pow2(-g.tscale[tab]);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    {
        const float* Tk = g.tables + (size_t)tab * TS * TS;
        for (int j = tid; j < TSZ; j += RT_THREADS) {
            const int Nn = j / WS, mu = j - Nn * WS - 2 * p, a = mu < 0 ? -mu : mu;
            const float t = Tk[Nn * TS + a];
            float wr = t * sPh[a], wi = t * sPh[RT_PH + a];
            if (mu < 0) {
                if (a & 1) wr = -wr; else wi = -wi;
            }
            sW[j] = make_float2(wr, wi);
        }
    }
    const double hl = g.levelh[lev];
    __syncthreads();  // W is in shared memory
    // gather unit of every chunk: row xj, 16-byte quarter xq; operator unit: row pair xj, quarter xq
    const int xj = tid >> 2, xq = tid & 3;
    const int src = xj < Np ? s_src[xj] : -1;
    const int4 rw = s_row[xj];
    const float2 rk = s_rk[xj];
    bool ok = true;
    int gr = 0;  // round counter over the vectors
    for (int r0 = 0; r0 < g.nr && ok; r0 += V) {
        const int nv = min(V, g.nr - r0);  // vectors of this pass
        const uint32_t idesc = tc_idesc_f16(128, nv * Np);
        for (int i = 0; i < nkc; ++i, ++gr) {
            const int kc = nkc - 1 - i, buf = gr & 1;  // falling degree
            if (gr >= 2 && !mbar_wait(&bar[buf], (uint32_t)(((gr - 2) >> 1) & 1))) s_abort = 1;
            unsigned char* sa = sm + (size_t)(S::KEEP ? kc : buf) * 2 * RT_A_CHUNK;
            unsigned char* sx = smx + (size_t)buf * S::XB;
            if (xj < Np) {
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    if (v >= nv) break;
                    const __half* gs = g.Ms + (size_t)(r0 + v) * g.ms_stride +
                                       (size_t)(src >= 0 ? src : 0) * (2 * S::MROW) + kc * TH_KC + xq * 8;
                    const uint32_t off = swz16(v * Np + xj, xq * 8);
#pragma unroll
                    for (int piece = 0; piece < 2; ++piece) {
                        unsigned char* dst = sx + piece * V * RT_X_CHUNK + off;
                        if (src >= 0)
                            cp_async16(smem_u32(dst), gs + piece * S::MROW);
                        else
                            *reinterpret_cast<float4*>(dst) = make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                }
            }
            cp_async_commit();
            if ((!S::KEEP || r0 == 0) && rw.x >= 0) {
                __align__(16) __half2 ha[4], la[4], hb[4], lb[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int cp = kc * (TH_KC / 2) + 4 * xq + e;
                    const int2 o = s_co[cp];
                    const float2 f = s_cf[cp];
                    const bool sg = o.y < 0;  // two real inputs
                    const int o2 = sg ? -1 - o.y : o.y;
                    const float2 x = sW[rw.z + o.x], y = sW[rw.z + o2];
                    float a0, a1, b0, b1;
                    if (rw.z == rw.w) {  // Re and Im of one output
                        const float fy = sg ? 0.f : f.y;
                        a0 = fmaf(f.x, x.x, fy * y.x);
                        b0 = fmaf(f.x, x.y, fy * y.y);
                        a1 = sg ? f.y * y.x : fmaf(-f.x, x.y, f.y * y.y);
                        b1 = sg ? f.y * y.y : fmaf(f.x, x.x, -f.y * y.x);
                    } else {  // two real outputs
                        const int w2 = max(rw.w, 0);
                        const float2 x2 = sW[w2 + o.x], y2 = sW[w2 + o2];
                        a0 = sg ? f.x * x.x : fmaf(f.x, x.x, f.y * y.x);
                        a1 = sg ? f.y * y.x : fmaf(-f.x, x.y, f.y * y.y);
                        b0 = sg ? f.x * x2.x : fmaf(f.x, x2.x, f.y * y2.x);
                        b1 = sg ? f.y * y2.x : fmaf(-f.x, x2.y, f.y * y2.y);
                    }
                    a0 *= rk.x;
                    a1 *= rk.x;
                    b0 *= rk.y;
                    b1 *= rk.y;
                    ha[e] = __floats2half2_rn(a0, a1);
                    hb[e] = __floats2half2_rn(b0, b1);
                    const float2 fa = __half22float2(ha[e]), fb = __half22float2(hb[e]);
                    la[e] = __floats2half2_rn(a0 - fa.x, a1 - fa.y);
                    lb[e] = __floats2half2_rn(b0 - fb.x, b1 - fb.y);
                }
                // (rows past the last coefficient are never read back)
                uint32_t off = swz16(xj, 8 * xq);
                *reinterpret_cast<uint4*>(sa + off) = *reinterpret_cast<const uint4*>(ha);
                *reinterpret_cast<uint4*>(sa + RT_A_CHUNK + off) = *reinterpret_cast<const uint4*>(la);
                if (rw.y >= 0) {
                    off = swz16(64 + xj, 8 * xq);
                    *reinterpret_cast<uint4*>(sa + off) = *reinterpret_cast<const uint4*>(hb);
                    *reinterpret_cast<uint4*>(sa + RT_A_CHUNK + off) = *reinterpret_cast<const uint4*>(lb);
                }
            }
            cp_async_wait<0>();
            fence_async_smem();
            tc_fence_before();
            __syncthreads();
            if (*(volatile int*)&s_abort) {  // block-uniform after the barrier
                ok = false;
                break;
            }
            if (tid == 0) {
                tc_fence_after();
                const uint32_t a0 = smem_u32(sa), x0 = smem_u32(sx);
                const int nks = (g.nk - kc * TH_KC) > 16 ? 2 : 1;
#pragma unroll
                for (int prod = 0; prod < 3; ++prod) {  // a2 x1, a1 x2, a1 x1
                    const uint32_t a = a0 + (prod == 0 ? RT_A_CHUNK : 0);
                    const uint32_t x = x0 + (prod == 1 ? V * RT_X_CHUNK : 0);
                    const uint32_t acc = tmem + (WIDE && prod < 2 ? 64 : 0);
#pragma unroll
                    for (int ks = 1; ks >= 0; --ks)
                        if (ks < nks)
                            tc_mma_f16(acc, smem_desc(a + 32 * ks), smem_desc(x + 32 * ks), idesc,
                                       (i == 0 && (prod == 0 || (WIDE && prod == 2)) && ks == nks - 1) ? 0u : 1u);
                }
                tc_commit(&bar[buf]);
            }
            __syncwarp();
        }
        // the last round's commit covers every MMA before it
        bool got = false;
        if (ok) got = mbar_wait(&bar[(gr - 1) & 1], (uint32_t)(((gr - 1) >> 1) & 1));
        ok = __syncthreads_and(got) != 0;  // block-uniform
        tc_fence_after();
        if (ok) {
            const int q4 = warp & 3, row = s_prow[32 * q4 + lane];
            const float rs = row >= 0 ? g.cscale[row] : 0.f;
            float sc[V];
#pragma unroll
            for (int v = 0; v < V; ++v)
                sc[v] = rs * (float)(1.0 / hl) /
                        tc_scale(g.gmax[(size_t)min(r0 + v, g.nr - 1) * 32 + lev]) * s_as;
            for (int c0 = 32 * (warp >> 2); c0 < nv * Np; c0 += 64) {
                float v[32];
                tc_ld32(tmem + ((uint32_t)(32 * q4) << 16) + (uint32_t)c0, v);
                if constexpr (WIDE) {
                    float u[32];
                    tc_ld32(tmem + ((uint32_t)(32 * q4) << 16) + (uint32_t)(64 + c0), u);
#pragma unroll
                    for (int i = 0; i < 32; ++i) v[i] += u[i];
                }
                if (row >= 0) {
#pragma unroll
                    for (int i = 0; i < 32; ++i) {
                        const int vj = (V > 1 && c0 + i >= Np) ? 1 : 0, j = c0 + i - vj * Np;
                        if (vj < nv && j < cnt)
                            atomicAdd(g.L + (size_t)(r0 + vj) * g.stride + (size_t)s_tgt[j] * nc + row,
                                      v[i] * (V > 1 && vj ? sc[V - 1] : sc[0]));
                    }
                }
            }
        } else if (tid == 0) {
            atomicAdd(g.err, 1);
        }
        tc_fence_before();
        __syncthreads();  // the accumulator is free again
        tc_fence_after();
    }
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(S::COLS)
                     : "memory");
}

// ---------------------------------------------------------------------------
// FP64 form, p <= 15: the key's operator applied by digit products on the
// tensor cores (scheme and bounds of lfmm_m2l_oz.cu: seven 9-bit digits per
// operand, the 28 products of the leading diagonals, one offset per sum).  One CTA per batch of
// pairs of one key (and 128-row part of the outputs), 32 columns at a time.
// The dense operator is formed in FP64 from the table W of the complex
// reaction coefficient in blocks of 2 x 2 (as k_m2r_tc: one addition per
// entry), turned into a 64-bit fixed-point number by shifts (the scales are
// powers of two, so no rounding but the last of 63 bits) and cut into digits;
// a biased add makes the signed digits plain bit fields, and 1024 + digit in
// float16 is the bit pattern itself.  The operator's scale comes from the key's
// largest table value with the smallest scale it meets (emin), so every entry
// is below 1/2.  The multipoles' digits are those of the free M2L.
//   Bound: the integer work of the digits (about 50 operations per entry) and
// the FP64 additions and conversions, which share an SM's 2 per clock; two CTAs
// per SM hide each other's gathers and read-backs.
// Measured: 65,536 charges, p = 10 (171,888 pairs): 3.75 ms (k_m2r_rot) -> 0.97 ms;
// 1,000 charges 0.215 -> 0.082 ms.
// ---------------------------------------------------------------------------
#define RZ_T 256
#define RZ_N 32                          // columns at a time (MMA N: 16 or 32)
#define RZ_X_BYTES (RZ_N * TC_ROWB)      // one multipole digit of a K chunk
#define RZ_STAGE (OZ_S * (OZ_A_BYTES + RZ_X_BYTES))
#define RZ_PMAX 15                       // largest order
#define RZ_PAIRS 128                     // row (column) pairs at that order

struct ROzArgs {
    int p, nc, nk, nkc, parts;  // order, coefficients, K positions and chunks, 128-row parts
    const int4* batches;        // key index, first sorted entry, count | key << 8, table
    const double* tables;       // [table][TS][TS]
    const LfmmComp* comps;
    const double* phase;        // [225 lateral offsets][cos | sin][RR_PH]
    const int2* pairs;          // (source box, target box) per sorted entry
    const double* levelh;
    const __half* Ms;           // digits [box][OZ_S][32 nkc]
    const double* cscale;       // 2^e per packed coefficient
    const int* perm;            // packed coefficient of each K position (and row), -1: none
    const int* emin;            // [TS][TS] smallest exponent of a table value
    const unsigned long long* gmax;  // largest scaled multipole per level (double bits), [16] per right-hand side
    double* L;
    size_t ms_stride, stride;
    int* err;
};

// a 2^sh, |a 2^sh| < 1/2, in units of 2^-63 (sign flipped by neg), biased so
// that its signed digits d_i are the bit fields d_i + 256 (the leading one unmasked)
__device__ __forceinline__ unsigned long long rz_fixed(double a, int sh, bool neg)
{
    constexpr unsigned long long BIAS = 256ull * (1ull + (1ull << 9) + (1ull << 18) + (1ull << 27) + (1ull << 36) +
                                                  (1ull << 45) + (1ull << 54));
    const unsigned long long b = (unsigned long long)__double_as_longlong(a);
    const int r = 1022 - (int)((b >> 52) & 0x7ffu) - sh;  // right shift of the significand in bits 62 .. 10
    const unsigned long long m = ((b & 0xfffffffffffffull) | 0x10000000000000ull) << 10;
    const unsigned long long f = r > 63 ? 0ull : (m + (1ull << (max(r, 1) - 1))) >> max(r, 1);
    return BIAS + ((((long long)b < 0) != neg) ? 0ull - f : f);
}

// digit i (0: leading) of two biased numbers as float16
template <int I>
__device__ __forceinline__ __half2 rz_digit(unsigned long long a, unsigned long long b)
{
    constexpr int S = OZ_B * (OZ_S - 1 - I);
    uint32_t x = (uint32_t)(a >> S), y = (uint32_t)(b >> S);
    if (I > 0) {
        x &= 511u;
        y &= 511u;
    }
    const uint32_t v = (x | y << 16) + 0x64006400u;  // 1024 + field
    return __hsub2(*reinterpret_cast<const __half2*>(&v), __half2half2(__ushort_as_half(0x6500)));  // - 1280
}

// the digits of 8 K values of one operator row
template <int I>
__device__ __forceinline__ void rz_store(unsigned char* sa, const unsigned long long w[8])
{
    __align__(16) __half2 h[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) h[e] = rz_digit<I>(w[2 * e], w[2 * e + 1]);
    *reinterpret_cast<uint4*>(sa + I * OZ_A_BYTES) = *reinterpret_cast<const uint4*>(h);
    if constexpr (I + 1 < OZ_S) rz_store<I + 1>(sa, w);
}

// x or -x by the sign bit (a selected negation ran on the FP64 pipe)
__device__ __forceinline__ double rz_flip(double x, int neg)
{
    return __hiloint2double(__double2hiint(x) ^ (neg ? 0x80000000 : 0), __double2loint(x));
}

__global__ void __launch_bounds__(RZ_T, 2) k_m2r_oz(ROzArgs g)
{
    extern __shared__ unsigned char smem_raw[];
    // 512-byte alignment: the period of the 64-byte swizzle
    unsigned char* sm = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 511) &
                                                         ~(uintptr_t)511);
    unsigned char* sx = sm + OZ_S * OZ_A_BYTES;
    double2* sW = reinterpret_cast<double2*>(sm + RZ_STAGE);  // [N][mu + 2p], rows of 4p + 1
    // column pairs: offsets of the two W terms from the row's; signs of the two
    // terms (bits 0, 1), two real inputs (bit 2); exponents
    __shared__ int4 s_co[RZ_PAIRS];
    __shared__ int s_prow[128];
    __shared__ double sPh[2 * RR_PH];
    __shared__ int s_src[R_TB], s_tgt[R_TB];
    __shared__ unsigned long long s_max;
    __shared__ double s_unit;  // output unit: 2^{-36 - sc} over the multipoles' scale and h
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t s_tmem;
    __shared__ int s_abort;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int p = g.p, nc = g.nc, nkc = g.nkc, TS = 2 * p + 1, WS = 4 * p + 1;
    const int part = blockIdx.x % g.parts;
    const int4 b = g.batches[blockIdx.x / g.parts];
    const int start = b.y, cnt = b.z & 255;
    if (cnt <= 0 || cnt > R_TB) return;
    int c, lev, ox, oy, oz;
    rkey_decode((uint32_t)b.z >> 8, c, lev, ox, oy, oz);
    const bool refl = g.comps[c].refl != 0;
    if (tid < RZ_PAIRS) {
        int4 o = make_int4(0, 0, 4, 0);
        if (2 * tid < g.nk) {
            const int j0 = g.perm[2 * tid], j1 = g.perm[2 * tid + 1];
            int n, m, im;
            lf_decode(p, j0, n, m, im);
            const int e0 = ilogb(g.cscale[j0]);
            // the multipole's reflection sign (-1)^{n+m} for s = -1 maps, and (-1)^m of the second term
            const int sg = refl && ((n + m) & 1) ? 1 : 0;
            if (m > 0) {
                o = make_int4(n * WS + m, n * WS - m, sg | (sg ^ (m & 1)) << 1, e0 | e0 << 16);
            } else {
                o = make_int4(n * WS, n * WS, 4 | sg, e0 | e0 << 16);
                if (j1 >= 0) {
                    lf_decode(p, j1, n, m, im);
                    o.y = n * WS;
                    o.z |= (refl && (n & 1)) ? 2 : 0;
                    o.w = e0 | ilogb(g.cscale[j1]) << 16;
                }
            }
        }
        s_co[tid] = o;
    } else {
        // rows t and 64 + t: the pair t of this part (so that 8 pairs' stores meet no bank twice)
        const int r = tid - 128, i = 128 * part + 2 * (r & 63) + (r >> 6);
        s_prow[r] = i < g.nk ? g.perm[i] : -1;
    }
    if (tid < R_TB) {
        const int2 pr = (tid < cnt) ? g.pairs[start + tid] : make_int2(-1, -1);
        s_src[tid] = pr.x;
        s_tgt[tid] = pr.y;
    } else if (tid < R_TB + 2 * RR_PH) {
        sPh[tid - R_TB] = g.phase[(size_t)((ox + R_OR) * R_OW + (oy + R_OR)) * 2 * RR_PH + (tid - R_TB)];
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(256)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        mbar_init(&bar, 1);
        s_abort = 0;
        s_max = 0ull;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    {
        const double* Tk = g.tables + (size_t)b.w * TS * TS;
        unsigned long long mx = 0;
        for (int j = tid; j < TS * TS; j += RZ_T) {
            const int N = j / TS, a = j - N * TS;
            const double t = Tk[j];
            const int e = g.emin[j];
            if (e < 1000) {
                const unsigned long long v = (unsigned long long)__double_as_longlong(
                    fabs(t) * __longlong_as_double((long long)(1023 - e) << 52));
                mx = v > mx ? v : mx;
            }
            const double wr = t * sPh[a], wi = t * sPh[RR_PH + a];
            double2* w = sW + N * WS + 2 * p;
            w[a] = make_double2(wr, wi);
            w[-a] = (a & 1) ? make_double2(-wr, wi) : make_double2(wr, -wi);
        }
        const unsigned h = __reduce_max_sync(0xffffffffu, (unsigned)(mx >> 32));
        const unsigned l = __reduce_max_sync(0xffffffffu, (unsigned)(mx >> 32) == h ? (unsigned)mx : 0u);
        if (lane == 0) atomicMax(&s_max, (unsigned long long)h << 32 | l);
    }
    __syncthreads();
    // two table values of at most s_max 2^{e_in + e_out} each make an entry: 2^sc takes it below 1/2
    const unsigned long long mx = s_max;
    const bool badt = mx >= 0x7ff0000000000000ull;
    const int sc = (mx == 0ull || badt) ? 0 : 1020 - (int)(mx >> 52);
    if (tid == 0) {  // (read after the chunks' barriers)
        const double u = ldexp(1.0, -36 - sc) / (oz_scale(g.gmax[(size_t)blockIdx.y * 16 + lev]) * g.levelh[lev]);
        s_unit = badt ? nan64() : u;
    }
    // operator unit: row pair xj, quarter xq of every chunk
    const int xj = tid >> 2, xq = tid & 3;
    const int r0 = s_prow[xj], r1 = s_prow[64 + xj];
    int z0 = 0, z1 = 0, er0 = 0, er1 = 0;
    bool ng0 = false, ng1 = false, cpx = false;  // cpx: Re and Im of one output
    if (r0 >= 0) {
        int k, l, im;
        lf_decode(p, r0, k, l, im);
        z0 = z1 = k * WS + l + 2 * p;
        er0 = er1 = ilogb(g.cscale[r0]);
        ng0 = ng1 = (k & 1) != 0;
        cpx = l > 0;
        if (!cpx && r1 >= 0) {
            lf_decode(p, r1, k, l, im);
            z1 = k * WS + l + 2 * p;
            er1 = ilogb(g.cscale[r1]);
            ng1 = (k & 1) != 0;
        }
    }
    const uint32_t off0 = swz16(xj, 8 * xq), off1 = swz16(64 + xj, 8 * xq);
    const __half* Ms = g.Ms + (size_t)blockIdx.y * g.ms_stride;
    double* L = g.L + (size_t)blockIdx.y * g.stride;
    const int mrow = nkc * TH_KC;
    bool ok = true;
    int gr = 0;  // chunks so far
    for (int q0 = 0; q0 < cnt && ok; q0 += RZ_N) {
        const int nq = min(RZ_N, cnt - q0), Np = (nq + 15) & ~15;
        const uint32_t idesc = tc_idesc_f16(128, Np);
        for (int kc = 0; kc < nkc; ++kc, ++gr) {
            unsigned long long w[8];
            const int4* co = s_co + kc * (TH_KC / 2) + 4 * xq;
            if (r0 >= 0)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int4 o = co[e];
                    const double2 x = sW[z0 + o.x], y = sW[z0 + o.y];
                    const double xr = rz_flip(x.x, o.z & 1), yr = rz_flip(y.x, o.z & 2);
                    const double u0 = (o.z & 4) ? xr : xr + yr;
                    const double u1 = (o.z & 4) ? yr : rz_flip(y.y, o.z & 2) - rz_flip(x.y, o.z & 1);
                    w[2 * e] = rz_fixed(u0, sc - (o.w & 0xffff) - er0, ng0);
                    w[2 * e + 1] = rz_fixed(u1, sc - (o.w >> 16) - er0, ng0);
                }
            // the previous chunk's MMAs have read the stage
            if (gr > 0 && !mbar_wait(&bar, (uint32_t)((gr - 1) & 1))) s_abort = 1;
            {
                const int row = (tid & 127) >> 2, q = tid & 3, d0 = tid < 128 ? 0 : 4, d1 = tid < 128 ? 4 : OZ_S;
                if (row < Np) {
                    const int src = s_src[q0 + row];
                    const __half* gs = Ms + (size_t)(src >= 0 ? src : 0) * (OZ_S * mrow) + kc * TH_KC + q * 8;
                    unsigned char* dst = sx + swz16(row, q * 8);
                    for (int i = d0; i < d1; ++i) {
                        if (src >= 0)
                            cp_async16(smem_u32(dst + i * RZ_X_BYTES), gs + (size_t)i * mrow);
                        else
                            *reinterpret_cast<float4*>(dst + i * RZ_X_BYTES) = make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                }
            }
            cp_async_commit();
            // (rows past the last coefficient are never read back)
            if (r0 >= 0) rz_store<0>(sm + off0, w);
            if (r1 >= 0) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int4 o = co[e];
                    const double2 x = sW[z1 + o.x], y = sW[z1 + o.y];
                    // the imaginary part of an output, or the second of two real ones
                    const double xr = rz_flip(cpx ? x.y : x.x, o.z & 1), yr = rz_flip(cpx ? y.y : y.x, o.z & 2);
                    const double xi = rz_flip(cpx ? x.x : x.y, o.z & 1), yi = rz_flip(cpx ? y.x : y.y, o.z & 2);
                    const double u0 = (o.z & 4) ? xr : xr + yr;
                    const double u1 = (o.z & 4) ? yr : (cpx ? xi - yi : yi - xi);
                    w[2 * e] = rz_fixed(u0, sc - (o.w & 0xffff) - er1, ng1);
                    w[2 * e + 1] = rz_fixed(u1, sc - (o.w >> 16) - er1, ng1);
                }
                rz_store<0>(sm + off1, w);
            }
            cp_async_wait<0>();
            fence_async_smem();
            tc_fence_before();
            __syncthreads();
            if (*(volatile int*)&s_abort) {  // block-uniform after the barrier
                ok = false;
                break;
            }
            if (tid == 0) {
                tc_fence_after();
                const uint32_t ab = smem_u32(sm), xb = smem_u32(sx);
                const int nks = (g.nk - kc * TH_KC) > 16 ? 2 : 1;
                for (int ks = 0; ks < nks; ++ks)
#pragma unroll
                    for (int i = 0; i < OZ_S; ++i)
#pragma unroll
                        for (int j = 0; j < OZ_S - i; ++j)
                            tc_mma_f16(tmem + (uint32_t)((i + j) * RZ_N), smem_desc(ab + i * OZ_A_BYTES + 32 * ks),
                                       smem_desc(xb + j * RZ_X_BYTES + 32 * ks), idesc,
                                       (kc == 0 && ks == 0 && i == 0) ? 0u : 1u);
                tc_commit(&bar);
            }
            __syncwarp();
        }
        bool got = false;
        if (ok) got = mbar_wait(&bar, (uint32_t)((gr - 1) & 1));
        ok = __syncthreads_and(got) != 0;  // block-uniform
        tc_fence_after();
        if (ok) {
            const int q4 = warp & 3, row = s_prow[32 * q4 + lane], cb = 16 * (warp >> 2);
            if (cb < Np) {
                long long hi[16], lo[16];  // units 2^-36 and 2^-72
#pragma unroll
                for (int d = 0; d < OZ_S; ++d) {
                    float v[16];
                    tc_ld16(tmem + ((uint32_t)(32 * q4) << 16) + (uint32_t)(d * RZ_N + cb), v);
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const long long n = __float2int_rn(v[i]);
                        if (d == 0)
                            hi[i] = n * (1ll << (2 * OZ_B));
                        else if (d < 3)
                            hi[i] += n * (1ll << (OZ_B * (2 - d)));
                        else if (d == 3)
                            lo[i] = n * (1ll << (3 * OZ_B));
                        else
                            lo[i] += n * (1ll << (OZ_B * (6 - d)));
                    }
                }
                if (row >= 0) {
                    const double sh = g.cscale[row] * s_unit, sl = sh * 0x1p-36;
#pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        if (cb + i >= nq) break;
                        // carry into hi, then both to FP64 by the bits of 1.5 2^52 + n
                        const long long h = hi[i] + (lo[i] >> 36), l = lo[i] & 0xfffffffffll;
                        const double dh = __longlong_as_double(0x4338000000000000ll + h) - 0x1.8p52;
                        const double dl = __longlong_as_double(0x4338000000000000ll + l) - 0x1.8p52;
                        atomicAdd(L + (size_t)s_tgt[q0 + cb + i] * nc + row, fma(dh, sh, dl * sl));
                    }
                }
            }
        } else if (tid == 0) {
            atomicAdd(g.err, 1);
        }
        tc_fence_before();
        __syncthreads();  // the accumulators are free again
        tc_fence_after();
    }
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256) : "memory");
}

// once per context (the first evaluation; a captured batch graph never sees it)
static LfErr m2r_phases64(lfmm_ctx* ctx, cudaStream_t st)
{
    if (ctx->m2r_phase64_ready) return LfErr();
    LF_TRY(lf_reserve(ctx->m2r_phase64, (size_t)R_OW * R_OW * 2 * RR_PH * sizeof(double)));
    ++ctx->launches, k_m2r_phase64<<<R_OW * R_OW, RR_PH, 0, st>>>(ctx->m2r_phase64.as<double>());
    LF_TRY(lf_cuda(cudaGetLastError(), "m2r phases"));
    ctx->m2r_phase64_ready = 1;
    return LfErr();
}

static LfErr m2r_apply_oz(lfmm_ctx* ctx, cudaStream_t st)
{
    LF_TRY(m2r_phases64(ctx, st));
    ROzArgs g;
    g.p = ctx->p;
    g.nc = lf_nc(ctx->p);
    g.nk = ctx->oz_nk;
    g.nkc = (g.nk + TH_KC - 1) / TH_KC;
    g.parts = (g.nk + 127) / 128;
    g.batches = ctx->m2r_batches.as<int4>();
    g.tables = ctx->m2r_tables.as<double>();
    g.comps = ctx->comp_dev.as<LfmmComp>();
    g.phase = ctx->m2r_phase64.as<double>();
    g.pairs = ctx->m2r_pairs.as<int2>();
    g.levelh = ctx->m2r_levelh.as<double>();
    g.Ms = ctx->oz_Ms.as<__half>();
    g.cscale = ctx->oz_cscale.as<double>();
    g.perm = ctx->oz_perm.as<int>();
    g.emin = ctx->m2r_emin.as<int>();
    g.gmax = reinterpret_cast<unsigned long long*>(ctx->counts.as<char>() + LFMM_TCMAX_OFF);
    g.L = ctx->Lexp.as<double>();
    g.ms_stride = (size_t)ctx->nbox_total * OZ_S * g.nkc * TH_KC;
    g.stride = (size_t)ctx->nbox_total * g.nc;
    g.err = reinterpret_cast<int*>(ctx->counts.as<char>() + LFMM_TIMEOUT_OFF);
    const size_t sm = 512 + RZ_STAGE + sizeof(double2) * (size_t)(2 * g.p + 1) * (4 * g.p + 1);
    LF_TRY(lf_smem_limit(k_m2r_oz, 512 + RZ_STAGE + sizeof(double2) * (2 * RZ_PMAX + 1) * (4 * RZ_PMAX + 1)));
    ++ctx->launches, k_m2r_oz<<<dim3(ctx->m2r_nbatch * g.parts, ctx->nrhs_b), RZ_T, sm, st>>>(g);
    return lf_cuda(cudaGetLastError(), "m2r digit products");
}

template <typename R>
static LfErr m2r_apply_rot(lfmm_ctx* ctx, cudaStream_t st)
{
    RRotArgs g;
    g.p = ctx->p;
    g.nc = lf_nc(ctx->p);
    // 32 columns (16 above p = 10) keep several blocks per SM
    g.cb = ctx->p <= 10 ? 32 : RR_CB;
    g.batches = ctx->m2r_batches.as<int4>();
    g.tables = ctx->m2r_tables.as<double>();
    g.comps = ctx->comp_dev.as<LfmmComp>();
    LF_TRY(m2r_phases64(ctx, st));
    g.phase = ctx->m2r_phase64.as<double>();
    g.keys = ctx->m2r_keys.as<uint32_t>();
    g.pairs = ctx->m2r_pairs.as<int2>();
    g.levelh = ctx->m2r_levelh.as<double>();
    g.M = ctx->Mexp.ptr;
    g.L = ctx->Lexp.ptr;
    g.stride = (size_t)ctx->nbox_total * g.nc;
    g.nr = ctx->nrhs_b;
    const int TS = 2 * ctx->p + 1;
    const size_t sm = sizeof(R) * ((size_t)2 * lf_nre(ctx->p) * g.cb + (size_t)TS * TS);
    constexpr int MS = 2 * LFMM_PMAX + 1;  // (more than p = 10 takes with its 32 columns)
    constexpr size_t most = sizeof(R) * (2 * ((LFMM_PMAX + 1) * (LFMM_PMAX + 2) / 2) * RR_CB + MS * MS);
    // share the rows of each batch between blocks, so that the longest batches
    // do not outlast the rest; four shares leave every SM quarter a warp
    int parts = 1;
    while ((parts < 4 && (int64_t)ctx->m2r_nbatch * parts < 64 * 152) ||
           (parts < 8 && (int64_t)ctx->m2r_nbatch * parts < 8 * 152))
        parts *= 2;
    LF_TRY(lf_smem_limit(k_m2r_rot<R>, most));
    ++ctx->launches, k_m2r_rot<R><<<dim3(ctx->m2r_nbatch, parts), R_T, sm, st>>>(g);
    return lf_cuda(cudaGetLastError(), "m2r rotated");
}

// the float32 form applies the keys on the tensor cores whenever the free M2L
// does (tensor-core option)
static bool m2r_tc_on(const lfmm_ctx* ctx) { return ctx->precision == 1 && lf_tc_on(ctx); }

template <int V, bool WIDE>
static LfErr m2r_launch_tc(lfmm_ctx* ctx, const RTcArgs& g, cudaStream_t st)
{
    constexpr int sm = RtShape<V, WIDE>::SMEM;
    LF_TRY(lf_smem_limit(k_m2r_tc<V, WIDE>, sm));
    ++ctx->launches, k_m2r_tc<V, WIDE><<<ctx->m2r_nbatch * g.parts, RT_THREADS, sm, st>>>(g);
    return lf_cuda(cudaGetLastError(), "m2r tensor-core GEMM");
}

static LfErr m2r_apply_tc(lfmm_ctx* ctx, cudaStream_t st)
{
    RTcArgs g;
    g.p = ctx->p;
    g.nc = lf_nc(ctx->p);
    g.nk = ctx->tc_nk;
    g.nkc = (g.nk + TH_KC - 1) / TH_KC;
    g.batches = ctx->m2r_batches.as<int4>();
    g.tables = ctx->m2r_tabf.as<float>();
    g.tscale = ctx->m2r_tscale.as<int>();
    g.comps = ctx->comp_dev.as<LfmmComp>();
    g.pairs = ctx->m2r_pairs.as<int2>();
    g.levelh = ctx->m2r_levelh.as<double>();
    g.Ms = ctx->m2l_Ms.as<__half>();
    g.cscale = ctx->tc_cscale.as<float>();
    g.perm = ctx->tc_perm.as<int>();
    g.gmax = reinterpret_cast<unsigned*>(ctx->counts.as<char>() + LFMM_TCMAX_OFF);
    g.parts = (g.nk + 127) / 128;
    g.ms_stride = (size_t)ctx->nbox_total * (g.parts > 1 ? 512 : 256);
    g.L = ctx->Lexp.as<float>();
    g.stride = (size_t)ctx->nbox_total * g.nc;
    g.nr = ctx->nrhs_b;
    g.err = reinterpret_cast<int*>(ctx->counts.as<char>() + LFMM_TIMEOUT_OFF);
    if (ctx->m2r_phase_p != ctx->p) {
        // once per context (the first evaluation; a captured batch graph never sees it)
        LF_TRY(lf_reserve(ctx->m2r_phase, (size_t)R_OW * R_OW * 2 * RT_PH * sizeof(float)));
        ++ctx->launches, k_m2r_phase<<<R_OW * R_OW, RT_PH, 0, st>>>(ctx->p, ctx->m2r_phase.as<float>());
        LF_TRY(lf_cuda(cudaGetLastError(), "m2r phases"));
        ctx->m2r_phase_p = ctx->p;
    }
    g.phase = ctx->m2r_phase.as<float>();
    if (g.parts > 1) return m2r_launch_tc<1, true>(ctx, g, st);
    return g.nr == 1 ? m2r_launch_tc<1, false>(ctx, g, st) : m2r_launch_tc<2, false>(ctx, g, st);
}

LfErr lf_m2r_apply(lfmm_ctx* ctx, cudaStream_t st)
{
    if (ctx->m2r_nbatch == 0) return LfErr();
    if (m2r_tc_on(ctx)) return m2r_apply_tc(ctx, st);
    if (ctx->precision) return m2r_apply_rot<float>(ctx, st);
    return lf_m2l_oz_ok(ctx) ? m2r_apply_oz(ctx, st) : m2r_apply_rot<double>(ctx, st);
}
