// Weight gradients of the depth prior's 3x3 convolutions on the tcgen05 tensor
// cores: dW_tap[ci x co] = sum over pixels p of X[p + tap][ci] dZ[p][co].
//
// The contraction runs over pixels, so both operands are read "MN-major" (channels
// contiguous, as NHWC stores them): eight channels of eight consecutive pixels are
// one core matrix, and nothing is transposed.  One operand S is shifted, the other U
// is not.  S is held three times, once per horizontal shift dx, each copy in planes
// of eight channels one plane pitch apart, so that the (dx, channel) pairs are the
// rows of one MMA (up to 128, the descriptor's stride offset one plane); the vertical
// shift dy moves the start address by a row, into the copies' halo rows, and has an
// accumulator of its own.  Padding a 16-channel layer's rows per tap instead would
// use 16 of an MMA's 64 rows; three shifts use 48.  The operand with fewer channels
// is the shifted one (shifting dZ by -tap is shifting X by tap), so S's rows are
// few and U's channels are the columns.
//
// k_conv3x3_wgrad does this for shifted operands of up to 32 channels.  With more, a
// tap's own channels fill an MMA's rows, nothing needs three copies, and
// k_conv3x3_wgrad_tap has the TMA load one halo tile per operand and gives each tap an
// accumulator.
//
// A CTA walks tiles of TX x TY pixels: warps 0-7 copy the next tile (zeros
// outside the image) while warp 8 issues the current
// tile's MMAs, 16 pixels an instruction.  The tensor core truncates as it accumulates
// (an all-positive sum of 505 steps came out 1.8e-5 low), so no accumulator runs for
// more than `chain` steps: four more warps then add it to dW with FP32 reductions,
// while the MMAs go on in a second set of accumulators where tensor memory holds two.
// `chain` is the depth the split-K gathered GEMM (gemm_tc.cu) gives the same layer.
//
// Scattering a transposed im2col into shared memory two bytes at a time took, for the
// 14 layers of a batch of 32 at 320x240, 2.57 ms; this takes 0.73 (0.67 with accumulators
// that run over all of a CTA's pixels, whose errors were twice the GEMM's).  Before the
// flushes, 16 -> 16 channels 282 -> 71 us (24 at the HBM rate), 96 -> 32 at a quarter of
// the pixels 347 -> 63 (24).
// Bounds: the loaders' latency with few channels, the 16-byte rows of the TMA's boxes
// with many.
#include <algorithm>

#include "tc_common.cuh"
#include "tensor_map.cuh"

namespace gevo {

gevo_status conv3x3_wgrad_gemm(int nb, int H, int W, int Cin, const void* X, int Cout,
                               const void* dZt, float* dWt, int ksplit, uint32_t* err,
                               cudaStream_t st);

constexpr int kWgLoaders = 8;                          // loader warps
constexpr int kWgThreads = 32 * (kWgLoaders + 1 + 4);  // + the MMA warp + four that flush

struct WgTile {
    int H, W, Cs, Cu;
    int kgs, kgu;          // 8-channel groups of S and U
    int nmt, mlast;        // MMA row tiles over the 3 kgs groups; rows of the last (64 or 128)
    int tx, ty;            // tile
    int nd, mper;          // a CTA's vertical shifts (3 or 1) and row tiles (mper divides nmt)
    int ps, pu;            // plane pitches of S and U (U K-major: pitch of 8 pixels)
    int nt, tcols;         // columns of an accumulator (U's channels, multiple of 16)
    int ntx, nty, ntiles;
    uint32_t sbytes, stage;
    int swap;              // S is dZ and U is X (taps reversed)
    int K9;                // 9 Cin: row length of dW
    int chain, sets;       // MMA steps an accumulator runs before it is flushed; accumulator sets
};

__device__ __forceinline__ void red_add4(float* p, float a, float b, float c, float d)
{
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d)
                 : "memory");
}

// The flush points of a CTA's walk: before a tile whose steps would take the running
// chain past its limit, and after the last tile.  The warp that issues and the warps
// that flush run through the same sequence.  Flush number f uses accumulator set
// f % sets, for the (f / sets)-th time.
struct WgChain {
    int steps = 0, flush = 0;
    __device__ bool full(int more, int limit) const { return steps > 0 && steps + more > limit; }
    __device__ int set(int sets) const { return sets == 2 ? flush & 1 : 0; }
    __device__ uint32_t use(int sets) const { return (uint32_t)(sets == 2 ? flush >> 1 : flush); }
    __device__ void next()
    {
        steps = 0;
        flush++;
    }
};

// Adds a row's 16 columns [c0, c0 + 16) of a tap's accumulator: row = channel c of S,
// column = channel of U.
__device__ __forceinline__ void wg_add(float* __restrict__ dW, const float v[16], int c, int c0,
                                       int tap, int swap, int Cs, int Cu, int K9)
{
    if (swap) {            // channels of U are X's: consecutive in dW
        float* o = dW + (size_t)c * K9 + tap * Cu + c0;
#pragma unroll
        for (int q = 0; q < 16; q += 4)
            if (c0 + q < Cu) red_add4(o + q, v[q], v[q + 1], v[q + 2], v[q + 3]);
    } else {
#pragma unroll
        for (int q = 0; q < 16; q++)
            if (c0 + q < Cu) atomicAdd(dW + (size_t)(c0 + q) * K9 + tap * Cs + c, v[q]);
    }
}

// KMAJ: U is dZ^T ([channel][pixel], W a multiple of 8) instead of NHWC.  ND vertical
// shifts and NM row tiles a CTA are compile-time counts: with run-time loops around
// it an MMA took 176 clocks to issue, unrolled it takes the 23 to 40 it runs.
template <bool KMAJ, int ND, int NM>
__global__ void __launch_bounds__(kWgThreads)
k_conv3x3_wgrad(WgTile t, const __nv_bfloat16* __restrict__ S, const __nv_bfloat16* __restrict__ U,
                float* __restrict__ dW, size_t P, uint32_t* __restrict__ err)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) unsigned long long s_full[2], s_empty[2], s_accfull[2], s_accempty[2];
    __shared__ uint32_t s_tmem;

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const uint32_t base = smem_u32(smem);
    if (tid == 0) {
        for (int i = 0; i < 2; i++) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&s_full[i])), "r"(kWgLoaders) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_empty[i])) : "memory");
        }
        for (int i = 0; i < 2; i++) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_accfull[i])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 4;" ::"r"(smem_u32(&s_accempty[i])) : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == kWgLoaders) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&s_tmem)),
                     "r"(t.tcols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;
    const int txy = t.ntx * t.nty;
    // this CTA's first vertical shift and its first row tile
    const int nmg = t.nmt / NM;
    const int dy0 = (int)blockIdx.y / nmg, m0 = ((int)blockIdx.y % nmg) * NM;
    const bool tail = m0 + NM == t.nmt;                    // holds the last row tile
    bool ok = true;

    if (warp < kWgLoaders) {
        // S: pieces (row, column -1 .. TX, channel group), consecutive in memory but for
        // the row ends; each is read once and stored into the three copies.  (Three
        // asynchronous copies of it instead tripled what an SM reads from L2, about
        // 20 bytes a clock whatever asks, and that was the kernel's time.)
        constexpr int NL = 32 * kWgLoaders, NB = 4;        // loader threads, pieces in flight
        const int hx = t.tx + 2;                           // columns with the halo
        const int dps = NL / t.kgs, dks = NL - dps * t.kgs, drs = dps / hx, dcs = dps - drs * hx;
        const int sp0 = tid / t.kgs, ks0 = tid - sp0 * t.kgs, rs0 = sp0 / hx, cs0 = sp0 - rs0 * hx;
        const int du = 32 / t.kgu, eu = 32 - du * t.kgu;
        const int cu0 = lane / t.kgu, ku0 = lane - cu0 * t.kgu;
        const uint32_t cps = (uint32_t)(t.kgs * t.ps);     // from one copy to the next
        const int srows = t.ty + ND - 1;
        int i = 0;
        for (int tile = blockIdx.x; tile < t.ntiles; tile += gridDim.x, i++) {
            const int s = i & 1;
            const int b = tile / txy, r = tile - b * txy, tyi = r / t.ntx, txi = r - tyi * t.ntx;
            const int x0 = txi * t.tx, y0 = tyi * t.ty;
            const uint32_t sS = base + s * t.stage, sU = sS + t.sbytes;
            const int wx = t.W - x0;                       // columns of the tile inside the image
            const __nv_bfloat16* img = S + (size_t)b * t.H * t.W * t.Cs;
            int kg = ks0, row = rs0, col = cs0;            // col 0: the halo column left of x0
            bool waited = false;
            do {
                uint4 v[NB];
                uint32_t dst[NB];
                int at[NB];
#pragma unroll
                for (int j = 0; j < NB; j++) {
                    const int gy = y0 + row + dy0 - 1, gx = x0 + col - 1;
                    v[j] = make_uint4(0u, 0u, 0u, 0u);
                    if (row < srows && (unsigned)gy < (unsigned)t.H && (unsigned)gx < (unsigned)t.W)
                        v[j] = *reinterpret_cast<const uint4*>(img + ((size_t)gy * t.W + gx) * t.Cs + kg * 8);
                    dst[j] = sS + kg * t.ps + (row * t.tx + col) * 16;
                    at[j] = row < srows ? col : 1 << 20;
                    kg += dks;
                    row += drs;
                    col += dcs;
                    if (kg >= t.kgs) { kg -= t.kgs; col++; }
                    if (col >= hx) { col -= hx; row++; }
                }
                if (!waited) {                             // the first pieces are on their way by now
                    waited = true;
                    if (i >= 2 && !mbar_wait(smem_u32(&s_empty[s]), (uint32_t)((i >> 1) - 1) & 1u)) {
                        ok = false;
                        break;
                    }
                }
#pragma unroll
                for (int j = 0; j < NB; j++) {
                    // the pixel at col is the left neighbour of column col of the tile, the
                    // centre of col - 1 and the right neighbour of col - 2.  Columns past
                    // the image are no pixels of U: zero there, so that no value meets
                    // U's padding
                    if (at[j] < t.tx)
                        st_shared_16(dst[j], at[j] < wx ? v[j] : make_uint4(0u, 0u, 0u, 0u));
                    if ((unsigned)(at[j] - 1) < (unsigned)t.tx) st_shared_16(dst[j] + cps - 16, v[j]);
                    if ((unsigned)(at[j] - 2) < (unsigned)t.tx) st_shared_16(dst[j] + 2 * cps - 32, v[j]);
                }
            } while (row < srows);
            if (!ok) break;
            if (KMAJ) {
                // a warp takes channels: the 8-pixel pieces of its tile
                const int t8 = t.tx >> 3, per = t.ty * t8;
                for (int c = warp; c < t.Cu; c += kWgLoaders) {
                    const __nv_bfloat16* img = U + (size_t)c * P + (size_t)b * t.H * t.W;
                    for (int e = lane; e < per; e += 32) {
                        const int row = e / t8, gx = x0 + 8 * (e - row * t8), gy = y0 + row;
                        const bool in = gy < t.H && gx < t.W;
                        cp_async16(sU + e * t.pu + c * 16, in ? img + (size_t)gy * t.W + gx : U, in);
                    }
                }
            } else {
                for (int row = warp; row < t.ty; row += kWgLoaders) {
                    const int gy = y0 + row;
                    const bool yin = gy < t.H;
                    const __nv_bfloat16* src = U + (((size_t)b * t.H + (yin ? gy : 0)) * t.W + x0) * t.Cu + lane * 8;
                    uint32_t d = sU + ku0 * t.pu + (row * t.tx + cu0) * 16;
                    int kg = ku0, col = cu0;
                    while (col < t.tx) {
                        const bool in = yin && col < wx;
                        cp_async16(d, in ? src : U, in);
                        src += 32 * 8;
                        kg += eu;
                        col += du;
                        d += eu * t.pu + du * 16;
                        if (kg >= t.kgu) { kg -= t.kgu; col++; d -= t.kgu * t.pu - 16; }
                    }
                }
            }
            cp_async_commit();
            cp_async_wait<0>();
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&s_full[s]));
        }
        cp_async_wait<0>();
    } else if (warp == kWgLoaders) {
        const uint32_t majors = (1u << 15) | (KMAJ ? 0u : 1u << 16);    // A, B MN-major
        const uint32_t id128 = idesc_bf16(128, t.nt) | majors;
        const uint32_t idlast = idesc_bf16(tail ? t.mlast : 128, t.nt) | majors;
        const uint64_t ver = (uint64_t)1 << 46;
        // stride offset: the next 8 rows (columns); leading offset: the next 8 pixels
        const uint64_t hiA = (uint64_t)(t.ps >> 4) << 32 | (uint64_t)(128 >> 4) << 16 | ver;
        const uint64_t hiB = KMAJ ? (uint64_t)(128 >> 4) << 32 | (uint64_t)(t.pu >> 4) << 16 | ver
                                  : (uint64_t)(t.pu >> 4) << 32 | (uint64_t)(128 >> 4) << 16 | ver;
        const uint64_t stepB = KMAJ ? (uint64_t)((2 * t.pu) >> 4) : (uint64_t)(256 >> 4);
        WgChain ch;
        int i = 0;
        for (int tile = blockIdx.x; tile < t.ntiles; tile += gridDim.x, i++) {
            const int s = i & 1;
            const int y0 = ((tile % txy) / t.ntx) * t.ty;
            // 16 pixels of one row a step; rows past the image are left out
            const int steps = min(t.ty, t.H - y0) * (t.tx >> 4);
            if (ch.full(steps, t.chain)) {
                if (elect_one()) mma_commit(smem_u32(&s_accfull[ch.set(t.sets)]));
                __syncwarp();
                ch.next();
                // the set was last flushed `sets` flushes ago
                if (ch.use(t.sets) > 0 &&
                    !mbar_wait(smem_u32(&s_accempty[ch.set(t.sets)]), (ch.use(t.sets) - 1) & 1u)) {
                    ok = false;
                    break;
                }
            }
            if (!mbar_wait(smem_u32(&s_full[s]), (uint32_t)(i >> 1) & 1u)) {
                ok = false;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (elect_one()) {
                const uint32_t sS = base + s * t.stage;
                const uint32_t tacc = tmem + ch.set(t.sets) * (ND * NM * t.nt);
                uint32_t acc = ch.steps > 0;
                uint64_t da = (hiA | (uint64_t)(sS >> 4)) + (uint64_t)(m0 * t.ps), db = hiB | (uint64_t)((sS + t.sbytes) >> 4);
                for (int k = 0; k < steps; k++) {
#pragma unroll
                    for (int e = 0; e < ND; e++)
#pragma unroll
                        for (int m = 0; m < NM; m++)       // 16 planes, a row: 16-byte units
                            mma_bf16(tacc + (e * NM + m) * t.nt, da + e * t.tx + (uint64_t)(m * t.ps),
                                     db, m + 1 == NM ? idlast : id128, acc);
                    acc = 1u;
                    da += 256 >> 4;
                    db += stepB;
                }
                mma_commit(smem_u32(&s_empty[s]));
            }
            __syncwarp();
            ch.steps += steps;
        }
        if (ok && elect_one()) mma_commit(smem_u32(&s_accfull[ch.set(t.sets)]));
        __syncwarp();
    } else {
        // the accumulators: row (dx, channel of S), one column per channel of U
        const int w4 = warp & 3;
        WgChain ch;
        auto flush = [&]() {
            const int set = ch.set(t.sets);
            if (!mbar_wait(smem_u32(&s_accfull[set]), ch.use(t.sets) & 1u)) return false;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
            for (int e = 0; e < ND; e++) {
#pragma unroll 1
                for (int m = m0; m < m0 + NM; m++) {
                    // 128 rows: lane = row; 64 rows: 16 of them per warp's 32 lanes
                    const int mr = m + 1 == t.nmt ? t.mlast : 128;
                    const int row = mr == 128 ? w4 * 32 + lane : (lane < 16 ? w4 * 16 + lane : 3 * t.Cs);
                    const int g = m * 128 + row;
                    const int dx = g / t.Cs, c = g - dx * t.Cs;
                    const int tap0 = (dy0 + e) * 3 + dx, tap = t.swap ? 8 - tap0 : tap0;
#pragma unroll 1
                    for (int c0 = 0; c0 < t.nt; c0 += 16) {
                        float v[16];
                        __syncwarp();
                        tmem_ld16(tmem + ((uint32_t)(w4 * 32) << 16) +
                                      (uint32_t)(((set * ND + e) * NM + m - m0) * t.nt + c0), v);
                        if (g < 3 * t.Cs) wg_add(dW, v, c, c0, tap, t.swap, t.Cs, t.Cu, t.K9);
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&s_accempty[set]));
            ch.next();
            return true;
        };
        for (int tile = blockIdx.x; tile < t.ntiles && ok; tile += gridDim.x) {
            const int y0 = ((tile % txy) / t.ntx) * t.ty;
            const int steps = min(t.ty, t.H - y0) * (t.tx >> 4);
            if (ch.full(steps, t.chain)) ok = flush();
            ch.steps += steps;
        }
        if (ok) ok = flush();
    }
    if (!ok && lane == 0) atomicOr(err, kErrTimeout);
    __syncthreads();
    if (warp == kWgLoaders)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(t.tcols)
                     : "memory");
}

// The weight gradient tap by tap: S is a tile with its halo (planes of eight
// channels, rows TX + 2 pixels apart, loaded by TMA), a tap moves the start address,
// and the CTA's 3 ND taps have an accumulator each: rows = mrows channels of S from
// m0, columns = nt channels of U from n0.  Warp 4 loads, warp 5 issues, warps 0-3 add
// the accumulators to dW at the end.  W is a multiple of 16: every pixel of a step is
// one of the image's.
struct WgTap {
    int H, Cs, Cu;
    int tx, ty, rp, ps;    // tile, row pitch (pixels) and plane pitch (bytes) of S
    int pu;                // pitch of U's planes (KMAJ: of its groups of 8 pixels)
    int mtiles, nt, nsplit, tcols;
    int ntx, nty, ntiles;
    uint32_t sbytes, stage, copied;   // offset of U, bytes of a buffer, bytes copied into it
    int swap, K9, chain, sets;
};

constexpr int kWgTapThreads = 192;

template <bool KMAJ, int ND>
__global__ void __launch_bounds__(kWgTapThreads)
k_conv3x3_wgrad_tap(WgTap t, const __grid_constant__ CUtensorMap mapS,
                    const __grid_constant__ CUtensorMap mapU, float* __restrict__ dW,
                    uint32_t* __restrict__ err)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) unsigned long long s_full[2], s_empty[2], s_accfull[2], s_accempty[2];
    __shared__ uint32_t s_tmem;

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const uint32_t base = smem_u32(smem);
    if (tid == 0) {
        for (int i = 0; i < 2; i++) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_full[i])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_empty[i])) : "memory");
        }
        for (int i = 0; i < 2; i++) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_accfull[i])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 4;" ::"r"(smem_u32(&s_accempty[i])) : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 5) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&s_tmem)),
                     "r"(t.tcols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;
    const int txy = t.ntx * t.nty;
    // blockIdx.y: (first vertical shift, row tile, column split)
    const int mi = (int)blockIdx.y % t.mtiles, ni = ((int)blockIdx.y / t.mtiles) % t.nsplit;
    const int dy0 = (int)blockIdx.y / (t.mtiles * t.nsplit);
    const int m0 = 128 * mi, n0 = t.nt * ni;
    const int mrows = t.Cs - m0 <= 64 ? 64 : 128;
    bool ok = true;

    if (warp == 4) {
        int i = 0;
        for (int tile = blockIdx.x; tile < t.ntiles; tile += gridDim.x, i++) {
            const int s = i & 1;
            if (i >= 2 && !mbar_wait(smem_u32(&s_empty[s]), (uint32_t)((i >> 1) - 1) & 1u)) {
                ok = false;
                break;
            }
            const int b = tile / txy, r = tile - b * txy, tyi = r / t.ntx, txi = r - tyi * t.ntx;
            const int x0 = txi * t.tx, y0 = tyi * t.ty;
            if (elect_one()) {
                const uint32_t sS = base + s * t.stage, bar = smem_u32(&s_full[s]);
                mbar_expect_tx(bar, t.copied);
                tma_load_5d(sS, &mapS, bar, 0, x0 - 1, y0 + dy0 - 1, m0 / 8, b);
                if (KMAJ) tma_load_5d(sS + t.sbytes, &mapU, bar, 0, n0, x0 / 8, y0, b);
                else tma_load_5d(sS + t.sbytes, &mapU, bar, 0, x0, y0, n0 / 8, b);
            }
            __syncwarp();
        }
        for (int j = i > 2 ? i - 2 : 0; j < i; j++)      // copies in flight land first
            if (!mbar_wait(smem_u32(&s_full[j & 1]), (uint32_t)(j >> 1) & 1u)) ok = false;
    } else if (warp == 5) {
        const uint32_t idesc = idesc_bf16(mrows, t.nt) | (1u << 15) | (KMAJ ? 0u : 1u << 16);
        const uint64_t ver = (uint64_t)1 << 46;
        const uint64_t hiA = (uint64_t)(t.ps >> 4) << 32 | (uint64_t)(128 >> 4) << 16 | ver;
        const uint64_t hiB = KMAJ ? (uint64_t)(128 >> 4) << 32 | (uint64_t)(t.pu >> 4) << 16 | ver
                                  : (uint64_t)(t.pu >> 4) << 32 | (uint64_t)(128 >> 4) << 16 | ver;
        const uint64_t stepB = KMAJ ? (uint64_t)((2 * t.pu) >> 4) : (uint64_t)(256 >> 4);
        WgChain ch;
        int i = 0;
        for (int tile = blockIdx.x; tile < t.ntiles; tile += gridDim.x, i++) {
            const int s = i & 1;
            const int rows = min(t.ty, t.H - ((tile % txy) / t.ntx) * t.ty);
            const int steps = rows * (t.tx >> 4);
            if (ch.full(steps, t.chain)) {
                if (elect_one()) mma_commit(smem_u32(&s_accfull[ch.set(t.sets)]));
                __syncwarp();
                ch.next();
                if (ch.use(t.sets) > 0 &&
                    !mbar_wait(smem_u32(&s_accempty[ch.set(t.sets)]), (ch.use(t.sets) - 1) & 1u)) {
                    ok = false;
                    break;
                }
            }
            if (!mbar_wait(smem_u32(&s_full[s]), (uint32_t)(i >> 1) & 1u)) {
                ok = false;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (elect_one()) {
                const uint32_t sS = base + s * t.stage;
                const uint32_t tacc = tmem + ch.set(t.sets) * (3 * ND * t.nt);
                uint32_t acc = ch.steps > 0;
                uint64_t da = hiA | (uint64_t)(sS >> 4), db = hiB | (uint64_t)((sS + t.sbytes) >> 4);
                for (int row = 0; row < rows; row++) {
                    uint64_t a = da;
                    for (int k = 0; k < t.tx; k += 16) {
#pragma unroll
                        for (int e = 0; e < ND; e++)
#pragma unroll
                            for (int dx = 0; dx < 3; dx++)
                                mma_bf16(tacc + (e * 3 + dx) * t.nt, a + e * t.rp + dx, db, idesc, acc);
                        acc = 1u;
                        a += 16;
                        db += stepB;
                    }
                    da += t.rp;
                }
                mma_commit(smem_u32(&s_empty[s]));
            }
            __syncwarp();
            ch.steps += steps;
        }
        if (ok && elect_one()) mma_commit(smem_u32(&s_accfull[ch.set(t.sets)]));
        __syncwarp();
    } else {
        const int row = mrows == 128 ? warp * 32 + lane : (lane < 16 ? warp * 16 + lane : t.Cs);
        const int c = m0 + row;
        WgChain ch;
        auto flush = [&]() {
            const int set = ch.set(t.sets);
            if (!mbar_wait(smem_u32(&s_accfull[set]), ch.use(t.sets) & 1u)) return false;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
            for (int e = 0; e < 3 * ND; e++) {
                const int tap0 = 3 * dy0 + e, tap = t.swap ? 8 - tap0 : tap0;
#pragma unroll 1
                for (int c0 = 0; c0 < t.nt; c0 += 16) {
                    float v[16];
                    __syncwarp();
                    tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)((set * 3 * ND + e) * t.nt + c0), v);
                    if (c < t.Cs) wg_add(dW, v, c, n0 + c0, tap, t.swap, t.Cs, t.Cu, t.K9);
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&s_accempty[set]));
            ch.next();
            return true;
        };
        for (int tile = blockIdx.x; tile < t.ntiles && ok; tile += gridDim.x) {
            const int steps = min(t.ty, t.H - ((tile % txy) / t.ntx) * t.ty) * (t.tx >> 4);
            if (ch.full(steps, t.chain)) ok = flush();
            ch.steps += steps;
        }
        if (ok) ok = flush();
    }
    if (!ok && lane == 0) atomicOr(err, kErrTimeout);
    __syncthreads();
    if (warp == 5)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(t.tcols)
                     : "memory");
}

static int ceil_div(int a, int b) { return (a + b - 1) / b; }

// MMA steps (16 pixels) an accumulator may run: what the gathered GEMM's split over
// the pixels gives this layer (gevo_conv3x3_wgrad's rule), so that no sum is truncated
// more often here than there.
static int wg_chain(int nb, int H, int W, int Cin)
{
    const long long P = (long long)nb * H * W, mtiles = (9 * Cin + 127) / 128;
    const long long want = ((long long)sm_count() * 8 + mtiles - 1) / mtiles;
    const long long split = std::max(2ll, std::min(P / 512, want)), slices = (P + 63) / 64;
    return (int)(4 * ((slices + split - 1) / split));
}

// Clocks of the MMAs of one K step (16 pixels, three vertical shifts) with Cs
// shifted and Cu unshifted channels (see conv_tc.cu for an MMA's cost).
static double wg_cost(int Cs, int Cu)
{
    const int g = 3 * Cs / 8, full = g / 16, rem = g % 16;
    const double nt = ceil_div(Cu, 16) * 16;
    double c = full * std::max(36.0 + nt / 4.0, nt / 2.0);
    if (rem) c += std::max((rem <= 8 ? 20.0 : 36.0) + nt / 4.0, nt / 2.0);
    return 3.0 * c;
}

// Shape of a layer's tiles, by estimated clocks; false where the operands do not
// fit.  A batch of 1024 pieces of S is 1500 clocks alone (its loads' latency) and 820
// of an SM's time, an asynchronous piece of U 0.6, a CTA 3000 to start; fitted to a
// sweep of tile and CTA counts over the prior's layers (within 4.5% of the fastest on
// average).
static bool wg_shape(WgTile& t, int nb, bool kmaj, size_t& smem, int& ctas_sm)
{
    t.kgs = t.Cs / 8;
    t.kgu = t.Cu / 8;
    const int g = 3 * t.kgs, full = g / 16, rem = g % 16;
    t.nmt = full + (rem ? 1 : 0);
    t.mlast = rem && rem <= 8 ? 64 : 128;
    t.nt = ceil_div(t.Cu, 16) * 16;
    if (t.nt > 256 || t.kgs > 128) return false;
    // all three vertical shifts in one CTA where their accumulators fit in tensor
    // memory; else a CTA per shift and as many row tiles as fit
    t.nd = t.nmt <= 4 && 3 * t.nmt * t.nt <= 512 ? 3 : 1;
    t.mper = t.nmt;
    if (t.nd == 1)
        while (t.nmt % t.mper || t.mper > 4 || t.mper * t.nt > 512) t.mper--;
    const int gy = t.nd == 3 ? 1 : 3 * t.nmt / t.mper;
    t.sets = 2 * t.nd * t.mper * t.nt <= 512 ? 2 : 1;
    t.tcols = 32;
    while (t.tcols < t.sets * t.nd * t.mper * t.nt) t.tcols *= 2;
    const size_t cap = (size_t)device_max_smem_optin() - 2048, sm_total = 228 * 1024;
    double best = 1e30;
    WgTile out = t;
    // the tile: TX a multiple of 16, so that a step of 16 pixels stays in one row
    for (int tx = 16; tx <= 64; tx += 16) {
        for (int ty = 2; ty <= 16; ty *= 2) {
            WgTile c = t;
            c.tx = tx;
            c.ty = ty;
            const int plane = (ty + c.nd - 1) * tx * 16;
            // pitches 64 / 32 / 16 bytes past a multiple of 128: the pieces eight
            // lanes store fall on distinct banks
            auto pad = [](int kg) { return kg == 2 ? 64 : kg == 4 ? 32 : 16; };
            c.ps = (plane + 127) / 128 * 128 + pad(c.kgs);
            c.pu = kmaj ? c.nt * 16 + 16 : (ty * tx * 16 + 127) / 128 * 128 + pad(c.kgu);
            c.sbytes = (uint32_t)(g * c.ps);
            const uint32_t ub = kmaj ? (uint32_t)(ty * tx / 8 * c.pu) : (uint32_t)(c.kgu * c.pu);
            c.stage = (c.sbytes + ub + 127) / 128 * 128;
            // the padding rows (columns) of the last row tile (U's last group) read
            // past their planes: keep them inside the allocation
            const size_t over_s = (size_t)(full * 16 + (rem ? (rem <= 8 ? 8 : 16) : 0)) * c.ps;
            const size_t over_u = c.sbytes + (kmaj ? (size_t)ub : (size_t)(c.nt / 8) * c.pu);
            const size_t bytes = c.stage + std::max({(size_t)c.stage, over_s, over_u}) + 128;
            if (bytes > cap || c.ps >= (1 << 18)) continue;
            c.ntx = ceil_div(c.W, tx);
            c.nty = ceil_div(c.H, ty);
            c.ntiles = c.ntx * c.nty * nb;
            const int fit = std::max(1, std::min({(int)(sm_total / (bytes + 1280)), 512 / c.tcols, 4}));
            const double mma = wg_cost(c.Cs, c.Cu) / gy * (tx * ty / 16);
            const double batches = std::ceil(c.kgs * (ty + 2) * (tx + 2) / 1024.0);
            const double pu = (double)c.kgu * tx * ty;
            const double lone = std::max(mma + 300.0, 500.0 + 1500.0 * batches + pu / 6.4);
            const double work = std::max(mma, 820.0 * batches + 0.6 * pu);
            for (int occ = 1; occ <= fit; occ++) {
                const double ctas = std::min((double)c.ntiles, std::max(1.0, std::floor((double)sm_count() * occ / gy)));
                const double act = std::min((double)occ, std::ceil(ctas * gy / sm_count()));
                const double time = 4000.0 + 3000.0 * act +
                                    std::ceil(c.ntiles / ctas) * std::max(lone, act * work);
                if (time < best) {
                    best = time;
                    out = c;
                    smem = bytes;
                    ctas_sm = occ;
                }
            }
        }
    }
    t = out;
    return best < 1e30;
}

template <bool KMAJ, int ND, int NM>
static gevo_status wg_launch(const WgTile& t, int nb, const void* S, const void* U, float* dWt,
                             size_t smem, int ctas_sm, uint32_t* err, cudaStream_t st)
{
    const int gy = t.nd == 3 ? 1 : 3 * t.nmt / t.mper;
    const int grid = std::max(1, std::min(t.ntiles, sm_count() * ctas_sm / gy));
    auto kern = k_conv3x3_wgrad<KMAJ, ND, NM>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    kern<<<dim3(grid, gy), kWgThreads, smem, st>>>(
        t, reinterpret_cast<const __nv_bfloat16*>(S), reinterpret_cast<const __nv_bfloat16*>(U), dWt,
        (size_t)nb * t.H * t.W, err);
    GEVO_CHECK_LAUNCH();
    return GEVO_OK;
}

template <bool KMAJ>
static gevo_status wg_dispatch(const WgTile& t, int nb, const void* S, const void* U, float* dWt,
                               size_t smem, int ctas_sm, uint32_t* err, cudaStream_t st)
{
#define GEVO_WG(ND, NM) \
    if (t.nd == ND && t.mper == NM) return wg_launch<KMAJ, ND, NM>(t, nb, S, U, dWt, smem, ctas_sm, err, st)
    GEVO_WG(3, 1);
    GEVO_WG(3, 2);
    GEVO_WG(3, 3);
    GEVO_WG(3, 4);
    GEVO_WG(1, 1);
    GEVO_WG(1, 2);
    GEVO_WG(1, 3);
    GEVO_WG(1, 4);
#undef GEVO_WG
    return GEVO_ERR_INVALID;
}

// Shape of the tap-by-tap kernel: tile, vertical shifts a CTA, column split.  A copy
// by TMA moves about 16 bytes a clock (its rows are 16 bytes).
static bool wt_shape(WgTap& t, int W, int nb, bool kmaj, int& nd_out, size_t& smem, int& ctas_sm, double& best)
{
    if (W % 16) return false;
    const size_t cap = (size_t)device_max_smem_optin() - 2048, sm_total = 228 * 1024;
    const double sms = sm_count();
    const int full = ceil_div(t.Cu, 16) * 16;
    best = 1e30;
    WgTap out = t;
    t.mtiles = ceil_div(t.Cs, 128);
    const int kS = std::min(t.Cs, 128) / 8;
    const int mlast = t.Cs - 128 * (t.mtiles - 1);
    for (int nd : {3, 1})
    for (int split = 1; split <= full / 16; split *= 2) {
        WgTap c = t;
        c.nt = ceil_div(ceil_div(full, split), 16) * 16;
        c.nsplit = ceil_div(full, c.nt);
        if (c.nt > 256 || 3 * nd * c.nt > 512) continue;
        c.sets = 2 * 3 * nd * c.nt <= 512 ? 2 : 1;
        c.tcols = 32;
        while (c.tcols < c.sets * 3 * nd * c.nt) c.tcols *= 2;
        const int gy = (3 / nd) * c.mtiles * c.nsplit;
        for (int tx = 16; tx <= 64; tx += 16) {
            if (W % tx) continue;
            for (int ty = 2; ty <= 16; ty *= 2) {
                c.tx = tx;
                c.ty = ty;
                c.rp = tx + 2;
                c.ps = c.rp * (ty + nd - 1) * 16;
                c.sbytes = ((uint32_t)(kS * c.ps) + 127) / 128 * 128;
                c.pu = kmaj ? c.nt * 16 : tx * ty * 16;
                const uint32_t ub = (uint32_t)(c.nt * tx * ty * 2);
                c.stage = (c.sbytes + ub + 127) / 128 * 128;
                c.copied = (uint32_t)(kS * c.ps) + ub;
                // an MMA's 64 or 128 rows may reach past the planes loaded
                const size_t over = (size_t)(mlast <= 64 && c.mtiles == 1 ? 8 : 16) * c.ps + 64;
                const size_t bytes = c.stage + std::max((size_t)c.stage, over) + 128;
                if (bytes > cap) continue;
                c.ntx = W / tx;
                c.nty = ceil_div(c.H, ty);
                c.ntiles = c.ntx * c.nty * nb;
                const int occ = std::max(1, std::min({(int)(sm_total / (bytes + 1280)), 512 / c.tcols, 3}));
                const double ctas = std::min((double)c.ntiles, std::max(1.0, std::floor(sms * occ / gy)));
                const double act = std::min((double)occ, std::ceil(ctas * gy / sms));
                const double one = std::max(36.0 + c.nt / 4.0, c.nt / 2.0);
                const double mma = tx * ty / 16 * 3.0 * nd * one;
                const double load = (double)kS * c.rp * (ty + nd - 1) + c.nt / 8.0 * tx * ty;
                const double tile = std::max({mma + 500.0, load + 1500.0, act * std::max(mma, load)});
                const double time = 5000.0 + std::ceil(c.ntiles / ctas) * tile +
                                    act * 3.0 * nd * (c.nt / 16) * 400.0;
                if (time < best) {
                    best = time;
                    out = c;
                    nd_out = nd;
                    smem = bytes;
                    ctas_sm = occ;
                }
            }
        }
    }
    t = out;
    return best < 1e30;
}

template <bool KMAJ, int ND>
static gevo_status wt_launch(const WgTap& t, int W, int nb, const void* S, const void* U, float* dWt,
                             size_t smem, int ctas_sm, uint32_t* err, cudaStream_t st)
{
    const int gy = (3 / ND) * t.mtiles * t.nsplit;
    const int grid = std::max(1, std::min(t.ntiles, sm_count() * ctas_sm / gy));
    CUtensorMap ms, mu;
    if (!nhwc_planes_map(ms, S, nb, t.H, W, t.Cs, t.rp, t.ty + ND - 1, std::min(t.Cs, 128) / 8))
        return GEVO_ERR_CUDA;
    const size_t HW = (size_t)t.H * W;
    if (KMAJ) {
        // dZ^T [channel][image][y][x]: boxes of 8 pixels, channels, pixel groups, rows
        const uint64_t dims[5] = {8, (uint64_t)t.Cu, (uint64_t)(W / 8), (uint64_t)t.H, (uint64_t)nb};
        const uint64_t strides[4] = {HW * nb * 2, 16, (uint64_t)W * 2, HW * 2};
        const uint32_t box[5] = {8, (uint32_t)t.nt, (uint32_t)(t.tx / 8), (uint32_t)t.ty, 1};
        if (!encode_map_bf16(mu, U, dims, strides, box)) return GEVO_ERR_CUDA;
    } else if (!nhwc_planes_map(mu, U, nb, t.H, W, t.Cu, t.tx, t.ty, t.nt / 8)) {
        return GEVO_ERR_CUDA;
    }
    auto kern = k_conv3x3_wgrad_tap<KMAJ, ND>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    kern<<<dim3(grid, gy), kWgTapThreads, smem, st>>>(t, ms, mu, dWt, err);
    GEVO_CHECK_LAUNCH();
    return GEVO_OK;
}

// dWt (zeroed by the caller) += the weight gradient.  Exactly one of dZ ([P][Cout])
// and dZt ([Cout][P]) is given.
gevo_status conv3x3_wgrad_bf16(int nb, int H, int W, int Cin, const void* X, int Cout,
                               const void* dZ, const void* dZt, float* dWt, uint32_t* err,
                               cudaStream_t st, bool& done)
{
    done = true;
    const bool kmaj = dZ == nullptr;
    if (kmaj && W % 8) {         // dZt's rows start off 16-byte boundaries
        done = false;
        return GEVO_OK;
    }
    // the roles: S the operand with fewer channels, except that dZt cannot be shifted
    const bool swap = !kmaj && Cout < Cin;
    const int Cs = swap ? Cout : Cin, Cu = swap ? Cin : Cout;
    const void* S = swap ? dZ : X;
    const void* U = swap ? X : kmaj ? dZt : dZ;
    size_t smem = 0;
    int ctas_sm = 1, nd = 3;
    if (Cs > 32) {
        WgTap t{};
        t.H = H;
        t.Cs = Cs;
        t.Cu = Cu;
        t.swap = swap;
        t.K9 = 9 * Cin;
        t.chain = wg_chain(nb, H, W, Cin);
        double clocks;
        if (wt_shape(t, W, nb, kmaj, nd, smem, ctas_sm, clocks)) {
            auto go = kmaj ? (nd == 3 ? wt_launch<true, 3> : wt_launch<true, 1>)
                           : (nd == 3 ? wt_launch<false, 3> : wt_launch<false, 1>);
            return go(t, W, nb, S, U, dWt, smem, ctas_sm, err, st);
        }
    }
    WgTile t{};
    t.H = H;
    t.W = W;
    t.K9 = 9 * Cin;
    t.swap = swap;
    t.Cs = Cs;
    t.Cu = Cu;
    t.chain = wg_chain(nb, H, W, Cin);
    // with dZt, more than 32 input channels and a width that is no multiple of 16 the
    // gathered GEMM is faster (64 -> 128 channels, 32 of 40x30: 38 us against 54)
    if (!(kmaj && Cs > 32) && wg_shape(t, nb, kmaj, smem, ctas_sm))
        return kmaj ? wg_dispatch<true>(t, nb, S, U, dWt, smem, ctas_sm, err, st)
                    : wg_dispatch<false>(t, nb, S, U, dWt, smem, ctas_sm, err, st);
    done = false;
    return GEVO_OK;
}

}  // namespace gevo
