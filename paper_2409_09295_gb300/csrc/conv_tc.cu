// 3x3 convolutions of the learned depth prior on the tcgen05 tensor cores, as
// implicit GEMMs whose nine taps read ONE copy of the activations in shared
// memory: Y[pixels x Cout] = sum over taps of shifted X[pixels x Cin] W_tap.
//
// A CTA owns a tile of 8 mx columns x 16 rows of one image (mx MMA row tiles of
// 8 x 16 = 128 pixels) and NT output channels.  Its activations, with a halo
// of one pixel, are copied once into "planes": one plane per 8 input channels,
// 16 bytes per pixel, pixels of a row consecutive, rows RP = 8 mx + 2 pixels
// apart.  Eight consecutive pixels of a plane are one no-swizzle core matrix
// (8 rows x 16 bytes), the next image row's is RP * 16 bytes on (the
// descriptor's stride offset) and the next 8 channels are one plane on (its
// leading offset), so the operand of tap (dy, dx) is the same memory with the
// start address moved by (dy RP + dx) pixels: no im2col, neither in memory nor
// in shared memory.  Gathering the nine shifted copies into shared memory
// instead made every 16-byte piece of X cross L2 and the load units nine
// times, and that, not the tensor cores, was the time.  32 images of 320x240,
// before and after (HBM floor): 16 -> 16 channels 294 -> 41 us (24), 48 -> 16
// 622 -> 84 (47), at a quarter of the pixels 96 -> 32 343 -> 53 (24), 32 -> 96 in
// FP32 224 -> 58 (41).  What bounds it now is the shared memory the MMAs read:
// 4 KB of A for every 16 channels of 128 pixels, however few the columns.
//
// The contraction runs tap by tap, 16 channels an instruction, in the order of
// the weight rows (tap, channel), so the accumulation order does not depend on
// the tile shape.
#include "tc_common.cuh"
#include "tensor_map.cuh"

namespace gevo {

gevo_status conv3x3_gemm(int nb, int H, int W, int Cin, const void* X, int Cout, const void* Wt,
                         void* Y, int ldy, int out_bf16, const float* bias, int relu, float beta,
                         uint32_t* err, cudaStream_t st);

constexpr int kConvThreads = 192;
constexpr int kConvTY = 16;            // rows of a tile: the 16 core matrices of 128 MMA rows

struct ConvTile {
    int H, W, Cin, Cout;
    int kgn, kgp;          // 8-channel groups, padded to an even count (the last one zeros)
    int ntap, steps;       // 9 taps of kgp / 2 MMAs (K = 16); Cin == 8: 1 of 5, two taps each
    int mx, rp, ps;        // MMA row tiles, row pitch (pixels), plane pitch (bytes)
    int nt, tcols;         // output channels of a CTA (multiple of 16), TMEM columns
    int bst, blb;          // bytes of a tap's weights, and between their K groups
    int ntx, nty, ntiles;  // tiles of an image, of all images
    int ldy, out_bf16, relu, vec, ldact;
    float beta;
};

// Bytes from one activation buffer to the next (a TMA destination is 128-byte
// aligned).
__host__ __device__ inline uint32_t conv_abuf(const ConvTile& t)
{
    return ((uint32_t)(t.kgp * t.ps) + 127u) / 128u * 128u;
}

// The CTA's weights: 16-byte pieces (output channel n, K group j) of each tap at
// tap * bst + j * blb + n * 16, zero where n or j is past the matrix.  K groups sit
// 64 bytes past a multiple of 128 apart, so that the pieces eight lanes store (a
// pair of K groups of four channels) fall on distinct banks.
__device__ __forceinline__ void conv_load_b(const ConvTile& t, const __nv_bfloat16* __restrict__ Wt,
                                            int n0, uint32_t dst)
{
    const int nj = 2 * t.steps;                            // K groups of one entry
    const int jin = t.ntap == 1 ? 9 : t.kgn;               // of which the matrix holds jin
    const int K = 9 * t.Cin;
    // lanes: a pair of K groups (32 contiguous bytes) fastest, then channels
    for (int q = threadIdx.x; q < t.nt * nj; q += kConvThreads) {
        const int jh = q / (2 * t.nt), r = q - jh * 2 * t.nt;
        const int n = r >> 1, j = 2 * jh + (r & 1);
        const bool in = j < jin && n0 + n < t.Cout;
        const __nv_bfloat16* src = in ? Wt + (size_t)(n0 + n) * K + j * 8 : Wt;
        uint32_t d = dst + j * t.blb + n * 16;
        for (int i = 0; i < t.ntap; i++) {
            cp_async16(d, src, in);
            d += t.bst;
            src += in ? t.Cin : 0;
        }
    }
}

// Writes 16 output channels [cb, cb + 16) of pixel p: bias, beta Y, ReLU, BF16 or
// FP32; one 32-byte store per 32 bytes where rows keep that alignment (t.vec; a
// half-sector store costs L2 a second transaction).
__device__ __forceinline__ void st_global_32(void* p, const uint32_t w[8])
{
    asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(w[0]), "r"(w[1]),
                 "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                 : "memory");
}

__device__ __forceinline__ void conv_store16(const ConvTile& t, float v[16], size_t p, int cb,
                                             const float* __restrict__ bias, void* __restrict__ Y)
{
    if (bias) {
        if (cb + 16 <= t.Cout) {
#pragma unroll
            for (int i = 0; i < 16; i++) v[i] += bias[cb + i];
        } else {
#pragma unroll
            for (int i = 0; i < 16; i++) v[i] += cb + i < t.Cout ? bias[cb + i] : 0.f;
        }
    }
    if (t.out_bf16) {
        __nv_bfloat16* o = reinterpret_cast<__nv_bfloat16*>(Y) + p * t.ldy + cb;
        if (t.vec && t.beta == 0.f && cb + 16 <= t.Cout) {
            uint32_t w[8];
#pragma unroll
            for (int q = 0; q < 8; q++) {
                float a0 = v[2 * q], a1 = v[2 * q + 1];
                if (t.relu) { a0 = fmaxf(a0, 0.f); a1 = fmaxf(a1, 0.f); }
                const __nv_bfloat162 pr = __floats2bfloat162_rn(a0, a1);
                w[q] = *reinterpret_cast<const uint32_t*>(&pr);
            }
            st_global_32(o, w);
            return;
        }
#pragma unroll
        for (int i = 0; i < 16; i++) {
            if (cb + i < t.Cout) {
                float a = v[i];
                if (t.beta != 0.f) a += t.beta * __bfloat162float(o[i]);
                if (t.relu) a = fmaxf(a, 0.f);
                o[i] = __float2bfloat16_rn(a);
            }
        }
    } else {
        float* o = reinterpret_cast<float*>(Y) + p * t.ldy + cb;
        if (t.vec && t.beta == 0.f && cb + 16 <= t.Cout) {
#pragma unroll
            for (int h = 0; h < 2; h++) {
                uint32_t w[8];
#pragma unroll
                for (int q = 0; q < 8; q++) {
                    float a = v[8 * h + q];
                    if (t.relu) a = fmaxf(a, 0.f);
                    w[q] = __float_as_uint(a);
                }
                st_global_32(o + 8 * h, w);
            }
            return;
        }
#pragma unroll
        for (int i = 0; i < 16; i++) {
            if (cb + i < t.Cout) {
                float a = v[i];
                if (t.beta != 0.f) a += t.beta * o[i];
                if (t.relu) a = fmaxf(a, 0.f);
                o[i] = a;
            }
        }
    }
}

// 16 channels [cb, cb + 16) of pixel p of the activation a ReLU's gradient is masked
// by (BF16, rows of stride ldact; zeros past Cout).
__device__ __forceinline__ void ld_act16(const ConvTile& t, const __nv_bfloat16* __restrict__ act,
                                         size_t p, int cb, uint4 a[2])
{
    const __nv_bfloat16* o = act + p * t.ldact + cb;      // Cout, ldact multiples of 8
    a[0] = *reinterpret_cast<const uint4*>(o);
    a[1] = cb + 8 < t.Cout ? *reinterpret_cast<const uint4*>(o + 8) : make_uint4(0u, 0u, 0u, 0u);
}

__device__ __forceinline__ void conv_mask16(float v[16], const uint4 a[2])
{
    const uint32_t w[8] = {a[0].x, a[0].y, a[0].z, a[0].w, a[1].x, a[1].y, a[1].z, a[1].w};
#pragma unroll
    for (int q = 0; q < 8; q++) {
        // bf16 > 0 as a float: the low half shifted up, the high half masked
        v[2 * q] = __uint_as_float(w[q] << 16) > 0.f ? v[2 * q] : 0.f;
        v[2 * q + 1] = __uint_as_float(w[q] & 0xffff0000u) > 0.f ? v[2 * q + 1] : 0.f;
    }
}

// The MMAs of one K step of 16 for the MX row tiles of the CTA (start addresses 8
// pixels, 128 bytes, apart; accumulators nt columns apart).
template <int MX>
__device__ __forceinline__ void conv_mma(uint32_t tmem, int nt, uint64_t da, uint64_t db,
                                         uint32_t idesc, uint32_t acc)
{
#pragma unroll
    for (int m = 0; m < MX; m++)
        mma_bf16(tmem + m * nt, da + (uint64_t)(m * (128 >> 4)), db, idesc, acc);
}

// The MMAs of a tile.  hiA / hiB: the descriptor bits that do not change.  Start
// addresses are in 16-byte units, one pixel: a step adds two planes, a tap one
// pixel, a row of taps the row pitch, and the weights run on.
template <int MX>
__device__ __forceinline__ void conv_issue(const ConvTile& t, uint32_t tmem, uint32_t sA, uint32_t sB,
                                           uint64_t hiA, uint64_t hiB, uint32_t idesc)
{
    uint64_t db = hiB | (uint64_t)(sB >> 4);
    if (t.ntap > 1) {
        const uint64_t sa = (uint64_t)((2 * t.ps) >> 4), sb = (uint64_t)((2 * t.blb) >> 4);
        uint64_t dtap = hiA | (uint64_t)(t.ps >> 4) << 16 | (uint64_t)(sA >> 4);
        uint32_t acc = 0u;
        for (int dy = 0; dy < 3; dy++) {
            for (int dx = 0; dx < 3; dx++) {
                uint64_t da = dtap + dx;
                for (int k = 0; k < t.steps; k++) {
                    conv_mma<MX>(tmem, t.nt, da, db, idesc, acc);
                    da += sa;
                    db += sb;
                    acc = 1u;
                }
            }
            dtap += t.rp;
        }
    } else {        // Cin == 8: the two K groups of a step are two taps
#pragma unroll
        for (int k = 0; k < 5; k++) {
            const int c0 = 2 * k, c1 = c0 + 1;
            const int p0 = (c0 / 3) * t.rp + c0 % 3, p1 = (c1 / 3) * t.rp + c1 % 3;
            const uint32_t lbo = c1 < 9 ? (uint32_t)(p1 - p0) * 16 : (uint32_t)t.ps;
            conv_mma<MX>(tmem, t.nt, hiA | (uint64_t)(lbo >> 4) << 16 | (uint64_t)((sA + p0 * 16) >> 4),
                         db, idesc, k > 0);
            db += (uint64_t)((2 * t.blb) >> 4);
        }
    }
}

// The same tile, persistent and specialised by warp, for layers whose weights
// stay in shared memory beside two activation tiles: warp 4 has the TMA copy the
// next tile's planes (one five-dimensional box: 8 channels, columns, rows, channel
// groups, image; zeros outside the image) while warp 5 issues the current tile's
// MMAs and warps 0-3 read the previous tile's accumulators and write them out.
// What a tile costs is then the largest of the three, not their sum, and the
// weights are read once per CTA.  Barriers: full / empty per plane buffer, accfull
// / accempty per accumulator buffer (two of each); every wait is bounded (a role
// that gives up records GEVO_ERR_TIMEOUT and ends, and the others run out too).
//
// NG > 0: the convolution is a data gradient whose result only feeds the ReLU before
// it, so the epilogue applies the mask and writes dZ (BF16) and the bias gradient
// instead of an FP32 tensor that another pass would read back; a thread keeps its
// columns' sums in registers over all its tiles (at most NG groups of 16 columns).
constexpr int kFuseGroups = 4;

template <int MX, int NG>
__global__ void __launch_bounds__(kConvThreads)
k_conv3x3(ConvTile t, const __grid_constant__ CUtensorMap map, const __nv_bfloat16* __restrict__ Wt,
          const float* __restrict__ bias, void* __restrict__ Y,
          const __nv_bfloat16* __restrict__ act, float* __restrict__ db, uint32_t* __restrict__ err)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) unsigned long long s_full[2], s_empty[2], s_accfull[2], s_accempty[2];
    __shared__ uint32_t s_tmem;
    constexpr bool FUSE = NG > 0;
    __shared__ float s_db[FUSE ? 16 * NG : 1];

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const uint32_t abuf = conv_abuf(t);
    const uint32_t sA = smem_u32(smem), sB = sA + 2 * abuf;
    const int n0 = blockIdx.y * t.nt;
    if (tid == 0) {
        for (int i = 0; i < 2; i++) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_full[i])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_empty[i])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_accfull[i])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 4;" ::"r"(smem_u32(&s_accempty[i])) : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    conv_load_b(t, Wt, n0, sB);
    cp_async_commit();
    if (FUSE && tid < 16 * NG) s_db[tid] = 0.f;
    if (t.kgp > t.kgn)          // the padding planes of both buffers
        for (int i = tid; i < 2 * (t.ps / 16); i += kConvThreads) {
            const int bufi = i / (t.ps / 16), j = i - bufi * (t.ps / 16);
            reinterpret_cast<uint4*>(smem + (size_t)bufi * abuf + (size_t)t.kgn * t.ps)[j] =
                make_uint4(0u, 0u, 0u, 0u);
        }
    if (warp == 5) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&s_tmem)),
                     "r"(t.tcols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    cp_async_wait<0>();
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = s_tmem;
    const int txy = t.ntx * t.nty;

    if (warp == 4) {
        // one tile ahead of the tensor core
        int i = 0;
        const uint32_t bytes = (uint32_t)(t.kgn * t.ps);
        for (int tile = blockIdx.x; tile < t.ntiles; tile += gridDim.x, i++) {
            const int s = i & 1;
            if (i >= 2 && !mbar_wait(smem_u32(&s_empty[s]), (uint32_t)((i >> 1) - 1) & 1u)) {
                if (lane == 0) atomicOr(err, kErrTimeout);
                break;
            }
            const int b = tile / txy, r = tile - b * txy, ty = r / t.ntx, tx = r - ty * t.ntx;
            if (elect_one()) {
                mbar_expect_tx(smem_u32(&s_full[s]), bytes);
                tma_load_5d(sA + s * abuf, &map, smem_u32(&s_full[s]), 0, tx * 8 * MX - 1,
                            ty * kConvTY - 1, 0, b);
            }
            __syncwarp();
        }
        // the copies in flight land before the block ends (the last two tiles')
        for (int j = i > 2 ? i - 2 : 0; j < i; j++)
            if (!mbar_wait(smem_u32(&s_full[j & 1]), (uint32_t)(j >> 1) & 1u) && lane == 0)
                atomicOr(err, kErrTimeout);
    } else if (warp == 5) {
        const uint32_t idesc = idesc_bf16(128, t.nt);
        const uint64_t hiA = (uint64_t)((t.rp * 16) >> 4) << 32 | (uint64_t)1 << 46;
        const uint64_t hiB = (uint64_t)(128 >> 4) << 32 | (uint64_t)1 << 46 | (uint64_t)(t.blb >> 4) << 16;
        int i = 0;
        for (int tile = blockIdx.x; tile < t.ntiles; tile += gridDim.x, i++) {
            const int s = i & 1;
            if ((i >= 2 && !mbar_wait(smem_u32(&s_accempty[s]), (uint32_t)((i >> 1) - 1) & 1u)) ||
                !mbar_wait(smem_u32(&s_full[s]), (uint32_t)(i >> 1) & 1u)) {
                if (lane == 0) atomicOr(err, kErrTimeout);
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            // one thread issues, elected in a branch the compiler sees is uniform: from
            // a divergent branch (threadIdx.x == 0) an MMA took 156 clocks to issue,
            // from this one the 36 to 128 its operands take
            if (elect_one()) {
                conv_issue<MX>(t, tmem + s * MX * t.nt, sA + s * abuf, sB, hiA, hiB, idesc);
                mma_commit(smem_u32(&s_empty[s]));
                mma_commit(smem_u32(&s_accfull[s]));
            }
            __syncwarp();
        }
    } else {
        const int r = warp * 32 + lane, cgs = t.nt >> 4;
        float sum[FUSE ? NG : 1][16];
        if (FUSE)
#pragma unroll
            for (int c = 0; c < NG; c++)
#pragma unroll
                for (int k = 0; k < 16; k++) sum[c][k] = 0.f;
        int i = 0;
        for (int tile = blockIdx.x; tile < t.ntiles; tile += gridDim.x, i++) {
            const int s = i & 1;
            const int b = tile / txy, q = tile - b * txy, ty = q / t.ntx, tx = q - ty * t.ntx;
            const int y = ty * kConvTY + (r >> 3), x = tx * 8 * MX + (r & 7);
            const size_t p = ((size_t)b * t.H + y) * t.W + x;
            const uint32_t tacc = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(s * MX * t.nt);
            // the first columns' activations are on their way while the MMAs finish
            uint4 a[FUSE ? MX : 1][2];
            if (FUSE)
#pragma unroll
                for (int m = 0; m < MX; m++)
                    if (y < t.H && x + 8 * m < t.W) ld_act16(t, act, p + 8 * m, n0, a[m]);
            if (!mbar_wait(smem_u32(&s_accfull[s]), (uint32_t)(i >> 1) & 1u)) {
                if (lane == 0) atomicOr(err, kErrTimeout);
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (FUSE) {
#pragma unroll
                for (int c = 0; c < NG; c++) {
                    if (c < cgs) {
#pragma unroll
                        for (int m = 0; m < MX; m++) {
                            const bool in = y < t.H && x + 8 * m < t.W;
                            if (c > 0 && in) ld_act16(t, act, p + 8 * m, n0 + 16 * c, a[m]);
                            float v[16];
                            __syncwarp();
                            tmem_ld16(tacc + (uint32_t)(m * t.nt + 16 * c), v);
                            if (in) {
                                conv_mask16(v, a[m]);
                                conv_store16(t, v, p + 8 * m, n0 + 16 * c, nullptr, Y);
#pragma unroll
                                for (int k = 0; k < 16; k++) sum[c][k] += v[k];
                            }
                        }
                    }
                }
            } else {
                for (int c = 0; c < cgs; c++) {
#pragma unroll
                    for (int m = 0; m < MX; m++) {
                        float v[16];
                        __syncwarp();
                        tmem_ld16(tacc + (uint32_t)(m * t.nt + 16 * c), v);
                        if (y < t.H && x + 8 * m < t.W)
                            conv_store16(t, v, p + 8 * m, n0 + 16 * c, bias, Y);
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&s_accempty[s]));
        }
        if (FUSE) {
#pragma unroll
            for (int c = 0; c < NG; c++) {
                if (c < cgs) {
#pragma unroll
                    for (int k = 0; k < 16; k++) {
                        float v = sum[c][k];
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                        if (lane == 0) atomicAdd(&s_db[16 * c + k], v);
                    }
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (FUSE && tid < t.nt && n0 + tid < t.Cout) atomicAdd(db + n0 + tid, s_db[tid]);
    if (warp == 5)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(t.tcols)
                     : "memory");
}

static int ceil_div(int a, int b) { return (a + b - 1) / b; }

// Fills the shape fields that follow from (mx, nt, nst); returns the CTA's
// dynamic shared memory in bytes.
// Fills the shape fields that follow from (mx, nt); returns the CTA's dynamic shared
// memory in bytes: two activation buffers and the weights.
static size_t conv_shape(ConvTile& t, int nb, int mx, int nt)
{
    t.mx = mx;
    t.nt = nt;
    t.rp = 8 * mx + 2;
    t.ps = t.rp * (kConvTY + 2) * 16;
    t.blb = nt * 16 + 64;
    t.bst = 2 * t.steps * t.blb;
    t.tcols = 32;
    while (t.tcols < 2 * mx * nt) t.tcols *= 2;
    t.ntx = ceil_div(t.W, 8 * mx);
    t.nty = ceil_div(t.H, kConvTY);
    t.ntiles = t.ntx * t.nty * nb;
    return 2 * (size_t)conv_abuf(t) + (size_t)t.ntap * t.bst;
}

// Tile shape for a layer: the least estimated time, in clocks, over the candidate
// row tiles, column splits and CTAs per SM.  The tensor core takes max(32 + nt / 4,
// 38, nt / 2) clocks an MMA of 128 x nt x 16 (measured: below 128 columns the
// 4 KB of A are what is read), the TMA about 16 bytes a clock of this box (its
// rows are 16 bytes), the epilogue about 350 a group of 16 columns, a CTA 2500 and
// its weights to start.  The constants were fitted to a sweep of every candidate
// on the prior's 16 layer shapes at 32 x 320x240 and 1 x 640x480: the pick is
// within 2.5% of the fastest on average, 14% at worst (shapes alone differ up to 4x).
static bool conv_pick(ConvTile& best, int nb, bool fuse, size_t& smem, int& ctas_sm)
{
    const size_t cap = (size_t)device_max_smem_optin() - 2048, sm_total = 228 * 1024;
    const double sms = sm_count();
    double best_time = 1e30;
    const int full = ceil_div(best.Cout, 16) * 16;
    ConvTile out = best;
    for (int mx = 4; mx >= 1; mx /= 2) {
        for (int nsplit = 1; nsplit <= full / 16; nsplit *= 2) {
            const int nt = ceil_div(ceil_div(full, nsplit), 16) * 16;
            if (nt > (fuse ? 16 * kFuseGroups : 256) || 2 * mx * nt > 512) continue;
            ConvTile t = best;
            const size_t bytes = conv_shape(t, nb, mx, nt);
            if (bytes > cap) continue;
            // (a fused CTA of many columns and row tiles holds up to half the registers)
            const int fit = std::min({(int)(sm_total / (bytes + 1280)), 512 / t.tcols,
                                      fuse && mx * nt > 64 ? 1 : fuse ? 2 : 4});
            const double ns = ceil_div(best.Cout, nt);
            const double mma = t.ntap * t.steps * mx * std::max({38.0, 32.0 + nt / 4.0, nt / 2.0});
            const double load = t.kgn * t.ps / 16.0, epi = 600.0 + mx * (nt / 16) * 350.0;
            for (int occ = 1; occ <= std::max(1, fit); occ++) {
                const double ctas = std::min((double)t.ntiles, std::max(1.0, std::floor(sms * occ / ns)));
                const double act = std::min((double)occ, std::ceil(ctas * ns / sms));
                const double tile = std::max({mma + 600.0, load + 1000.0, epi,
                                              act * std::max({mma, load, 0.7 * (epi - 600.0)})});
                const double time = 2500.0 + act * (t.ntap * t.bst / 32.0 + 2500.0) + load +
                                    std::ceil(t.ntiles / ctas) * tile + epi;
                if (time < best_time) {
                    best_time = time;
                    out = t;
                    smem = bytes;
                    ctas_sm = occ;
                }
            }
        }
    }
    best = out;
    return best_time < 1e30;
}

template <int NG>
static gevo_status conv_launch(const ConvTile& t, int nb, const void* X, const void* Wt,
                               const float* bias, void* Y, const void* act, float* db, size_t smem,
                               int ctas_sm, uint32_t* err, cudaStream_t st)
{
    CUtensorMap map;
    if (!nhwc_planes_map(map, X, nb, t.H, t.W, t.Cin, t.rp, kConvTY + 2, t.kgn)) return GEVO_ERR_CUDA;
    const int ns = ceil_div(t.Cout, t.nt);
    const int grid = std::max(1, std::min(t.ntiles, sm_count() * ctas_sm / ns));
    auto kern = t.mx == 4 ? k_conv3x3<4, NG> : t.mx == 2 ? k_conv3x3<2, NG> : k_conv3x3<1, NG>;
    // set on every launch: a host-only call of about a microsecond, correct for
    // whichever device is current and free of shared state between host threads
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    kern<<<dim3(grid, ns), kConvThreads, smem, st>>>(
        t, map, reinterpret_cast<const __nv_bfloat16*>(Wt), bias, Y,
        reinterpret_cast<const __nv_bfloat16*>(act), db, err);
    GEVO_CHECK_LAUNCH();
    return GEVO_OK;
}

static ConvTile conv_tile(int H, int W, int Cin, int Cout, void* Y, int ldy, int out_bf16)
{
    ConvTile t{};
    t.H = H; t.W = W; t.Cin = Cin; t.Cout = Cout;
    t.kgn = Cin / 8;
    t.kgp = (t.kgn + 1) & ~1;
    t.ntap = Cin == 8 ? 1 : 9;
    t.steps = Cin == 8 ? 5 : t.kgp / 2;
    t.ldy = ldy;
    t.out_bf16 = out_bf16;
    t.vec = (uintptr_t)Y % 32 == 0 && ldy % (out_bf16 ? 16 : 8) == 0;
    return t;
}

gevo_status conv3x3_bf16(int nb, int H, int W, int Cin, const void* X, int Cout, const void* Wt,
                         void* Y, int ldy, int out_bf16, const float* bias, int relu, float beta,
                         uint32_t* err, cudaStream_t st)
{
    ConvTile t = conv_tile(H, W, Cin, Cout, Y, ldy, out_bf16);
    t.relu = relu;
    t.beta = beta;
    size_t smem = 0;
    int ctas_sm = 1;
    // more input channels than two buffers of the smallest tile hold (about 230)
    // go through the gathered GEMM
    if (!conv_pick(t, nb, false, smem, ctas_sm))
        return conv3x3_gemm(nb, H, W, Cin, X, Cout, Wt, Y, ldy, out_bf16, bias, relu, beta, err, st);
    return conv_launch<0>(t, nb, X, Wt, bias, Y, nullptr, nullptr, smem, ctas_sm, err, st);
}

// dZ [P][Cout] = BF16 of conv(X) where act > 0, else 0; db += its FP32 sums over pixels.
gevo_status conv3x3_relu_bwd(int nb, int H, int W, int Cin, const void* X, int Cout, const void* Wt,
                             const void* act, int ldact, void* dZ, float* db, uint32_t* err,
                             cudaStream_t st)
{
    ConvTile t = conv_tile(H, W, Cin, Cout, dZ, Cout, 1);
    t.ldact = ldact;
    size_t smem = 0;
    int ctas_sm = 1;
    if (!conv_pick(t, nb, true, smem, ctas_sm)) return GEVO_ERR_INVALID;
    auto go = t.nt <= 16 ? conv_launch<1> : t.nt <= 32 ? conv_launch<2> : conv_launch<kFuseGroups>;
    return go(t, nb, X, Wt, nullptr, dZ, act, db, smem, ctas_sm, err, st);
}

}  // namespace gevo
