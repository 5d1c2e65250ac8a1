// Initialisation of new Gaussians from depth (Section III-A).
//
// The paper builds a photometric cost volume over N keyframes (Eq. 1): for each
// pixel u of the newest keyframe I_{N-1}, downsampled 4x, and each of 64 depth
// hypotheses spaced linearly over 0.25-25 m, V(u, d) = mean over the other
// keyframes of |I_{N-1}(u) - I_i(pi(u, d, T^i_{N-1}))|, then extracts depth with
// belief propagation and upsamples it edge-aware before SPGF* makes Gaussians.
// Here: the cost volume as Eq. 1 defines it (grey = mean of RGB, bilinear
// sampling, out-of-image samples left out of the mean), winner-take-all over
// hypotheses in place of belief propagation, nearest x4 upsampling in place of
// the edge-aware filter, and one Gaussian per selected pixel in place of SPGF*
// (the parts the paper only cites).  The learned depth prior feeds the same
// unprojection.
#include "../../include/gevo_prior.h"
#include "gevo_internal.cuh"

namespace gevo {

// 4x4 box average of the mean of RGB: planar [nk][3][H][W] -> [nk][H/4][W/4]
// vec: rows start on 16-byte boundaries, one load per row of a box
__global__ void k_grey4(int nk, int H, int W, const float* __restrict__ rgb, float* __restrict__ g, int vec)
{
    const int h = H / 4, w = W / 4;
    const size_t n = (size_t)nk * h * w;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const int x = (int)(i % w);
        const size_t t = i / w;
        const int y = (int)(t % h);
        const size_t k = t / h;
        float acc = 0.f;
        for (int ch = 0; ch < 3; ch++) {
            const float* p = rgb + (k * 3 + ch) * (size_t)H * W;
#pragma unroll
            for (int dy = 0; dy < 4; dy++) {
                const float* r = p + (size_t)(4 * y + dy) * W + 4 * x;
                if (vec) {
                    const float4 q = *reinterpret_cast<const float4*>(r);
                    acc += q.x;
                    acc += q.y;
                    acc += q.z;
                    acc += q.w;
                } else {
                    for (int dx = 0; dx < 4; dx++) acc += r[dx];
                }
            }
        }
        g[i] = acc * (1.f / 48.f);
    }
}

// Bilinear sample; pixel i is sampled at coordinate i.  ok false outside the image (the
// value is then some pixel's): no branch, so that several samples' loads are in flight.
__device__ __forceinline__ float bilinear(const float* __restrict__ img, int w, int h, float u, float v,
                                          bool& ok)
{
    ok = u >= 0.f && v >= 0.f && u <= (float)(w - 1) && v <= (float)(h - 1);
    const int x0 = ok ? min((int)u, w - 2 < 0 ? 0 : w - 2) : 0, y0 = ok ? min((int)v, h - 2 < 0 ? 0 : h - 2) : 0;
    const float fx = u - (float)x0, fy = v - (float)y0;
    const float* q = img + y0 * w + x0;
    const float a = q[0], b = q[1];
    const float c = q[w], d = q[w + 1];
    return (1.f - fy) * ((1.f - fx) * a + fx * b) + fy * ((1.f - fx) * c + fx * d);
}

// cams: [nk][16] (R, t, fx, fy, cx, cy) of the full-resolution keyframes;
// the reference is keyframe `ref`, the sources all the others.
// A block takes 32 neighbouring pixels and 32 hypotheses, a warp four hypotheses of the
// 32 pixels: its lanes' samples lie side by side in a source, where 32 hypotheses of one
// pixel lie strewn along its epipolar line, a cache line each.  A source's camera is
// four 16-byte loads from shared memory for the four hypotheses, whose samples are
// independent chains; the costs turn round in shared memory for the store.  Eight 640x480
// keyframes, 64 hypotheses: 44 us with a thread per (pixel, hypothesis), 32 now, bound by
// the arithmetic of a sample (two IEEE divisions, four taps).
constexpr int kCostMaxCams = 64;     // cameras in shared memory; more are read from memory
constexpr int kCostPer = 4;          // hypotheses per thread

__global__ void __launch_bounds__(256)
k_cost_volume(int nk, int ref, int h, int w, const float* __restrict__ grey,
              const float* __restrict__ cams, int nd, float d0, float d1, float* __restrict__ V)
{
    __shared__ float4 s_cams[4 * kCostMaxCams];
    __shared__ float s_v[32][33];
    const bool in_smem = nk <= kCostMaxCams;
    if (in_smem)
        for (int i = threadIdx.x; i < 16 * nk; i += 256)
            reinterpret_cast<float*>(s_cams)[i] = cams[i];
    __syncthreads();
    const float* cr = cams + 16 * ref;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, hw = h * w;
    const int nq = (hw + 31) / 32, nkb = (nd + 31) / 32;
    const float fx = cr[12] * 0.25f, fy = cr[13] * 0.25f, cx = cr[14] * 0.25f, cy = cr[15] * 0.25f;
    for (size_t t = blockIdx.x; t < (size_t)nq * nkb; t += gridDim.x) {
        const int q0 = (int)(t / nkb) * 32, kb = (int)(t % nkb) * 32;
        const int q = min(q0 + lane, hw - 1), x = q % w, y = q / w;
        const float I0 = grey[(size_t)ref * hw + q];
        float pw[kCostPer][3], acc[kCostPer];
        int cnt[kCostPer];
#pragma unroll
        for (int i = 0; i < kCostPer; i++) {
            const float d = d0 + (d1 - d0) * (float)(kb + warp + 8 * i) / (float)(nd - 1);
            // camera-frame point of pixel (x, y) at depth d (pixel i sits at i + 0.5 - c)
            const float pc[3] = {((float)x + 0.5f - cx) / fx * d, ((float)y + 0.5f - cy) / fy * d, d};
#pragma unroll
            for (int j = 0; j < 3; j++)
                pw[i][j] = cr[j] * (pc[0] - cr[9]) + cr[3 + j] * (pc[1] - cr[10]) +
                           cr[6 + j] * (pc[2] - cr[11]);
            acc[i] = 0.f;
            cnt[i] = 0;
        }
#pragma unroll 1
        for (int s = 0; s < nk; s++) {
            if (s == ref) continue;
            float cs[16];
            if (in_smem) {
#pragma unroll
                for (int j = 0; j < 4; j++) {
                    const float4 c = s_cams[4 * s + j];
                    cs[4 * j] = c.x; cs[4 * j + 1] = c.y; cs[4 * j + 2] = c.z; cs[4 * j + 3] = c.w;
                }
            } else {
#pragma unroll
                for (int j = 0; j < 16; j++) cs[j] = cams[16 * s + j];
            }
            const float* img = grey + (size_t)s * hw;
#pragma unroll
            for (int i = 0; i < kCostPer; i++) {
                float p[3];
#pragma unroll
                for (int j = 0; j < 3; j++)
                    p[j] = cs[3 * j] * pw[i][0] + cs[3 * j + 1] * pw[i][1] + cs[3 * j + 2] * pw[i][2] +
                           cs[9 + j];
                const float u = cs[12] * 0.25f * p[0] / p[2] + cs[14] * 0.25f - 0.5f;
                const float v = cs[13] * 0.25f * p[1] / p[2] + cs[15] * 0.25f - 0.5f;
                bool ok;
                const float Is = bilinear(img, w, h, u, v, ok);
                ok = ok && p[2] > 1e-3f;
                acc[i] += ok ? fabsf(I0 - Is) : 0.f;
                cnt[i] += ok ? 1 : 0;
            }
        }
#pragma unroll
        for (int i = 0; i < kCostPer; i++)
            s_v[lane][warp + 8 * i] = cnt[i] > 0 ? acc[i] / (float)cnt[i] : 1.f;
        __syncthreads();
        for (int r = warp; r < 32 && q0 + r < hw; r += 8)
            if (kb + lane < nd) V[(size_t)(q0 + r) * nd + kb + lane] = s_v[r][lane];
        __syncthreads();
    }
}

// winner-take-all over hypotheses (lowest cost, then lowest index), nearest x4
// upsampling to full resolution
// A warp per quarter-resolution pixel: the lanes read its costs together and the
// winner fills the 4 x 4 pixels (one thread per full-resolution pixel read the same
// costs sixteen times over, one after another: 640x480 and 64 hypotheses, 29 us against 5.7).
__global__ void __launch_bounds__(256)
k_wta_up4(int h, int w, int nd, float d0, float d1, const float* __restrict__ V,
          float* __restrict__ depth)
{
    const int lane = threadIdx.x & 31, W = 4 * w;
    const size_t hw = (size_t)h * w, warps = ((size_t)gridDim.x * blockDim.x) >> 5;
    for (size_t p = (blockIdx.x * (size_t)blockDim.x + threadIdx.x) >> 5; p < hw; p += warps) {
        const float* v = V + p * nd;
        float bv = INFINITY;
        int bi = 0x7fffffff;
        for (int k = lane; k < nd; k += 32) {
            const float c = v[k];
            if (c < bv || (c == bv && k < bi)) { bv = c; bi = k; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (ov < bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
        }
        // nothing is below a NaN in first place, and NaNs elsewhere never win
        const float v0 = v[0];
        if (v0 != v0 || bi == 0x7fffffff) bi = 0;
        if (lane < 16) {
            const int x = (int)(p % w), y = (int)(p / w);
            depth[(size_t)(4 * y + (lane >> 2)) * W + 4 * x + (lane & 3)] =
                d0 + (d1 - d0) * (float)bi / (float)(nd - 1);
        }
    }
}

__device__ __forceinline__ uint32_t hash32(uint32_t x)
{
    x ^= x >> 16; x *= 0x7feb352du; x ^= x >> 15; x *= 0x846ca68bu; x ^= x >> 16;
    return x;
}

// New Gaussians from a depth map: every masked pixel whose hash falls under
// `keep` becomes one Gaussian at its back-projected point, coloured by the
// pixel (SH DC (c - 0.5) / Y00, higher bands 0), isotropic scale
// scale_px * depth / f, identity rotation, opacity `opac`.
__global__ void k_unproject(int H, int W, const float* __restrict__ rgb, const float* __restrict__ depth,
                            const float* __restrict__ mask, const float* __restrict__ cam,
                            uint32_t keep, uint32_t seed, float scale_px, float opac, int K,
                            uint32_t* __restrict__ counter, int cap, float* __restrict__ means,
                            float* __restrict__ scales, float* __restrict__ quats,
                            float* __restrict__ opacities, float* __restrict__ sh)
{
    const size_t P = (size_t)H * W;
    const float fx = cam[12], fy = cam[13], cx = cam[14], cy = cam[15];
    const float kY00 = 0.28209479177387814f;
    for (size_t p = blockIdx.x * (size_t)blockDim.x + threadIdx.x; p < P; p += (size_t)gridDim.x * blockDim.x) {
        if (!(mask[p] > 0.5f)) continue;
        if (hash32((uint32_t)p * 2654435761u + seed) > keep) continue;
        const uint32_t slot = atomicAdd(counter, 1u);
        if ((int)slot >= cap) continue;
        const int x = (int)(p % W), y = (int)(p / W);
        const float d = depth[p];
        const float pc[3] = {((float)x + 0.5f - cx) / fx * d, ((float)y + 0.5f - cy) / fy * d, d};
        for (int j = 0; j < 3; j++)
            means[3 * slot + j] = cam[j] * (pc[0] - cam[9]) + cam[3 + j] * (pc[1] - cam[10]) +
                                  cam[6 + j] * (pc[2] - cam[11]);
        const float s = scale_px * d / fx;
        scales[3 * slot] = s; scales[3 * slot + 1] = s; scales[3 * slot + 2] = s;
        quats[4 * slot] = 1.f; quats[4 * slot + 1] = 0.f; quats[4 * slot + 2] = 0.f; quats[4 * slot + 3] = 0.f;
        opacities[slot] = opac;
        for (int ch = 0; ch < 3; ch++) {
            sh[(size_t)slot * K * 3 + ch] = (rgb[ch * P + p] - 0.5f) / kY00;
            for (int k = 1; k < K; k++) sh[((size_t)slot * K + k) * 3 + ch] = 0.f;
        }
    }
}

// ---------------------------------------------------------------------------
// Belief propagation over the cost volume (Section III-A2; the min-sum
// algorithm of Felzenszwalb and Huttenlocher, 2006): 4-connected grid, data
// cost V(p, d_f), discontinuity cost min(s |f_p - f_q|, tau), synchronous
// iterations from zero messages, each message shifted to minimum 0.
// The minimisation over f_p of h(f_p) + min(s |f_p - f|, tau) splits into
//   min( s f + min_{f_p <= f} (h(f_p) - s f_p),  -s f + min_{f_p >= f} (h(f_p) + s f_p),
//        min h + tau ),
// a prefix and a suffix minimum.
// msgs: [4][h * w][nd], direction d = message sent to the left, right, upper,
// lower neighbour.
// ---------------------------------------------------------------------------
__device__ __constant__ int c_bp_dy[4] = {0, 0, -1, 1};
__device__ __constant__ int c_bp_dx[4] = {-1, 1, 0, 0};
__device__ __constant__ int c_bp_opp[4] = {1, 0, 3, 2};

// Loads the data cost and the four incoming messages of pixel (x, y) for
// labels f0 = lane, f1 = lane + 32 of a warp (INF past nd for the data cost, 0 for
// messages).
__device__ __forceinline__ void bp_load(int h, int w, int nd, const float* __restrict__ V,
                                        const float* __restrict__ msg, int x, int y, float D[2],
                                        float inc[4][2])
{
    const int lane = threadIdx.x & 31;
    const size_t hw = (size_t)h * w;
    const size_t p = (size_t)y * w + x;
    for (int j = 0; j < 2; j++) {
        const int f = lane + 32 * j;
        D[j] = f < nd ? V[p * nd + f] : INFINITY;
    }
    for (int d = 0; d < 4; d++) {
        const int ny = y + c_bp_dy[d], nx = x + c_bp_dx[d];
        const bool in = ny >= 0 && ny < h && nx >= 0 && nx < w;
        const float* src = msg + (size_t)c_bp_opp[d] * hw * nd + ((size_t)ny * w + nx) * nd;
        for (int j = 0; j < 2; j++) {
            const int f = lane + 32 * j;
            inc[d][j] = (in && f < nd) ? src[f] : 0.f;
        }
    }
}

// Eight lanes a pixel, lane l of the eight holding labels 8 l .. 8 l + 7: the prefix and
// suffix minima are chains of eight in registers and three shuffles over the lanes, where
// a warp a pixel took five shuffles for each of four half scans, and a lane's labels
// are two 16-byte loads (nd a multiple of 4; VEC).  Minima do not round, so the messages
// are the same bits.  A direction's incoming message is read again from L1 when its turn
// comes: all four in registers took 131 of them, one block an SM.  160x120 pixels, 64
// labels: 14.9 us an iteration with a warp a pixel, 10.0 now, bound by the 44 MB it moves
// through L2 (sixteen lanes of four labels: 10.4).
constexpr int kBpLanes = 8, kBpPer = 8;

template <bool VEC>
__device__ __forceinline__ void bp_load(const float* __restrict__ src, bool in, int f0, int nd,
                                         float pad, float v[kBpPer])
{
#pragma unroll
    for (int k = 0; k < kBpPer; k++) v[k] = f0 + k < nd ? 0.f : pad;
    if (!in) return;
    if (VEC) {
#pragma unroll
        for (int k = 0; k < kBpPer; k += 4) {
            if (f0 + k >= nd) break;
            const float4 q = *reinterpret_cast<const float4*>(src + f0 + k);
            v[k] = q.x; v[k + 1] = q.y; v[k + 2] = q.z; v[k + 3] = q.w;
        }
    } else {
#pragma unroll
        for (int k = 0; k < kBpPer; k++)
            if (f0 + k < nd) v[k] = src[f0 + k];
    }
}

template <bool VEC>
__global__ void __launch_bounds__(256, 4)
k_bp_iter(int h, int w, int nd, const float* __restrict__ V, const float* __restrict__ msg_in,
          float* __restrict__ msg_out, float s, float tau)
{
    const int l = threadIdx.x % kBpLanes, f0 = kBpPer * l;
    const size_t hw = (size_t)h * w, groups = (size_t)gridDim.x * blockDim.x / kBpLanes;
    // every lane of a warp runs the same number of rounds (the shuffles)
    const size_t rounds = (hw + groups - 1) / groups;
    const size_t g0 = (blockIdx.x * (size_t)blockDim.x + threadIdx.x) / kBpLanes;
    for (size_t r = 0; r < rounds; r++) {
        const size_t p = g0 + r * groups;
        const bool on = p < hw;
        const int y = on ? (int)(p / w) : 0, x = on ? (int)(p - (size_t)y * w) : 0;
        float tot[kBpPer];
        bp_load<VEC>(V + p * nd, on, f0, nd, INFINITY, tot);
#pragma unroll
        for (int d = 0; d < 4; d++) {
            const int ny = y + c_bp_dy[d], nx = x + c_bp_dx[d];
            const bool in = on && ny >= 0 && ny < h && nx >= 0 && nx < w;
            const float* src = msg_in + (size_t)c_bp_opp[d] * hw * nd + ((size_t)ny * w + nx) * nd;
            float inc[kBpPer];
            bp_load<VEC>(src, in, f0, nd, 0.f, inc);
#pragma unroll
            for (int k = 0; k < kBpPer; k++) tot[k] += inc[k];
        }
#pragma unroll 1
        for (int d = 0; d < 4; d++) {
            const int ny = y + c_bp_dy[d], nx = x + c_bp_dx[d];
            const bool in = on && ny >= 0 && ny < h && nx >= 0 && nx < w;
            const float* src = msg_in + (size_t)c_bp_opp[d] * hw * nd + ((size_t)ny * w + nx) * nd;
            float inc[kBpPer];
            bp_load<VEC>(src, in, f0, nd, 0.f, inc);       // from L1
            float a[kBpPer], b[kBpPer], hmin = INFINITY;
#pragma unroll
            for (int k = 0; k < kBpPer; k++) {
                const float f = (float)(f0 + k), hv = tot[k] - inc[k];      // INF past nd
                hmin = fminf(hmin, hv);
                a[k] = __fmaf_rn(-s, f, hv);
                b[k] = __fmaf_rn(s, f, hv);
            }
#pragma unroll
            for (int k = 1; k < kBpPer; k++) {
                a[k] = fminf(a[k], a[k - 1]);
                b[kBpPer - 1 - k] = fminf(b[kBpPer - 1 - k], b[kBpPer - k]);
            }
            // minima of the lanes before (prefix) and after (suffix) this one
            float pa = __shfl_up_sync(0xffffffffu, a[kBpPer - 1], 1, kBpLanes);
            float pb = __shfl_down_sync(0xffffffffu, b[0], 1, kBpLanes);
            if (l == 0) pa = INFINITY;
            if (l == kBpLanes - 1) pb = INFINITY;
#pragma unroll
            for (int o = 1; o < kBpLanes; o <<= 1) {
                const float ua = __shfl_up_sync(0xffffffffu, pa, o, kBpLanes);
                const float ub = __shfl_down_sync(0xffffffffu, pb, o, kBpLanes);
                if (l >= o) pa = fminf(pa, ua);
                if (l + o < kBpLanes) pb = fminf(pb, ub);
                hmin = fminf(hmin, __shfl_xor_sync(0xffffffffu, hmin, o));
            }
            float m[kBpPer], mmin = INFINITY;
#pragma unroll
            for (int k = 0; k < kBpPer; k++) {
                const float f = (float)(f0 + k);
                m[k] = fminf(fminf(__fmaf_rn(s, f, fminf(a[k], pa)), __fmaf_rn(-s, f, fminf(b[k], pb))),
                             hmin + tau);
                if (f0 + k >= nd) m[k] = INFINITY;
                mmin = fminf(mmin, m[k]);
            }
#pragma unroll
            for (int o = 1; o < kBpLanes; o <<= 1) mmin = fminf(mmin, __shfl_xor_sync(0xffffffffu, mmin, o));
            if (on) {
                float* dst = msg_out + (size_t)d * hw * nd + p * nd + f0;
                if (VEC) {
#pragma unroll
                    for (int k = 0; k < kBpPer; k += 4)
                        if (f0 + k < nd)
                            *reinterpret_cast<float4*>(dst + k) =
                                make_float4(m[k] - mmin, m[k + 1] - mmin, m[k + 2] - mmin,
                                            m[k + 3] - mmin);
                } else {
#pragma unroll
                    for (int k = 0; k < kBpPer; k++)
                        if (f0 + k < nd) dst[k] = m[k] - mmin;
                }
            }
        }
    }
}

// Beliefs D + all incoming messages; label = argmin (lowest on ties); depth
// of the label written to the 4 x 4 full-resolution pixels it covers.
__global__ void __launch_bounds__(256)
k_bp_labels(int h, int w, int nd, const float* __restrict__ V, const float* __restrict__ msg,
            float d0, float d1, float* __restrict__ depth, int* __restrict__ labels,
            float* __restrict__ beliefs)
{
    const int lane = threadIdx.x & 31;
    const size_t hw = (size_t)h * w;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    for (size_t p = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; p < hw; p += warps) {
        const int x = (int)(p % w), y = (int)(p / w);
        float D[2], inc[4][2];
        bp_load(h, w, nd, V, msg, x, y, D, inc);
        float bv = INFINITY;
        int bi = 0x7fffffff;
        for (int j = 0; j < 2; j++) {
            const int f = lane + 32 * j;
            if (f >= nd) continue;
            const float b = D[j] + inc[0][j] + inc[1][j] + inc[2][j] + inc[3][j];
            if (beliefs) beliefs[p * nd + f] = b;
            if (b < bv) { bv = b; bi = f; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (ov < bv || (ov == bv && oi < bi)) { bv = ov; bi = oi; }
        }
        if (labels && lane == 0) labels[p] = bi;
        if (lane < 16) {
            const int W = 4 * w;
            depth[(size_t)(4 * y + (lane >> 2)) * W + 4 * x + (lane & 3)] =
                d0 + (d1 - d0) * (float)bi / (float)(nd - 1);
        }
    }
}

static int gridn(size_t n) { return (int)std::max<size_t>(1, std::min<size_t>((n + 255) / 256, (size_t)sm_count() * 16)); }

}  // namespace gevo

using namespace gevo;

extern "C" {

gevo_status gevo_cost_volume(int32_t nk, int32_t ref, int32_t H, int32_t W, const float* rgb,
                             const float* cams, int32_t nd, float d0, float d1, float* grey,
                             float* volume, float* depth, void* stream)
{
    if (nk < 2 || ref < 0 || ref >= nk || H % 4 || W % 4 || H < 8 || W < 8 || !rgb || !cams ||
        nd < 2 || !(d1 > d0) || !grey || !volume || !depth)
        return GEVO_ERR_INVALID;
    cudaStream_t st = (cudaStream_t)stream;
    const int h = H / 4, w = W / 4;
    k_grey4<<<gridn((size_t)nk * h * w), 256, 0, st>>>(nk, H, W, rgb, grey, gevo_aligned(rgb, 16));
    GEVO_CHECK_LAUNCH();
    const size_t tiles = (((size_t)h * w + 31) / 32) * ((nd + 31) / 32);
    k_cost_volume<<<gridn(tiles * 256), 256, 0, st>>>(nk, ref, h, w, grey, cams, nd, d0, d1, volume);
    GEVO_CHECK_LAUNCH();
    k_wta_up4<<<gridn((size_t)h * w * 32), 256, 0, st>>>(h, w, nd, d0, d1, volume, depth);
    GEVO_CHECK_LAUNCH();
    return GEVO_OK;
}

gevo_status gevo_unproject(int32_t H, int32_t W, const float* rgb, const float* depth,
                           const float* mask, const float* cam, uint32_t keep, uint32_t seed,
                           float scale_px, float opacity, int32_t sh_degree, uint32_t* counter,
                           int32_t cap, float* means, float* scales, float* quats,
                           float* opacities, float* sh, void* stream)
{
    if (H <= 0 || W <= 0 || !rgb || !depth || !mask || !cam || !counter || cap < 0 || !means ||
        !scales || !quats || !opacities || !sh || sh_degree < 0 || sh_degree > 3)
        return GEVO_ERR_INVALID;
    const int K = (sh_degree + 1) * (sh_degree + 1);
    k_unproject<<<gridn((size_t)H * W), 256, 0, (cudaStream_t)stream>>>(
        H, W, rgb, depth, mask, cam, keep, seed, scale_px, opacity, K, counter, cap, means, scales,
        quats, opacities, sh);
    GEVO_CHECK_LAUNCH();
    return GEVO_OK;
}

gevo_status gevo_depth_bp(int32_t h, int32_t w, int32_t nd, const float* volume, float s,
                          float tau, int32_t iters, float d0, float d1, float* msgs, float* depth,
                          int32_t* labels, float* beliefs, void* stream)
{
    if (h < 1 || w < 1 || nd < 2 || nd > 64 || !volume || !(s >= 0.f) || !(tau >= 0.f) ||
        iters < 0 || !(d1 > d0) || !msgs || !depth)
        return GEVO_ERR_INVALID;
    cudaStream_t st = (cudaStream_t)stream;
    const size_t per = (size_t)4 * h * w * nd;
    float* a = msgs;
    float* b = msgs + per;
    if (cudaMemsetAsync(a, 0, sizeof(float) * per, st) != cudaSuccess) return GEVO_ERR_CUDA;
    const int grid = gridn((size_t)h * w * 32);
    const bool vec = nd % 4 == 0 && gevo_aligned(volume, 16) && gevo_aligned(msgs, 16);
    const int igrid = gridn((size_t)h * w * kBpLanes);
    for (int it = 0; it < iters; it++) {
        if (vec) k_bp_iter<true><<<igrid, 256, 0, st>>>(h, w, nd, volume, a, b, s, tau);
        else k_bp_iter<false><<<igrid, 256, 0, st>>>(h, w, nd, volume, a, b, s, tau);
        GEVO_CHECK_LAUNCH();
        float* t = a; a = b; b = t;
    }
    k_bp_labels<<<grid, 256, 0, st>>>(h, w, nd, volume, a, d0, d1, depth, labels, beliefs);
    GEVO_CHECK_LAUNCH();
    return GEVO_OK;
}

}  // extern "C"
