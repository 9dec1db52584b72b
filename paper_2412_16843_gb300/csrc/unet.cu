// Warm-start U-Net on the tensor cores: forward, backward and Adam.
//
// Convolutions are implicit GEMMs on channels-last BF16 activations
// [voxel][channel] with FP32 accumulation:
//   forward      y[v][co] = b[co] + sum_t sum_ci x[v + off(t)][ci] W[t][co][ci]
//   data grad    dx = forward(dy) with the taps flipped and W transposed,
//                because the adjoint of a zero-padded correlation is the
//                correlation with the mirrored kernel
//   weight grad  dW[t][co][ci] = sum_v dy[v][co] x[v + off(t)][ci]
// By default on tcgen05 with accumulators in tensor memory: k_conv_zb (forward
// and data gradient; M = 128 voxels, the three dz taps folded into N) and
// k_wgrad_tc (weight and bias gradients; M = rows of taps x input channels,
// K = voxels, split sums added in a fixed order).  The alternative (k_conv,
// k_wgrad) runs mma.sync m16n8k16: M = 16 voxels per warp, N = all output
// channels, K = 27 taps x Cin, and for the weight gradient M = 16 output
// channels, K = voxels, partial sums added with atomics.
// Pooling (2x2x2 mean), nearest upsampling, channel concatenation, ReLU
// masks, the mean-squared-error loss and Adam are elementwise kernels; at
// inference the last layer's read-out applies the 1x1x1 head.
// Master weights and Adam moments are FP32; the tensor cores see BF16 copies.
#include "unet.cuh"
#include "ops.cuh"
#include "../../include/cdi.h"

#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <vector>

namespace cdi {
namespace {

using bf16 = __nv_bfloat16;

struct CG {
    int nx, ny, nz, N;
};

constexpr int kLayers = 8;
// name order e0, e1, e2, b, d2, d1, d0, head: Cin, Cout, taps
constexpr int kCin[kLayers] = {2, 16, 32, 64, 192, 96, 48, 16};
constexpr int kCout[kLayers] = {16, 32, 64, 128, 64, 32, 16, 1};
constexpr int kTaps[kLayers] = {27, 27, 27, 27, 27, 27, 27, 1};

inline int pad16(int c) { return (c + 15) / 16 * 16; }

__device__ __forceinline__ unsigned ld_pair(const bf16* p) { return *reinterpret_cast<const unsigned*>(p); }
__device__ __forceinline__ unsigned pack2(bf16 lo, bf16 hi) {
    return (unsigned)__bfloat16_as_ushort(lo) | ((unsigned)__bfloat16_as_ushort(hi) << 16);
}
__device__ __forceinline__ void mma_bf16(float* c, unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0,
                                         unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// tap t = (dz+1)*9 + (dy+1)*3 + (dx+1); a 1-tap layer is the centre only
__device__ __forceinline__ void tap_off(int tap, int ntaps, int& dz, int& dy, int& dx) {
    if (ntaps == 1) {
        dz = dy = dx = 0;
        return;
    }
    dz = tap / 9 - 1;
    dy = (tap / 3) % 3 - 1;
    dx = tap % 3 - 1;
}

struct Vox {
    int x, y, z;
    bool in;
};
__device__ __forceinline__ Vox vox(const CG& g, int v) {
    Vox o;
    o.in = v < g.N;
    const int vv = o.in ? v : 0;
    o.x = vv % g.nx;
    const int r = vv / g.nx;
    o.y = r % g.ny;
    o.z = r / g.ny;
    return o;
}
// neighbour index or -1 (zero padding)
__device__ __forceinline__ int nbr(const CG& g, const Vox& p, int dz, int dy, int dx) {
    const int x = p.x + dx, y = p.y + dy, z = p.z + dz;
    if (!p.in || x < 0 || x >= g.nx || y < 0 || y >= g.ny || z < 0 || z >= g.nz) return -1;
    return x + g.nx * (y + g.ny * z);
}

// forward convolution (also the data gradient with flipped, transposed W)
template <int NF, bool OUTF32>
__global__ void __launch_bounds__(128) k_conv(CG g, const bf16* __restrict__ in, int cin_pad,
                                              const bf16* __restrict__ w, int cout_pad, const float* __restrict__ bias,
                                              int cout, void* out, int out_stride, int out_off, int relu, int ntaps) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
    const int r0 = (blockIdx.x * 4 + warp) * 16 + gid, r1 = r0 + 8;
    const Vox v0 = vox(g, r0), v1 = vox(g, r1);
    float acc[NF][4];
#pragma unroll
    for (int j = 0; j < NF; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
    for (int tap = 0; tap < ntaps; ++tap) {
        int dz, dy, dx;
        tap_off(tap, ntaps, dz, dy, dx);
        const int n0 = nbr(g, v0, dz, dy, dx), n1 = nbr(g, v1, dz, dy, dx);
        const bf16* p0 = in + (size_t)(n0 < 0 ? 0 : n0) * cin_pad + 2 * tig;
        const bf16* p1 = in + (size_t)(n1 < 0 ? 0 : n1) * cin_pad + 2 * tig;
        const bf16* wt = w + ((size_t)tap * cout_pad + gid) * cin_pad + 2 * tig;
        for (int k0 = 0; k0 < cin_pad; k0 += 16) {
            const unsigned a0 = n0 >= 0 ? ld_pair(p0 + k0) : 0u;
            const unsigned a1 = n1 >= 0 ? ld_pair(p1 + k0) : 0u;
            const unsigned a2 = n0 >= 0 ? ld_pair(p0 + k0 + 8) : 0u;
            const unsigned a3 = n1 >= 0 ? ld_pair(p1 + k0 + 8) : 0u;
#pragma unroll
            for (int j = 0; j < NF; ++j) {
                const bf16* wj = wt + (size_t)j * 8 * cin_pad + k0;
                mma_bf16(acc[j], a0, a1, a2, a3, ld_pair(wj), ld_pair(wj + 8));
            }
        }
    }
#pragma unroll
    for (int j = 0; j < NF; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = h ? r1 : r0;
            if (r >= g.N) continue;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int co = j * 8 + 2 * tig + e;
                if (co >= cout) continue;
                float v = acc[j][2 * h + e] + (bias ? bias[co] : 0.f);
                if (relu) v = fmaxf(v, 0.f);
                const size_t o = (size_t)r * out_stride + out_off + co;
                if (OUTF32) reinterpret_cast<float*>(out)[o] = v;
                else reinterpret_cast<bf16*>(out)[o] = __float2bfloat16(v);
            }
        }
}

// weight gradient: dW[t][co][ci] += sum over a voxel chunk of dy[v][co] x[v+off(t)][ci]
template <int NF>
__global__ void __launch_bounds__(128) k_wgrad(CG g, const bf16* __restrict__ in, int cin_pad,
                                               const bf16* __restrict__ dyv, int cout_pad, float* dW, int cout, int cin,
                                               int ntaps, int chunk) {
    const int tap = blockIdx.x, co0 = blockIdx.y * 16;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
    int dz, dy, dx;
    tap_off(tap, ntaps, dz, dy, dx);
    float acc[NF][4];
#pragma unroll
    for (int j = 0; j < NF; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
    const int per_warp = chunk / 4;
    const int vbeg = blockIdx.z * chunk + warp * per_warp;
    const int vend = min(vbeg + per_warp, g.N);
    const bf16 zero = __float2bfloat16(0.f);
    auto dyat = [&](int v, int co) { return (v < g.N && co < cout_pad) ? dyv[(size_t)v * cout_pad + co] : zero; };
    for (int vb = vbeg; vb < vend; vb += 16) {
        const int vk[4] = {vb + 2 * tig, vb + 2 * tig + 1, vb + 2 * tig + 8, vb + 2 * tig + 9};
        const int ca = co0 + gid, cb = co0 + gid + 8;
        const unsigned a0 = pack2(dyat(vk[0], ca), dyat(vk[1], ca));
        const unsigned a1 = pack2(dyat(vk[0], cb), dyat(vk[1], cb));
        const unsigned a2 = pack2(dyat(vk[2], ca), dyat(vk[3], ca));
        const unsigned a3 = pack2(dyat(vk[2], cb), dyat(vk[3], cb));
        int nb[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) nb[i] = (vk[i] < vend) ? nbr(g, vox(g, vk[i]), dz, dy, dx) : -1;
#pragma unroll
        for (int j = 0; j < NF; ++j) {
            const int ci = j * 8 + gid;
            auto xin = [&](int n) { return n >= 0 ? in[(size_t)n * cin_pad + ci] : zero; };
            mma_bf16(acc[j], a0, a1, a2, a3, pack2(xin(nb[0]), xin(nb[1])), pack2(xin(nb[2]), xin(nb[3])));
        }
    }
#pragma unroll
    for (int j = 0; j < NF; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int co = co0 + gid + 8 * h, ci = j * 8 + 2 * tig + e;
                if (co < cout && ci < cin) atomicAdd(&dW[((size_t)tap * cout + co) * cin + ci], acc[j][2 * h + e]);
            }
}

__global__ void k_bias_grad(int N, const bf16* dy, int stride, int C, float* db) {
    const int c = blockIdx.y;
    float s = 0.f;
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < N; v += gridDim.x * blockDim.x)
        s += __bfloat162float(dy[(size_t)v * stride + c]);
    __shared__ float sh[256];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(&db[c], sh[0]);
}

// 2x2x2 mean of the fine grid gf into the coarse grid; 8 channels (16 bytes) per thread
__global__ void k_pool(CG gf, const bf16* in, int C, bf16* out) {
    const int Nc = gf.N / 8, C8 = C / 8;
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long)Nc * C8) return;
    const int g8 = (int)(t % C8), V = (int)(t / C8);
    const int cx = gf.nx / 2, cy = gf.ny / 2;
    const int X = V % cx, Y = (V / cx) % cy, Z = V / (cx * cy);
    float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int k = 0; k < 2; ++k)
        for (int j = 0; j < 2; ++j)
            for (int i = 0; i < 2; ++i) {
                const size_t v = (size_t)((2 * X + i) + gf.nx * ((2 * Y + j) + gf.ny * (2 * Z + k)));
                const uint4 q = *reinterpret_cast<const uint4*>(in + v * C + 8 * g8);
                const bf16* h = reinterpret_cast<const bf16*>(&q);
#pragma unroll
                for (int e = 0; e < 8; ++e) s[e] += __bfloat162float(h[e]);
            }
    __align__(16) bf16 o[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) o[e] = __float2bfloat16(0.125f * s[e]);
    *reinterpret_cast<uint4*>(out + (size_t)V * C + 8 * g8) = *reinterpret_cast<const uint4*>(o);
}

// din[v][off+c] += dout[parent(v)][c] / 8 on the fine grid gf; 8 channels (16 bytes) per thread
__global__ void k_pool_bwd_add(CG gf, const bf16* dout, int C, bf16* din, int stride, int off) {
    const int C8 = C / 8;
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long)gf.N * C8) return;
    const int g8 = (int)(t % C8), v = (int)(t / C8);
    const int x = v % gf.nx, y = (v / gf.nx) % gf.ny, z = v / (gf.nx * gf.ny);
    const int P = (x / 2) + (gf.nx / 2) * ((y / 2) + (gf.ny / 2) * (z / 2));
    uint4* dst = reinterpret_cast<uint4*>(din + (size_t)v * stride + off + 8 * g8);
    uint4 d = *dst;
    const uint4 q = *reinterpret_cast<const uint4*>(dout + (size_t)P * C + 8 * g8);
    bf16* a = reinterpret_cast<bf16*>(&d);
    const bf16* h = reinterpret_cast<const bf16*>(&q);
#pragma unroll
    for (int e = 0; e < 8; ++e) a[e] = __float2bfloat16(__bfloat162float(a[e]) + 0.125f * __bfloat162float(h[e]));
    *dst = d;
}

// nearest upsampling of the coarse input into channels [off, off+C) of the fine output; 8 channels per thread
__global__ void k_up(CG gf, const bf16* in, int C, bf16* out, int stride, int off) {
    const int C8 = C / 8;
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long)gf.N * C8) return;
    const int g8 = (int)(t % C8), v = (int)(t / C8);
    const int x = v % gf.nx, y = (v / gf.nx) % gf.ny, z = v / (gf.nx * gf.ny);
    const int P = (x / 2) + (gf.nx / 2) * ((y / 2) + (gf.ny / 2) * (z / 2));
    *reinterpret_cast<uint4*>(out + (size_t)v * stride + off + 8 * g8) =
        *reinterpret_cast<const uint4*>(in + (size_t)P * C + 8 * g8);
}

// adjoint of k_up: din[V][c] = sum of the 8 children dout[child][off+c]
__global__ void k_up_bwd(CG gf, const bf16* dout, int stride, int off, int C, bf16* din) {
    const int Nc = gf.N / 8;
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long)Nc * C) return;
    const int c = (int)(t % C), V = (int)(t / C);
    const int cx = gf.nx / 2, cy = gf.ny / 2;
    const int X = V % cx, Y = (V / cx) % cy, Z = V / (cx * cy);
    float s = 0.f;
    for (int k = 0; k < 2; ++k)
        for (int j = 0; j < 2; ++j)
            for (int i = 0; i < 2; ++i)
                s += __bfloat162float(
                    dout[(size_t)((2 * X + i) + gf.nx * ((2 * Y + j) + gf.ny * (2 * Z + k))) * stride + off + c]);
    din[t] = __float2bfloat16(s);
}

// channel block copy, 8 channels (16 bytes) per thread; strides, offsets and C multiples of 8
__global__ void k_copy_ch(int N, const bf16* src, int sstride, int soff, bf16* dst, int dstride, int doff, int C) {
    const int C8 = C / 8;
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long)N * C8) return;
    const int g8 = (int)(t % C8), v = (int)(t / C8);
    *reinterpret_cast<uint4*>(dst + (size_t)v * dstride + doff + 8 * g8) =
        *reinterpret_cast<const uint4*>(src + (size_t)v * sstride + soff + 8 * g8);
}

// g *= (y > 0) (ReLU backward), both n contiguous values, a multiple of 8; 8 per thread
__global__ void k_relu_mask(long n, bf16* g, const bf16* y) {
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (8 * t >= n) return;
    uint4 d = reinterpret_cast<const uint4*>(g)[t];
    const uint4 q = reinterpret_cast<const uint4*>(y)[t];
    bf16* a = reinterpret_cast<bf16*>(&d);
    const bf16* h = reinterpret_cast<const bf16*>(&q);
#pragma unroll
    for (int e = 0; e < 8; ++e)
        if (!(__bfloat162float(h[e]) > 0.f)) a[e] = __float2bfloat16(0.f);
    reinterpret_cast<uint4*>(g)[t] = d;
}

// mean squared error: partial sums of (y-t)^2 and the BF16 gradient 2(y-t)/N in channel 0 of 16
__global__ void k_loss(int N, const float* y, const float* t, bf16* gy, float* part) {
    float s = 0.f;
    for (int v = blockIdx.x * blockDim.x + threadIdx.x; v < N; v += gridDim.x * blockDim.x) {
        const float d = y[v] - t[v];
        s += d * d;
        gy[(size_t)v * 16] = __float2bfloat16(2.f * d / (float)N);
    }
    __shared__ float sh[256];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(part, sh[0]);
}

// the parameter arrays of the network, one segment each, for one launch over all of them (16 launches of a few
// microseconds each otherwise)
struct ParamSegs {
    long end[2 * kLayers];  // running ends of the segments
    float *w[2 * kLayers], *g[2 * kLayers], *m[2 * kLayers], *v[2 * kLayers];
};

// Adam (Kingma and Ba, 2015) with bias corrections bc1 = 1 - b1^t, bc2 = 1 - b2^t
__global__ void k_adam(const __grid_constant__ ParamSegs p, float lr, float b1, float b2, float eps, float bc1,
                       float bc2) {
    long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= p.end[2 * kLayers - 1]) return;
    int k = 0;
    while (i >= p.end[k]) ++k;
    if (k) i -= p.end[k - 1];
    const float gi = p.g[k][i];
    const float mi = b1 * p.m[k][i] + (1.f - b1) * gi;
    const float vi = b2 * p.v[k][i] + (1.f - b2) * gi * gi;
    p.m[k][i] = mi;
    p.v[k][i] = vi;
    p.w[k][i] -= lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
}

// output channels of one CTA of the tcgen05 convolution with n output channels
__host__ __device__ constexpr int conv_nb(int n) {
    return n % 64 == 0 ? 64 : n % 48 == 0 ? 48 : n % 32 == 0 ? 32 : 16;
}
// element of tap t, output channel o (of n), input channel i (of cin) in the tcgen05 convolution's weights:
// [block of NB][block of 16 input channels][tap (dy, dx)][dz = +1, 0, -1][8 channels][2 x 8 inputs][8][8]
__device__ __forceinline__ size_t conv_w_at(int t, int o, int n, int i, int cin) {
    const int NB = conv_nb(n), row = (2 - t / 9) * NB + o % NB;
    const size_t blk = (size_t)(o / NB) * (cin / 16) + i / 16;
    return (blk * 9 + t % 9) * (3 * NB * 16) + (row >> 3) * 128 + ((i >> 3) & 1) * 64 + (row & 7) * 8 + (i & 7);
}

// the weights of every layer and their BF16 copies, one segment a layer (padded elements)
struct WeightSegs {
    long end[kLayers];
    const float* W[kLayers];
    int taps[kLayers], cout[kLayers], cin[kLayers], co_pad[kLayers], ci_pad[kLayers];
    bf16 *wb[kLayers], *wt[kLayers], *wk[kLayers], *wkt[kLayers];
};

// BF16 copies: wb[t][co_pad][ci_pad] = W[t][co][ci]; wt[t][ci_pad][co_pad] = W[T-1-t][co][ci]; for 27 taps
// also both in the order of the tcgen05 convolution (wk, wkt)
__global__ void k_weights_bf16(const __grid_constant__ WeightSegs p) {
    long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= p.end[kLayers - 1]) return;
    int l = 0;
    while (i >= p.end[l]) ++l;
    if (l) i -= p.end[l - 1];
    const int ci_pad = p.ci_pad[l], co_pad = p.co_pad[l], taps = p.taps[l], cout = p.cout[l], cin = p.cin[l];
    const unsigned r = (unsigned)i / (unsigned)ci_pad;
    const int ci = (int)((unsigned)i - r * (unsigned)ci_pad), t = (int)(r / (unsigned)co_pad), co = (int)r - t * co_pad;
    const bf16 val = __float2bfloat16((co < cout && ci < cin) ? p.W[l][((size_t)t * cout + co) * cin + ci] : 0.f);
    p.wb[l][i] = val;
    const int tf = taps - 1 - t;
    p.wt[l][((size_t)tf * ci_pad + ci) * co_pad + co] = val;
    if (taps == 27) {
        p.wk[l][conv_w_at(t, co, co_pad, ci, ci_pad)] = val;
        p.wkt[l][conv_w_at(tf, ci, ci_pad, co, co_pad)] = val;
    }
}

// network input in two forms: pairs xp [N][2] for the first layer's tcgen05 convolution and, where x is not null,
// padded to 16 channels for the mma.sync kernels and the weight gradient
__device__ __forceinline__ void put_input(int v, float a, float b, bf16* xp, bf16* x) {
    const unsigned p = pack2(__float2bfloat16(a), __float2bfloat16(b));
    reinterpret_cast<unsigned*>(xp)[v] = p;
    if (x) {
        uint4* q = reinterpret_cast<uint4*>(x + (size_t)v * 16);
        q[0] = make_uint4(p, 0u, 0u, 0u);
        q[1] = make_uint4(0u, 0u, 0u, 0u);
    }
}
__global__ void k_input_host(int N, const double* x2, bf16* xp, bf16* x) {  // x2: [N][2] from the host
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v < N) put_input(v, (float)x2[(size_t)v * 2], (float)x2[(size_t)v * 2 + 1], xp, x);
}

__global__ void k_input_dev16(int N, const float* x2, bf16* xp, bf16* x) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v < N) put_input(v, x2[(size_t)v * 2], x2[(size_t)v * 2 + 1], xp, x);
}

// x2: [N][2] on the device (4-byte aligned), N even; two voxels a thread.  The 16-channel form it replaces wrote
// 32 bytes a voxel, a channel a thread (615 us at 256^3).
__global__ void k_input_dev(int N, const float* x2, bf16* xp) {
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (2 * t >= N) return;
    const float* q = x2 + 4 * t;
    const bool al = (reinterpret_cast<uintptr_t>(q) & 15) == 0;
    const float4 v = al ? *reinterpret_cast<const float4*>(q) : make_float4(q[0], q[1], q[2], q[3]);
    uint2 o;
    o.x = pack2(__float2bfloat16(v.x), __float2bfloat16(v.y));
    o.y = pack2(__float2bfloat16(v.z), __float2bfloat16(v.w));
    reinterpret_cast<uint2*>(xp)[t] = o;
}

// scales of one prediction from ||f||_2 (one thread): sd = {1/rms(f), rms(f) max(rho) h^2}
// in FP64 and sf the same in FP32; a zero right-hand side gives a zero guess
__global__ void k_solver_scales(const double* fnorm, int N, double rho_h2, double* sd, float* sf) {
    const double rms = *fnorm / sqrt((double)N);
    sd[0] = rms > 0.0 ? 1.0 / rms : 0.0;
    sd[1] = rms * rho_h2;
    sf[0] = (float)sd[0];
    sf[1] = (float)sd[1];
}

// network input from the solver's f (its mean already removed in the FP64
// form; removed here with the double-float mean in the FP32-mixed form) and phi
template <typename T>
__global__ void k_input_solver(int N, const FT<T>* f, const float* fmean_df, const T* phi, float drho, float rho2,
                               float inv_rmax, const double* sd, const float* sf, bf16* xp, bf16* x) {
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= N) return;
    float val;
    if constexpr (sizeof(T) == 8) val = (float)(f[v] * sd[0]);
    else val = ((f[v] - fmean_df[0]) - fmean_df[1]) * sf[0];
    put_input(v, val, (drho * (float)phi[v] + rho2) * inv_rmax, xp, x);
}

template <typename T>
__global__ void k_output_solver(int N, const float* y, const double* sd, const float* sf, PT<T>* p) {
    const long v = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= N) return;
    if constexpr (sizeof(T) == 8) p[v] = (double)y[v] * sd[1];
    else p[v] = make_float2(y[v] * sf[1], 0.f);
}

unsigned blocks(long n, int t = 256) { return (unsigned)((n + t - 1) / t); }

// ---------------------------------------------------------------------------
// 3x3x3 convolution on the 5th-generation tensor cores (tcgen05).
//
// What bounds it: an M = 128, K = 16 BF16 MMA reads 4 KB of A and 32 N bytes
// of B from shared memory at 128 B a cycle and multiplies for N / 2 cycles, so
// with N = 16 (the layers of the finest level) it is bound by the A reads
// (36 cycles for 8 of arithmetic).  The kernel therefore folds the three dz
// taps into N: an input plane meets the weights of all three in one MMA of
// N = 3 NB columns, whose column blocks are the accumulators of the output
// planes below, at and above it, which lie side by side in tensor memory.
//
// A CTA (one per SM, persistent) computes tiles of 8 (x) x 16 (y) x zt voxels
// for a block of NB output channels: accumulator column j NB + c of tensor
// memory lane m is channel c of voxel m of output plane j.  Its work is a
// sequence of stages, one a 16-input-channel block: the input tile with a
// one-voxel halo (zt + 2 planes of 18 x 10 voxels) and the block's weights of
// all 27 taps, both in the canonical K-major layout without swizzling (a core
// matrix is 8 rows of 16 bytes stored contiguously; the descriptor's leading
// offset steps to the next 8 channels, its stride offset to the next 8 rows).
// A tap (dy, dx) only shifts the start address of the A descriptor by whole
// 16-byte rows.  Input plane zi feeds output planes zi-2 .. zi of the tile
// (clipped at its ends), a contiguous window of the column blocks and of the
// weight rows, stored in the order dz = +1, 0, -1.  Every accumulator still
// receives its products in the order channel block, dz, dy, dx.
//
// The first layer has two input channels (PAIRS): its rows are staged as one
// 16-byte unit a voxel, 4 bytes of it copied and the rest zero, and the second
// half of K reads a block of zeros.  (Packing dx and dy into K would need two
// MMAs a plane instead of nine, but sums the products in another order: the
// BF16 roundings that flip then, about one in 10^6, grow through the layers
// to the rounding noise of the whole network, 1e-3 of the output.)
//
// Roles: warps 0-3 read the accumulators of a finished tile (bias, ReLU, BF16
// rounding, 16-byte stores), warp 4 issues the MMAs (one thread), warps 5-7
// stage the input with cp.async, one thread of them the weights with one bulk
// copy a stage.  Stages form a ring of 2 to 4 buffers, accumulators two sets,
// so copies, MMAs and read-out of consecutive tiles overlap.  zt is chosen by
// conv_planes (below).
//
// Measured, forward pass of the network (GB300): 256^3 8.05 -> 2.07 ms (650
// TFLOP/s), 128^3 1.20 -> 0.34 ms, 40 x 24 x 16 283 -> 102 us against one MMA
// of N = NB a tap and plane with a CTA barrier every 18 MMAs, an input kernel
// of 32 bytes a voxel (615 us at 256^3, now 31) and a separate head (396 us,
// now in the last layer's read-out, whose output is not stored).  The three
// dz taps in N alone gave 3.50 ms; handing a stage over as soon as its copies
// land, instead of after the next stage's have been issued, 460 -> 311 us on
// the 96 -> 32 layer at 128^3.
// ---------------------------------------------------------------------------
constexpr int kZbThreads = 256, kZbProd = 96, kZbMmaWarp = 4;
constexpr int kTileX = 8, kTileY = 16;
constexpr int kHX = kTileX + 2, kHY = kTileY + 2;
constexpr int kPlaneUnits = kHY * 2 * kHX;       // 16-byte units of one staged plane: [y][8-channel half][x]
constexpr int kZbMaxStages = 4;
// PAIRS: 16-byte units of a plane [y][x], and the block of zeros (with the same row stride) of channels 8..15
constexpr int kPairUnits = kHY * kHX, kPairZeroBytes = kTileY * kHX * 16;

// bytes of one stage's weights and of one staged plane
__host__ __device__ constexpr uint32_t zb_wbytes(int NB) { return 27u * 32u * NB; }
__host__ __device__ constexpr uint32_t zb_plane(bool pairs) { return 16u * (pairs ? kPairUnits : kPlaneUnits); }

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mbar_test_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long tc_globaltimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// wait (at most about one second) for the phase of the given parity to complete
// Wait for phase `parity` of an mbarrier.  It gives up only after 1 s of
// wall time AND 2^20 polls: a context switched out by time slicing does not
// poll, so a long preemption alone cannot end the wait.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity) {
    const unsigned long long t0 = tc_globaltimer();
    long polls = 0;
    while (!mbar_try_wait(bar, parity))
        if (++polls > (1L << 20) && tc_globaltimer() - t0 > 1000000000ull) return false;
    return true;
}
// A second wait for a phase whose first wait gave up, bounded by polls only
// (2^22 polls with a 1 us back-off, about 4 s of running time); true once
// the phase completed.
__device__ __forceinline__ bool mbar_drain(uint64_t* bar, uint32_t parity) {
    for (long it = 0; it < (1L << 22); ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        __nanosleep(1000);
    }
    return false;
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// shared-memory matrix descriptor: start address, leading byte offset (next 8
// channels), stride byte offset (next 8 rows), descriptor version 1, no swizzle
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}
// instruction descriptor of kind::f16: FP32 D, BF16 A and B, both K-major, M x N
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void tc_mma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                       uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}
// 8 consecutive FP32 columns of this thread's TMEM lane
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void cp_async16(uint32_t saddr, const void* g, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(saddr), "l"(g), "r"(valid ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t saddr, const void* g, bool valid) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(saddr), "l"(g), "r"(valid ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// 16 (and, from a second place, 16 more) consecutive FP32 columns of this thread's TMEM lane, complete on return
#define TM_OUT16(r, o)                                                                                            \
    "=r"(r[o]), "=r"(r[o + 1]), "=r"(r[o + 2]), "=r"(r[o + 3]), "=r"(r[o + 4]), "=r"(r[o + 5]), "=r"(r[o + 6]),    \
        "=r"(r[o + 7]), "=r"(r[o + 8]), "=r"(r[o + 9]), "=r"(r[o + 10]), "=r"(r[o + 11]), "=r"(r[o + 12]),         \
        "=r"(r[o + 13]), "=r"(r[o + 14]), "=r"(r[o + 15])
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : TM_OUT16(r, 0)
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,"
        "%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        "tcgen05.wait::ld.sync.aligned;"
        : TM_OUT16(r, 0), TM_OUT16(r, 16)
        : "r"(taddr)
        : "memory");
}
#undef TM_OUT16
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("{\n .reg .b64 t;\n mbarrier.arrive.shared::cta.b64 t, [%0];\n}\n" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("{\n .reg .b64 t;\n mbarrier.arrive.expect_tx.shared::cta.b64 t, [%0], %1;\n}\n" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}
// bulk copy of bytes (a multiple of 16) from 16-byte aligned global memory, counted on bar
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
// mbar_wait_bounded that also ends (false) once another role of the CTA has given up
__device__ __forceinline__ bool mbar_wait_role(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* err) {
    const unsigned long long t0 = tc_globaltimer();
    long polls = 0;
    while (!mbar_try_wait(bar, parity)) {
        if (*abort_flag) return false;
        if (++polls > (1L << 20) && tc_globaltimer() - t0 > 1000000000ull) {
            *abort_flag = 1;
            atomicMax(err, 1);
            return false;
        }
    }
    return true;
}
// mbar_wait_role of a whole warp whose lanes go on together: a lane may see the phase complete where another, a poll
// earlier, saw a role give up, and a warp barrier or tcgen05.ld without all 32 lanes never ends
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* err) {
    return __all_sync(0xffffffffu, mbar_wait_role(bar, parity, abort_flag, err));
}

struct ConvArgs {
    CG g;
    const bf16* in;     // [voxel][cin - cup]; PAIRS: [voxel][2]
    const bf16* up;     // coarse input of the first cup channels (nearest upsampling of half the extents), or null
    int cin, cup;       // multiples of 16
    const bf16* w;      // blocked weights (k_weights_bf16): [channel block of NB][16 input channels][9][3 NB][16]
    const float* bias;  // [N] or null
    bf16* out;          // [voxel][N], or null (NB = 16 with the head only)
    const bf16* head_w;   // NB = 16: also y[voxel] = head_b + sum_c head_w[c] (this layer's BF16 output c), or null
    const float* head_b;
    float* y;
    int N, relu;
    int zt, nstage, nblk, ncols;  // planes of a tile, staging buffers, N / NB, TMEM columns (a power of two >= 2 zt NB)
    int* err;
};

// out[v][co] = act(bias[co] + sum_t sum_ci in[v + off(t)][ci] w[t][co][ci]).  A wait that runs out sets
// *err to 1, and every role of the CTA stops.  Tensor memory is released only once every MMA the CTA
// issued has been seen complete (a last commit, waited for with a poll bound); if that wait runs out too,
// *err is set to 2 (the CTA must still release its columns before it exits, so their contents are not to
// be trusted by any later kernel of the context).
template <int NB, bool PAIRS>
__global__ void __launch_bounds__(kZbThreads, PAIRS ? 2 : 1) k_conv_zb(const ConvArgs a) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t b_full[kZbMaxStages], b_wfull[kZbMaxStages], b_empty[kZbMaxStages];
    __shared__ __align__(8) uint64_t b_acc[2], b_accfree[2], b_end;
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;
    const CG& g = a.g;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    constexpr uint32_t kWBytes = zb_wbytes(NB), kPlane = zb_plane(PAIRS);
    const uint32_t stage_bytes = kWBytes + (uint32_t)(a.zt + 2) * kPlane;
    const uint32_t base = smem_u32(smem);

    if (warp == kZbMmaWarp) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(a.ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        for (int i = 0; i < kZbMaxStages; ++i) {
            mbar_init(&b_full[i], kZbProd);
            mbar_init(&b_wfull[i], 1);
            mbar_init(&b_empty[i], 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(&b_acc[i], 1);
            mbar_init(&b_accfree[i], 128);
        }
        mbar_init(&b_end, 1);
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (PAIRS) {  // the rows' other channels and the block of zeros after the stages stay zero
        const uint4 z = make_uint4(0u, 0u, 0u, 0u);
        uint4* q = reinterpret_cast<uint4*>(smem);
        for (int i = tid; i < (int)(a.nstage * stage_bytes + kPairZeroBytes) / 16; i += kZbThreads) q[i] = z;
        fence_proxy_async();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;

    const int tiles_x = (g.nx + kTileX - 1) / kTileX, tiles_y = (g.ny + kTileY - 1) / kTileY;
    const int tiles_z = (g.nz + a.zt - 1) / a.zt;
    const int items = tiles_x * tiles_y * tiles_z * a.nblk;  // item = tile nblk + channel block
    const int ncb = a.cin / 16;
    auto origin = [&](int item, int& x0, int& y0, int& z0, int& blk) {
        const int tile = item / a.nblk;
        blk = item - tile * a.nblk;
        const int r = tile / tiles_x;
        x0 = (tile - r * tiles_x) * kTileX;
        const int tz = r / tiles_y;
        y0 = (r - tz * tiles_y) * kTileY;
        z0 = tz * a.zt;
    };

    if (warp > kZbMmaWarp) {
        // ---- staging ----
        const int pt = tid - (kZbMmaWarp + 1) * 32;
        int st = 0, issued = 0;
        uint32_t ph = 1u;  // a buffer's first use finds it empty
        bool ok = true;
        uint64_t* prev = nullptr;
        for (int item = blockIdx.x; item < items && ok; item += gridDim.x) {
            int x0, y0, z0, blk;
            origin(item, x0, y0, z0, blk);
            for (int cb = 0; cb < ncb; ++cb) {
                ok = mbar_wait_role(&b_empty[st], ph, &s_abort, a.err);
                if (!ok) break;
                const uint32_t wbase = base + (uint32_t)st * stage_bytes, hbase = wbase + kWBytes;
                if (pt == 0) {
                    mbar_arrive_tx(&b_wfull[st], kWBytes);
                    bulk_load(wbase, a.w + (size_t)(blk * ncb + cb) * (kWBytes / 2), kWBytes, &b_wfull[st]);
                    ++issued;
                }
                if (PAIRS) {
                    for (int u = pt; u < kPairUnits; u += kZbProd) {
                        const int hy = u / kHX, gx = x0 + (u - hy * kHX) - 1, gy = y0 + hy - 1;
                        const bool in2 = gx >= 0 && gx < g.nx && gy >= 0 && gy < g.ny;
                        const bf16* p = a.in + (in2 ? 2 * ((long)gy * g.nx + gx) : 0);
                        uint32_t dst = hbase + (uint32_t)u * 16u;
                        for (int hz = 0; hz < a.zt + 2; ++hz, dst += kPlane) {
                            const int gz = z0 + hz - 1;
                            const bool in3 = in2 && gz >= 0 && gz < g.nz;
                            cp_async4(dst, in3 ? p + 2 * (long)gz * g.nx * g.ny : a.in, in3);
                        }
                    }
                } else {
                const bool isup = cb * 16 < a.cup;
                const int sh = isup ? 1 : 0, C = isup ? a.cup : a.cin - a.cup;
                const int snx = g.nx >> sh, sny = g.ny >> sh;
                const bf16* src0 = (isup ? a.up + cb * 16 : a.in + (cb * 16 - a.cup));
                const size_t zstride = (size_t)snx * sny * C;
                for (int u = pt; u < kPlaneUnits; u += kZbProd) {
                    const int kc = u & 1, r = u >> 1, hy = r / kHX, hx = r - hy * kHX;
                    const int gx = x0 + hx - 1, gy = y0 + hy - 1;
                    const bool in2 = gx >= 0 && gx < g.nx && gy >= 0 && gy < g.ny;
                    const bf16* p = src0 + (in2 ? ((size_t)(gy >> sh) * snx + (gx >> sh)) * C : 0) + kc * 8;
                    uint32_t dst = hbase + (uint32_t)((hy * 2 + kc) * kHX + hx) * 16u;
                    for (int hz = 0; hz < a.zt + 2; ++hz, dst += kPlane) {
                        const int gz = z0 + hz - 1;
                        const bool in3 = in2 && gz >= 0 && gz < g.nz;
                        cp_async16(dst, in3 ? p + (size_t)(gz >> sh) * zstride : a.in, in3);
                    }
                }
                }
                cp_async_commit();
                // hand over the stage before this one: its copies are done when at most one group is open
                if (prev) {
                    asm volatile("cp.async.wait_group 1;" ::: "memory");
                    fence_proxy_async();
                    mbar_arrive(prev);
                }
                prev = &b_full[st];
                if (++st == a.nstage) {
                    st = 0;
                    ph ^= 1u;
                }
                // and this one at once where the next buffer is not free yet
                if (!mbar_test_wait(&b_empty[st], ph)) {
                    cp_async_wait_all();
                    fence_proxy_async();
                    mbar_arrive(prev);
                    prev = nullptr;
                }
            }
        }
        cp_async_wait_all();
        if (prev) {
            fence_proxy_async();
            mbar_arrive(prev);
        }
        // the CTA ends only once its bulk copies have landed (bounded), also where another role gives up after this one
        // is through
        if (pt == 0)
            for (int i = max(0, issued - a.nstage); i < issued; ++i)
                if (!mbar_drain(&b_wfull[i % a.nstage], (uint32_t)(i / a.nstage) & 1u)) atomicMax(a.err, 1);
    } else if (warp == kZbMmaWarp) {
        // ---- MMA issue ----
        if (lane == 0) {
            int st = 0, k = 0;
            uint32_t ph = 0u;
            bool ok = true;
            const uint32_t zeros = base + (uint32_t)a.nstage * stage_bytes;  // PAIRS
            for (int item = blockIdx.x; item < items && ok; item += gridDim.x, ++k) {
                const uint32_t acc = tmem + (uint32_t)((k & 1) * a.zt * NB);
                ok = mbar_wait_role(&b_accfree[k & 1], (uint32_t)((k >> 1) & 1) ^ 1u, &s_abort, a.err);
                if (!ok) break;
                for (int cb = 0; cb < ncb; ++cb) {
                    ok = mbar_wait_role(&b_full[st], ph, &s_abort, a.err) &&
                         mbar_wait_role(&b_wfull[st], ph, &s_abort, a.err);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t wbase = base + (uint32_t)st * stage_bytes, hbase = wbase + kWBytes;
                    for (int zi = 0; zi < a.zt + 2; ++zi) {
                        const int lo = max(0, zi - 2), nw = min(a.zt - 1, zi) - lo + 1;
                        const uint32_t d = acc + (uint32_t)(lo * NB);
                        const uint32_t pl = hbase + (uint32_t)zi * kPlane;
                        const uint64_t ad0 = smem_desc(pl, kHX * 16, 2 * kHX * 16);
                        const uint64_t bd0 =
                            smem_desc(wbase + (uint32_t)((lo - (zi - 2)) * NB * 32), 8 * 16, 2 * 8 * 16);
                        const uint32_t id = idesc_bf16(128, nw * NB);
                        // the newest output plane of the window starts at its first tap
                        const bool start = cb == 0 && zi < a.zt;
#pragma unroll
                        for (int t = 0; t < 9; ++t) {
                            // start addresses are in 16-byte units in the low bits of the descriptors
                            const uint32_t tp = pl + (uint32_t)((t / 3) * kHX + t % 3) * 16u;
                            const uint64_t ad = PAIRS ? smem_desc(tp, zeros - tp, kHX * 16)
                                                      : ad0 + (uint64_t)((t / 3) * 2 * kHX + t % 3);
                            const uint64_t bd = bd0 + (uint64_t)(t * 6 * NB);
                            if (t == 0 && start) {
                                if (nw > 1) tc_mma(d, ad, bd, idesc_bf16(128, (nw - 1) * NB), 1u);
                                tc_mma(d + (uint32_t)((nw - 1) * NB), ad, bd + (uint64_t)((nw - 1) * 2 * NB),
                                       idesc_bf16(128, NB), 0u);
                            } else {
                                tc_mma(d, ad, bd, id, 1u);
                            }
                        }
                    }
                    tc_commit(&b_empty[st]);
                    if (++st == a.nstage) {
                        st = 0;
                        ph ^= 1u;
                    }
                }
                if (ok) tc_commit(&b_acc[k & 1]);
            }
            tc_commit(&b_end);
            if (!mbar_drain(&b_end, 0u)) atomicMax(a.err, 2);
        }
        __syncwarp();
    } else {
        // ---- read-out ----
        const int m = warp * 32 + lane;
        const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16);
        // NB = 16: one channel block, so its biases and the head's weights stay in registers
        float bias0[16], head[16], hbias = 0.f;
        if (NB == 16) {
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                bias0[e] = a.bias ? a.bias[e] : 0.f;
                head[e] = a.y ? __bfloat162float(a.head_w[e]) : 0.f;
            }
            if (a.y) hbias = a.head_b[0];
        }
        int k = 0;
        for (int item = blockIdx.x; item < items; item += gridDim.x, ++k) {
            int x0, y0, z0, blk;
            origin(item, x0, y0, z0, blk);
            const int gx = x0 + (m & 7), gy = y0 + (m >> 3);
            const bool in2 = gx < g.nx && gy < g.ny;
            if (!mbar_wait_warp(&b_acc[k & 1], (uint32_t)((k >> 1) & 1), &s_abort, a.err)) break;
            tc_fence_after();
            const uint32_t acc = lane_base + (uint32_t)((k & 1) * a.zt * NB);
            const size_t v0 = in2 ? ((size_t)z0 * g.ny + gy) * g.nx + gx : 0;
            const int chunks = min(a.zt, g.nz - z0) * (NB / 16);
            for (int q0 = 0; q0 < chunks; q0 += 2) {  // 16 columns each, two at a time
                uint32_t r[32];
                if (q0 + 1 < chunks) tmem_ld32(acc + (uint32_t)(q0 * 16), r);
                else tmem_ld16(acc + (uint32_t)(q0 * 16), r);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int q = q0 + h, j = q / (NB / 16), c0 = (q - j * (NB / 16)) * 16 + blk * NB;
                    if (q >= chunks || !in2) continue;
                    const size_t v = v0 + (size_t)j * g.nx * g.ny;
                    __align__(16) bf16 o[16];
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        float x = __uint_as_float(r[16 * h + e]) + (NB == 16 ? bias0[e] : a.bias ? __ldg(a.bias + c0 + e) : 0.f);
                        if (a.relu) x = fmaxf(x, 0.f);
                        o[e] = __float2bfloat16(x);
                    }
                    if (NB > 16 || a.out) {
                        bf16* orow = a.out + v * a.N + c0;
                        *reinterpret_cast<uint4*>(orow) = *reinterpret_cast<const uint4*>(o);
                        *reinterpret_cast<uint4*>(orow + 8) = *reinterpret_cast<const uint4*>(o + 8);
                    }
                    if (NB == 16 && a.y) {
                        float sum = 0.f;
#pragma unroll
                        for (int e = 0; e < 16; ++e) sum = fmaf(__bfloat162float(o[e]), head[e], sum);
                        a.y[v] = sum + hbias;
                    }
                }
            }
            tc_fence_before();
            mbar_arrive(&b_accfree[k & 1]);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == kZbMmaWarp)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(a.ncols) : "memory");
}

// ---------------------------------------------------------------------------
// Weight and bias gradients on the tcgen05 tensor cores.
//
// dW[t][co][ci] = sum_v x[v + off(t)][ci] dy[v][co] and dB[co] = sum_v dy[v][co]
// form one GEMM D[m][n] = sum_k A[m][k] B[n][k]: rows m = t Cin_pad + ci
// (taps x padded input channels), then one row of ones (m = R = taps
// Cin_pad) whose product is the bias gradient, further rows zero; columns n =
// output channels (N = Cout_pad); K = voxels.  A CTA takes a block of 128
// rows and a contiguous range of voxel chunks (a K split), accumulates
// D[128][N] in tensor memory over chunks of kWgK voxels (eight MMAs of K =
// 16 each, M = 128) and stores it as FP32 partial sums; k_wgrad_reduce adds
// the splits in a fixed order, so no atomics are involved.  The operands
// arrive channels-last, so staging transposes them into the canonical K-major
// layout without swizzling (a core matrix is 8 rows of 16 bytes: 8 voxels of
// one row): a thread loads the 16-byte 8-channel groups of 8 voxels and
// stores eight 16-byte core-matrix rows, one per channel, after an 8 x 8
// transpose in registers.  Core matrices of consecutive row groups are
// kWgSbo = 272 bytes apart (not 256), so the eight threads of a store phase
// hit different bank groups.  Chunks are double-buffered: the MMAs of one
// chunk run while the next one is staged.  Waits are bounded and tensor
// memory is released under the same rules as in k_conv_zb.  Staging is bound by
// its index arithmetic and load latency: where nx is a multiple of 8 an octet of
// voxels lies in one row and is decoded once, and 256 threads load a chunk in
// one round (48 -> 16 layer at 64^3: 412 -> 203 us; a decode a voxel, 128
// threads and two rounds before).
// ---------------------------------------------------------------------------
constexpr int kWgK = 128;        // voxels per chunk
constexpr int kWgThreads = 256;  // staging; the accumulators are read out by the first 128
constexpr int kWgSbo = 272;      // bytes between the core matrices of consecutive 8-row groups
constexpr int kWgAStep = 16 * kWgSbo;   // bytes of one K = 16 step of A (16 row groups)
constexpr int kWgABytes = (kWgK / 16) * kWgAStep;
constexpr int kWgMaxCtas = 304;  // row blocks x splits of a launch (about two per SM)

__host__ __device__ constexpr int wg_bstep(int N) { return (N / 8) * kWgSbo; }
__host__ __device__ constexpr int wg_buf_bytes(int N) { return kWgABytes + (kWgK / 16) * wg_bstep(N); }

// 8 x 8 transpose of BF16 values: in[e] holds channels 0..7 of voxel e, out[j]
// voxels 0..7 of channel j (element i of a 16-byte group in bytes 2i, 2i+1)
__device__ __forceinline__ void transpose8(const uint4* in, uint4* out) {
    const uint32_t* w = reinterpret_cast<const uint32_t*>(in);  // w[4 e + k]: channels 2k (low), 2k+1 of voxel e
    uint32_t* o = reinterpret_cast<uint32_t*>(out);              // o[4 j + m]: voxels 2m (low), 2m+1 of channel j
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const uint32_t a = w[4 * (2 * m) + k], b = w[4 * (2 * m + 1) + k];
            o[4 * (2 * k) + m] = __byte_perm(a, b, 0x5410);
            o[4 * (2 * k + 1) + m] = __byte_perm(a, b, 0x7632);
        }
}

// Partial GEMM of row block blockIdx.x over voxel chunks [blockIdx.y cps,
// (blockIdx.y + 1) cps) into part[(split nrb + rb) 128 + row][N] (FP32).
// x: [voxel][cin_pad], dy: [voxel][N]; N a multiple of 16 in [16, 128].
__global__ void __launch_bounds__(kWgThreads) k_wgrad_tc(CG g, const bf16* __restrict__ x, int cin_pad, int ntaps,
                                                         const bf16* __restrict__ dy, int N, int cps,
                                                         float* __restrict__ part, int ncols, int* err) {
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ __align__(8) uint64_t mbar[2];
    __shared__ uint32_t s_tmem;
    // a wait gave up: in an even chunk, an odd chunk, after the chunks.  One word for all would let a fast thread set it
    // in its next wait before a slow one has read it after this chunk's barrier, and the two wait at other barriers.
    __shared__ int s_abort[3];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rb = blockIdx.x, nrb = gridDim.x;
    const int bstep = wg_bstep(N), bufb = wg_buf_bytes(N);

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        mbar_init(&mbar[0], 1);
        mbar_init(&mbar[1], 1);
        s_abort[0] = s_abort[1] = s_abort[2] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    const uint32_t idesc = idesc_bf16(128, N);

    const int R = ntaps * cin_pad;  // weight rows; row R is the row of ones
    const int nchunks = (g.N + kWgK - 1) / kWgK;
    const int ch0 = blockIdx.y * cps, nch = max(0, min(ch0 + cps, nchunks) - ch0);
    uint32_t phase[2] = {0u, 0u};
    bool pending[2] = {false, false};
    bool unconfirmed[2] = {false, false};
    uint32_t uphase[2] = {0u, 0u};
    auto wait_mma = [&](int b, int flag) {
        if (pending[b]) {
            if (!mbar_wait_bounded(&mbar[b], phase[b])) {
                s_abort[flag] = 1;
                atomicExch(err, 1);
                unconfirmed[b] = true;
                uphase[b] = phase[b];
            }
            phase[b] ^= 1u;
            pending[b] = false;
        }
    };
    const uint4 zero4 = make_uint4(0u, 0u, 0u, 0u);
    const bool rows8 = g.nx % 8 == 0;
    // stage chunk ch0 + c into buffer b
    auto stage = [&](int c, int b) {
        unsigned char* A = smem + b * bufb;
        unsigned char* B = A + kWgABytes;
        const int vbase = (ch0 + c) * kWgK;
        // A: 16 row groups x kWgK / 8 voxel octets (consecutive threads: consecutive row groups)
        for (int u = tid; u < 16 * (kWgK / 8); u += kWgThreads) {
            const int gq = u & 15, o = u >> 4;
            const int row0 = rb * 128 + gq * 8;
            uint4 in[8];
            if (row0 < R) {
                const int tap = row0 / cin_pad, ci0 = row0 - tap * cin_pad;
                int dz, dyy, dx;
                tap_off(tap, ntaps, dz, dyy, dx);
                if (rows8) {
                    // the octet lies in one x row: one decode, and only the row's ends can miss a neighbour
                    const Vox q = vox(g, vbase + 8 * o);
                    const int y = q.y + dyy, z = q.z + dz;
                    const bool ok = q.in && y >= 0 && y < g.ny && z >= 0 && z < g.nz;
                    const uint4* src = reinterpret_cast<const uint4*>(
                        x + ((ptrdiff_t)((long)(ok ? z : 0) * g.ny + (ok ? y : 0)) * g.nx + q.x + dx) * cin_pad + ci0);
                    const int step = cin_pad / 8;
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const int xe = q.x + dx + e;
                        in[e] = ok && xe >= 0 && xe < g.nx ? __ldg(src + e * step) : zero4;
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < 8; ++e) {
                        const int n = nbr(g, vox(g, vbase + 8 * o + e), dz, dyy, dx);
                        in[e] = n >= 0 ? __ldg(reinterpret_cast<const uint4*>(x + (size_t)n * cin_pad + ci0)) : zero4;
                    }
                }
            } else {
                // the row of ones (channel 0 of the group starting at row R), then zeros
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    in[e] = zero4;
                    if (row0 == R && vbase + 8 * o + e < g.N) in[e].x = 0x3F80u;  // BF16 1.0 in element 0
                }
            }
            uint4 out[8];
            transpose8(in, out);
            unsigned char* dst = A + (o >> 1) * kWgAStep + gq * kWgSbo + (o & 1) * 128;
#pragma unroll
            for (int j = 0; j < 8; ++j) *reinterpret_cast<uint4*>(dst + j * 16) = out[j];
        }
        // B: N / 8 column groups x kWgK / 8 voxel octets
        const int ng = N >> 3;
        for (int u = tid; u < ng * (kWgK / 8); u += kWgThreads) {
            const int gq = u % ng, o = u / ng;
            uint4 in[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int v = vbase + 8 * o + e;
                in[e] = v < g.N ? __ldg(reinterpret_cast<const uint4*>(dy + (size_t)v * N + gq * 8)) : zero4;
            }
            uint4 out[8];
            transpose8(in, out);
            unsigned char* dst = B + (o >> 1) * bstep + gq * kWgSbo + (o & 1) * 128;
#pragma unroll
            for (int j = 0; j < 8; ++j) *reinterpret_cast<uint4*>(dst + j * 16) = out[j];
        }
    };

    for (int c = 0; c < nch; ++c) {
        const int b = c & 1;
        wait_mma(b, b);  // the MMAs of chunk c - 2 read this buffer
        stage(c, b);
        fence_proxy_async();
        __syncthreads();
        if (s_abort[b]) break;
        if (tid == 0) {
            tc_fence_after();
            const uint32_t a0 = smem_u32(smem + b * bufb), b0 = a0 + kWgABytes;
#pragma unroll
            for (int q = 0; q < kWgK / 16; ++q) {
                const uint64_t ad = smem_desc(a0 + (uint32_t)(q * kWgAStep), 128, kWgSbo);
                const uint64_t bd = smem_desc(b0 + (uint32_t)(q * bstep), 128, kWgSbo);
                tc_mma(tmem, ad, bd, idesc, (c == 0 && q == 0) ? 0u : 1u);
            }
            tc_commit(&mbar[b]);
        }
        pending[b] = true;
    }
    for (int b = 0; b < 2; ++b) wait_mma(b, 2);
    __syncthreads();
    if (!(s_abort[0] | s_abort[1] | s_abort[2]) && nch > 0 && warp < 4) {
        tc_fence_after();
        const int row = warp * 32 + lane;
        float* dst = part + ((size_t)(blockIdx.y * nrb + rb) * 128 + row) * N;
        for (int c0 = 0; c0 < N; c0 += 8) {
            float v[8];
            tmem_ld8(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
            *reinterpret_cast<float4*>(dst + c0) = make_float4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<float4*>(dst + c0 + 4) = make_float4(v[4], v[5], v[6], v[7]);
        }
    }
    // a phase whose wait gave up must be seen complete before the dealloc
    for (int b = 0; b < 2; ++b)
        if (unconfirmed[b] && !mbar_drain(&mbar[b], uphase[b])) atomicMax(err, 2);
    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols) : "memory");
}

// dW[t][co][ci] (ci < cin, co < cout) and dB[co] from the partial sums of the
// nsplit voxel splits, added in split order
__global__ void k_wgrad_reduce(const float* __restrict__ part, int nsplit, int nrb, int N, int ntaps, int cin_pad,
                               int cin, int cout, float* __restrict__ dW, float* __restrict__ dB) {
    const long t = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const int R = ntaps * cin_pad;
    if (t >= (long)(R + 1) * cout) return;
    const int n = (int)(t % cout);
    const int m = (int)(t / cout);  // row, 0 .. R
    const int rb = m >> 7, row = m & 127;
    // added in split order, sixteen loads in flight (the head has 304 splits for 17 outputs: 47 us one at a time)
    float s = 0.f;
    const float* src = part + ((size_t)rb * 128 + row) * N + n;
    const size_t step = (size_t)nrb * 128 * N;
    for (int k0 = 0; k0 < nsplit; k0 += 16) {
        float v[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) v[u] = k0 + u < nsplit ? __ldg(src + (k0 + u) * step) : 0.f;
#pragma unroll
        for (int u = 0; u < 16; ++u)
            if (k0 + u < nsplit) s += v[u];
    }
    if (m == R) {
        dB[n] = s;
        return;
    }
    const int tap = m / cin_pad, ci = m - tap * cin_pad;
    if (ci < cin) dW[((size_t)tap * cout + n) * cin + ci] = s;
}

}  // namespace
}  // namespace cdi

using namespace cdi;

struct cdi_unet {
    int n[3] = {0, 0, 0};
    CG g[4];  // levels 0..3
    char* ws = nullptr;
    size_t ws_bytes = 0;
    cudaStream_t stream = nullptr;
    // parameters
    float *W[kLayers], *B[kLayers], *gW[kLayers], *gB[kLayers];
    float *mW[kLayers], *vW[kLayers], *mB[kLayers], *vB[kLayers];
    bf16 *Wb[kLayers], *Wt[kLayers];    // weights of the mma.sync kernels
    bf16 *Wk[kLayers], *Wkt[kLayers];   // weights of the tcgen05 convolution (forward, data gradient)
    int ci_pad[kLayers], co_pad[kLayers];
    // activations and gradients (BF16, channels last)
    bf16 *xp;  // input pairs [N][2]
    bf16 *x, *e0, *p0, *e1, *p1, *e2, *p2, *b, *c2, *d2, *c1, *d1, *c0, *d0;
    bf16 *gy, *gd0, *gc0, *gd1, *gc1, *gd2, *gc2, *gb, *gp2, *ge2, *gp1, *ge1, *gp0, *ge0;
    float *y, *t, *part;
    float* wpart;  // FP32 partial sums of the tcgen05 weight gradients (voxel splits x rows x columns)
    double* x2;  // host-input staging [N][2]
    double* sd;  // prediction scales (FP64 and FP32 copies)
    float* sf;
    int* tc_err;          // set by a tcgen05 convolution whose bounded wait ran out
    bool use_tc = true;   // 3x3x3 convolutions on tcgen05 (else mma.sync)
    bool wgrad_tc = true; // weight and bias gradients on tcgen05 (else mma.sync with FP32 atomics)
    long adam_t = 0;
    bool weights_ready = false;
    std::string err;
};

namespace {

std::string g_unet_error;

cdi_status ufail(cdi_unet* u, cdi_status st, const std::string& m) {
    if (u) u->err = m;
    else g_unet_error = m;
    return st;
}

struct UCarver {
    char* base;
    size_t off = 0;
    void* take(size_t bytes) {
        off = (off + 255) & ~size_t(255);
        void* p = base ? base + off : nullptr;
        off += bytes;
        return p;
    }
};

// level of the grid each layer works on (e0 e1 e2 b d2 d1 d0 head)
constexpr int kLevelOf[kLayers] = {0, 1, 2, 3, 2, 1, 0, 0};

// work split of the tcgen05 weight gradient of one layer: row blocks of 128
// (taps x padded input channels, plus the row of ones), voxel splits of cps
// chunks each (every split holds at least one chunk), about kWgMaxCtas CTAs
struct WgPlan {
    int nrb, nsplit, cps;
};
WgPlan wg_plan(int l, long nvox, int ci_pad) {
    WgPlan p;
    p.nrb = (kTaps[l] * ci_pad + 1 + 127) / 128;
    const int nchunks = (int)std::max(1L, (nvox + kWgK - 1) / kWgK);
    const int s = std::max(1, std::min(nchunks, (kWgMaxCtas + p.nrb - 1) / p.nrb));
    p.cps = (nchunks + s - 1) / s;
    p.nsplit = (nchunks + p.cps - 1) / p.cps;
    return p;
}

void unet_carve(cdi_unet* u, char* base, size_t* total) {
    UCarver cv{base};
    for (int l = 0; l < kLayers; ++l) {
        const size_t nw = (size_t)kTaps[l] * kCout[l] * kCin[l], nb = kCout[l];
        u->ci_pad[l] = pad16(kCin[l]);
        u->co_pad[l] = pad16(kCout[l]);
        u->W[l] = (float*)cv.take(nw * 4);
        u->B[l] = (float*)cv.take(nb * 4);
        u->gW[l] = (float*)cv.take(nw * 4);
        u->gB[l] = (float*)cv.take(nb * 4);
        u->mW[l] = (float*)cv.take(nw * 4);
        u->vW[l] = (float*)cv.take(nw * 4);
        u->mB[l] = (float*)cv.take(nb * 4);
        u->vB[l] = (float*)cv.take(nb * 4);
        const size_t np = (size_t)kTaps[l] * u->ci_pad[l] * u->co_pad[l];
        u->Wb[l] = (bf16*)cv.take(np * 2);
        u->Wt[l] = (bf16*)cv.take(np * 2);
        u->Wk[l] = (bf16*)cv.take(np * 2);
        u->Wkt[l] = (bf16*)cv.take(np * 2);
    }
    const long N0 = u->g[0].N, N1 = u->g[1].N, N2 = u->g[2].N, N3 = u->g[3].N;
    auto act = [&](long n, int c) { return (bf16*)cv.take((size_t)n * c * 2); };
    u->x = act(N0, 16);
    u->xp = act(N0, 2);
    u->e0 = act(N0, 16);
    u->p0 = act(N1, 16);
    u->e1 = act(N1, 32);
    u->p1 = act(N2, 32);
    u->e2 = act(N2, 64);
    u->p2 = act(N3, 64);
    u->b = act(N3, 128);
    u->c2 = act(N2, 192);
    u->d2 = act(N2, 64);
    u->c1 = act(N1, 96);
    u->d1 = act(N1, 32);
    u->c0 = act(N0, 48);
    u->d0 = act(N0, 16);
    u->gy = act(N0, 16);
    u->gd0 = act(N0, 16);
    u->gc0 = act(N0, 48);
    u->gd1 = act(N1, 32);
    u->gc1 = act(N1, 96);
    u->gd2 = act(N2, 64);
    u->gc2 = act(N2, 192);
    u->gb = act(N3, 128);
    u->gp2 = act(N3, 64);
    u->ge2 = act(N2, 64);
    u->gp1 = act(N2, 32);
    u->ge1 = act(N1, 32);
    u->gp0 = act(N1, 16);
    u->ge0 = act(N0, 16);
    u->y = (float*)cv.take((size_t)N0 * 4);
    u->t = (float*)cv.take((size_t)N0 * 4);
    u->part = (float*)cv.take(256);
    size_t wp = 0;
    for (int l = 0; l < kLayers; ++l) {
        const WgPlan p = wg_plan(l, u->g[kLevelOf[l]].N, pad16(kCin[l]));
        wp = std::max(wp, (size_t)p.nsplit * p.nrb * 128 * pad16(kCout[l]));
    }
    u->wpart = (float*)cv.take(wp * 4);
    u->sd = (double*)cv.take(4 * sizeof(double));
    u->sf = (float*)cv.take(4 * sizeof(float));
    u->tc_err = (int*)cv.take(sizeof(int));
    u->x2 = (double*)cv.take((size_t)N0 * 2 * 8);
    *total = cv.off + 256;
}

// Planes of a tile of the tcgen05 convolution.  More planes share each staged halo plane and fill the
// MMAs' N (planes 2 .. zt-1 of a tile feed three output planes at once), fewer give more tiles to spread
// over the SMs.  Takes the zt of least estimated cycles: rounds of the persistent grid times the MMA cycles
// of a tile (32 cycles of A and NB / 4 of B a column block, or NB / 2 of arithmetic, whichever is larger)
// plus 2500 for staging and reading out its ends.  NB zt <= 256 (two accumulator sets in 512 columns).
int conv_planes(const CG& g, int NB, int nblk, int ncb, int nsm) {
    const int cap = std::min(8, 256 / NB);
    long best = 0;
    int zt_best = 1;
    for (int zt = 1; zt <= cap; zt *= 2) {
        if (zt > 1 && zt / 2 >= g.nz) break;
        const long items = (long)((g.nx + kTileX - 1) / kTileX) * ((g.ny + kTileY - 1) / kTileY) *
                           ((g.nz + zt - 1) / zt) * nblk;
        long cyc = 0;
        for (int zi = 0; zi < zt + 2; ++zi) {
            const int nw = std::min(zt - 1, zi) - std::max(0, zi - 2) + 1;
            cyc += std::max(32 + nw * NB / 4, nw * NB / 2);
        }
        const long cost = (items + nsm - 1) / nsm * (9 * cyc * ncb + 2500);
        if (zt == 1 || cost < best) {
            best = cost;
            zt_best = zt;
        }
    }
    return zt_best;
}

constexpr size_t kConvSmem = 220 * 1024;  // of the 227 KB a CTA may use

template <int NB, bool PAIRS = false>
void conv_zb(const ConvArgs& a, size_t smem, unsigned grid, cudaStream_t s) {
    cudaFuncSetAttribute(k_conv_zb<NB, PAIRS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kConvSmem);
    k_conv_zb<NB, PAIRS><<<grid, kZbThreads, smem, s>>>(a);
}

// launch of the tcgen05 convolution of the layer a describes (all but its split): a persistent grid of one CTA per
// SM, or two for PAIRS, whose shared memory lets no more in, so no TMEM allocation waits for another CTA of the launch
void conv_launch(ConvArgs a, bool pairs, cudaStream_t s) {
    int dev = 0, nsm = 148;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const int per = pairs ? 2 : 1;
    const int NB = conv_nb(a.N);
    a.nblk = a.N / NB;
    a.zt = conv_planes(a.g, NB, a.nblk, a.cin / 16, nsm * per);
    const size_t stage = zb_wbytes(NB) + (size_t)(a.zt + 2) * zb_plane(pairs);
    const size_t extra = pairs ? kPairZeroBytes : 0;
    a.nstage = (int)std::min<size_t>(kZbMaxStages, (kConvSmem / per - extra - (per - 1) * 2048) / stage);
    a.ncols = 32;
    while (a.ncols < 2 * a.zt * NB) a.ncols *= 2;
    const long items = (long)((a.g.nx + kTileX - 1) / kTileX) * ((a.g.ny + kTileY - 1) / kTileY) *
                       ((a.g.nz + a.zt - 1) / a.zt) * a.nblk;
    const unsigned grid = (unsigned)std::min<long>(items, (long)nsm * per);
    // at least what keeps another CTA out of the SM
    const size_t smem = std::max(a.nstage * stage + extra, (size_t)(pairs ? 78 : 116) * 1024);
    if (pairs) {
        conv_zb<16, true>(a, smem, grid, s);
        return;
    }
    switch (NB) {
        case 16: conv_zb<16>(a, smem, grid, s); break;
        case 32: conv_zb<32>(a, smem, grid, s); break;
        case 48: conv_zb<48>(a, smem, grid, s); break;
        default: conv_zb<64>(a, smem, grid, s); break;
    }
}

void conv_tc(cdi_unet* u, const CG& gl, const bf16* in, int cin, const bf16* w, int N, const float* bias, bf16* out,
             bool relu, const bf16* up = nullptr, int cup = 0) {
    conv_launch({gl, in, up, cin, cup, w, bias, out, nullptr, nullptr, nullptr, N, relu ? 1 : 0, 0, 0, 0, 0, u->tc_err},
                false, u->stream);
}

// the first layer from the input pairs
void conv_first(cdi_unet* u) {
    conv_launch({u->g[0], u->xp, nullptr, 16, 0, u->Wk[0], u->B[0], u->e0, nullptr, nullptr, nullptr, 16, 1, 0, 0, 0, 0,
                 u->tc_err}, true, u->stream);
}

// the last 3x3x3 layer with the head in its read-out (y only; d0 is not stored); in: [up (32 channels), in (16)]
void conv_last(cdi_unet* u, const bf16* in, const bf16* up, float* y) {
    conv_launch({u->g[0], in, up, 48, 32, u->Wk[6], u->B[6], nullptr, u->Wb[7], u->B[7], y, 16, 1, 0, 0, 0, 0,
                 u->tc_err}, false, u->stream);
}

// y = conv(in) for layer l on level grid gl into out (stride, offset)
template <bool OUTF32>
void conv_fwd(cdi_unet* u, int l, const CG& gl, const bf16* in, void* out, int stride, int off, bool relu) {
    if (!OUTF32 && kTaps[l] == 27 && u->use_tc && off == 0 && stride == u->co_pad[l]) {
        conv_tc(u, gl, in, u->ci_pad[l], u->Wk[l], u->co_pad[l], u->B[l], (bf16*)out, relu);
        return;
    }
    const unsigned gb = (unsigned)((gl.N + 63) / 64);
    const int nf = u->co_pad[l] / 8;
    const int cin = u->ci_pad[l], cop = u->co_pad[l];
    cudaStream_t s = u->stream;
#define CONV_CASE(NFV)                                                                                          \
    case NFV:                                                                                                   \
        k_conv<NFV, OUTF32><<<gb, 128, 0, s>>>(gl, in, cin, u->Wb[l], cop, u->B[l], kCout[l], out, stride, off, \
                                                relu ? 1 : 0, kTaps[l]);                                        \
        break;
    switch (nf) {
        CONV_CASE(2)
        CONV_CASE(4)
        CONV_CASE(8)
        CONV_CASE(16)
        default: break;
    }
#undef CONV_CASE
}

// dx (BF16 [N][ci_pad]) = adjoint of layer l applied to dy (BF16 [N][co_pad])
void conv_dgrad(cdi_unet* u, int l, const CG& gl, const bf16* dy, bf16* dx) {
    if (kTaps[l] == 27 && u->use_tc) {
        conv_tc(u, gl, dy, u->co_pad[l], u->Wkt[l], u->ci_pad[l], nullptr, dx, false);
        return;
    }
    const unsigned gb = (unsigned)((gl.N + 63) / 64);
    const int nf = u->ci_pad[l] / 8;
    cudaStream_t s = u->stream;
#define DG_CASE(NFV)                                                                                              \
    case NFV:                                                                                                     \
        k_conv<NFV, false><<<gb, 128, 0, s>>>(gl, dy, u->co_pad[l], u->Wt[l], u->ci_pad[l], nullptr,             \
                                               u->ci_pad[l], dx, u->ci_pad[l], 0, 0, kTaps[l]);                   \
        break;
    switch (nf) {
        DG_CASE(2)
        DG_CASE(4)
        DG_CASE(6)
        DG_CASE(8)
        DG_CASE(12)
        DG_CASE(24)
        default: break;
    }
#undef DG_CASE
}

// weight and bias gradients of layer l on the tcgen05 tensor cores (no atomics)
void wgrad_tc(cdi_unet* u, int l, const CG& gl, const bf16* in, const bf16* dy) {
    static bool attr = false;
    if (!attr) {
        cudaFuncSetAttribute(k_wgrad_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * wg_buf_bytes(128));
        attr = true;
    }
    const int N = u->co_pad[l];
    const WgPlan p = wg_plan(l, gl.N, u->ci_pad[l]);
    const int ncols = N <= 32 ? 32 : N <= 64 ? 64 : 128;
    k_wgrad_tc<<<dim3((unsigned)p.nrb, (unsigned)p.nsplit), kWgThreads, 2 * (size_t)wg_buf_bytes(N), u->stream>>>(
        gl, in, u->ci_pad[l], kTaps[l], dy, N, p.cps, u->wpart, ncols, u->tc_err);
    const long nt = (long)(kTaps[l] * u->ci_pad[l] + 1) * kCout[l];
    k_wgrad_reduce<<<blocks(nt), 256, 0, u->stream>>>(u->wpart, p.nsplit, p.nrb, N, kTaps[l], u->ci_pad[l], kCin[l],
                                                      kCout[l], u->gW[l], u->gB[l]);
}

void conv_wgrad(cdi_unet* u, int l, const CG& gl, const bf16* in, const bf16* dy) {
    if (u->wgrad_tc) {
        wgrad_tc(u, l, gl, in, dy);
        return;
    }
    const int chunk = 1024;
    dim3 grid((unsigned)kTaps[l], (unsigned)((u->co_pad[l] + 15) / 16), (unsigned)((gl.N + chunk - 1) / chunk));
    const int nf = u->ci_pad[l] / 8;
    cudaStream_t s = u->stream;
#define WG_CASE(NFV)                                                                                                \
    case NFV:                                                                                                       \
        k_wgrad<NFV><<<grid, 128, 0, s>>>(gl, in, u->ci_pad[l], dy, u->co_pad[l], u->gW[l], kCout[l], kCin[l],     \
                                           kTaps[l], chunk);                                                        \
        break;
    switch (nf) {
        WG_CASE(2)
        WG_CASE(4)
        WG_CASE(6)
        WG_CASE(8)
        WG_CASE(12)
        WG_CASE(24)
        default: break;
    }
#undef WG_CASE
    k_bias_grad<<<dim3(64, (unsigned)kCout[l]), 256, 0, s>>>(gl.N, dy, u->co_pad[l], kCout[l], u->gB[l]);
}

void refresh_weights(cdi_unet* u) {
    WeightSegs p;
    long n = 0;
    for (int l = 0; l < kLayers; ++l) {
        n += (long)kTaps[l] * u->co_pad[l] * u->ci_pad[l];
        p.end[l] = n;
        p.W[l] = u->W[l];
        p.taps[l] = kTaps[l];
        p.cout[l] = kCout[l];
        p.cin[l] = kCin[l];
        p.co_pad[l] = u->co_pad[l];
        p.ci_pad[l] = u->ci_pad[l];
        p.wb[l] = u->Wb[l];
        p.wt[l] = u->Wt[l];
        p.wk[l] = u->Wk[l];
        p.wkt[l] = u->Wkt[l];
    }
    k_weights_bf16<<<blocks(n), 256, 0, u->stream>>>(p);
    u->weights_ready = true;
}

// forward pass from the input (u->xp; u->x for the mma.sync kernels) to y (FP32).  With keep (training) every
// activation the gradients read is stored: the decoder inputs [up(coarser), skip] and d0; otherwise the tcgen05
// convolution gathers the former while staging its input tiles and only uses the latter for the head.
void forward(cdi_unet* u, bool keep, float* y) {
    const CG* g = u->g;
    cudaStream_t s = u->stream;
    const bool fuse = !keep && u->use_tc;
    if (u->use_tc) conv_first(u);
    else conv_fwd<false>(u, 0, g[0], u->x, u->e0, 16, 0, true);
    k_pool<<<blocks(g[1].N * 2L), 256, 0, s>>>(g[0], u->e0, 16, u->p0);
    conv_fwd<false>(u, 1, g[1], u->p0, u->e1, 32, 0, true);
    k_pool<<<blocks(g[2].N * 4L), 256, 0, s>>>(g[1], u->e1, 32, u->p1);
    conv_fwd<false>(u, 2, g[2], u->p1, u->e2, 64, 0, true);
    k_pool<<<blocks(g[3].N * 8L), 256, 0, s>>>(g[2], u->e2, 64, u->p2);
    conv_fwd<false>(u, 3, g[3], u->p2, u->b, 128, 0, true);
    g_launches += 7;
    if (fuse) {
        conv_tc(u, g[2], u->e2, 192, u->Wk[4], 64, u->B[4], u->d2, true, u->b, 128);
        conv_tc(u, g[1], u->e1, 96, u->Wk[5], 32, u->B[5], u->d1, true, u->d2, 64);
        conv_last(u, u->e0, u->d1, y);
        g_launches += 3;
        return;
    }
    k_up<<<blocks(g[2].N * 16L), 256, 0, s>>>(g[2], u->b, 128, u->c2, 192, 0);
    k_copy_ch<<<blocks(g[2].N * 8L), 256, 0, s>>>(g[2].N, u->e2, 64, 0, u->c2, 192, 128, 64);
    conv_fwd<false>(u, 4, g[2], u->c2, u->d2, 64, 0, true);
    k_up<<<blocks(g[1].N * 8L), 256, 0, s>>>(g[1], u->d2, 64, u->c1, 96, 0);
    k_copy_ch<<<blocks(g[1].N * 4L), 256, 0, s>>>(g[1].N, u->e1, 32, 0, u->c1, 96, 64, 32);
    conv_fwd<false>(u, 5, g[1], u->c1, u->d1, 32, 0, true);
    k_up<<<blocks(g[0].N * 4L), 256, 0, s>>>(g[0], u->d1, 32, u->c0, 48, 0);
    k_copy_ch<<<blocks(g[0].N * 2L), 256, 0, s>>>(g[0].N, u->e0, 16, 0, u->c0, 48, 32, 16);
    conv_fwd<false>(u, 6, g[0], u->c0, u->d0, 16, 0, true);
    conv_fwd<true>(u, 7, g[0], u->d0, y, 1, 0, false);
    g_launches += 10;
}

// gradients of the mean squared error (u->y against u->t) into gW, gB
void backward(cdi_unet* u) {
    const CG* g = u->g;
    cudaStream_t s = u->stream;
    for (int l = 0; l < kLayers && !u->wgrad_tc; ++l) {  // summed with atomics (the tcgen05 form stores every entry)
        cudaMemsetAsync(u->gW[l], 0, (size_t)kTaps[l] * kCout[l] * kCin[l] * 4, s);
        cudaMemsetAsync(u->gB[l], 0, (size_t)kCout[l] * 4, s);
    }
    cudaMemsetAsync(u->gy, 0, (size_t)g[0].N * 16 * 2, s);
    cudaMemsetAsync(u->part, 0, 4, s);
    k_loss<<<256, 256, 0, s>>>(g[0].N, u->y, u->t, u->gy, u->part);
    // head and d0
    conv_wgrad(u, 7, g[0], u->d0, u->gy);
    conv_dgrad(u, 7, g[0], u->gy, u->gd0);
    k_relu_mask<<<blocks(g[0].N * 2L), 256, 0, s>>>(g[0].N * 16L, u->gd0, u->d0);
    conv_wgrad(u, 6, g[0], u->c0, u->gd0);
    conv_dgrad(u, 6, g[0], u->gd0, u->gc0);
    k_up_bwd<<<blocks(g[1].N * 32L), 256, 0, s>>>(g[0], u->gc0, 48, 0, 32, u->gd1);
    k_relu_mask<<<blocks(g[1].N * 4L), 256, 0, s>>>(g[1].N * 32L, u->gd1, u->d1);
    k_copy_ch<<<blocks(g[0].N * 2L), 256, 0, s>>>(g[0].N, u->gc0, 48, 32, u->ge0, 16, 0, 16);
    // d1
    conv_wgrad(u, 5, g[1], u->c1, u->gd1);
    conv_dgrad(u, 5, g[1], u->gd1, u->gc1);
    k_up_bwd<<<blocks(g[2].N * 64L), 256, 0, s>>>(g[1], u->gc1, 96, 0, 64, u->gd2);
    k_relu_mask<<<blocks(g[2].N * 8L), 256, 0, s>>>(g[2].N * 64L, u->gd2, u->d2);
    k_copy_ch<<<blocks(g[1].N * 4L), 256, 0, s>>>(g[1].N, u->gc1, 96, 64, u->ge1, 32, 0, 32);
    // d2
    conv_wgrad(u, 4, g[2], u->c2, u->gd2);
    conv_dgrad(u, 4, g[2], u->gd2, u->gc2);
    k_up_bwd<<<blocks(g[3].N * 128L), 256, 0, s>>>(g[2], u->gc2, 192, 0, 128, u->gb);
    k_relu_mask<<<blocks(g[3].N * 16L), 256, 0, s>>>(g[3].N * 128L, u->gb, u->b);
    k_copy_ch<<<blocks(g[2].N * 8L), 256, 0, s>>>(g[2].N, u->gc2, 192, 128, u->ge2, 64, 0, 64);
    // bottleneck
    conv_wgrad(u, 3, g[3], u->p2, u->gb);
    conv_dgrad(u, 3, g[3], u->gb, u->gp2);
    k_pool_bwd_add<<<blocks(g[2].N * 8L), 256, 0, s>>>(g[2], u->gp2, 64, u->ge2, 64, 0);
    k_relu_mask<<<blocks(g[2].N * 8L), 256, 0, s>>>(g[2].N * 64L, u->ge2, u->e2);
    // e2
    conv_wgrad(u, 2, g[2], u->p1, u->ge2);
    conv_dgrad(u, 2, g[2], u->ge2, u->gp1);
    k_pool_bwd_add<<<blocks(g[1].N * 4L), 256, 0, s>>>(g[1], u->gp1, 32, u->ge1, 32, 0);
    k_relu_mask<<<blocks(g[1].N * 4L), 256, 0, s>>>(g[1].N * 32L, u->ge1, u->e1);
    // e1
    conv_wgrad(u, 1, g[1], u->p0, u->ge1);
    conv_dgrad(u, 1, g[1], u->ge1, u->gp0);
    k_pool_bwd_add<<<blocks(g[0].N * 2L), 256, 0, s>>>(g[0], u->gp0, 16, u->ge0, 16, 0);
    k_relu_mask<<<blocks(g[0].N * 2L), 256, 0, s>>>(g[0].N * 16L, u->ge0, u->e0);
    // e0
    conv_wgrad(u, 0, g[0], u->x, u->ge0);
    g_launches += 50;
}

void adam(cdi_unet* u, double lr) {
    ++u->adam_t;
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float bc1 = (float)(1.0 - std::pow(0.9, (double)u->adam_t));
    const float bc2 = (float)(1.0 - std::pow(0.999, (double)u->adam_t));
    ParamSegs p;
    long n = 0;
    for (int l = 0; l < kLayers; ++l) {
        const int i = 2 * l;
        p.end[i] = n += (long)kTaps[l] * kCout[l] * kCin[l];
        p.end[i + 1] = n += kCout[l];
        p.w[i] = u->W[l]; p.g[i] = u->gW[l]; p.m[i] = u->mW[l]; p.v[i] = u->vW[l];
        p.w[i + 1] = u->B[l]; p.g[i + 1] = u->gB[l]; p.m[i + 1] = u->mB[l]; p.v[i + 1] = u->vB[l];
    }
    k_adam<<<blocks(n), 256, 0, u->stream>>>(p, (float)lr, b1, b2, eps, bc1, bc2);
    refresh_weights(u);
}

size_t param_count() {
    size_t n = 0;
    for (int l = 0; l < kLayers; ++l) n += (size_t)kTaps[l] * kCout[l] * kCin[l] + kCout[l];
    return n;
}

// after a synchronisation: did a tcgen05 convolution give up on a wait?
cdi_status check_tc(cdi_unet* u) {
    int e = 0;
    if (cudaMemcpy(&e, u->tc_err, sizeof e, cudaMemcpyDeviceToHost) != cudaSuccess)
        return ufail(u, CDI_ECUDA, "error flag read failed");
    if (e) {
        cudaMemset(u->tc_err, 0, sizeof(int));
        return ufail(u, CDI_ETIMEOUT,
                     e == 1 ? "a tensor-core convolution timed out waiting for its MMAs"
                            : "a tensor-core convolution released tensor memory with an MMA still unconfirmed "
                              "after its waits ran out: treat the device state as unknown");
    }
    return CDI_OK;
}

cdi_status upload_x(cdi_unet* u, const double* x_host) {
    const long N = u->g[0].N;
    if (cudaMemcpyAsync(u->x2, x_host, (size_t)N * 2 * 8, cudaMemcpyHostToDevice, u->stream) != cudaSuccess)
        return ufail(u, CDI_ECUDA, "input upload failed");
    k_input_host<<<blocks(N), 256, 0, u->stream>>>((int)N, u->x2, u->xp, u->x);
    return CDI_OK;
}

}  // namespace

namespace cdi {

template <typename T>
cudaError_t unet_predict_device(cdi_unet* u, const MG& mg, const T* phi_dev, double rho1, double rho2, double h,
                                cudaStream_t s) {
    cudaStream_t keep = u->stream;
    u->stream = s;
    if (!u->weights_ready) refresh_weights(u);
    const long N = u->g[0].N;
    const double rmax = fmax(rho1, rho2);
    k_solver_scales<<<1, 1, 0, s>>>(mg.scal + S_FNORM, (int)N, rmax * h * h, u->sd, u->sf);
    k_input_solver<T><<<blocks(N), 256, 0, s>>>((int)N, ops::fbuf<T>(mg.lv[0]), mg.scalf + SF_FMEAN_HI, phi_dev,
                                                (float)(rho1 - rho2), (float)rho2, (float)(1.0 / rmax), u->sd, u->sf,
                                                u->xp, u->use_tc ? nullptr : u->x);
    forward(u, false, u->y);
    k_output_solver<T><<<blocks(N), 256, 0, s>>>((int)N, u->y, u->sd, u->sf, ops::pbuf<T>(mg.lv[0]));
    g_launches += 3;
    u->stream = keep;
    return cudaGetLastError();
}

void unet_extents(const cdi_unet* u, int* n) {
    n[0] = u->n[0];
    n[1] = u->n[1];
    n[2] = u->n[2];
}

template cudaError_t unet_predict_device<double>(cdi_unet*, const MG&, const double*, double, double, double,
                                                 cudaStream_t);
template cudaError_t unet_predict_device<float>(cdi_unet*, const MG&, const float*, double, double, double,
                                                cudaStream_t);

}  // namespace cdi

extern "C" {

cdi_status cdi_unet_create(cdi_unet** out, int nx, int ny, int nz) {
    if (!out) return ufail(nullptr, CDI_EINVAL, "out is NULL");
    *out = nullptr;
    if (nx < 8 || ny < 8 || nz < 8 || nx % 8 || ny % 8 || nz % 8)
        return ufail(nullptr, CDI_EINVAL, "network extents must be multiples of 8 (three 2x2x2 poolings)");
    if ((long)nx * ny * nz > (1L << 28)) return ufail(nullptr, CDI_EINVAL, "grid too large for the network");
    cdi_unet* u = new (std::nothrow) cdi_unet();
    if (!u) return ufail(nullptr, CDI_EINVAL, "out of host memory");
    u->n[0] = nx;
    u->n[1] = ny;
    u->n[2] = nz;
    for (int l = 0; l < 4; ++l) {
        u->g[l].nx = nx >> l;
        u->g[l].ny = ny >> l;
        u->g[l].nz = nz >> l;
        u->g[l].N = u->g[l].nx * u->g[l].ny * u->g[l].nz;
    }
    size_t total = 0;
    unet_carve(u, nullptr, &total);
    u->ws_bytes = total;
    *out = u;
    return CDI_OK;
}

cdi_status cdi_unet_workspace_bytes(const cdi_unet* u, size_t* bytes) {
    if (!u || !bytes) return ufail(nullptr, CDI_EINVAL, "null argument");
    *bytes = u->ws_bytes;
    return CDI_OK;
}

cdi_status cdi_unet_bind_workspace(cdi_unet* u, void* dev_ptr, size_t bytes, void* stream) {
    if (!u) return ufail(nullptr, CDI_EINVAL, "null network");
    if (!dev_ptr || bytes < u->ws_bytes) return ufail(u, CDI_EINVAL, "workspace missing or too small");
    if (((uintptr_t)dev_ptr) & 255u) return ufail(u, CDI_EINVAL, "workspace must be 256-byte aligned");
    u->ws = (char*)dev_ptr;
    u->stream = (cudaStream_t)stream;
    size_t total = 0;
    unet_carve(u, u->ws, &total);
    if (cudaMemsetAsync(u->ws, 0, u->ws_bytes - 256, u->stream) != cudaSuccess ||
        cudaStreamSynchronize(u->stream) != cudaSuccess)
        return ufail(u, CDI_ECUDA, "workspace clear failed");
    u->adam_t = 0;
    u->weights_ready = false;
    return CDI_OK;
}

cdi_status cdi_unet_param_count(size_t* n) {
    if (!n) return ufail(nullptr, CDI_EINVAL, "null argument");
    *n = param_count();
    return CDI_OK;
}

// flat parameter order: for each layer (e0, e1, e2, b, d2, d1, d0, head) the
// weights [taps][Cout][Cin] then the biases [Cout]
cdi_status cdi_unet_set_params(cdi_unet* u, const double* host, size_t n) {
    if (!u || !u->ws) return ufail(u, CDI_ESTATE, "network workspace not bound");
    if (!host || n != param_count()) return ufail(u, CDI_EINVAL, "parameter array has the wrong length");
    std::vector<float> tmp(host, host + n);
    size_t o = 0;
    for (int l = 0; l < kLayers; ++l) {
        const size_t nw = (size_t)kTaps[l] * kCout[l] * kCin[l];
        cudaMemcpyAsync(u->W[l], tmp.data() + o, nw * 4, cudaMemcpyHostToDevice, u->stream);
        o += nw;
        cudaMemcpyAsync(u->B[l], tmp.data() + o, (size_t)kCout[l] * 4, cudaMemcpyHostToDevice, u->stream);
        o += kCout[l];
        cudaMemsetAsync(u->mW[l], 0, nw * 4, u->stream);
        cudaMemsetAsync(u->vW[l], 0, nw * 4, u->stream);
        cudaMemsetAsync(u->mB[l], 0, (size_t)kCout[l] * 4, u->stream);
        cudaMemsetAsync(u->vB[l], 0, (size_t)kCout[l] * 4, u->stream);
    }
    u->adam_t = 0;
    refresh_weights(u);
    if (cudaStreamSynchronize(u->stream) != cudaSuccess) return ufail(u, CDI_ECUDA, "parameter upload failed");
    return CDI_OK;
}

cdi_status cdi_unet_get_params(cdi_unet* u, double* host, size_t n) {
    if (!u || !u->ws) return ufail(u, CDI_ESTATE, "network workspace not bound");
    if (!host || n != param_count()) return ufail(u, CDI_EINVAL, "parameter array has the wrong length");
    std::vector<float> tmp(n);
    size_t o = 0;
    for (int l = 0; l < kLayers; ++l) {
        const size_t nw = (size_t)kTaps[l] * kCout[l] * kCin[l];
        cudaMemcpyAsync(tmp.data() + o, u->W[l], nw * 4, cudaMemcpyDeviceToHost, u->stream);
        o += nw;
        cudaMemcpyAsync(tmp.data() + o, u->B[l], (size_t)kCout[l] * 4, cudaMemcpyDeviceToHost, u->stream);
        o += kCout[l];
    }
    if (cudaStreamSynchronize(u->stream) != cudaSuccess) return ufail(u, CDI_ECUDA, "parameter download failed");
    for (size_t i = 0; i < n; ++i) host[i] = tmp[i];
    return CDI_OK;
}

// x_host: [N][2] (channels last), y_host: [N]
cdi_status cdi_unet_forward(cdi_unet* u, const double* x_host, double* y_host) {
    if (!u || !u->ws) return ufail(u, CDI_ESTATE, "network workspace not bound");
    if (!x_host || !y_host) return ufail(u, CDI_EINVAL, "null array");
    if (!u->weights_ready) refresh_weights(u);
    cdi_status st = upload_x(u, x_host);
    if (st) return st;
    forward(u, false, u->y);
    const long N = u->g[0].N;
    std::vector<float> y(N);
    if (cudaMemcpyAsync(y.data(), u->y, (size_t)N * 4, cudaMemcpyDeviceToHost, u->stream) != cudaSuccess ||
        cudaStreamSynchronize(u->stream) != cudaSuccess)
        return ufail(u, CDI_ECUDA, std::string("forward: ") + cudaGetErrorString(cudaGetLastError()));
    for (long i = 0; i < N; ++i) y_host[i] = y[i];
    return check_tc(u);
}

// forward pass on device arrays (FP32 [N][2] -> FP32 [N]), stream-ordered, no host copies
cdi_status cdi_unet_forward_device(cdi_unet* u, const float* x_dev, float* y_dev) {
    if (!u || !u->ws) return ufail(u, CDI_ESTATE, "network workspace not bound");
    if (!x_dev || !y_dev) return ufail(u, CDI_EINVAL, "null array");
    if (!u->weights_ready) refresh_weights(u);
    const long N = u->g[0].N;
    if (u->use_tc) k_input_dev<<<blocks(N / 2), 256, 0, u->stream>>>((int)N, x_dev, u->xp);
    else k_input_dev16<<<blocks(N), 256, 0, u->stream>>>((int)N, x_dev, u->xp, u->x);
    forward(u, false, y_dev);
    g_launches += 1;
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return ufail(u, CDI_ECUDA, std::string("forward_device: ") + cudaGetErrorString(e));
    return CDI_OK;
}

// one training step on (x, target): loss before the update; grads (FP32,
// flat parameter order) if grads_host is not NULL; Adam update if lr > 0
cdi_status cdi_unet_train_step(cdi_unet* u, const double* x_host, const double* t_host, double lr, double* loss,
                               double* grads_host) {
    if (!u || !u->ws) return ufail(u, CDI_ESTATE, "network workspace not bound");
    if (!x_host || !t_host) return ufail(u, CDI_EINVAL, "null array");
    if (!(lr >= 0.0) || !std::isfinite(lr)) return ufail(u, CDI_EINVAL, "lr must be >= 0");
    if (!u->weights_ready) refresh_weights(u);
    const long N = u->g[0].N;
    cdi_status st = upload_x(u, x_host);
    if (st) return st;
    std::vector<float> t(t_host, t_host + N);
    cudaMemcpyAsync(u->t, t.data(), (size_t)N * 4, cudaMemcpyHostToDevice, u->stream);
    forward(u, true, u->y);
    backward(u);
    float part = 0.f;
    cudaMemcpyAsync(&part, u->part, 4, cudaMemcpyDeviceToHost, u->stream);
    if (grads_host) {
        std::vector<float> g(param_count());
        size_t o = 0;
        for (int l = 0; l < kLayers; ++l) {
            const size_t nw = (size_t)kTaps[l] * kCout[l] * kCin[l];
            cudaMemcpyAsync(g.data() + o, u->gW[l], nw * 4, cudaMemcpyDeviceToHost, u->stream);
            o += nw;
            cudaMemcpyAsync(g.data() + o, u->gB[l], (size_t)kCout[l] * 4, cudaMemcpyDeviceToHost, u->stream);
            o += kCout[l];
        }
        if (cudaStreamSynchronize(u->stream) != cudaSuccess) return ufail(u, CDI_ECUDA, "gradient download failed");
        for (size_t i = 0; i < g.size(); ++i) grads_host[i] = g[i];
    }
    if (lr > 0.0) adam(u, lr);
    if (cudaStreamSynchronize(u->stream) != cudaSuccess)
        return ufail(u, CDI_ECUDA, std::string("train step: ") + cudaGetErrorString(cudaGetLastError()));
    if (loss) *loss = (double)part / (double)N;
    return check_tc(u);
}

cdi_status cdi_unet_set_conv_kernel(cdi_unet* u, int tensor_core) {
    if (!u) return ufail(nullptr, CDI_EINVAL, "null network");
    if (tensor_core < 0 || tensor_core > 2) return ufail(u, CDI_EINVAL, "tensor_core must be 0, 1 or 2");
    u->use_tc = tensor_core != 0;
    u->wgrad_tc = tensor_core == 1;
    return CDI_OK;
}

const char* cdi_unet_last_error(const cdi_unet* u) { return u ? u->err.c_str() : g_unet_error.c_str(); }

void cdi_unet_destroy(cdi_unet* u) { delete u; }

}  // extern "C"
