// Kernels of the warm-start U-Net (3x3x3 periodic convolutions on voxel grids).
//
// Activations are bfloat16, channels-last [V][C] with a row stride (so a
// tensor can be a channel slice of a concatenation buffer); accumulation is
// FP32.  The convolutions are implicit GEMMs on the tensor cores
// (mma.sync m16n8k16 bf16 -> f32): M = voxels (16 per warp, 64 per block),
// N = output channels (<= 64), K = 27 taps x input channels (16 per step);
// the A fragment of a tap reads the 16 voxels' periodic neighbours.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace gff {
namespace unet {

using bf16 = __nv_bfloat16;

struct Dims {
    int nz, ny, nx;
    long long V;
};

// periodic neighbour of voxel (z, y, x) at offset (dz, dy, dx) of tap t = 9 (dz+1) + 3 (dy+1) + (dx+1)
__device__ __forceinline__ long long neighbour_of(const Dims& d, int z, int y, int x, int t) {
    z += t / 9 - 1;
    y += (t / 3) % 3 - 1;
    x += t % 3 - 1;
    z = z < 0 ? z + d.nz : (z >= d.nz ? z - d.nz : z);
    y = y < 0 ? y + d.ny : (y >= d.ny ? y - d.ny : y);
    x = x < 0 ? x + d.nx : (x >= d.nx ? x - d.nx : x);
    return ((long long)z * d.ny + y) * d.nx + x;
}
__device__ __forceinline__ long long neighbour(const Dims& d, long long v, int t) {
    const long long plane = (long long)d.ny * d.nx;
    const int z = (int)(v / plane);
    const long long rem = v - (long long)z * plane;
    const int y = (int)(rem / d.nx);
    return neighbour_of(d, z, y, (int)(rem - (long long)y * d.nx), t);
}

// negative-side slope of the activation: plain ReLU let whole layers die in training
constexpr float LEAK = 0.125f;

__device__ __forceinline__ void mma_bf16(float* c, const uint32_t* a, const uint32_t* b) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// out[v, co] = act(bias[co] + sum_{t, ci} W[t][co][ci] in[nb(v, t), ci])
// in: cin channels (multiple of 16) at stride sin; W: [27][cout][cin] bf16;
// out: cout channels at stride sout.  RELU: leaky ReLU (slope LEAK for z <= 0).
// A warp takes MW tiles of 16 voxels and NT tiles of 8 output channels (blockIdx.y: which of cout / (8 NT) groups), a
// block four warps = 64 MW voxels.  Each output's sum runs over t and then ci whatever the split, so the bits do not
// depend on it.  Bound: the loads of the weight fragments (two 4-byte loads per tile of 8 channels and k16 step), hence
// MW tiles of voxels per fragment where the grid is large enough to fill the GPU all the same, and the channels split
// over blocks where it is not (launch_conv_nt in unet.cu).
template <int NT, int MW, bool RELU>
__global__ void __launch_bounds__(128) k_conv3(const bf16* __restrict__ in, int sin, int cin,
                                               const bf16* __restrict__ W, int cout, const float* __restrict__ bias,
                                               bf16* __restrict__ out, int sout, Dims d) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, tq = lane & 3;
    const int co0 = blockIdx.y * (NT * 8);
    const long long v0 = ((long long)blockIdx.x * 4 + warp) * (16 * MW);
    if (v0 >= d.V) return;
    // this lane's rows g and g + 8 of every tile (clamped to the first voxel past the end)
    int z[2 * MW], y[2 * MW], x[2 * MW];
#pragma unroll
    for (int m = 0; m < 2 * MW; ++m) {
        const long long v = v0 + 8 * m + g, vc = v < d.V ? v : v0;
        const int plane = d.ny * d.nx;
        z[m] = (int)(vc / plane);
        const int rem = (int)(vc - (long long)z[m] * plane);
        y[m] = rem / d.nx;
        x[m] = rem - y[m] * d.nx;
    }
    float acc[MW][NT][4];
#pragma unroll
    for (int m = 0; m < MW; ++m)
#pragma unroll
        for (int j = 0; j < NT; ++j) acc[m][j][0] = acc[m][j][1] = acc[m][j][2] = acc[m][j][3] = 0.f;
    for (int t = 0; t < 27; ++t) {
        const bf16* r[2 * MW];
#pragma unroll
        for (int m = 0; m < 2 * MW; ++m) r[m] = in + neighbour_of(d, z[m], y[m], x[m], t) * sin + 2 * tq;
        const bf16* wt = W + ((long long)t * cout + co0 + g) * cin + 2 * tq;
        for (int kc = 0; kc < cin; kc += 16) {
            uint32_t a[MW][4];
#pragma unroll
            for (int m = 0; m < MW; ++m) {
                a[m][0] = *reinterpret_cast<const uint32_t*>(r[2 * m] + kc);
                a[m][1] = *reinterpret_cast<const uint32_t*>(r[2 * m + 1] + kc);
                a[m][2] = *reinterpret_cast<const uint32_t*>(r[2 * m] + kc + 8);
                a[m][3] = *reinterpret_cast<const uint32_t*>(r[2 * m + 1] + kc + 8);
            }
#pragma unroll
            for (int j = 0; j < NT; ++j) {
                uint32_t b[2];
                const bf16* wj = wt + (long long)j * 8 * cin + kc;
                b[0] = __ldg(reinterpret_cast<const unsigned int*>(wj));
                b[1] = __ldg(reinterpret_cast<const unsigned int*>(wj + 8));
#pragma unroll
                for (int m = 0; m < MW; ++m) mma_bf16(acc[m][j], a[m], b);
            }
        }
    }
#pragma unroll
    for (int m = 0; m < MW; ++m) {
        const long long va = v0 + 16 * m + g, vb = va + 8;
#pragma unroll
        for (int j = 0; j < NT; ++j) {
            const int co = co0 + j * 8 + 2 * tq;
            const float b0 = bias ? bias[co] : 0.f, b1 = bias ? bias[co + 1] : 0.f;
            float r0 = acc[m][j][0] + b0, r1 = acc[m][j][1] + b1, r2 = acc[m][j][2] + b0, r3 = acc[m][j][3] + b1;
            if (RELU) {
                r0 = r0 > 0.f ? r0 : LEAK * r0;
                r1 = r1 > 0.f ? r1 : LEAK * r1;
                r2 = r2 > 0.f ? r2 : LEAK * r2;
                r3 = r3 > 0.f ? r3 : LEAK * r3;
            }
            if (va < d.V) *reinterpret_cast<__nv_bfloat162*>(out + va * sout + co) = __floats2bfloat162_rn(r0, r1);
            if (vb < d.V) *reinterpret_cast<__nv_bfloat162*>(out + vb * sout + co) = __floats2bfloat162_rn(r2, r3);
        }
    }
}

// dz = da * (act > 0 ? 1 : LEAK), C channels (exact in bfloat16: LEAK is a power of two)
__global__ void k_relu_mask(const bf16* __restrict__ da, int sda, const bf16* __restrict__ act, int sact,
                            bf16* __restrict__ dz, int sdz, int C, long long V) {
    const long long n = V * C;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const long long v = i / C;
        const int c = (int)(i - v * C);
        const float a = __bfloat162float(act[v * sact + c]);
        dz[v * sdz + c] = a > 0.f ? da[v * sda + c] : __float2bfloat16(LEAK * __bfloat162float(da[v * sda + c]));
    }
}

// ---- weight gradients on the tensor cores
//   dW[t][co][ci] += sum_v dz[v, co] in[nb(v, t), ci]
// One GEMM per tap: M = cout, N = cin, K = voxels.  A block takes TG taps and a chunk of
// voxels, walked in tiles of WG_KV = 64: the tile of dz and, per tap, the tile of the
// neighbours' rows arrive by 16-byte asynchronous copies (two buffers), stored [voxel][channel]
// with rows padded by 16 bytes, so that the transposing 8x8 loads (ldmatrix.trans) that turn
// voxels into the K index hit distinct banks.  A warp keeps the dz fragments of one 16-channel
// slice for the whole tile and walks its (tap, 8 input channels) tiles; each tile's four k-steps
// accumulate from zero in the tensor core and are then added to the FP32 sums, so that a sum
// over the chunk rounds like the FP32 additions it replaces.  Chunks are added atomically.
// Bound: shared-memory loads (two 16-byte-row wavefront groups per k16 step and MMA).
// Why: a scalar kernel here did one FMA per two shared-memory loads, 72.6 of the 75.6 ms of GPU
// time of a 64^3 gradient; the fourteen launches of this form take 0.66 ms.
constexpr int WG_KV = 64;
template <int CO, int CI, int TG> constexpr size_t wgrad_smem() {
    return 2 * (size_t)WG_KV * ((CO * 2 + 16) + (size_t)TG * (CI * 2 + 16));
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ void ldm_x4_trans(uint32_t* r, uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}

template <int CO, int CI, int TG>
__global__ void __launch_bounds__(256) k_wgrad(const bf16* __restrict__ in, int sin, const bf16* __restrict__ dz, int sdz,
                                               float* __restrict__ dW, Dims d, long long chunk) {
    constexpr int MT = CO / 16, NT = CI / 8, WM = 8 / MT;  // warps per 16-channel slice of dz
    constexpr int TILES = TG * NT, PER = (TILES + WM - 1) / WM;
    constexpr int RD = CO * 2 + 16, RI = CI * 2 + 16;       // row bytes
    constexpr uint32_t BUF = WG_KV * (RD + TG * RI);
    extern __shared__ __align__(16) unsigned char wsm[];
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(wsm);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int mt = warp % MT, wm = warp / MT;
    const int t0 = blockIdx.x * TG;
    const long long vbeg = (long long)blockIdx.y * chunk;
    const long long vend = min(vbeg + chunk, d.V);
    float acc[PER][4];
#pragma unroll
    for (int i = 0; i < PER; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.f;

    // four threads per voxel row; rows past the end of the chunk are zero-filled
    const int r = tid >> 2, part = tid & 3;
    const int plane = d.ny * d.nx;
    auto load = [&](long long vb, uint32_t buf) {
        const bool ok = vb + r < vend;
        const long long v = ok ? vb + r : vbeg;
        const int z = (int)(v / plane), rem = (int)(v - (long long)z * plane);
        const int y = rem / d.nx, x = rem - y * d.nx;
        for (int q = part; q < CO / 8; q += 4) cp_async16(buf + r * RD + q * 16, dz + v * sdz + 8 * q, ok);
#pragma unroll
        for (int c = part; c < TG * (CI / 8); c += 4) {
            const int t = c / (CI / 8), q = c - t * (CI / 8);
            cp_async16(buf + WG_KV * RD + (t * WG_KV + r) * RI + q * 16,
                       in + neighbour_of(d, z, y, x, t0 + t) * sin + 8 * q, ok);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };

    int cur = 0;
    if (vbeg < vend) load(vbeg, sbase);
    for (long long vb = vbeg; vb < vend; vb += WG_KV) {
        if (vb + WG_KV < vend) {
            load(vb + WG_KV, sbase + (cur ^ 1) * BUF);
            asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        }
        __syncthreads();
        const uint32_t sd = sbase + cur * BUF, si = sd + WG_KV * RD;
        // dz fragments of the four k-steps: 8x8 blocks (k, m), (k, m + 8), (k + 8, m), (k + 8, m + 8)
        uint32_t a[4][4];
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)
            ldm_x4_trans(a[ks], sd + (16 * ks + (lane & 7) + ((lane >> 4) & 1) * 8) * RD + (16 * mt + ((lane >> 3) & 1) * 8) * 2);
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int tile = wm + i * WM;
            if (PER * WM != TILES && tile >= TILES) break;  // warp-uniform
            const int t = tile / NT, nt = tile - t * NT;
            const uint32_t st = si + (t * WG_KV + lane) * RI + nt * 16;  // lane = row k of blocks k, k + 8, k + 16, k + 24
            uint32_t b0[4], b1[4];
            ldm_x4_trans(b0, st);
            ldm_x4_trans(b1, st + 32 * RI);
            float s[4] = {0.f, 0.f, 0.f, 0.f};
            mma_bf16(s, a[0], b0);
            mma_bf16(s, a[1], b0 + 2);
            mma_bf16(s, a[2], b1);
            mma_bf16(s, a[3], b1 + 2);
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[i][k] += s[k];
        }
        __syncthreads();
        cur ^= 1;
    }
    const int g = lane >> 2, tq = lane & 3;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int tile = wm + i * WM;
        if (PER * WM != TILES && tile >= TILES) break;
        const int t = tile / NT, nt = tile - t * NT;
        float* o = dW + ((long long)(t0 + t) * CO + 16 * mt + g) * CI + 8 * nt + 2 * tq;
        atomicAdd(o, acc[i][0]);
        atomicAdd(o + 1, acc[i][1]);
        atomicAdd(o + 8 * CI, acc[i][2]);
        atomicAdd(o + 8 * CI + 1, acc[i][3]);
    }
}

// db[c] += sum_v dz[v, c]
__global__ void __launch_bounds__(256) k_bias_grad(const bf16* __restrict__ dz, int sdz, int C, long long V,
                                                   float* __restrict__ db) {
    __shared__ float part[64];
    if (threadIdx.x < 64) part[threadIdx.x] = 0.f;
    __syncthreads();
    const int c = threadIdx.x % C;
    const int rows_per = blockDim.x / C;
    float s = 0.f;
    if (threadIdx.x < rows_per * C)
        for (long long v = (long long)blockIdx.x * rows_per + threadIdx.x / C; v < V; v += (long long)gridDim.x * rows_per)
            s += __bfloat162float(dz[v * sdz + c]);
    if (threadIdx.x < rows_per * C) atomicAdd(part + c, s);
    __syncthreads();
    if (threadIdx.x < C) atomicAdd(db + threadIdx.x, part[threadIdx.x]);
}

// 2x2x2 average pooling: out (coarse dims dc) from in (fine)
__global__ void k_pool(const bf16* __restrict__ in, int sin, bf16* __restrict__ out, int sout, int C, Dims dc) {
    const long long n = dc.V * C;
    const int fx = 2 * dc.nx, fy = 2 * dc.ny;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const long long v = i / C;
        const int c = (int)(i - v * C);
        const int z = (int)(v / ((long long)dc.ny * dc.nx)), y = (int)((v / dc.nx) % dc.ny), x = (int)(v % dc.nx);
        float s = 0.f;
        for (int a = 0; a < 2; ++a)
            for (int b = 0; b < 2; ++b)
                for (int e = 0; e < 2; ++e)
                    s += __bfloat162float(in[(((long long)(2 * z + a) * fy + 2 * y + b) * fx + 2 * x + e) * sin + c]);
        out[v * sout + c] = __float2bfloat16(s * 0.125f);
    }
}

// out[child] = in[parent] (fine dims df)
__global__ void k_up(const bf16* __restrict__ in, int sin, bf16* __restrict__ out, int sout, int C, Dims df) {
    const long long n = df.V * C;
    const int cy = df.ny / 2, cx = df.nx / 2;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const long long v = i / C;
        const int c = (int)(i - v * C);
        const int z = (int)(v / ((long long)df.ny * df.nx)), y = (int)((v / df.nx) % df.ny), x = (int)(v % df.nx);
        out[v * sout + c] = in[(((long long)(z / 2) * cy + y / 2) * cx + x / 2) * sin + c];
    }
}

// gradient of nearest upsampling: din[parent] = sum of the 8 children (coarse dims dc)
__global__ void k_up_grad(const bf16* __restrict__ dout, int sdo, bf16* __restrict__ din, int sdi, int C, Dims dc) {
    const long long n = dc.V * C;
    const int fx = 2 * dc.nx, fy = 2 * dc.ny;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const long long v = i / C;
        const int c = (int)(i - v * C);
        const int z = (int)(v / ((long long)dc.ny * dc.nx)), y = (int)((v / dc.nx) % dc.ny), x = (int)(v % dc.nx);
        float s = 0.f;
        for (int a = 0; a < 2; ++a)
            for (int b = 0; b < 2; ++b)
                for (int e = 0; e < 2; ++e)
                    s += __bfloat162float(dout[(((long long)(2 * z + a) * fy + 2 * y + b) * fx + 2 * x + e) * sdo + c]);
        din[v * sdi + c] = __float2bfloat16(s);
    }
}

// out[child] = skip[child] + dpool[parent] / 8   (fine dims df)
__global__ void k_pool_grad_add(const bf16* __restrict__ skip, int ssk, const bf16* __restrict__ dp, int sdp,
                                bf16* __restrict__ out, int sout, int C, Dims df) {
    const long long n = df.V * C;
    const int cy = df.ny / 2, cx = df.nx / 2;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const long long v = i / C;
        const int c = (int)(i - v * C);
        const int z = (int)(v / ((long long)df.ny * df.nx)), y = (int)((v / df.nx) % df.ny), x = (int)(v % df.nx);
        const float s = __bfloat162float(skip[v * ssk + c]) +
                        0.125f * __bfloat162float(dp[(((long long)(z / 2) * cy + y / 2) * cx + x / 2) * sdp + c]);
        out[v * sout + c] = __float2bfloat16(s);
    }
}

// 1x1 head: y[v][o] = b[o] + sum_i Wr[o][i] a[v][i]   (Wr: bfloat16-rounded weights held in FP32)
__global__ void k_head_fwd(const bf16* __restrict__ a, int sa, const float* __restrict__ Wr, const float* __restrict__ b,
                           float* __restrict__ y, int cin, int cout, long long V) {
    for (long long v = (long long)blockIdx.x * blockDim.x + threadIdx.x; v < V; v += (long long)gridDim.x * blockDim.x) {
        float xi[16];
        for (int i = 0; i < cin; ++i) xi[i] = __bfloat162float(a[v * sa + i]);
        for (int o = 0; o < cout; ++o) {
            float s = b[o];
            for (int i = 0; i < cin; ++i) s = fmaf(Wr[o * cin + i], xi[i], s);
            y[v * cout + o] = s;
        }
    }
}

// head backward: da[v][i] = bf16(sum_o Wr[o][i] dy[v][o]); dW[o][i] += sum_v dy[v][o] a[v][i]; db[o] += sum_v dy[v][o]
// A block walks tiles of 256 voxels: each thread loads and back-propagates one voxel (32 and 36 contiguous
// bytes) and leaves a and dy in shared memory; then thread t < CO CI + CO keeps one weight's or bias's sum over the
// tile in a register.  One atomic addition per sum and block: with one voxel per thread and shared-memory
// atomics for all 153 sums of every voxel a 64^3 call took 816 us.
template <int CI, int CO>
__global__ void __launch_bounds__(256) k_head_bwd(const bf16* __restrict__ a, int sa, const float* __restrict__ Wr,
                                                  const float* __restrict__ dy, bf16* __restrict__ da, int sda,
                                                  float* __restrict__ dW, float* __restrict__ db, long long V) {
    static_assert(CI % 8 == 0 && CO * CI + CO <= 256, "one thread per sum");
    __shared__ float sx[256][CI + 1], sg[256][CO];  // odd strides: a thread's row and a column of rows hit distinct banks
    __shared__ float sw[CO * CI];
    const int tid = threadIdx.x;
    for (int e = tid; e < CO * CI; e += 256) sw[e] = Wr[e];
    const int o = tid < CO * CI ? tid / CI : tid - CO * CI, i = tid < CO * CI ? tid % CI : CI;  // i = CI: the bias
    float acc = 0.f;
    for (long long v0 = (long long)blockIdx.x * 256; v0 < V; v0 += (long long)gridDim.x * 256) {
        const int nv = (int)min(256LL, V - v0);
        __syncthreads();  // the previous tile's readers are done (and sw is loaded)
        if (tid < nv) {
            const long long v = v0 + tid;
            float g[CO];
#pragma unroll
            for (int k = 0; k < CO; ++k) sg[tid][k] = g[k] = dy[v * CO + k];
#pragma unroll
            for (int q = 0; q < CI / 8; ++q) {
                const uint4 raw = *reinterpret_cast<const uint4*>(a + v * sa + 8 * q);
                const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&raw);
                uint4 outv;
                __nv_bfloat162* d2 = reinterpret_cast<__nv_bfloat162*>(&outv);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int c = 8 * q + 2 * e;
                    sx[tid][c] = __low2float(h[e]);
                    sx[tid][c + 1] = __high2float(h[e]);
                    float s0 = 0.f, s1 = 0.f;
#pragma unroll
                    for (int k = 0; k < CO; ++k) {
                        s0 = fmaf(sw[k * CI + c], g[k], s0);
                        s1 = fmaf(sw[k * CI + c + 1], g[k], s1);
                    }
                    d2[e] = __floats2bfloat162_rn(s0, s1);
                }
                *reinterpret_cast<uint4*>(da + v * sda + 8 * q) = outv;
            }
            sx[tid][CI] = 1.f;
        }
        __syncthreads();
        if (tid < CO * CI + CO)
            for (int r = 0; r < nv; ++r) acc = fmaf(sg[r][o], sx[r][i], acc);
    }
    if (tid < CO * CI)
        atomicAdd(dW + tid, acc);
    else if (tid < CO * CI + CO)
        atomicAdd(db + o, acc);
}

// y = bfloat16(x), n a multiple of 4 (host arrays arrive as FP32 and are rounded here: the same rounding on one host
// thread took 4 ms for the inputs of a 64^3 grid)
__global__ void __launch_bounds__(256) k_to_bf16(const float* __restrict__ x, bf16* __restrict__ y, long long n) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n / 4; i += (long long)gridDim.x * blockDim.x) {
        const float4 v = reinterpret_cast<const float4*>(x)[i];
        __nv_bfloat162 p[2] = {__floats2bfloat162_rn(v.x, v.y), __floats2bfloat162_rn(v.z, v.w)};
        reinterpret_cast<uint2*>(y)[i] = *reinterpret_cast<const uint2*>(p);
    }
}

// mean squared error: dy = 2 (y - t) / n, loss += sum (y - t)^2 / n
__global__ void __launch_bounds__(256) k_mse(const float* __restrict__ y, const float* __restrict__ t, float* __restrict__ dy,
                                             long long n, double* __restrict__ loss) {
    __shared__ double part[8];
    double s = 0.0;
    const double inv = 1.0 / (double)n;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float d = y[i] - t[i];
        dy[i] = (float)(2.0 * d * inv);
        s += (double)d * d;
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += part[w];
        atomicAdd(loss, tot * inv);
    }
}

// out += sum_i g[i]^2
__global__ void __launch_bounds__(256) k_sumsq(const float* __restrict__ g, long long n, double* __restrict__ out) {
    __shared__ double part[8];
    double s = 0.0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        s += (double)g[i] * g[i];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += part[w];
        atomicAdd(out, tot);
    }
}

// Adam on the flat parameter vector (FP32 master weights); the gradient is
// scaled down to global norm `clip` when sqrt(*gn2) exceeds it
__global__ void k_adam(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                       long long n, float lr, float b1, float b2, float eps, float c1, float c2,
                       const double* __restrict__ gn2, float clip) {
    const double gn = sqrt(*gn2);
    const float sc = gn > clip ? (float)(clip / gn) : 1.f;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const float gi = sc * g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

// bfloat16 copies of one conv layer: forward [27][co][ci] and data-gradient [27][ci][co] with flipped taps
__global__ void k_refresh(const float* __restrict__ w, bf16* __restrict__ wf, bf16* __restrict__ wd, int cout, int cin) {
    const long long n = 27LL * cout * cin;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
        const int t = (int)(e / ((long long)cout * cin));
        const int rem = (int)(e - (long long)t * cout * cin);
        const int o = rem / cin, i = rem - o * cin;
        const bf16 r = __float2bfloat16(w[e]);
        wf[e] = r;
        wd[((long long)(26 - t) * cin + i) * cout + o] = r;
    }
}

__global__ void k_round_f32(const float* __restrict__ w, float* __restrict__ wr, int n) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x)
        wr[e] = __bfloat162float(__float2bfloat16(w[e]));
}

}  // namespace unet
}  // namespace gff
