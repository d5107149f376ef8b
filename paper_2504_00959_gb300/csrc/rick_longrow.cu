// rick_longrow.cu -- the row transforms of the split transform for n = 8192 and
// 16384 (step 3 of the workflow, Sec. 2.1), in place, over what is not empty:
// imaging reads only the tiles with entries (the gridder leaves the others
// unwritten) of the rows in the plane's range of non-empty tile rows; the
// adjoint writes only the tiles that the measurements' footprints touch.  The
// column factor (k_colfft) takes rows outside the range as zeros and leaves
// them out.
//
// One row per block (64 or 128 KB of shared memory), n / 16 threads with 16
// values each: n = 16 x 16 x 16 x q, q = n / 4096.  With x = j + (n / 16) a, j
// = t2 + r b (r = n / 256), t2 = s + q c and output k1 + 16 k2 + 256 k3 + 4096 k4:
//   pass 1  DFT over a, times w_n^(j k1);         block k1, element j
//   pass 2  DFT over b, times w_(n/16)^(t2 k2);   element r k2 + t2
//   pass 3  DFT over c, times w_r^(s k3);         element r k2 + q k3 + s
//   pass 4  DFT over s (2 or 4 points): 16 adjacent columns per half warp.
// Blocks k1 lie at an odd pitch, and pass 3's half warps take q values of s and
// every q-th block: all four passes read and write without bank conflicts.
#include <algorithm>
#include <atomic>

#include "rick_dft.cuh"
#include "rick_internal.cuh"

namespace rick {
namespace {

template <int N>
struct LongShape {
    static constexpr int kPer = N / 16, r = N / 256, q = N / 4096, P = kPer + 1;
    static constexpr size_t kSmem = 16 * (size_t)P * sizeof(float2);
};

__device__ __forceinline__ cpx ld_c(const float2* p)
{
    return cpx{f2{*reinterpret_cast<const unsigned long long*>(p)}};
}
__device__ __forceinline__ void st_c(float2* p, cpx x) { *reinterpret_cast<unsigned long long*>(p) = x.v.v; }

// grid (blocks per plane, planes); DIR +1 imaging, -1 adjoint.  A block takes
// every gridDim.x-th row of the plane's range; the next row's loads are in
// flight during the last pass.
// Bound: 16 planes of 16384^2 (2.5e7 measurements of an Earth-rotation track)
// take 13.6 ms, cuFFT's rows of everything 18.3; 9.4 us per row of a plane whose
// tiles are nearly all full (cuFFT: 10.6), of which ~4 are issue slots and ~5.5
// shared-memory passes that one block of 32 warps per SM (its shared memory and
// registers are full) does not overlap with the row's 256 KB of memory traffic.
// Loading the next row after the last pass instead of before it: 16.4 ms.
template <int N, int DIR>
__global__ void __launch_bounds__(N / 16, N >= 16384 ? 1 : 2)
    k_longrows(const float2* __restrict__ tw1, const float2* __restrict__ tw2, const float2* __restrict__ tw3,
               const uint32_t* __restrict__ bits, const int2* __restrict__ range, int k0, int wpr, int log2T,
               int row_perm, float2* __restrict__ planes)
{
    using Sh = LongShape<N>;
    constexpr int kPer = Sh::kPer, r = Sh::r, Q = Sh::q, P = Sh::P;
    extern __shared__ float2 long_smem[];
    const int plane = blockIdx.y, k = k0 + plane;
    // the thread index anew in every pass: addresses kept across passes cost spills
    auto tid = [] {
        int x = threadIdx.x;
        asm volatile("" : "+r"(x));
        return x;
    };
    const int2 rg = __ldg(range + k);
    const int v1 = rg.y << log2T;
    int v = (rg.x << log2T) + (int)blockIdx.x;
    if (v >= v1) return;
    float2* base = planes + (size_t)plane * N * N;
    const uint32_t* tb = bits + (size_t)k * (N >> log2T) * wpr;
    auto row_at = [&](int g) {  // memory row of grid row g (GridCfg::row_perm)
        return base + (size_t)(row_perm ? ((g & 15) << row_perm) | (g >> 4) : g) * N;
    };
    auto tile = [&](int g, int col) {
        const int tu = col >> log2T;
        return (__ldg(tb + (g >> log2T) * wpr + (tu >> 5)) >> (tu & 31)) & 1u;
    };
    // bit o of a thread's mask: whether the tile of column col(o) of its half
    // warp is wanted (16 adjacent columns lie in one tile); lane o looks up o
    auto mask = [&](int g, int col) {
        return (__ballot_sync(0xffffffffu, tile(g, col)) >> (threadIdx.x & 16)) & 0xffffu;
    };
    cpx x[16];
    auto load = [&](int g) {
        const int t = tid();
        const float2* src = row_at(g) + t;
        const uint32_t want = DIR > 0 ? mask(g, (t & ~15) + (t & 15) * kPer) : 0xffffu;
#pragma unroll
        for (int a = 0; a < 16; ++a) {
            x[a] = cpx_make(0.f, 0.f);
            if ((want >> a) & 1u) {
                const float2 z = __ldcs(src + a * kPer);
                x[a] = cpx_make(z.x, z.y);
            }
        }
    };
    load(v);
    for (; v < v1; v += gridDim.x) {
        {
            const int t = tid();
            dft16<DIR>(x);
            st_c(long_smem + t, x[0]);
#pragma unroll
            for (int k1 = 1; k1 < 16; ++k1) {
                float2 w = __ldg(tw1 + (k1 - 1) * kPer + t);
                if (DIR < 0) w.y = -w.y;
                st_c(long_smem + k1 * P + t, c_mul(x[k1], w));
            }
        }
        __syncthreads();
        {
            const int t = tid(), t2 = t % r;
            float2* blk = long_smem + (t / r) * P + t2;
#pragma unroll
            for (int b = 0; b < 16; ++b) x[b] = ld_c(blk + r * b);
            dft16<DIR>(x);
            st_c(blk, x[0]);
#pragma unroll
            for (int k2 = 1; k2 < 16; ++k2) {
                float2 w = __ldg(tw2 + (k2 - 1) * r + t2);
                if (DIR < 0) w.y = -w.y;
                st_c(blk + r * k2, c_mul(x[k2], w));
            }
        }
        __syncthreads();
        {
            // lanes: s | blocks Q apart | the block's remainder; then k2
            const int t = tid(), s = t % Q, k1 = Q * ((t / Q) % (16 / Q)) + (t / 16) % Q, k2 = t / (16 * Q);
            float2* blk = long_smem + k1 * P + k2 * r + s;
#pragma unroll
            for (int c = 0; c < 16; ++c) x[c] = ld_c(blk + Q * c);
            dft16<DIR>(x);
            st_c(blk, x[0]);
#pragma unroll
            for (int k3 = 1; k3 < 16; ++k3) {
                float2 w = __ldg(tw3 + (k3 - 1) * Q + s);
                if (DIR < 0) w.y = -w.y;
                st_c(blk + Q * k3, c_mul(x[k3], w));
            }
        }
        __syncthreads();
        float2* dst = row_at(v);
        const int g = v;
        if (v + (int)gridDim.x < v1) load(v + gridDim.x);
        {
            const int t = tid(), k1 = t & 15, k2 = (t >> 4) & 15, k30 = t >> 8;  // k30 < Q
            const float2* blk = long_smem + k1 * P + k2 * r;
            const uint32_t want =
                DIR > 0 ? 0xffffu : mask(g, 16 * k2 + 256 * (k30 + Q * (k1 / Q)) + 4096 * (k1 % Q));  // o = Q i + k4
#pragma unroll 1  // the next row's values take the registers
            for (int i = 0; i < 16 / Q; ++i) {
                const int k3 = k30 + Q * i;
                cpx y[Q];
#pragma unroll
                for (int s = 0; s < Q; ++s) y[s] = ld_c(blk + Q * k3 + s);
                dft_small<Q, DIR>(y);
#pragma unroll
                for (int k4 = 0; k4 < Q; ++k4) {
                    const int col = k1 + 16 * k2 + 256 * k3 + 4096 * k4;
                    if ((want >> (Q * i + k4)) & 1u) st_c(dst + col, y[k4]);
                }
            }
        }
        __syncthreads();  // the next row overwrites the shared memory
    }
}

template <int N, int DIR>
cudaError_t launch_long_n(const StripArgs& s, int k0, int nk, int row_perm, float2* planes, cudaStream_t st)
{
    // SMs of a device, once its shared-memory opt-in is done (handles on several
    // threads: written after both, read before either is relied on)
    static std::atomic<int> ready[64];
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool known = dev >= 0 && dev < 64;
    if (known) sms = ready[dev].load(std::memory_order_acquire);
    if (!sms) {
        e = cudaFuncSetAttribute(k_longrows<N, DIR>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)LongShape<N>::kSmem);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        if (known) ready[dev].store(sms, std::memory_order_release);
    }
    const dim3 grid((unsigned)(sms * (N >= 16384 ? 1 : 2)), (unsigned)nk);
    const float2* tw3 = s.tw2 + 15 * LongShape<N>::r;
    k_longrows<N, DIR><<<grid, N / 16, LongShape<N>::kSmem, st>>>(s.tw1, s.tw2, tw3, s.bits, s.range, k0, s.wpr, s.log2T,
                                                                 row_perm, planes);
    return cudaGetLastError();
}

}  // namespace

bool longrow_shape(int n) { return n == 8192 || n == 16384; }

cudaError_t launch_longrows(int n, int dir, const StripArgs& s, int k0, int nk, int row_perm, float2* planes,
                            cudaStream_t st)
{
    if (nk <= 0) return cudaSuccess;
    if (nk > 65535) return cudaErrorInvalidValue;
    if (n == 8192)
        return dir > 0 ? launch_long_n<8192, 1>(s, k0, nk, row_perm, planes, st)
                       : launch_long_n<8192, -1>(s, k0, nk, row_perm, planes, st);
    if (n == 16384)
        return dir > 0 ? launch_long_n<16384, 1>(s, k0, nk, row_perm, planes, st)
                       : launch_long_n<16384, -1>(s, k0, nk, row_perm, planes, st);
    return cudaErrorInvalidValue;
}

}  // namespace rick
