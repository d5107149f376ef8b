// rick_strip.cu -- step 3 and 4 of the workflow (Sec. 2.1: the 2D FFT of every
// w-plane, the w-term screen and the sum over planes, Eq. 1) in two passes
// over the planes, and their adjoint, for n = 1024, 2048 and 4096.
//
// The uv coverage leaves most of a plane empty (an Earth-rotation synthesis
// touches about a quarter of the 32 x 32 tiles of a plane, in about two thirds
// of its tile rows), so the passes move only what is there:
//   k_occupancy  one bit per tile of every plane (the tile lists any entry)
//                and the range of each plane's non-empty tile rows;
//   k_rows       the row transforms of the rows in that range: reads the
//                non-empty tiles only (the gridder does not write the others)
//                and writes the transformed rows in strip order: plane, strip
//                of two adjacent columns, row, the two values, so that a
//                strip's rows are one contiguous run of 16 bytes per row;
//   k_colimage   for each strip: per plane one bulk copy of the run of
//                transformed rows into shared memory, the n-point column
//                transform, the w-screen and the sum over planes in registers,
//                and the finished pixels: the planes are read once here and
//                never written back.
// The adjoint runs the mirror image: k_colspread (screened pixels -> column
// transforms -> the rows of the range, strip order) and k_rows (-> the tiles
// that the measurements' footprints touch, natural order, for the gather).
//
// The n = 256 r-point transforms (r = 4, 8, 16) are 16 x 16 x r: with rows
// v = j + (n / 16) a and j = t2 + r b, outputs y = k1 + 16 k2 + 256 k3,
//   pass 1  DFT over a (16 points), times w_n^(j k1);
//   pass 2  within block k1: DFT over b (16 points), times w_(n/16)^(t2 k2);
//   pass 3  DFT over t2 (r points), output k3;
// the DFT matrix is symmetric, so the same passes in reverse order (3, 2, 1)
// also transform y to v, which k_colspread uses.
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "rick_dft.cuh"
#include "rick_internal.cuh"
#include "rick_screen.cuh"
#include "rick_tma.cuh"

#include <cudaTypedefs.h>

namespace rick {
namespace {

int sm_count_strip()
{
    static std::atomic<int> cached[64];
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    const bool known = dev >= 0 && dev < 64;
    if (known && (v = cached[dev].load(std::memory_order_relaxed)) > 0) return v;
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    v = v > 0 ? v : 1;
    if (known) cached[dev].store(v, std::memory_order_relaxed);
    return v;
}

// ------------------------------------------------------------- occupancy

constexpr int kOccThreads = 1024;
constexpr int kOccBatch = 8;
constexpr int kOccWords = kOccThreads / 32 * kOccBatch;

// grid (parts, planes): the plane's tile bits (wpr words per tile row) and its
// range of non-empty tile rows [lo, hi).  A block takes kOccWords words, all of a
// plane up to n = 2048 with tiles of 32; of several blocks the last to finish
// writes the range, from maxima in `occ` (which it leaves zero again).  With one
// block per plane, planes of 4096^2, 8192^2 and 16384^2 took 12, 34 and 118 us (16,
// 49 and 185 in the adjoint); now 9 (11) each, the offsets' latency.  Lists: a tile is non-empty when any
// of them has entries there.  Adjoint (reach > 0, one list, sorted by the tile
// of the first footprint cell on the first plane of the w-footprint): a tile
// of plane k is needed when it or its left, upper or upper left neighbour
// holds a measurement of the planes k - reach + 1 .. k.
__global__ void __launch_bounds__(kOccThreads) k_occupancy(GridCfg c, ChunkList ch, int reach, int wpr,
                                                           uint32_t* __restrict__ bits, int2* __restrict__ range,
                                                           int4* __restrict__ occ)
{
    __shared__ int s_lo, s_hi;
    const int k = blockIdx.y, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        s_lo = c.ntu;
        s_hi = 0;
    }
    __syncthreads();
    const int words = c.ntu * wpr;
    int lo = c.ntu, hi = 0;
    // kOccBatch words per warp: their first list's offsets are in flight together
    constexpr int kWarps = kOccThreads / 32;
    {
        const int i0 = blockIdx.x * kOccWords + wid;
        uint32_t o0[kOccBatch], o1[kOccBatch];
#pragma unroll
        for (int b = 0; b < kOccBatch; ++b) {
            const int i = i0 + b * kWarps, tv = i / wpr, tu = (i - tv * wpr) * 32 + lane;
            o0[b] = o1[b] = 0;
            if (i < words && tu < c.ntu && ch.count > 0) {
                const uint32_t* off = ch.off[0] + (int64_t)k * c.ntp + (int64_t)tv * c.ntu;
                o0[b] = __ldg(off + (reach && tu > 0 ? tu - 1 : tu));
                o1[b] = __ldg(off + tu + 1);
            }
        }
#pragma unroll
        for (int b = 0; b < kOccBatch; ++b) {
            const int i = i0 + b * kWarps, tv = i / wpr, tu = (i - tv * wpr) * 32 + lane;
            if (i >= words) break;
            bool any = false;
            if (tu < c.ntu) {
                const int64_t t = (int64_t)k * c.ntp + (int64_t)tv * c.ntu + tu;
                any = ch.count < 0 || o0[b] != o1[b];  // count < 0: every tile
                for (int q = 1; q < ch.count; ++q) any |= __ldg(ch.off[q] + t + 1) != __ldg(ch.off[q] + t);
                if (reach) {
                    const int k0 = k - reach + 1 > 0 ? k - reach + 1 : 0, l = tu > 0 ? 1 : 0;
                    for (int kk = k0; kk <= k; ++kk) {
                        const uint32_t* off = ch.off[0] + (int64_t)kk * c.ntp + (int64_t)tv * c.ntu + tu;
                        if (kk < k) any |= __ldg(off + 1) != __ldg(off - l);
                        if (tv > 0) any |= __ldg(off - c.ntu + 1) != __ldg(off - c.ntu - l);
                    }
                }
            }
            const uint32_t m = __ballot_sync(0xffffffffu, any);
            if (lane == 0) bits[(int64_t)k * words + i] = m;
            if (m) {
                lo = min(lo, tv);
                hi = max(hi, tv + 1);
            }
        }
    }
    if (lane == 0) {
        atomicMin(&s_lo, lo);
        atomicMax(&s_hi, hi);
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    if (gridDim.x == 1) {
        range[k] = s_hi > s_lo ? make_int2(s_lo, s_hi) : make_int2(0, 0);
        return;
    }
    int* o = reinterpret_cast<int*>(occ + k);  // tile rows from lo on, hi, blocks that are done
    if (s_hi > s_lo) {
        atomicMax(o, c.ntu - s_lo);
        atomicMax(o + 1, s_hi);
    }
    __threadfence();
    if (atomicAdd(o + 2, 1) == (int)gridDim.x - 1) {
        __threadfence();
        const int from = atomicExch(o, 0), to = atomicExch(o + 1, 0);
        atomicExch(o + 2, 0);
        range[k] = to > 0 ? make_int2(c.ntu - from, to) : make_int2(0, 0);
    }
}

// ------------------------------------------------------------------- rows

constexpr unsigned long long kStripWaitNs = 1000000000ull;  // bound of one wait: 1 s
__device__ __forceinline__ cpx lds_c(const float2* p)
{
    return cpx{f2{*reinterpret_cast<const unsigned long long*>(p)}};
}
__device__ __forceinline__ void sts_c(float2* p, cpx x) { *reinterpret_cast<unsigned long long*>(p) = x.v.v; }

constexpr int kRowThreads = 512;

// Shared memory of k_rows: R = 8192 / N rows of 16 blocks k1 of N / 16 values
// at an odd pitch, the rows 16 / R (mod 16) values apart.  In pass 3 of the
// forward direction a half warp holds R rows of 16 / R adjacent blocks: with
// these pitches its elements fall in 16 different bank pairs.
template <int N>
struct RowShape {
    static constexpr int r = N / 256, kPer = N / 16, R = 8192 / N, P = kPer + 1;
    static constexpr int kRowPitch = N + 16 + 16 / R;
};

// The row transforms of R rows at a time (64 KB of shared memory, two blocks
// per SM; grid (blocks per plane, planes)).  DIR +1: natural rows
// (non-empty tiles) -> strips; -1: strips -> natural rows (needed tiles).  The
// strips' side moves by TMA, from and to a [strip][row][2] image of the rows
// in shared memory (map: the strip buffer as [strips][2 n] values, boxes of 2 R
// values x 256 strips): each 16 R-byte piece would cost a store or load
// instruction of the SM one pass of its own (direct stores: 1.24 instead of
// 1.09 ms for 32 planes of 4096^2, 1.72 instead of 1.13 for 128 of 2048^2).  The
// next rows' loads are in flight while the image is written out (+1) or the
// last pass runs (-1).  A
// warp's 32 lanes are 16 adjacent columns of 2 rows (natural rows: 128
// contiguous bytes per half warp), or pairs of adjacent columns of all R rows
// (16 R contiguous bytes of the image each).
// Bound: 32 planes of 4096^2 (0.26 of the tiles, 0.68 of the rows: 4.0 GB) take
// 1.10 ms, 3.6 TB/s; the passes alone, without loads and stores, 0.71 ms of
// issue and shared-memory time at 16 warps per block and two blocks per SM
// (registers), which the loads and stores overlap in part.  cuFFT's rows of all
// tiles and rows took 1.37 ms.
template <int N, bool STRIP>
__device__ __forceinline__ void row_lane(int t, int& row, int& low, int& g)
{
    constexpr int R = RowShape<N>::R;
    const int lane = t & 31, w = t >> 5;
    if (STRIP) {
        // lane bits: column parity | row | next columns; 32 / R columns per warp
        row = (lane >> 1) % R;
        const int q = (lane & 1) + 2 * ((lane >> 1) / R) + (32 / R) * w;
        low = q & 15;
        g = q >> 4;
    } else {
        low = lane & 15;
        row = (lane >> 4) + 2 * (w % (R / 2));
        g = w / (R / 2);
    }
}

constexpr int kRowBox = 256;  // strips per TMA box

template <int N, int DIR, int LOG2T>
__global__ void __launch_bounds__(kRowThreads, 2) k_rows(const __grid_constant__ CUtensorMap map,
                                                         const float2* __restrict__ tw1,
                                                         const float2* __restrict__ tw2,
                                                         const uint32_t* __restrict__ bits,
                                                         const int2* __restrict__ range, int k0,
                                                         float2* __restrict__ planes, unsigned long long wait_ns,
                                                         unsigned long long* __restrict__ err)
{
    using Sh = RowShape<N>;
    constexpr int r = Sh::r, kPer = Sh::kPer, R = Sh::R, P = Sh::P;
    constexpr int kTiles = N >> LOG2T, kWords = (kTiles + 31) / 32;  // tiles and words of tile bits per tile row
    extern __shared__ __align__(128) unsigned char row_smem[];
    __shared__ __align__(8) unsigned long long bar;
    __shared__ int s_abort;
    float2* sm = reinterpret_cast<float2*>(row_smem);
    const int plane = blockIdx.y, k = k0 + plane;
    const int2 rg = __ldg(range + k);
    // this block's rows: every gridDim.x-th group of R of the range, so that
    // the blocks in flight write (read) neighbouring rows of the strips: with a
    // run of rows per block the 32-byte pieces of a DRAM access came at
    // different times and cost it twice (757 -> 1450 MB written for 8 planes)
    const int stride = (int)gridDim.x * R, v1 = rg.y << LOG2T;
    int v0 = (rg.x << LOG2T) + (int)blockIdx.x * R;
    if (v0 >= v1) return;
    const int t = threadIdx.x;
    float2* nat = planes + (size_t)plane * N * N;
    const uint32_t* tb = bits + (size_t)k * kTiles * kWords;
    const unsigned long long limit = wait_ns ? wait_ns : kStripWaitNs;

    // the lane maps are evaluated where they are used: kept, they cost spills
    struct Lane {
        int row, low, g;
    };
    auto lane_map = [&](auto strip) {
        int tt = t;
        asm volatile("" : "+r"(tt));
        Lane l;
        row_lane<N, decltype(strip)::value>(tt, l.row, l.low, l.g);
        return l;
    };
    using Strip = std::integral_constant<bool, true>;
    using Natural = std::integral_constant<bool, false>;
    using First = std::integral_constant<bool, (DIR < 0)>;  // the map of pass 1
    using Last = std::integral_constant<bool, (DIR > 0)>;   // the map of pass 3

    cpx x[16];
    // the tile bits of row v's tile row, shifted to the tile of column `col` <
    // kPer; the tile `off` columns (a multiple of 64) further is bit (off >>
    // LOG2T) % 32 of word (off >> LOG2T) / 32 (no carry: col < kPer)
    struct Bits {
        uint32_t w[kWords];
        __device__ __forceinline__ bool at(int off) const { return (w[(off >> LOG2T) >> 5] >> ((off >> LOG2T) & 31)) & 1u; }
    };
    auto tile_bits = [&](int v, int col) {
        Bits b;
#pragma unroll
        for (int i = 0; i < kWords; ++i) b.w[i] = __ldg(tb + (v >> LOG2T) * kWords + i) >> (col >> LOG2T);
        return b;
    };
    // +1: the rows' values from the non-empty tiles into registers
    auto load = [&](int v) {
        const Lane l = lane_map(Natural());
        const int j = l.low + 16 * l.g;
        const float2* src = nat + (size_t)(v + l.row) * N + j;
        const Bits b = tile_bits(v, j);
#pragma unroll
        for (int a = 0; a < 16; ++a) {
            x[a] = cpx_make(0.f, 0.f);
            if (b.at(a * kPer)) {
                const float2 z = __ldcs(src + a * kPer);
                x[a] = cpx_make(z.x, z.y);
            }
        }
    };
    // -1: the rows' image from the strips into shared memory (thread 0)
    auto fetch = [&](int v) {
        mbar_expect(smem_u32(&bar), (uint32_t)(8192 * sizeof(float2)));
        for (int q = 0; q < N / 2; q += kRowBox)
            tma_load_2d(smem_u32(sm + q * 2 * R), &map, 2 * v, plane * (N / 2) + q, smem_u32(&bar));
    };
    uint32_t phase = 0;
    if (DIR > 0) {
        load(v0);
    } else {
        if (t == 0) {
            s_abort = 0;
            mbar_init(smem_u32(&bar), 1);
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
            fetch(v0);
        }
        __syncthreads();
    }
    for (; v0 < v1; v0 += stride) {
        if (DIR < 0) {
            const bool ok = mbar_wait(smem_u32(&bar), phase, &s_abort, limit);
            if (__syncthreads_or(!ok)) {
                if (t == 0) {  // leave no copy in flight into this block's shared memory
                    atomicOr(err, 1ull);
                    const unsigned long long t0 = global_ns();
                    while (!mbar_try(smem_u32(&bar), phase) && global_ns() - t0 <= limit) {
                    }
                }
                __syncthreads();
                return;
            }
            phase ^= 1;
            const Lane l = lane_map(Strip());
#pragma unroll
            for (int a = 0; a < 16; ++a) {
                const int col = l.low + 16 * l.g + a * kPer;
                x[a] = lds_c(sm + (col >> 1) * (2 * R) + 2 * l.row + (col & 1));
            }
            __syncthreads();
        }
        {
            const Lane l = lane_map(First());
            const int j = l.low + 16 * l.g;
            float2* buf = sm + l.row * Sh::kRowPitch + j;
            dft16<DIR>(x);
            sts_c(buf, x[0]);
#pragma unroll
            for (int k1 = 1; k1 < 16; ++k1) {
                float2 w = __ldg(tw1 + (k1 - 1) * kPer + j);
                if (DIR < 0) w.y = -w.y;
                sts_c(buf + k1 * P, c_mul(x[k1], w));
            }
        }
        __syncthreads();
        {
            const Lane l = lane_map(Natural());
            const int j = l.low + 16 * l.g, k1 = j / r, t2 = j % r;
            float2* blk = sm + l.row * Sh::kRowPitch + k1 * P + t2;
#pragma unroll
            for (int b = 0; b < 16; ++b) x[b] = lds_c(blk + r * b);
            dft16<DIR>(x);
            sts_c(blk, x[0]);
#pragma unroll
            for (int k2 = 1; k2 < 16; ++k2) {
                float2 w = __ldg(tw2 + (k2 - 1) * r + t2);
                if (DIR < 0) w.y = -w.y;
                sts_c(blk + r * k2, c_mul(x[k2], w));
            }
        }
        __syncthreads();
        const Lane l = lane_map(Last());
        const int row = l.row, k1 = l.low, g = l.g;
        {
            const float2* blk = sm + row * Sh::kRowPitch + k1 * P;
#pragma unroll
            for (int o = 0; o < 16; ++o) x[o] = lds_c(blk + (g + r * (o / r)) * r + o % r);
        }
        __syncthreads();  // the rows are read: their place takes an image
        if (DIR < 0 && t == 0 && v0 + stride < v1) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            fetch(v0 + stride);
        }
        Bits need;
        if (DIR < 0) need = tile_bits(v0, k1 + 16 * g);
#pragma unroll
        for (int i = 0; i < 16 / r; ++i) {
            cpx y[r];
#pragma unroll
            for (int q = 0; q < r; ++q) y[q] = x[i * r + q];
            dft_small<r, DIR>(y);
#pragma unroll
            for (int k3 = 0; k3 < r; ++k3) {
                const int col = k1 + 16 * (g + r * i) + 256 * k3;
                if (DIR > 0) {
                    sts_c(sm + (col >> 1) * (2 * R) + 2 * row + (col & 1), y[k3]);
                } else {
                    if (need.at(16 * r * i + 256 * k3)) sts_c(nat + (size_t)(v0 + row) * N + col, y[k3]);
                }
            }
        }
        if (DIR > 0) {
            if (v0 + stride < v1) load(v0 + stride);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncthreads();
            if (t == 0) {
                for (int q = 0; q < N / 2; q += kRowBox)
                    tma_store_2d(&map, 2 * v0, plane * (N / 2) + q, smem_u32(sm + q * 2 * R));
                bulk_store_drain();  // the image is read until here
            }
            __syncthreads();
        }
    }
}

template <int N>
constexpr size_t rows_smem()
{
    return (size_t)RowShape<N>::R * RowShape<N>::kRowPitch * sizeof(float2);
}

// ------------------------------------------------------- the pixels' screen

// Per pixel, with n - 1 of the pixel: the rotation between planes rho = exp(2
// pi i dw (n - 1)), and for every run of kScreenRun planes fin = exp(2 pi i w_k
// (n - 1)) of the run's first plane k, times the finalisation's factors that do
// not depend on the data (taper, n and w correction per flags, 0 outside the
// sky).  Within a run the screen is a power of the binary32 rho; fin is
// evaluated directly, so that what the powers miss does not add up from run to
// run (RMS error of a sum of random planes over its RMS: 4e-7 for one run and
// for 64; with a binary32 correction per run in its place 1e-6 at 4 runs, 2e-5
// at 64).  The tables depend on |x - n / 2| and |y - n / 2| only and are
// symmetric in the two: one quadrant [a][b], a, b <= n / 2, is kept, and the
// column kernels bring in the rows of their columns' a.  A handle makes them
// once: evaluated per pixel inside the column kernel, on 8 to 16 warps per SM,
// they took as long as 16 of its planes.  Entry b is stored at b ^ (b / 16 %
// 16): lanes whose pixels are 16 rows apart then read 16 different banks.
__host__ __device__ __forceinline__ int screen_pitch(int n) { return n / 2 + 16; }
__device__ __forceinline__ int screen_at(int b) { return b ^ ((b >> 4) & 15); }

// grid z: run of a channel (tab.runs each)
__global__ void __launch_bounds__(256) k_screen(StackArgs a_in, const float* __restrict__ taper, ScreenTab tab)
{
    StackArgs a = a_in;
    const int chan = (int)blockIdx.z / tab.runs, run = (int)blockIdx.z - chan * tab.runs;
    if (a_in.chan_screen) {
        const float4 cs = __ldg(a_in.chan_screen + chan);
        a.wb_hi = cs.x;
        a.wb_lo = cs.y;
        a.dw_hi = cs.z;
        a.dw_lo = cs.w;
    }
    const int hn = a.n / 2, pitch = screen_pitch(a.n);
    const int ib = blockIdx.x * 256 + threadIdx.x, ia = blockIdx.y;
    if (ib > hn) return;
    const int x = hn - ia, y = hn - ib;  // pixels 0 .. n / 2
    const PixelScreen ps = pixel_screen(a, x, y);
    if (run == 0)
        tab.rho[((size_t)chan * (hn + 1) + ia) * pitch + screen_at(ib)] = turns_to_phasor(ps.B.hi, ps.B.lo);
    float f = ps.sky ? 1.0f : 0.0f;
    if (a.flags & RICK_GRID_CORRECT) f = f / (__ldg(taper + x) * __ldg(taper + y));
    if (a.flags & RICK_APPLY_N) f *= 1.0f + ps.nm1;
    if (a.wcorr) f /= wcorr_at(a, ps.nm1);
    const float2 z = screen(ps.A, ps.B, run * kScreenRun);
    tab.fin[((size_t)blockIdx.z * (hn + 1) + ia) * pitch + screen_at(ib)] = make_float2(z.x * f, z.y * f);
}

// ---------------------------------------------------------------- columns

// Blocks of the column kernels: kStrips strips of 2 x N / 16 threads; a thread
// holds 16 positions of one column, and the Horner sum and the rotation of 16
// pixels (96 registers of state, at most 128 in all: 512 threads per SM).
template <int N>
__host__ __device__ constexpr int strips_per_block()
{
    return N >= 2048 ? 1 : 2;
}
template <int N>
__host__ __device__ constexpr int col_threads()
{
    return strips_per_block<N>() * N / 8;
}
constexpr int kStripStages = 3;
template <int N>
constexpr size_t col_tw_bytes()
{
    return (size_t)(15 * (N / 16) + 15 * (N / 256)) * sizeof(float2);
}
template <int N>
constexpr size_t colimage_smem()
{
    return (size_t)kStripStages * strips_per_block<N>() * N * sizeof(float4) + col_tw_bytes<N>() +
           kStripStages * sizeof(unsigned long long);
}
// two exchange buffers | w_n^(j k1), k1 < 16 | w_(n/16)^(t2 k2), [t2][k2]
template <int N>
constexpr size_t colspread_smem()
{
    return 2 * (size_t)strips_per_block<N>() * N * sizeof(float4) + (size_t)(16 * (N / 16) + 16 * (N / 256)) * sizeof(float2);
}

// Positions in shared memory, in rows of two columns (16 bytes; a lane takes
// one of them).  Block k1 of a transform holds N / 16 rows; the XORs keep the
// 8 rows of each half warp in 8 different 16-byte bank groups in pass 2 (lanes
// over t2, then blocks) and pass 3 (lanes over k2, then blocks).
template <int N>
__device__ __forceinline__ int pos1(int k1, int j)
{
    constexpr int r = N / 256;
    return k1 * (N / 16) + (r == 4 ? j ^ ((k1 & 1) << 2) : j);
}
template <int N>
__device__ __forceinline__ int pos2(int k1, int k2, int t2)
{
    constexpr int r = N / 256;
    if constexpr (r == 4) {
        const int s = ((k2 >> 1) & 1) | ((k1 & 1) << 1);
        return k1 * (N / 16) + ((k2 * 4 + (t2 ^ s)) ^ ((k1 & 1) << 2));
    } else {
        return k1 * (N / 16) + k2 * r + (t2 ^ (k2 & 7));
    }
}

// A thread's place in the column kernels: column c of strip `sub` of the block's
// S, position j < N / 16 of the passes, and its pixels' rows y(o), o = i r + k3,
// y = k1 + 16 (g + r i) + 256 k3.
template <int N>
struct ColThread {
    static constexpr int r = N / 256, kPer = N / 16;
    int c, j, sub, k1, g;
    __device__ __forceinline__ explicit ColThread(int t)
    {
        c = t & 1;
        j = (t >> 1) % kPer;
        sub = (t >> 1) / kPer;
        k1 = j / r;
        g = j % r;
    }
    __device__ __forceinline__ int y(int o) const { return k1 + 16 * (g + r * (o / r)) + 256 * (o % r); }
    // the pixel's entry of its column's row of a screen table
    __device__ __forceinline__ int entry(int o) const
    {
        const int d = y(o) - N / 2;
        return screen_at(d < 0 ? -d : d);
    }
};

// the row of column x in table `t` (channel, or channel and run) of a ScreenTab member
template <int N>
__device__ __forceinline__ size_t screen_row(int t, int x)
{
    const int d = x - N / 2;
    return ((size_t)t * (N / 2 + 1) + (d < 0 ? -d : d)) * screen_pitch(N);
}

// Persistent blocks (as many as are co-resident) over the units of a launch:
// a unit is kStrips strips of one channel, its slots are the rho rows of its
// columns, then the planes from the last to the first, and after each run's
// first plane (and the unit's) the run's fin rows.  The
// slots of consecutive units follow one another through three shared-memory
// stages (bulk copies completing on the stage's mbarrier), so that a unit's
// first copies are in flight while the last planes of the one before are
// transformed.  Every slot has one block barrier, at which all threads are
// done with the slot before: the copy of the slot two further on is issued
// there.  The planes of a run are summed per pixel by Horner's rule, h <- h rho +
// v, and the runs' sums, times their fin, in `part` (a unit of one run does
// without it; 64 KB per SM, which stay in L2): registers are full.
// range: the ranges of tile rows of the group's planes, from plane 0 of the
// strip buffer.  err: bit 0 when a bounded wait ran out.
// Bound: 32 planes of 4096^2 take 1.22 ms, the sum of the column factor (1.21)
// and the fused stack (0.91) that it replaces 2.12; 5000 cycles per plane and
// SM, of which ~3300 are issue slots (830 warp instructions per 16 values and
// lane) and ~3000 shared-memory passes, at 16 warps per SM (registers); the
// copies need 2100.
template <int N>
__global__ void __launch_bounds__(col_threads<N>(), 512 / col_threads<N>())
    k_colimage(StackArgs a, const float2* __restrict__ tw1, const float2* __restrict__ tw2,
               const int2* __restrict__ range, int log2T, const float4* __restrict__ strips, ScreenTab tab,
               float2* __restrict__ part, float2* __restrict__ acc, const double* __restrict__ sum_w, void* image,
               int units, unsigned long long* __restrict__ err)
{
    constexpr int r = N / 256, kPer = N / 16, S = strips_per_block<N>(), kThreads = col_threads<N>();
    constexpr int kUnits = N / 2 / S;  // units per channel
    constexpr int kRow = N / 2 + 16;   // screen_pitch(N)
    static_assert(2 * kRow <= 2 * N, "two table rows fit in a strip's share of a stage");
    extern __shared__ __align__(128) unsigned char strip_smem[];
    float4* stage = reinterpret_cast<float4*>(strip_smem);  // [stages][S][N]
    float2* s1 = reinterpret_cast<float2*>(stage + kStripStages * S * N);  // [15][kPer]
    float2* s2 = s1 + 15 * kPer;                                           // [15][r]
    unsigned long long* full = reinterpret_cast<unsigned long long*>(s2 + 15 * r);
    __shared__ int s_abort;

    const int t = threadIdx.x, nk = a.nk;
    const ColThread<N> me(t);
    const unsigned long long limit = a.wait_ns ? a.wait_ns : kStripWaitNs;
    if (t == 0) {
        s_abort = 0;
        for (int st = 0; st < kStripStages; ++st) mbar_init(smem_u32(full + st), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    // whether plane p of the group is the first of its run (or of the group)
    auto run_start = [&](int p) { return p == 0 || (a.k0 + p) % kScreenRun == 0; };
    // thread 0: issue the next slot in order, if any: of unit iu the rho rows (ip
    // = nk), plane ip, or the fin rows after it (ifin)
    int iu = blockIdx.x, ip = nk, ist = 0, issued = 0;
    bool ifin = false;
    auto issue = [&]() {
        if (iu >= units) return;
        const int chan = iu / kUnits, strip0 = (iu - chan * kUnits) * S;
        const uint32_t bar = smem_u32(full + ist);
        float4* dst = stage + (size_t)ist * S * N;
        if (ip == nk || ifin) {
            const float2* src = ifin ? tab.fin : tab.rho;
            const int table = ifin ? (a.chan0 + chan) * tab.runs + (a.k0 + ip) / kScreenRun : a.chan0 + chan;
            mbar_expect(bar, S * 2 * kRow * (uint32_t)sizeof(float2));
            for (int q = 0; q < 2 * S; ++q)
                bulk_load(smem_u32(reinterpret_cast<float2*>(dst + (q >> 1) * N) + (q & 1) * kRow),
                          src + screen_row<N>(table, 2 * strip0 + q), kRow * (uint32_t)sizeof(float2), bar);
        } else if (nk - ip != a.skip_slot1) {
            const int p = a.plane0 + chan * nk + ip;
            const int2 rg = __ldg(range + p);
            const uint32_t row0 = (uint32_t)rg.x << log2T, bytes = ((uint32_t)(rg.y - rg.x) << log2T) * 16u;
            mbar_expect(bar, S * bytes);
            if (bytes)
                for (int q = 0; q < S; ++q)
                    bulk_load(smem_u32(dst + (size_t)q * N + row0), strips + ((size_t)p * (N / 2) + strip0 + q) * N + row0,
                              bytes, bar);
        }
        ++issued;
        if (++ist == kStripStages) ist = 0;
        if (ip < nk && !ifin && run_start(ip)) {
            ifin = true;
            return;
        }
        ifin = false;
        if (--ip < 0) {
            ip = nk;
            iu += gridDim.x;
        }
    };
    if (t == 0)
        for (int i = 0; i < kStripStages; ++i) issue();
    for (int i = t; i < 15 * kPer; i += kThreads) s1[i] = __ldg(tw1 + i);
    for (int i = t; i < 15 * r; i += kThreads) s2[i] = __ldg(tw2 + i);
    const float2* w1 = s1 + me.j;
    const float2* w2 = s2 + me.g;

    // wait for the next slot's copy; false (in every thread of the block, at
    // the slot's barrier) once a wait ran out
    int st = 0;
    uint32_t phase = 0;
    bool ok = true;
    auto wait = [&]() -> float2* {
        ok = mbar_wait(smem_u32(full + st), phase, &s_abort, limit);
        return reinterpret_cast<float2*>(stage + ((size_t)st * S + me.sub) * N);
    };
    auto next = [&]() {
        if (++st == kStripStages) {
            st = 0;
            phase ^= 1;
        }
    };
    // the slot's barrier: every thread is done with the slot before, whose
    // stage is refilled (not at the block's first slot: nothing was read yet)
    bool first = true;
    auto barrier = [&]() -> bool {
        if (__syncthreads_or(!ok)) return false;
        if (t == 0 && !first) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            issue();
        }
        first = false;
        return true;
    };

    for (int u = blockIdx.x; u < units; u += gridDim.x) {
        const int chan = u / kUnits, strip0 = (u - chan * kUnits) * S;
        const int plane0 = a.plane0 + chan * nk, px = 2 * (strip0 + me.sub) + me.c;
        float2 rho[16], h[16];
        {
            const float2* row = wait() + me.c * kRow;
#pragma unroll
            for (int o = 0; o < 16; ++o) {
                rho[o] = row[me.entry(o)];
                h[o] = make_float2(0.f, 0.f);
            }
            if (!barrier()) break;
            next();
        }
        bool bad = false;
        for (int phi = nk; phi > 0 && !bad;) {
            // the run [plo, phi)
            const int plo = max(0, (a.k0 + phi - 1) / kScreenRun * kScreenRun - a.k0);
            for (int p = phi - 1; p >= plo; --p) {
                const int2 rg = __ldg(range + plane0 + p);
                // rows j + kPer q of the range: q from qlo to qhi - 1
                const int qlo = ((rg.x << log2T) + kPer - 1 - me.j) / kPer, qhi = ((rg.y << log2T) + kPer - 1 - me.j) / kPer;
                const uint32_t in = (1u << qhi) - (1u << qlo);
                float2* buf = wait() + me.c;
                cpx x[16];
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    x[q] = cpx_make(0.f, 0.f);
                    if (in & (1u << q)) x[q] = lds_c(buf + 2 * (me.j + kPer * q));
                }
                if (r == 4) __syncwarp();  // pos1 moves values between neighbouring lanes
                dft16<1>(x);
                sts_c(buf + 2 * pos1<N>(0, me.j), x[0]);
#pragma unroll
                for (int q = 1; q < 16; ++q) sts_c(buf + 2 * pos1<N>(q, me.j), c_mul(x[q], w1[(q - 1) * kPer]));
                if (!barrier()) {
                    bad = true;
                    break;
                }
#pragma unroll
                for (int b = 0; b < 16; ++b) x[b] = lds_c(buf + 2 * pos1<N>(me.k1, me.g + r * b));
                __syncwarp();  // the block's reads (pos1) before its writes (pos2)
                dft16<1>(x);
                sts_c(buf + 2 * pos2<N>(me.k1, 0, me.g), x[0]);
#pragma unroll
                for (int k2 = 1; k2 < 16; ++k2) sts_c(buf + 2 * pos2<N>(me.k1, k2, me.g), c_mul(x[k2], w2[(k2 - 1) * r]));
                __syncwarp();
#pragma unroll
                for (int ii = 0; ii < 16 / r; ++ii) {
                    cpx y[r];
#pragma unroll
                    for (int q = 0; q < r; ++q) y[q] = lds_c(buf + 2 * pos2<N>(me.k1, me.g + r * ii, q));
                    dft_small<r, 1>(y);
#pragma unroll
                    for (int k3 = 0; k3 < r; ++k3) {
                        const int o = ii * r + k3;
                        const float2 v = cpx_get(y[k3]), g = h[o];
                        h[o].x = fmaf(g.x, rho[o].x, fmaf(-g.y, rho[o].y, v.x));
                        h[o].y = fmaf(g.x, rho[o].y, fmaf(g.y, rho[o].x, v.y));
                    }
                }
                next();
            }
            if (bad) break;
            // a group that begins within a run: on to the run's first plane, by
            // the rotation's powers (the unit needs rho no more)
            for (int z = (a.k0 + plo) % kScreenRun; z > 0; z >>= 1) {
#pragma unroll
                for (int o = 0; o < 16; ++o) {
                    if (z & 1) h[o] = c_mul(h[o], rho[o]);
                    rho[o] = c_mul(rho[o], rho[o]);
                }
            }
            const float2* row = wait() + me.c * kRow;
            if (!barrier()) {
                bad = true;
                break;
            }
            const bool top = phi == nk;  // the unit's first run
            float2* mine = part + (size_t)blockIdx.x * 16 * kThreads + t;
            const int ch = a.chan_screen ? a.chan0 + chan : 0;
            const double sw = sum_w[ch];
            const float inv_sw = (sw != 0.0) ? (float)(1.0 / sw) : 0.0f;
            float* out = reinterpret_cast<float*>(image) + (size_t)ch * a.img_stride;
#pragma unroll
            for (int o = 0; o < 16; ++o) {
                const int y = me.y(o);
                const int64_t pix = (int64_t)y * N + px;
                const float2 f = row[me.entry(o)];
                // outside the sky (f = 0) the pixel is 0 whatever the planes hold, infinities too
                float2 v = f.x != 0.f || f.y != 0.f ? c_mul(h[o], f) : make_float2(0.f, 0.f);
                h[o] = make_float2(0.f, 0.f);
                if (!top) v = c_add(v, mine[o * kThreads]);
                if (plo > 0) {
                    mine[o * kThreads] = v;
                    continue;
                }
                if ((px + y) & 1) v = make_float2(-v.x, -v.y);  // fftshift sign
                if (!a.first) v = c_add(v, acc[pix]);
                if (!a.last)
                    acc[pix] = v;
                else if (a.flags & RICK_REAL_IMAGE)
                    out[pix] = v.x * inv_sw;
                else
                    reinterpret_cast<float2*>(out)[pix] = make_float2(v.x * inv_sw, v.y * inv_sw);
            }
            next();
            phi = plo;
        }
        if (bad) break;
    }
    if (!ok) s_abort = 1;
    __syncthreads();
    if (s_abort && t == 0) {
        // leave no bulk copy in flight into this block's shared memory: wait
        // (bounded) for the last slot issued into every stage
        atomicOr(err, 1ull);
        for (int i = issued > kStripStages ? issued - kStripStages : 0; i < issued; ++i) {
            const unsigned long long t0 = global_ns();
            while (!mbar_try(smem_u32(full + i % kStripStages), (uint32_t)((i / kStripStages) & 1)) &&
                   global_ns() - t0 <= limit) {
            }
        }
    }
    __syncthreads();
}

// Adjoint of k_colimage: for every plane of the group, the rows of its range
// of the (forward) column transforms of R conj(screen), R the adjoint of the
// finalisation applied to the image gradient, in strip order.  The pixels'
// conjugate rotation advances the screened value from plane to plane within a
// run of planes, whose first value is made from the pixels again.  Planes
// alternate between two exchange buffers, so that the barrier between passes 2
// and 1 of a plane also covers the reads of the plane before.  32 planes of
// 4096^2: 1.38 ms, the rows after it 0.91 (0.26 of the tiles written): together
// 2.3 where the adjoint stack, column factor and cuFFT's rows took 3.6.  Bound by
// latency: issue slots 39 % busy, the shared-memory pipe 43 %, at 16 warps per SM
// (registers).
template <int N>
__global__ void __launch_bounds__(col_threads<N>(), 512 / col_threads<N>())
    k_colspread(StackArgs a, const float2* __restrict__ tw1, const float2* __restrict__ tw2,
                const int2* __restrict__ range, int log2T, const void* __restrict__ rimg, ScreenTab tab,
                const double* __restrict__ sum_w, float4* __restrict__ strips)
{
    constexpr int r = N / 256, kPer = N / 16, S = strips_per_block<N>(), kThreads = col_threads<N>();
    extern __shared__ __align__(128) unsigned char strip_smem[];
    const int t = threadIdx.x;
    const ColThread<N> me(t);
    const int x0 = 2 * (blockIdx.x * S + me.sub) + me.c;
    float4* bufs = reinterpret_cast<float4*>(strip_smem);
    float2* s1 = reinterpret_cast<float2*>(bufs + 2 * S * N);  // [16][kPer]
    float2* s2 = s1 + 16 * kPer;                               // [r][16]
    const float2 one = make_float2(1.f, 0.f);
    for (int i = t; i < 16 * kPer; i += kThreads) s1[i] = i < kPer ? one : __ldg(tw1 + i - kPer);
    for (int i = t; i < 16 * r; i += kThreads) s2[i] = (i & 15) ? __ldg(tw2 + ((i & 15) - 1) * r + (i >> 4)) : one;

    const double sw = *sum_w;
    const float inv_sw = (sw != 0.0) ? (float)(1.0 / sw) : 0.0f;
    float2 rho[16], q[16];  // conjugate rotation, screened value of the current plane
    // the table rows of the block's columns, through shared memory
    constexpr int kRow = N / 2 + 16;
    float2* rows = reinterpret_cast<float2*>(strip_smem) + (size_t)(2 * me.sub + me.c) * kRow;
    auto load_rows = [&](const float2* src, int table) {
        __syncthreads();
        for (int i = t; i < 2 * S * kRow; i += kThreads) {
            const int col = i / kRow;
            reinterpret_cast<float2*>(strip_smem)[i] = __ldg(src + screen_row<N>(table, 2 * blockIdx.x * S + col) + i - col * kRow);
        }
        __syncthreads();
    };
    auto load_rho = [&]() {
        load_rows(tab.rho, 0);
#pragma unroll
        for (int o = 0; o < 16; ++o) {
            rho[o] = rows[me.entry(o)];
            rho[o].y = -rho[o].y;
        }
    };
    load_rho();
    // the screened values of plane p: the run's first plane's, rotated on to it
    auto start = [&](int p) {
        const int run = (a.k0 + p) / kScreenRun;
        load_rows(tab.fin, run);
#pragma unroll
        for (int o = 0; o < 16; ++o) {
            const int y = me.y(o);
            const int64_t pix = (int64_t)y * N + x0;
            float2 z = rows[me.entry(o)];
            const float s = ((x0 + y) & 1) ? -inv_sw : inv_sw;  // fftshift sign
            z = make_float2(z.x * s, -z.y * s);
            const float2 v = (a.flags & RICK_REAL_IMAGE) ? make_float2(reinterpret_cast<const float*>(rimg)[pix], 0.f)
                                                         : reinterpret_cast<const float2*>(rimg)[pix];
            q[o] = c_mul(v, z);
        }
        const int from = (a.k0 + p) - run * kScreenRun;  // > 0: a group that begins within a run
        for (int z = from; z > 0; z >>= 1) {
#pragma unroll
            for (int o = 0; o < 16; ++o) {
                if (z & 1) q[o] = c_mul(q[o], rho[o]);
                rho[o] = c_mul(rho[o], rho[o]);
            }
        }
        if (from > 0) load_rho();
        __syncthreads();
    };

    float2* dst0 = reinterpret_cast<float2*>(strips + (size_t)(blockIdx.x * S + me.sub) * N) + me.c;
    int which = 0;
    for (int p = 0; p < a.nk; ++p) {
        const int2 rg = __ldg(range + p);
        const int vlo = rg.x << log2T, vhi = rg.y << log2T;
        if (p == 0 || (a.k0 + p) % kScreenRun == 0) {
            start(p);
        } else {
#pragma unroll
            for (int o = 0; o < 16; ++o) q[o] = c_mul(q[o], rho[o]);
        }
        if (vhi <= vlo) continue;  // nothing on this plane (the same in every thread)
        float2* buf = reinterpret_cast<float2*>(bufs + (size_t)(which * S + me.sub) * N) + me.c;
        which ^= 1;
        // pass 3: over k3, output t2, times conj(w_(n/16)^(t2 k2))
#pragma unroll
        for (int ii = 0; ii < 16 / r; ++ii) {
            const int k2 = me.g + r * ii;
            cpx y[r];
#pragma unroll
            for (int k3 = 0; k3 < r; ++k3) y[k3] = cpx_make(q[ii * r + k3].x, q[ii * r + k3].y);
            dft_small<r, -1>(y);
#pragma unroll
            for (int t2 = 0; t2 < r; ++t2) {
                if (t2 > 0) {
                    const float2 w = s2[t2 * 16 + k2];
                    y[t2] = c_mul(y[t2], make_float2(w.x, -w.y));
                }
                sts_c(buf + 2 * pos2<N>(me.k1, k2, t2), y[t2]);
            }
        }
        __syncwarp();
        // pass 2: over k2, output b (t2 = g), times conj(w_n^(j' k1)), j' = t2 + r b
        cpx x[16];
#pragma unroll
        for (int k2 = 0; k2 < 16; ++k2) x[k2] = lds_c(buf + 2 * pos2<N>(me.k1, k2, me.g));
        __syncwarp();
        dft16<-1>(x);
#pragma unroll
        for (int b = 0; b < 16; ++b) {
            const int jj = me.g + r * b;
            const float2 w = s1[me.k1 * kPer + jj];
            sts_c(buf + 2 * pos1<N>(me.k1, jj), c_mul(x[b], make_float2(w.x, -w.y)));
        }
        __syncthreads();
        // pass 1: over k1, output a: rows v = j + (n / 16) a
#pragma unroll
        for (int q1 = 0; q1 < 16; ++q1) x[q1] = lds_c(buf + 2 * pos1<N>(q1, me.j));
        dft16<-1>(x);
        float2* dst = dst0 + (size_t)p * N * N;
#pragma unroll
        for (int q1 = 0; q1 < 16; ++q1) {
            const int v = me.j + kPer * q1;
            if (v >= vlo && v < vhi) sts_c(dst + 2 * v, x[q1]);
        }
    }
}

template <typename K>
cudaError_t opt_in(K kernel, size_t bytes, std::atomic<bool> (&done)[64])
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64 && done[dev].load(std::memory_order_acquire)) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev].store(true, std::memory_order_release);
    return e;
}

template <int N, int DIR, int LOG2T>
cudaError_t launch_rows_n(const StripArgs& s, int k0, int nk, float2* planes, unsigned long long wait_ns,
                          unsigned long long* err, cudaStream_t st)
{
    static std::atomic<bool> done[64];
    const cudaError_t e = opt_in(k_rows<N, DIR, LOG2T>, rows_smem<N>(), done);
    if (e != cudaSuccess) return e;
    // two blocks per SM and plane (a plane at a time); n = 4096 gives each several row groups
    const int groups = N / RowShape<N>::R, want = 2 * sm_count_strip();
    const dim3 grid((unsigned)std::min(groups, want), (unsigned)nk);
    k_rows<N, DIR, LOG2T><<<grid, kRowThreads, rows_smem<N>(), st>>>(*reinterpret_cast<const CUtensorMap*>(s.map), s.tw1,
                                                                    s.tw2, s.bits, s.range, k0, planes, wait_ns, err);
    return cudaGetLastError();
}

template <int N>
cudaError_t launch_rows_t(int dir, const StripArgs& s, int k0, int nk, float2* planes,
                          unsigned long long wait_ns, unsigned long long* err, cudaStream_t st)
{
    switch (s.log2T) {
#define RICK_ROWS_CASE(L)                                                               \
    case L:                                                                             \
        return dir > 0 ? launch_rows_n<N, 1, L>(s, k0, nk, planes, wait_ns, err, st) \
                       : launch_rows_n<N, -1, L>(s, k0, nk, planes, wait_ns, err, st);
        RICK_ROWS_CASE(4)
        RICK_ROWS_CASE(5)
        RICK_ROWS_CASE(6)
#undef RICK_ROWS_CASE
        default: return cudaErrorInvalidValue;
    }
}

template <int N>
cudaError_t launch_colimage_n(const StripArgs& s, const StackArgs& a, const float2* strips, float2* acc,
                              const double* sum_w, void* image, unsigned long long* err, int nchan, cudaStream_t st)
{
    static std::atomic<bool> done[64];
    const cudaError_t e = opt_in(k_colimage<N>, colimage_smem<N>(), done);
    if (e != cudaSuccess) return e;
    const int units = nchan * (N / 2 / strips_per_block<N>());
    const int resident = sm_count_strip() * (512 / col_threads<N>());
    k_colimage<N><<<(unsigned)std::min(units, resident), col_threads<N>(), colimage_smem<N>(), st>>>(
        a, s.tw1, s.tw2, s.range + s.k0, s.log2T, reinterpret_cast<const float4*>(strips), s.tab, s.part, acc, sum_w,
        image, units, err);
    return cudaGetLastError();
}

template <int N>
cudaError_t launch_colspread_n(const StripArgs& s, const StackArgs& a, const void* rimg, const double* sum_w,
                               float2* strips, cudaStream_t st)
{
    static std::atomic<bool> done[64];
    const cudaError_t e = opt_in(k_colspread<N>, colspread_smem<N>(), done);
    if (e != cudaSuccess) return e;
    k_colspread<N><<<(unsigned)(N / 2 / strips_per_block<N>()), col_threads<N>(), colspread_smem<N>(), st>>>(
        a, s.tw1, s.tw2, s.range + s.k0, s.log2T, rimg, s.tab, sum_w, reinterpret_cast<float4*>(strips));
    return cudaGetLastError();
}

}  // namespace

// The strip buffer of `planes` planes as [strips][2 n] values; a box is the
// block's R rows of kRowBox strips.
cudaError_t encode_rows_map(void* map, const float2* strips, int n, int planes)
{
    static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
    if (!encode) {
        cudaDriverEntryPointQueryResult q;
        void* fn = nullptr;
        const cudaError_t e =
            cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
        if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
        encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    }
    const cuuint64_t dims[2] = {(cuuint64_t)n * 2, (cuuint64_t)planes * (n / 2)};
    const cuuint64_t strides[1] = {(cuuint64_t)n * 2 * sizeof(float2)};
    const cuuint32_t box[2] = {(cuuint32_t)(2 * (8192 / n)), (cuuint32_t)kRowBox};
    const cuuint32_t estr[2] = {1, 1};
    const CUresult r = encode(reinterpret_cast<CUtensorMap*>(map), CU_TENSOR_MAP_DATA_TYPE_UINT64, 2,
                              const_cast<float2*>(strips), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                              CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

bool strip_shape(int n) { return n == 1024 || n == 2048 || n == 4096; }

cudaError_t launch_occupancy(const GridCfg& c, const ChunkList& ch, int reach, const StripArgs& s, cudaStream_t st)
{
    const int parts = (c.ntu * s.wpr + kOccWords - 1) / kOccWords;
    k_occupancy<<<dim3((unsigned)parts, (unsigned)c.nw), kOccThreads, 0, st>>>(c, ch, reach, s.wpr, s.bits, s.range, s.occ);
    return cudaGetLastError();
}

cudaError_t launch_rows(int n, int dir, const StripArgs& s, int k0, int nk, float2* planes,
                        unsigned long long wait_ns, unsigned long long* err, cudaStream_t st)
{
    if (nk <= 0) return cudaSuccess;
    if (nk > 65535) return cudaErrorInvalidValue;
    switch (n) {
        case 1024: return launch_rows_t<1024>(dir, s, k0, nk, planes, wait_ns, err, st);
        case 2048: return launch_rows_t<2048>(dir, s, k0, nk, planes, wait_ns, err, st);
        case 4096: return launch_rows_t<4096>(dir, s, k0, nk, planes, wait_ns, err, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_screen(const StripArgs& s, const StackArgs& a, const float* taper, int nchan, cudaStream_t st)
{
    const int64_t tables = (int64_t)nchan * s.tab.runs;
    if (nchan < 1 || tables < 1 || tables > 65535) return cudaErrorInvalidValue;
    const int side = a.n / 2 + 1;
    k_screen<<<dim3((unsigned)((side + 255) / 256), (unsigned)side, (unsigned)tables), 256, 0, st>>>(a, taper, s.tab);
    return cudaGetLastError();
}

// k_colimage's `part`: 16 values of each thread that is resident (512 per SM).
size_t strip_part_bytes(int runs) { return runs > 1 ? (size_t)sm_count_strip() * 512 * 16 * sizeof(float2) : 0; }

cudaError_t launch_colimage(const StripArgs& s, const StackArgs& a, const float2* strips, float2* acc,
                            const double* sum_w, void* image, unsigned long long* err, cudaStream_t st, int nchan)
{
    if (a.nk <= 0 || nchan <= 0) return cudaSuccess;
    if (nchan > 65535 || (nchan > 1 && !a.chan_screen)) return cudaErrorInvalidValue;
    switch (a.n) {
        case 1024: return launch_colimage_n<1024>(s, a, strips, acc, sum_w, image, err, nchan, st);
        case 2048: return launch_colimage_n<2048>(s, a, strips, acc, sum_w, image, err, nchan, st);
        case 4096: return launch_colimage_n<4096>(s, a, strips, acc, sum_w, image, err, nchan, st);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_colspread(const StripArgs& s, const StackArgs& a, const void* rimg, const double* sum_w,
                             float2* strips, cudaStream_t st)
{
    if (a.nk <= 0) return cudaSuccess;
    switch (a.n) {
        case 1024: return launch_colspread_n<1024>(s, a, rimg, sum_w, strips, st);
        case 2048: return launch_colspread_n<2048>(s, a, rimg, sum_w, strips, st);
        case 4096: return launch_colspread_n<4096>(s, a, rimg, sum_w, strips, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace rick
