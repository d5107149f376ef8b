// rick_prep.cu -- sub-step 1 of gridding (Sec. 2.1: the measurements are
// gathered into one array per sector of the uv plane), done as a device
// counting sort by (w-plane, uv tile):
//   k_density  nearest-cell counts for uniform weighting
//   k_count    entries per tile (a footprint straddling tiles is listed in
//              every tile it touches)
//   k_scan_*   exclusive prefix sum of the counts -> tile start offsets
//   k_scatter  one 16-byte entry (pu, pv, s*Re V, s*Im V), s = weight / (sum of
//              u taps * sum of v taps), per (measurement, tile), written at
//              its tile's cursor; weight sum and counters.
// Grids are sized to the SM count; each block takes a contiguous range of the
// measurements (split at channel boundaries in batched imaging) and reads it
// coalesced; writes of entries are scattered 16-byte stores.
#include "rick_internal.cuh"

namespace rick {
namespace {

int sm_count()
{
    static int cached[64] = {0};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) dev = 0;
    if (!cached[dev]) {
        int v = 0;
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        cached[dev] = v > 0 ? v : 1;
    }
    return cached[dev];
}

constexpr int kPrepThreads = 256;

int prep_blocks(int64_t m, int bpsm = 8)
{
    int64_t want = (m + kPrepThreads - 1) / kPrepThreads;
    int64_t cap = (int64_t)sm_count() * (bpsm > 0 ? bpsm : 8);
    if (want > cap) want = cap;
    return (int)(want < 1 ? 1 : want);
}

struct Inputs {
    const float* u;
    const float* v;
    const float* w;
    const float* wt;
    const float2* vis;
};

__device__ __forceinline__ bool load_and_place(const GridCfg& c, const Inputs& in, int64_t i, int chan, Place& p,
                                               float& wi, float2& V)
{
    wi = in.wt ? __ldg(in.wt + i) : 1.0f;
    V = __ldg(in.vis + i);
    if (!place(c, __ldg(in.u + i), __ldg(in.v + i), __ldg(in.w + i), p, chan)) return false;
    if (p.conj) V.y = -V.y;
    return finite_value(wi, V);
}

// Each block takes one contiguous range of the m measurements and walks it
// channel by channel (one segment when there is a single channel): body(chan,
// i0, i1) is called for every non-empty segment, by all threads of the block.
template <typename Body>
__device__ __forceinline__ void for_each_segment(const GridCfg& c, int64_t m, Body&& body)
{
    const int64_t per = (m + gridDim.x - 1) / gridDim.x;
    int64_t r0 = (int64_t)blockIdx.x * per;
    const int64_t r1 = r0 + per < m ? r0 + per : m;
    if (r0 >= r1) return;
    int chan = 0;
    if (c.nchan > 1) {
        int lo = 0, hi = c.nchan - 1;  // last channel whose first measurement is <= r0
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (__ldg(c.chan_off + mid) <= r0) lo = mid; else hi = mid - 1;
        }
        chan = lo;
    }
    while (r0 < r1) {
        const int64_t end = (c.nchan > 1) ? min(r1, (int64_t)__ldg(c.chan_off + chan + 1)) : r1;
        if (end > r0) body(chan, r0, end);
        r0 = end > r0 ? end : r0;
        ++chan;
        if (chan >= c.nchan && r0 < r1) break;  // measurements past the last channel: none by construction
    }
}

__global__ void __launch_bounds__(kPrepThreads) k_density(GridCfg c, Inputs in, int64_t m,
                                                          uint32_t* __restrict__ density)
{
    for_each_segment(c, m, [&](int chan, int64_t i0, int64_t i1) {
        for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
            Place p;
            float wi;
            float2 V;
            if (!load_and_place(c, in, i, chan, p, wi, V)) continue;
            atomicAdd(density + (int64_t)nearest_cell(c, p.pv) * c.n + nearest_cell(c, p.pu), 1u);
        }
    });
}

// Tiles of plane `plane` touched by the uv footprint of a placed measurement: t[0] always, t[1]
// (right neighbour), t[2] (lower), t[3] (lower right) when the footprint
// straddles; -1 otherwise.
__device__ __forceinline__ void footprint_tiles(const GridCfg& c, const Place& p, int plane, int64_t (&t)[4])
{
    const int tu0 = p.fu >> c.log2T, tu1 = (p.fu + c.S - 1) >> c.log2T;
    const int tv0 = p.fv >> c.log2T, tv1 = (p.fv + c.S - 1) >> c.log2T;
    const int64_t base = (int64_t)plane * c.ntp;
    t[0] = base + tv0 * c.ntu + tu0;
    t[1] = tu1 != tu0 ? base + tv0 * c.ntu + tu1 : -1;
    t[2] = tv1 != tv0 ? base + tv1 * c.ntu + tu0 : -1;
    t[3] = (tu1 != tu0 && tv1 != tv0) ? base + tv1 * c.ntu + tu1 : -1;
}

// Measurements per thread and loop trip: their loads, and then their atomics,
// are in flight together.  Two rather than four: the scatter then needs 78
// instead of 128 registers and runs three CTAs per SM instead of two
// (measured 0.426 -> 0.392 ms at 4096^2 x 32 x 1e7, 34.1 -> 33.2 ms at
// 16384^2 x 128 x 2e8).
constexpr int kVisPerThread = 2;

__global__ void __launch_bounds__(kPrepThreads) k_count(GridCfg c, Inputs in, int64_t m,
                                                        uint32_t* __restrict__ counts)
{
    for_each_segment(c, m, [&](int chan, int64_t i0, int64_t i1) {
        for (int64_t ib = i0 + threadIdx.x; ib < i1; ib += (int64_t)kVisPerThread * blockDim.x) {
            Place p[kVisPerThread];
            bool ok[kVisPerThread];
#pragma unroll
            for (int q = 0; q < kVisPerThread; ++q) {
                const int64_t i = ib + (int64_t)q * blockDim.x;
                float wi;
                float2 V;
                ok[q] = i < i1 && load_and_place(c, in, i, chan, p[q], wi, V);
            }
#pragma unroll
            for (int q = 0; q < kVisPerThread; ++q) {
                if (!ok[q]) continue;
                // the measurement's planes: its own (Sw = 1) or its w-footprint
                for (int tw = 0; tw < c.Sw; ++tw) {
                    const int plane = p[q].k + tw;
                    if (plane < c.plane_lo || plane >= c.plane_hi) continue;
                    int64_t t[4];
                    footprint_tiles(c, p[q], plane, t);
#pragma unroll
                    for (int r = 0; r < 4; ++r)
                        if (t[r] >= 0) atomicAdd(counts + t[r] * c.cstride, 1u);
                }
            }
        }
    });
}

template <typename T>
__device__ __forceinline__ T warp_sum(T x)
{
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// Sum of one float over the block (all threads call it); result valid in thread 0.
__device__ __forceinline__ float block_sum(float x)
{
    __shared__ float s[kPrepThreads / 32];
    x = warp_sum(x);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) s[wid] = x;
    __syncthreads();
    float t = 0.0f;
    if (threadIdx.x == 0)
        for (int j = 0; j < kPrepThreads / 32; ++j) t += s[j];
    return t;
}

// chan_sw[chan] accumulates the weight sum of each channel (one entry when
// there is a single channel).
__global__ void __launch_bounds__(kPrepThreads) k_scatter(GridCfg c, Inputs in, int64_t m,
                                                          const uint32_t* __restrict__ density,
                                                          uint32_t* __restrict__ cursor,
                                                          float4* __restrict__ entries, Counters* ctr,
                                                          double* __restrict__ chan_sw)
{
    unsigned gridded = 0, dropped = 0, nent = 0;
    for_each_segment(c, m, [&](int chan, int64_t i0, int64_t i1) {
        float sw = 0.0f;
        for (int64_t ib = i0 + threadIdx.x; ib < i1; ib += (int64_t)kVisPerThread * blockDim.x) {
            Place p[kVisPerThread];
            float wi[kVisPerThread];
            float2 V[kVisPerThread];
            bool ok[kVisPerThread];
#pragma unroll
            for (int q = 0; q < kVisPerThread; ++q) {
                const int64_t i = ib + (int64_t)q * blockDim.x;
                ok[q] = false;
                if (i < i1) {
                    ok[q] = load_and_place(c, in, i, chan, p[q], wi[q], V[q]);
                    if (!ok[q]) ++dropped;
                }
            }
            // the gridder reads the visibility already weighted and divided by
            // the two tap sums (normalised taps), once per measurement here
            // instead of once per (measurement, tile) entry there
            float4 rec[kVisPerThread];
            uint32_t slot[kVisPerThread][4];
            int64_t t[kVisPerThread][4];
#pragma unroll
            for (int q = 0; q < kVisPerThread; ++q) {
                if (!ok[q]) continue;
                if (c.uniform) {
                    const uint32_t cnt =
                        __ldg(density + (int64_t)nearest_cell(c, p[q].pv) * c.n + nearest_cell(c, p[q].pu));
                    wi[q] = wi[q] / (float)cnt;
                }
                const float scale = wi[q] / (tap_sum(c, p[q].pu, p[q].fu) * tap_sum(c, p[q].pv, p[q].fv));
                rec[q] = make_float4(p[q].pu, p[q].pv, scale * V[q].x, scale * V[q].y);
                sw += wi[q];
                ++gridded;
                if (c.Sw > 1) {
                    // w-footprint: one set of entries per plane, the w-tap in the scale
                    const float hn = w_tap_norm(c, p[q]);
                    for (int tw = 0; tw < c.Sw; ++tw) {
                        const int plane = p[q].k + tw;
                        if (plane < c.plane_lo || plane >= c.plane_hi) continue;
                        const float ht = w_kernel(c, __fsub_rn((float)plane, p[q].pw)) * hn;
                        const float4 rw = make_float4(rec[q].x, rec[q].y, ht * rec[q].z, ht * rec[q].w);
                        int64_t tt[4];
                        footprint_tiles(c, p[q], plane, tt);
#pragma unroll
                        for (int r = 0; r < 4; ++r)
                            if (tt[r] >= 0) {
                                entries[atomicAdd(cursor + tt[r] * c.cstride, 1u)] = rw;
                                ++nent;
                            }
                    }
                    ok[q] = false;  // written: skip the nearest-plane stores below
                    continue;
                }
                if (p[q].k < c.plane_lo || p[q].k >= c.plane_hi) {
                    ok[q] = false;  // weighted and counted, no entries: another rank's plane
                    continue;
                }
                footprint_tiles(c, p[q], p[q].k, t[q]);
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    if (t[q][r] >= 0) slot[q][r] = atomicAdd(cursor + t[q][r] * c.cstride, 1u);
            }
#pragma unroll
            for (int q = 0; q < kVisPerThread; ++q) {
                if (!ok[q]) continue;
#pragma unroll
                for (int r = 0; r < 4; ++r)
                    if (t[q][r] >= 0) {
                        entries[slot[q][r]] = rec[q];
                        ++nent;
                    }
            }
        }
        const float tot = block_sum(sw);
        if (threadIdx.x == 0 && tot != 0.0f) atomicAdd(chan_sw + chan, (double)tot);
    });
    // counters: one set of atomics per block
    __shared__ unsigned s_g[kPrepThreads / 32], s_d[kPrepThreads / 32], s_e[kPrepThreads / 32];
    gridded = warp_sum(gridded);
    dropped = warp_sum(dropped);
    nent = warp_sum(nent);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
        s_g[wid] = gridded;
        s_d[wid] = dropped;
        s_e[wid] = nent;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long g = 0, d = 0, e = 0;
        for (int j = 0; j < kPrepThreads / 32; ++j) {
            g += s_g[j];
            d += s_d[j];
            e += s_e[j];
        }
        if (g) atomicAdd(&ctr->gridded, g);
        if (d) atomicAdd(&ctr->dropped, d);
        if (e) atomicAdd(&ctr->entries, e);
    }
}

// ------------------------------------------------ adjoint: primary-tile sort

// Placement for the adjoint: coordinates and weight only (no visibility value).
__device__ __forceinline__ bool place_coords(const GridCfg& c, const Inputs& in, int64_t i, Place& p, float& wi)
{
    wi = in.wt ? __ldg(in.wt + i) : 1.0f;
    return place(c, __ldg(in.u + i), __ldg(in.v + i), __ldg(in.w + i), p, 0) && isfinite(wi);
}

// Sort key of the adjoint: the tile of the first footprint cell on the
// measurement's plane (Sw = 1) or on the first plane of its w-footprint,
// clamped to the plane range (Sw > 1).
__device__ __forceinline__ int64_t primary_tile(const GridCfg& c, const Place& p)
{
    const int k = p.k < 0 ? 0 : (p.k > c.nw - 1 ? c.nw - 1 : p.k);
    return (int64_t)k * c.ntp + (p.fv >> c.log2T) * c.ntu + (p.fu >> c.log2T);
}

__global__ void __launch_bounds__(kPrepThreads) k_primary_count(GridCfg c, Inputs in, int64_t m,
                                                                uint32_t* __restrict__ counts)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * blockDim.x) {
        Place p;
        float wi;
        if (place_coords(c, in, i, p, wi)) atomicAdd(counts + primary_tile(c, p) * c.cstride, 1u);
    }
}

// The sorted measurements of the adjoint: (pu, pv, effective weight, index with
// the top bit set for a mirrored one) and the first plane of the w-footprint,
// so that the gather reads its list in order instead of the inputs at random
// (ent, plane); or, where that scratch does not fit, the indices alone (perm).
struct PrimaryList {
    float4* ent;
    int* plane;
    uint32_t* perm;
};

__global__ void __launch_bounds__(kPrepThreads) k_primary_scatter(GridCfg c, Inputs in, int64_t m,
                                                                  const uint32_t* __restrict__ density,
                                                                  uint32_t* __restrict__ cursor, PrimaryList list)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m;
         i += (int64_t)gridDim.x * blockDim.x) {
        Place p;
        float wi;
        if (!place_coords(c, in, i, p, wi)) continue;
        const uint32_t slot = atomicAdd(cursor + primary_tile(c, p) * c.cstride, 1u);
        if (!list.ent) {
            list.perm[slot] = (uint32_t)i;
            continue;
        }
        if (c.uniform)
            wi = wi / (float)__ldg(density + (int64_t)nearest_cell(c, p.pv) * c.n + nearest_cell(c, p.pu));
        list.ent[slot] = make_float4(p.pu, p.pv, wi, __uint_as_float((uint32_t)i | (p.conj ? 0x80000000u : 0u)));
        list.plane[slot] = p.k;
    }
}

// The list in its scratch of primary_list_bytes(m, with_entries).
PrimaryList primary_list(void* p, int64_t m, bool with_entries)
{
    if (!with_entries) return PrimaryList{nullptr, nullptr, static_cast<uint32_t*>(p)};
    float4* ent = static_cast<float4*>(p);
    return PrimaryList{ent, reinterpret_cast<int*>(ent + m), nullptr};
}

// Lanes that gather one measurement in k_degrid_gather: one per footprint
// column (supports 4, 7 and 8: gather_by_columns).
template <int S>
__host__ __device__ constexpr int gather_lanes()
{
    return S <= 4 ? 4 : 8;
}

// Each sorted measurement of planes [k0, k0+nk) gathers its S x S footprint
// of the (forward-transformed) adjoint planes with the gridding taps, times
// its effective weight.  A warp takes 32 consecutive measurements, one per
// lane; groups of L lanes then gather them one after another, a lane per
// footprint column: a row of a footprint is one contiguous read of S cells, and
// the lane keeps its column's tap polynomial in registers.  With a lane per
// measurement every read of the warp touched up to 32 lines (one pass of the
// load pipe each); consecutive measurements lie in the same tile, so the
// footprints overlap in L1.  1e7 measurements of support 7 on 4096^2 x 32
// planes: 1.07 -> 0.55 ms (a copy of each tile in shared memory and a lane per
// measurement: 1.04); reading the inputs through the list of indices instead
// of sorted entries costs 0.41 ms more here, and 0.11 less in the scatter.
template <int S>
__global__ void __launch_bounds__(kPrepThreads) k_degrid_gather(GridCfg c, PrimaryList list,
                                                                const uint32_t* __restrict__ off, int k0, int nk,
                                                                const float2* __restrict__ planes, Inputs in,
                                                                const uint32_t* __restrict__ density,
                                                                float2* __restrict__ grad)
{
    constexpr int L = gather_lanes<S>();
    const uint32_t full = 0xffffffffu;
    const int lane = threadIdx.x & 31, q = lane & (L - 1);
    // the tap polynomial of column (and row) q, with the checkerboard sign of odd taps
    float coef[kPolyTerms];
#pragma unroll
    for (int j = 0; j < kPolyTerms; ++j) {
        coef[j] = 0.f;
#pragma unroll
        for (int t = 0; t < S; ++t)
            if (t == q) coef[j] = (t & 1) ? -c.coef[t][j] : c.coef[t][j];
    }
    // measurements whose planes reach [k0, k0 + nk): sort key plane in
    // [k0 - Sw + 1, k0 + nk) (a contiguous run of the sorted list)
    const int klo = k0 - (c.Sw - 1) > 0 ? k0 - (c.Sw - 1) : 0;
    const uint32_t b = off[(int64_t)klo * c.ntp], e = off[(int64_t)(k0 + nk) * c.ntp];
    for (uint64_t j0 = (uint64_t)b + (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x - lane); j0 < e;
         j0 += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t j = j0 + lane;
        bool valid = j < e;
        Place p;
        p.pu = p.pv = c.half_s;
        p.k = -c.Sw;  // on no plane
        p.conj = false;
        p.pw = 0.f;
        float wi = 0.f;
        uint32_t i = 0;
        if (valid) {
            if (list.ent) {
                const float4 x = __ldg(list.ent + j);
                p.pu = x.x;
                p.pv = x.y;
                wi = x.z;
                i = __float_as_uint(x.w) & 0x7fffffffu;
                p.conj = (__float_as_uint(x.w) >> 31) != 0;
                p.k = __ldg(list.plane + j);
                if (c.Sw > 1) {
                    const float w = __ldg(in.w + i);
                    p.pw = __fsub_rn(__fmul_rn(__fsub_rn(p.conj ? -w : w, c.wmin), c.invdw), 0.5f);
                }
            } else {
                i = __ldg(list.perm + j);
                valid = place_coords(c, in, i, p, wi);  // always: the list holds placed ones
                if (c.uniform)
                    wi = wi / (float)__ldg(density + (int64_t)nearest_cell(c, p.pv) * c.n + nearest_cell(c, p.pu));
            }
        }
        p.fu = first_cell(c, p.pu);
        p.fv = first_cell(c, p.pv);
        // its planes in this group: the one plane (Sw = 1), or the w-footprint
        // with the normalised w-taps (Sw > 1)
        const float hn = c.Sw > 1 && valid ? w_tap_norm(c, p) : 1.0f;
        float ar = 0.f, ai = 0.f;
        for (int tw = 0; tw < c.Sw; ++tw) {
            const int plane = p.k + tw;
            const bool act = valid && plane >= k0 && plane < k0 + nk;
            if (!__any_sync(full, act)) continue;
            const int kl = act ? plane - k0 : -1;
            float cr = 0.f, ci = 0.f;
#pragma unroll 2
            for (int s = 0; s < L; ++s) {
                const float pu = __shfl_sync(full, p.pu, s, L), pv = __shfl_sync(full, p.pv, s, L);
                const int k = __shfl_sync(full, kl, s, L);
                const int fu = first_cell(c, pu), fv = first_cell(c, pv);
                float2 x[S];
#pragma unroll
                for (int rr = 0; rr < S; ++rr) x[rr] = make_float2(0.f, 0.f);
                if (k >= 0 && q < S) {
                    const float2* P = planes + (int64_t)k * c.n * c.n + fu + q;
#pragma unroll
                    for (int rr = 0; rr < S; ++rr) x[rr] = __ldg(P + (int64_t)plane_row(c, fv + rr) * c.n);
                }
                const float zu = __fmaf_rn(2.0f, __fsub_rn(__fsub_rn(pu, c.half_s), (float)(fu - 1)), -1.0f);
                const float zv = __fmaf_rn(2.0f, __fsub_rn(__fsub_rn(pv, c.half_s), (float)(fv - 1)), -1.0f);
                float gu = coef[kPolyTerms - 1], gv = coef[kPolyTerms - 1];
#pragma unroll
                for (int jj = kPolyTerms - 2; jj >= 0; --jj) {
                    gu = __fmaf_rn(gu, zu, coef[jj]);
                    gv = __fmaf_rn(gv, zv, coef[jj]);
                }
                float br = 0.f, bi = 0.f;
#pragma unroll
                for (int rr = 0; rr < S; ++rr) {
                    const float g = __shfl_sync(full, gv, rr, L);
                    br = fmaf(g, x[rr].x, br);
                    bi = fmaf(g, x[rr].y, bi);
                }
                br *= gu;
                bi *= gu;
#pragma unroll
                for (int o = L / 2; o > 0; o >>= 1) {
                    br += __shfl_xor_sync(full, br, o);
                    bi += __shfl_xor_sync(full, bi, o);
                }
                if (q == s) {
                    cr = br;
                    ci = bi;
                }
            }
            const float ht = c.Sw > 1 && act ? w_kernel(c, __fsub_rn((float)plane, p.pw)) * hn : 1.0f;
            ar = fmaf(ht, cr, ar);
            ai = fmaf(ht, ci, ai);
        }
        if (!valid) continue;
        float scale = wi / (tap_sum(c, p.pu, p.fu) * tap_sum(c, p.pv, p.fv));
        if ((p.fu + p.fv) & 1) scale = -scale;
        // a mirrored measurement enters as conj(V): its gradient is conjugated
        const float2 gi = make_float2(ar * scale, p.conj ? -ai * scale : ai * scale);
        if (c.Sw == 1) {
            grad[i] = gi;
        } else {  // a w-footprint can span plane groups: add this group's part
            const float2 prev = grad[i];
            grad[i] = make_float2(prev.x + gi.x, prev.y + gi.y);
        }
    }
}

// Each sorted measurement of planes [k0, k0+nk) gathers its S x S footprint
// of the (forward-transformed) adjoint planes with the gridding taps, times
// its effective weight, one thread per measurement, the taps summed row by
// row.  For kernels whose grid correction amplifies rounding (kGatherAmp):
// there the sum of a footprint cancels to far below its terms, and another
// order of summation is another result; and where gather_by_columns measured
// it the faster one.
template <int S>
__global__ void __launch_bounds__(kPrepThreads) k_degrid_gather_rows(GridCfg c, const uint32_t* __restrict__ perm,
                                                                     const uint32_t* __restrict__ off, int k0, int nk,
                                                                const float2* __restrict__ planes, Inputs in,
                                                                const uint32_t* __restrict__ density,
                                                                float2* __restrict__ grad)
{
    // measurements whose planes reach [k0, k0 + nk): sort key plane in
    // [k0 - Sw + 1, k0 + nk) (a contiguous run of the sorted list)
    const int klo = k0 - (c.Sw - 1) > 0 ? k0 - (c.Sw - 1) : 0;
    const uint32_t b = off[(int64_t)klo * c.ntp], e = off[(int64_t)(k0 + nk) * c.ntp];
    for (int64_t j = b + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < e;
         j += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t i = perm[j];
        Place p;
        float wi;
        if (!place_coords(c, in, i, p, wi)) continue;  // cannot happen: perm holds placed ones
        if (c.uniform) wi = wi / (float)__ldg(density + (int64_t)nearest_cell(c, p.pv) * c.n + nearest_cell(c, p.pu));
        float gu[S], gv[S];
        eval_taps<S>(c, p.pu, p.fu, gu);
        eval_taps<S>(c, p.pv, p.fv, gv);
        float su = 0.f, sv = 0.f;
#pragma unroll
        for (int t = 0; t < S; ++t) {
            su += gu[t];
            sv += gv[t];
        }
#pragma unroll
        for (int t = 1; t < S; t += 2) {
            gu[t] = -gu[t];
            gv[t] = -gv[t];
        }
        // its planes in this group: the one plane (Sw = 1), or the w-footprint
        // with the normalised w-taps (Sw > 1)
        const float hn = c.Sw > 1 ? w_tap_norm(c, p) : 1.0f;
        float ar = 0.f, ai = 0.f;
        for (int tw = 0; tw < c.Sw; ++tw) {
            const int plane = p.k + tw;
            if (plane < k0 || plane >= k0 + nk) continue;
            const float ht = c.Sw > 1 ? w_kernel(c, __fsub_rn((float)plane, p.pw)) * hn : 1.0f;
            const float2* P = planes + (int64_t)(plane - k0) * c.n * c.n + p.fu;
            float cr = 0.f, ci = 0.f;
#pragma unroll
            for (int rr = 0; rr < S; ++rr) {
                const float2* R = P + (int64_t)plane_row(c, p.fv + rr) * c.n;
                float br = 0.f, bi = 0.f;
#pragma unroll
                for (int t = 0; t < S; ++t) {
                    const float2 x = __ldg(R + t);
                    br = fmaf(gu[t], x.x, br);
                    bi = fmaf(gu[t], x.y, bi);
                }
                cr = fmaf(gv[rr], br, cr);
                ci = fmaf(gv[rr], bi, ci);
            }
            ar = fmaf(ht, cr, ar);
            ai = fmaf(ht, ci, ai);
        }
        float scale = wi / (su * sv);
        if ((p.fu + p.fv) & 1) scale = -scale;
        // a mirrored measurement enters as conj(V): its gradient is conjugated
        const float2 gi = make_float2(ar * scale, p.conj ? -ai * scale : ai * scale);
        if (c.Sw == 1) {
            grad[i] = gi;
        } else {  // a w-footprint can span plane groups: add this group's part
            const float2 prev = grad[i];
            grad[i] = make_float2(prev.x + gi.x, prev.y + gi.y);
        }
    }
}

// ------------------------------------------------------------------ scan

// Exclusive scan of one value per thread across a 1024-thread block.
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* total)
{
    __shared__ uint32_t ws[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t x = v;
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) ws[wid] = x;
    __syncthreads();
    if (wid == 0) {
        uint32_t t = ws[lane];
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        ws[lane] = t;
    }
    __syncthreads();
    const uint32_t prefix = wid ? ws[wid - 1] : 0u;
    *total = ws[31];
    __syncthreads();
    return prefix + x - v;
}

__global__ void __launch_bounds__(kScanBlock) k_scan_local(const uint32_t* __restrict__ in, int64_t len,
                                                           int stride, uint32_t* __restrict__ out,
                                                           uint32_t* __restrict__ block_sums)
{
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    uint32_t x[kScanItems];
    uint32_t s = 0;
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        x[j] = (base + j < len) ? in[(base + j) * stride] : 0u;
        s += x[j];
    }
    uint32_t total;
    uint32_t run = block_exclusive_scan(s, &total);
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        if (base + j < len) out[base + j] = run;
        run += x[j];
    }
    if (threadIdx.x == 0) block_sums[blockIdx.x] = total;
}

// Exclusive scan of the block totals in place (one block, any length), and
// the grand total into out[len].
__global__ void __launch_bounds__(kScanBlock) k_scan_sums(uint32_t* __restrict__ sums, int64_t nb,
                                                          uint32_t* __restrict__ out, int64_t len)
{
    uint32_t carry = 0;
    for (int64_t s0 = 0; s0 < nb; s0 += kScanBlock) {
        const int64_t i = s0 + threadIdx.x;
        const uint32_t v = (i < nb) ? sums[i] : 0u;
        uint32_t total;
        const uint32_t ex = block_exclusive_scan(v, &total);
        if (i < nb) sums[i] = carry + ex;
        carry += total;
    }
    if (threadIdx.x == 0) out[len] = carry;
}

__global__ void __launch_bounds__(kScanBlock) k_scan_add(const uint32_t* __restrict__ sums, int64_t len,
                                                         int stride, uint32_t* __restrict__ out,
                                                         uint32_t* __restrict__ cursor)
{
    const uint32_t add = sums[blockIdx.x];
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
#pragma unroll
    for (int j = 0; j < kScanItems; ++j) {
        if (base + j < len) {
            const uint32_t o = out[base + j] + add;
            out[base + j] = o;
            cursor[(base + j) * stride] = o;
        }
    }
}

// The whole scan in one launch for up to kScanMax counters: one thread-block
// cluster, each CTA a run of `per` counters (a multiple of kScanTile) in
// registers; the CTAs exchange their totals through distributed shared memory,
// which a CTA may write only once the owner is known to run: every CTA arrives
// at the cluster's barrier at its start and waits for it ahead of the stores
// (by then the loads and the block scan have covered the wait).  `in` and
// `cursor` may be the same array: every thread reads its counters before it
// writes them, and neither pointer is declared free of aliases.
// The sort of 1e5 measurements into 512 tiles took 35 us with three launches
// for the scan and takes 28 with one.  Eight SMs fall behind beyond kScanMax: the
// sort of 5e5 with three launches and with one takes 51 and 44.5 us for 16384
// tiles, 50.4 and 44 for 32768, 50.5 and 50 for 49152, 50.4 and 50.3 for 65536, and
// took 54.8 and 65 for 105300 and 131072.
constexpr int kScanCluster = 8;
constexpr int kScanSub = 2;  // tiles of kScanTile counters per CTA at most
constexpr int64_t kScanMax = (int64_t)kScanCluster * kScanSub * kScanTile;

__global__ void __cluster_dims__(kScanCluster, 1, 1) __launch_bounds__(kScanBlock)
    k_scan_one(const uint32_t* in, int len, int stride, int subs, uint32_t* __restrict__ out, uint32_t* cursor)
{
    __shared__ uint32_t s_total[kScanCluster];
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    const int rank = blockIdx.x, base = rank * subs * kScanTile + threadIdx.x * kScanItems;
    uint32_t x[kScanSub][kScanItems], run[kScanSub];
#pragma unroll
    for (int q = 0; q < kScanSub; ++q)
#pragma unroll
        for (int j = 0; j < kScanItems; ++j) {
            const int i = base + q * kScanTile + j;
            x[q][j] = q < subs && i < len ? in[(int64_t)i * stride] : 0u;
        }
    uint32_t carry = 0;
#pragma unroll
    for (int q = 0; q < kScanSub; ++q) {
        if (q < subs) {  // the same in every thread
            uint32_t s = 0, total;
#pragma unroll
            for (int j = 0; j < kScanItems; ++j) s += x[q][j];
            run[q] = carry + block_exclusive_scan(s, &total);
            carry += total;
        }
    }
    // this CTA's total into every CTA's s_total, once all of them run
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (threadIdx.x < kScanCluster) {
        uint32_t dst;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                     : "=r"(dst)
                     : "r"((uint32_t)__cvta_generic_to_shared(s_total + rank)), "r"(threadIdx.x));
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(dst), "r"(carry) : "memory");
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    uint32_t before = 0;
    for (int r = 0; r < rank; ++r) before += s_total[r];
#pragma unroll
    for (int q = 0; q < kScanSub; ++q) {
        if (q >= subs) break;
        uint32_t o = before + run[q];
#pragma unroll
        for (int j = 0; j < kScanItems; ++j) {
            const int i = base + q * kScanTile + j;
            if (i < len) {
                out[i] = o;
                cursor[(int64_t)i * stride] = o;
            }
            o += x[q][j];
        }
    }
    if (rank == kScanCluster - 1 && threadIdx.x == 0) out[len] = before + carry;
}

}  // namespace

cudaError_t launch_primary_count(const GridCfg& c, const float* u, const float* v, const float* w,
                                 const float* wt, int64_t m, uint32_t* counts, cudaStream_t s)
{
    if (m <= 0) return cudaSuccess;
    k_primary_count<<<prep_blocks(m), kPrepThreads, 0, s>>>(c, Inputs{u, v, w, wt, nullptr}, m, counts);
    return cudaGetLastError();
}

cudaError_t launch_primary_scatter(const GridCfg& c, const float* u, const float* v, const float* w,
                                   const float* wt, int64_t m, const uint32_t* density, uint32_t* cursor,
                                   void* list, bool with_entries, cudaStream_t s)
{
    if (m <= 0) return cudaSuccess;
    k_primary_scatter<<<prep_blocks(m), kPrepThreads, 0, s>>>(c, Inputs{u, v, w, wt, nullptr}, m, density, cursor,
                                                              primary_list(list, m, with_entries));
    return cudaGetLastError();
}

template <int S>
cudaError_t launch_gather_rows_s(const GridCfg& c, const uint32_t* perm, const uint32_t* off, int k0, int nk,
                                 const float2* planes, const Inputs& in, const uint32_t* density, float2* grad,
                                 cudaStream_t s)
{
    // the launch is sized for the whole input; threads beyond the group's range exit at once
    const int64_t m = (int64_t)sm_count() * 8 * kPrepThreads;
    k_degrid_gather_rows<S><<<prep_blocks(m), kPrepThreads, 0, s>>>(c, perm, off, k0, nk, planes, in, density, grad);
    return cudaGetLastError();
}

template <int S>
cudaError_t launch_gather_s(const GridCfg& c, const PrimaryList& list, const uint32_t* off, int k0, int nk,
                            const float2* planes, const Inputs& in, const uint32_t* density, float2* grad,
                            int64_t m, cudaStream_t s)
{
    // blocks beyond the group's run of the list exit at once
    k_degrid_gather<S><<<prep_blocks(m), kPrepThreads, 0, s>>>(c, list, off, k0, nk, planes, in, density, grad);
    return cudaGetLastError();
}

// Whether k_degrid_gather (a lane per footprint column) is to gather m
// measurements per launch (a plane group's share of a call's), and
// k_degrid_gather_rows otherwise: supports that fill its groups of 4 or 8 lanes,
// and lists that fill the chip's warps, each of which takes 32 measurements one
// group step after another.  Predictions, row by row and by columns, us: support
// 8 at 2000^2 x 8 planes, 5e4 measurements 350 and 349, 3e5 378 and 374, 6e6 973
// and 861, at 512^2 5e4 71 and 79, 3e5 97 and 96, 6e6 771 and 681; support 4 at
// 2000^2 6e6 785 and 693.  Lanes without a column cost what the kernel gains:
// support 6 at 512^2, 3e5 85 and 100, 6e6 610 and 631; support 9 at 2000^2 6e6 1069
// and 1184; support 12 1403 and 1350 there, but 411 and 432 at 3e5.  Per launch:
// 1.1e6 measurements of support 7 at 256^2 x 43 planes take 403 and 485 in groups
// of 3 planes (7.7e4 each), 148 by columns and 158 by rows in one.
bool gather_by_columns(const GridCfg& c, int64_t m)
{
    return (c.S == 4 || c.S == 7 || c.S == 8) && m >= ((int64_t)1 << 18);
}

cudaError_t launch_degrid_gather(const GridCfg& c, void* list, bool with_entries, bool by_rows, int64_t m,
                                 const uint32_t* offsets, int k0, int nk, const float2* planes, const float* u, const float* v, const float* w,
                                 const float* wt, const uint32_t* density, float2* grad, cudaStream_t s)
{
    if (m <= 0) return cudaSuccess;
    if (by_rows && with_entries) return cudaErrorInvalidValue;  // takes the indices
    const Inputs in{u, v, w, wt, nullptr};
    const PrimaryList pl = primary_list(list, m, with_entries);
    if (!by_rows) {
        switch (c.S) {
            case 4: return launch_gather_s<4>(c, pl, offsets, k0, nk, planes, in, density, grad, m, s);
            case 7: return launch_gather_s<7>(c, pl, offsets, k0, nk, planes, in, density, grad, m, s);
            case 8: return launch_gather_s<8>(c, pl, offsets, k0, nk, planes, in, density, grad, m, s);
            default: return cudaErrorInvalidValue;
        }
    }
    switch (c.S) {
#define RICK_GATHER_CASE(SS) \
    case SS:                       \
        return launch_gather_rows_s<SS>(c, pl.perm, offsets, k0, nk, planes, in, density, grad, s);
        RICK_GATHER_CASE(1) RICK_GATHER_CASE(2) RICK_GATHER_CASE(3) RICK_GATHER_CASE(4)
        RICK_GATHER_CASE(5) RICK_GATHER_CASE(6) RICK_GATHER_CASE(7) RICK_GATHER_CASE(8)
        RICK_GATHER_CASE(9) RICK_GATHER_CASE(10) RICK_GATHER_CASE(11) RICK_GATHER_CASE(12)
        RICK_GATHER_CASE(13) RICK_GATHER_CASE(14) RICK_GATHER_CASE(15) RICK_GATHER_CASE(16)
#undef RICK_GATHER_CASE
        default: return cudaErrorInvalidValue;
    }
}

size_t primary_list_bytes(int64_t m, bool with_entries)
{
    return (size_t)m * (with_entries ? sizeof(float4) + sizeof(int) : sizeof(uint32_t));
}

size_t scan_block_sums_len(int64_t len)
{
    return (size_t)((len + kScanTile - 1) / kScanTile) + 1;
}

cudaError_t launch_density(const GridCfg& c, const float* u, const float* v, const float* w,
                           const float* wt, const float2* vis, int64_t m, uint32_t* density,
                           cudaStream_t s)
{
    if (m <= 0) return cudaSuccess;
    k_density<<<prep_blocks(m), kPrepThreads, 0, s>>>(c, Inputs{u, v, w, wt, vis}, m, density);
    return cudaGetLastError();
}

cudaError_t launch_count(const GridCfg& c, const float* u, const float* v, const float* w,
                         const float* wt, const float2* vis, int64_t m, uint32_t* counts,
                         cudaStream_t s)
{
    if (m <= 0) return cudaSuccess;
    k_count<<<prep_blocks(m, c.prep_bpsm), kPrepThreads, 0, s>>>(c, Inputs{u, v, w, wt, vis}, m, counts);
    return cudaGetLastError();
}

int scan_launches(int64_t len) { return len <= 0 ? 0 : len <= kScanMax ? 1 : 3; }

cudaError_t launch_scan(const uint32_t* counts, int64_t len, int stride, uint32_t* offsets, uint32_t* cursor,
                        uint32_t* block_sums, cudaStream_t s)
{
    const int64_t nb = (len + kScanTile - 1) / kScanTile;
    if (nb > 0x7fffffff) return cudaErrorInvalidValue;
    if (nb == 0) return cudaMemsetAsync(offsets, 0, sizeof(uint32_t), s);
    if (len <= kScanMax) {
        const int subs = (int)((len + kScanCluster * kScanTile - 1) / (kScanCluster * kScanTile));
        k_scan_one<<<kScanCluster, kScanBlock, 0, s>>>(counts, (int)len, stride, subs, offsets, cursor);
        return cudaGetLastError();
    }
    k_scan_local<<<(unsigned)nb, kScanBlock, 0, s>>>(counts, len, stride, offsets, block_sums);
    k_scan_sums<<<1, kScanBlock, 0, s>>>(block_sums, nb, offsets, len);
    k_scan_add<<<(unsigned)nb, kScanBlock, 0, s>>>(block_sums, len, stride, offsets, cursor);
    return cudaGetLastError();
}

cudaError_t launch_scatter(const GridCfg& c, const float* u, const float* v, const float* w,
                           const float* wt, const float2* vis, int64_t m, const uint32_t* density,
                           uint32_t* cursor, float4* entries, Counters* ctr, double* chan_sw, cudaStream_t s)
{
    if (m <= 0) return cudaSuccess;
    k_scatter<<<prep_blocks(m, c.prep_bpsm), kPrepThreads, 0, s>>>(c, Inputs{u, v, w, wt, vis}, m, density, cursor,
                                                      entries, ctr, chan_sw ? chan_sw : &ctr->sum_w);
    return cudaGetLastError();
}

}  // namespace rick
