// Data restructuring of Phi on the device (Sec. 4.1.2): validation, sort by a
// packed (v, a, f) key, duplicate merge, and the layouts the SpMV kernels stream.
#include <algorithm>
#include <cstdarg>

#include "life_internal.cuh"

namespace life {

// ------------------------------------------------------------------ scans

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

// Block-wide exclusive scan of one 2048-element tile; writes the tile total.
__global__ void scan_tile_kernel(const int32_t* __restrict__ in, int32_t* __restrict__ out, int64_t n,
                                 int32_t* __restrict__ tile_sums) {
    __shared__ int32_t warp_tot[SCAN_THREADS / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)tid * SCAN_ITEMS;
    int32_t v[SCAN_ITEMS];
    // a thread's 8 consecutive items as two 16-byte accesses where the whole tile exists
    const bool vec = base + SCAN_ITEMS <= n &&
                     ((reinterpret_cast<uintptr_t>(in) | reinterpret_cast<uintptr_t>(out)) & 15) == 0;
    if (vec) {
        const int4 p = *reinterpret_cast<const int4*>(in + base), q = *reinterpret_cast<const int4*>(in + base + 4);
        v[0] = p.x; v[1] = p.y; v[2] = p.z; v[3] = p.w;
        v[4] = q.x; v[5] = q.y; v[6] = q.z; v[7] = q.w;
    } else {
#pragma unroll
        for (int i = 0; i < SCAN_ITEMS; ++i) v[i] = base + i < n ? in[base + i] : 0;
    }
    int32_t run = 0;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        const int32_t t = v[i];
        v[i] = run;
        run += t;
    }
    // inclusive warp scan of per-thread totals
    int32_t x = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int32_t t = lane < SCAN_THREADS / 32 ? warp_tot[lane] : 0;
        int32_t s = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int32_t y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        if (lane < SCAN_THREADS / 32) warp_tot[lane] = s - t;  // exclusive
        if (lane == SCAN_THREADS / 32 - 1 && tile_sums) tile_sums[blockIdx.x] = s;
    }
    __syncthreads();
    const int32_t offset = warp_tot[warp] + (x - run);
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) v[i] += offset;
    if (vec) {
        *reinterpret_cast<int4*>(out + base) = make_int4(v[0], v[1], v[2], v[3]);
        *reinterpret_cast<int4*>(out + base + 4) = make_int4(v[4], v[5], v[6], v[7]);
        return;
    }
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i)
        if (base + i < n) out[base + i] = v[i];
}

__global__ void scan_add_kernel(int32_t* __restrict__ out, int64_t n, const int32_t* __restrict__ tile_off) {
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
    const int32_t add = tile_off[blockIdx.x];
    for (int i = threadIdx.x; i < SCAN_TILE; i += blockDim.x) {
        int64_t idx = base + i;
        if (idx < n) out[idx] += add;
    }
}

life_status exclusive_scan_i32(const int32_t* in, int32_t* out, int64_t n, cudaStream_t s) {
    if (n <= 0) return LIFE_OK;
    const int64_t tiles = (n + SCAN_TILE - 1) / SCAN_TILE;
    if (tiles == 1) {
        scan_tile_kernel<<<1, SCAN_THREADS, 0, s>>>(in, out, n, nullptr);
        LIFE_CHECK_LAUNCH();
        return LIFE_OK;
    }
    TmpBuf sums, sums_scan;
    LIFE_TRY(sums.alloc(sizeof(int32_t) * tiles, s));
    LIFE_TRY(sums_scan.alloc(sizeof(int32_t) * tiles, s));
    scan_tile_kernel<<<(unsigned)tiles, SCAN_THREADS, 0, s>>>(in, out, n, sums.as<int32_t>());
    LIFE_CHECK_LAUNCH();
    LIFE_TRY(exclusive_scan_i32(sums.as<int32_t>(), sums_scan.as<int32_t>(), tiles, s));
    scan_add_kernel<<<(unsigned)tiles, SCAN_THREADS, 0, s>>>(out, n, sums_scan.as<int32_t>());
    LIFE_CHECK_LAUNCH();
    return LIFE_OK;
}

// ------------------------------------------------------------- radix sort
// Stable LSD radix sort of (uint64 key, uint32 payload) pairs by the key bits
// [bit0, bit1), in digits of at most 8 bits.  Each pass: per-tile digit histograms
// (digit-major), an exclusive scan of the histograms, and a stable scatter ranked
// with warp match + per-warp counters.
//
// A pass is bound by memory: 12 B per pair read and written, 8 B more read by the
// histograms.  The scatter orders its tile by digit in shared memory before it
// writes, so that a warp writes a few runs of consecutive pairs instead of 32
// scattered ones (32-byte sectors of which 12 B were used): 6144 pairs a tile give
// runs of 24 pairs at 8 bits, 48 at 7, and two CTAs of 512 threads share an SM.
// A new index of the paper-scale workload (80M entries, BF16 storage) with its first
// DSC and WC took 80.0 ms with 22 passes of an unstaged scatter (1.9 ms each), 44.0 ms
// with this one, 16 passes (the callers sort only the bits that are not in order yet)
// and the merge below in two passes; 16.4 ms since the tile layout is counted.

constexpr int RS_THREADS = 512;
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_ROUNDS = 12;                     // items per lane (16 spill: the paper-scale build alone 14.7 ms, 14.1 with 12)
constexpr int RS_TILE = RS_THREADS * RS_ROUNDS;   // 6144 items per block
constexpr int RS_DIGITS = 256;
constexpr int RS_COPIES = 8;                      // histogram copies: two warps add to each
constexpr size_t RS_SMEM = (size_t)RS_TILE * 12 + sizeof(uint16_t) * RS_WARPS * RS_DIGITS;

__global__ void __launch_bounds__(RS_THREADS) rs_hist_kernel(const uint64_t* __restrict__ keys, int64_t n, int shift,
                                                             uint32_t mask, int32_t* __restrict__ hist, int nblocks) {
    __shared__ int32_t h[RS_COPIES][RS_DIGITS];
    for (int i = threadIdx.x; i < RS_COPIES * RS_DIGITS; i += RS_THREADS) (&h[0][0])[i] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * RS_TILE;
    int32_t* hw = h[(threadIdx.x >> 5) % RS_COPIES];
#pragma unroll
    for (int i = 0; i < RS_ROUNDS; ++i) {
        const int64_t idx = base + (int64_t)i * RS_THREADS + threadIdx.x;
        if (idx < n) atomicAdd(&hw[(uint32_t)(keys[idx] >> shift) & mask], 1);
    }
    __syncthreads();
    if (threadIdx.x <= mask) {
        int32_t t = 0;
#pragma unroll
        for (int c = 0; c < RS_COPIES; ++c) t += h[c][threadIdx.x];
        hist[(int64_t)threadIdx.x * nblocks + blockIdx.x] = t;
    }
}

__global__ void __launch_bounds__(RS_THREADS, 2)
rs_scatter_kernel(const uint64_t* __restrict__ kin, const uint32_t* __restrict__ vin, uint64_t* __restrict__ kout,
                  uint32_t* __restrict__ vout, int64_t n, int shift, uint32_t mask,
                  const int32_t* __restrict__ offs, int nblocks) {
    extern __shared__ __align__(16) unsigned char rs_smem[];
    uint64_t* sk = reinterpret_cast<uint64_t*>(rs_smem);
    uint32_t* sv = reinterpret_cast<uint32_t*>(sk + RS_TILE);
    uint16_t* wcnt = reinterpret_cast<uint16_t*>(sv + RS_TILE);  // [warp][digit]: at most 384 items a warp
    __shared__ int32_t gofs[RS_DIGITS], wtot[RS_DIGITS / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int i = tid; i < RS_WARPS * RS_DIGITS / 2; i += RS_THREADS) reinterpret_cast<uint32_t*>(wcnt)[i] = 0u;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * RS_TILE;
    const int64_t wbase = base + (int64_t)warp * (32 * RS_ROUNDS) + lane;
    const int count = (int)min((int64_t)RS_TILE, n - base);
    const unsigned lt_mask = (1u << lane) - 1u;
    uint16_t* cnt = wcnt + warp * RS_DIGITS;
    uint64_t k[RS_ROUNDS];
    uint16_t r[RS_ROUNDS];
#pragma unroll
    for (int j = 0; j < RS_ROUNDS; ++j) k[j] = wbase + 32 * j < n ? kin[wbase + 32 * j] : 0ull;
#pragma unroll
    for (int j = 0; j < RS_ROUNDS; ++j) {
        const bool valid = wbase + 32 * j < n;
        const uint32_t d = valid ? (uint32_t)(k[j] >> shift) & mask : (uint32_t)RS_DIGITS;
        const unsigned peers = __match_any_sync(0xffffffffu, d);
        const uint32_t cnt0 = valid ? cnt[d] : 0u;
        __syncwarp();
        if (valid && lane == __ffs(peers) - 1) cnt[d] = (uint16_t)(cnt0 + __popc(peers));
        __syncwarp();
        r[j] = (uint16_t)(cnt0 + __popc(peers & lt_mask));
    }
    __syncthreads();
    int32_t run = 0, incl = 0;
    if (tid < RS_DIGITS) {
        // per digit: exclusive prefix over the warps, then over the digits
#pragma unroll
        for (int w = 0; w < RS_WARPS; ++w) {
            const int32_t t = wcnt[w * RS_DIGITS + tid];
            wcnt[w * RS_DIGITS + tid] = (uint16_t)run;
            run += t;
        }
        incl = run;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) wtot[warp] = incl;
    }
    __syncthreads();
    if (tid < RS_DIGITS) {
        int32_t loc = incl - run;
        for (int w = 0; w < warp; ++w) loc += wtot[w];
#pragma unroll
        for (int w = 0; w < RS_WARPS; ++w) wcnt[w * RS_DIGITS + tid] = (uint16_t)(wcnt[w * RS_DIGITS + tid] + loc);
        gofs[tid] = (uint32_t)tid <= mask ? offs[(int64_t)tid * nblocks + blockIdx.x] - loc : 0;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < RS_ROUNDS; ++j) {
        if (wbase + 32 * j < n) {
            const int p = cnt[(uint32_t)(k[j] >> shift) & mask] + r[j];
            sk[p] = k[j];
            sv[p] = vin[wbase + 32 * j];
        }
    }
    __syncthreads();
#pragma unroll 4
    for (int i = tid; i < count; i += RS_THREADS) {
        const uint64_t key = sk[i];
        const int64_t pos = (int64_t)gofs[(uint32_t)(key >> shift) & mask] + i;
        kout[pos] = key;
        vout[pos] = sv[i];
    }
}

// Sorts n pairs by the key bits [bit0, bit1); keys and vals are exchanged for
// buffers of the same size when the number of passes is odd.
life_status radix_sort_pairs(TmpBuf& keys, TmpBuf& vals, int64_t n, int bit0, int bit1, cudaStream_t s) {
    if (n <= 1 || bit1 <= bit0) return LIFE_OK;
    if (n >= (int64_t)INT32_MAX) {
        set_error("radix sort: %lld items exceed the int32 position range", (long long)n);
        return LIFE_ERANGE;
    }
    const int nblocks = (int)((n + RS_TILE - 1) / RS_TILE);
    TmpBuf k2, v2, hist, offs;
    LIFE_TRY(k2.alloc(sizeof(uint64_t) * n, s));
    LIFE_TRY(v2.alloc(sizeof(uint32_t) * n, s));
    LIFE_TRY(hist.alloc(sizeof(int32_t) * RS_DIGITS * (int64_t)nblocks, s));
    LIFE_TRY(offs.alloc(sizeof(int32_t) * RS_DIGITS * (int64_t)nblocks, s));
    LIFE_CUDA_TRY(cudaFuncSetAttribute(rs_scatter_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RS_SMEM));
    const int bits = bit1 - bit0, passes = (bits + 7) / 8;
    for (int p = 0, shift = bit0; p < passes; ++p) {
        const int width = (bit1 - shift + passes - p - 1) / (passes - p);  // equal digits: 28 bits are 4 of 7
        const uint32_t mask = (1u << width) - 1u;
        rs_hist_kernel<<<nblocks, RS_THREADS, 0, s>>>(keys.as<uint64_t>(), n, shift, mask, hist.as<int32_t>(), nblocks);
        LIFE_CHECK_LAUNCH();
        LIFE_TRY(exclusive_scan_i32(hist.as<int32_t>(), offs.as<int32_t>(), ((int64_t)mask + 1) * nblocks, s));
        rs_scatter_kernel<<<nblocks, RS_THREADS, RS_SMEM, s>>>(keys.as<uint64_t>(), vals.as<uint32_t>(),
                                                               k2.as<uint64_t>(), v2.as<uint32_t>(), n, shift, mask,
                                                               offs.as<int32_t>(), nblocks);
        LIFE_CHECK_LAUNCH();
        keys.swap(k2);
        vals.swap(v2);
        shift += width;
    }
    return LIFE_OK;
}

// ------------------------------------------------------------ validation

static inline int nbits(int64_t n) {
    if (n <= 1) return 0;
    uint64_t x = (uint64_t)(n - 1);
    int b = 0;
    while (x) { ++b; x >>= 1; }
    return b;
}

// Checks ranges and finiteness and packs key = v | a | f (v most significant); also
// tells whether the fascicle ids come in non-decreasing order (DEV_UNSORTED when
// not).  Four entries a thread, by 16-byte accesses where the arrays allow it.
__global__ void __launch_bounds__(256) pack_vaf_kernel(const int32_t* __restrict__ atom, const int32_t* __restrict__ voxel,
                                const int32_t* __restrict__ fasc, const float* __restrict__ val, int64_t n,
                                int32_t na, int32_t nv, int32_t nf, int sa, int sv, int vec, uint64_t* __restrict__ key,
                                uint32_t* __restrict__ payload, uint32_t* __restrict__ err) {
    const int64_t i0 = 4 * (blockIdx.x * (int64_t)blockDim.x + threadIdx.x);
    uint32_t bad = 0;
    if (i0 < n) {
        // (aligned: written and read 16 bytes at a time where they do not stay in registers)
        __align__(16) int32_t a[4], v[4], f[4];
        __align__(16) float x[4];
        const int m = (int)min((int64_t)4, n - i0);
        if (vec && m == 4) {
            *reinterpret_cast<int4*>(a) = __ldg(reinterpret_cast<const int4*>(atom + i0));
            *reinterpret_cast<int4*>(v) = __ldg(reinterpret_cast<const int4*>(voxel + i0));
            *reinterpret_cast<int4*>(f) = __ldg(reinterpret_cast<const int4*>(fasc + i0));
            *reinterpret_cast<float4*>(x) = __ldg(reinterpret_cast<const float4*>(val + i0));
        } else {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                a[e] = e < m ? atom[i0 + e] : 0;
                v[e] = e < m ? voxel[i0 + e] : 0;
                f[e] = e < m ? fasc[i0 + e] : 0;
                x[e] = e < m ? val[i0 + e] : 0.0f;
            }
        }
        int32_t fp = i0 > 0 ? __ldg(fasc + i0 - 1) : f[0];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            if (e >= m) break;
            if (a[e] < 0 || a[e] >= na || v[e] < 0 || v[e] >= nv || f[e] < 0 || f[e] >= nf) bad |= DEV_BAD_INDEX;
            else if (!isfinite(x[e])) bad |= DEV_BAD_VALUE;
            if (f[e] < fp) bad |= DEV_UNSORTED;
            fp = f[e];
        }
        uint64_t k[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) k[e] = ((uint64_t)v[e] << sv) | ((uint64_t)a[e] << sa) | (uint64_t)f[e];
        if (m == 4) {  // key and payload are 256-byte aligned allocations
            *reinterpret_cast<ulonglong2*>(key + i0) = make_ulonglong2(k[0], k[1]);
            *reinterpret_cast<ulonglong2*>(key + i0 + 2) = make_ulonglong2(k[2], k[3]);
            *reinterpret_cast<float4*>(payload + i0) = *reinterpret_cast<const float4*>(x);
        } else {
#pragma unroll
            for (int e = 0; e < 3; ++e) {  // (unrolled: the arrays stay in registers)
                if (e >= m) break;
                key[i0 + e] = k[e];
                payload[i0 + e] = __float_as_uint(x[e]);
            }
        }
    }
    if (bad & ~*reinterpret_cast<volatile uint32_t*>(err)) atomicOr(err, bad);
}

// Duplicate merge and the voxel layout, in two passes over the sorted keys, each
// block taking MG_TILE consecutive ones: the run heads of each block are counted,
// the counts scanned, and each head then writes its merged entry at its rank (a
// run of equal keys is summed in FP64 and rounded once), with the (v, a, f)
// streams and the CSR voxel pointer of the voxel layout.  The flags and their
// scan never reach memory, and the layout is written from the sorted keys.
constexpr int MG_THREADS = 256;
constexpr int MG_ROUNDS = 8;
constexpr int MG_TILE = MG_THREADS * MG_ROUNDS;

__global__ void __launch_bounds__(MG_THREADS) head_count_kernel(const uint64_t* __restrict__ key, int64_t n,
                                                                int32_t* __restrict__ count) {
    __shared__ int32_t total;
    if (threadIdx.x == 0) total = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * MG_TILE + threadIdx.x;
    int c = 0;
#pragma unroll
    for (int j = 0; j < MG_ROUNDS; ++j) {
        const int64_t i = base + (int64_t)j * MG_THREADS;
        c += __popc(__ballot_sync(0xffffffffu, i < n && (i == 0 || key[i] != key[i - 1])));
    }
    if ((threadIdx.x & 31) == 0) atomicAdd(&total, c);
    __syncthreads();
    if (threadIdx.x == 0) count[blockIdx.x] = total;
}

template <class VT>
__global__ void __launch_bounds__(MG_THREADS)
merge_layout_kernel(const uint64_t* __restrict__ key, const uint32_t* __restrict__ payload, int64_t n,
                    const int32_t* __restrict__ offset, int32_t m, int sa, int sv, uint64_t amask, uint64_t fmask,
                    int32_t nv, float* __restrict__ uval, uint16_t* __restrict__ atom16,
                    int32_t* __restrict__ fasc, VT* __restrict__ valout, int32_t* __restrict__ vox_ptr) {
    __shared__ int32_t wsum[MG_ROUNDS][MG_THREADS / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t base = (int64_t)blockIdx.x * MG_TILE + tid;
    uint64_t k[MG_ROUNDS], kp[MG_ROUNDS];
    uint32_t ball[MG_ROUNDS];
#pragma unroll
    for (int j = 0; j < MG_ROUNDS; ++j) {
        const int64_t i = base + (int64_t)j * MG_THREADS;
        k[j] = i < n ? key[i] : 0ull;
        kp[j] = (i > 0 && i < n) ? key[i - 1] : 0ull;
    }
#pragma unroll
    for (int j = 0; j < MG_ROUNDS; ++j) {
        const int64_t i = base + (int64_t)j * MG_THREADS;
        ball[j] = __ballot_sync(0xffffffffu, i < n && (i == 0 || k[j] != kp[j]));
        if (lane == 0) wsum[j][warp] = __popc(ball[j]);
    }
    __syncthreads();
    if (tid < 32) {  // exclusive scan of the 64 (round, warp) counts, two a lane
        int32_t* p = &wsum[0][0];
        const int32_t x0 = p[2 * lane], x1 = p[2 * lane + 1];
        int32_t incl = x0 + x1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        p[2 * lane] = incl - x0 - x1;
        p[2 * lane + 1] = incl - x1;
    }
    __syncthreads();
    const int32_t off = offset[blockIdx.x];
#pragma unroll
    for (int j = 0; j < MG_ROUNDS; ++j) {
        if (!((ball[j] >> lane) & 1u)) continue;
        const int64_t i = base + (int64_t)j * MG_THREADS;
        const int32_t pos = off + wsum[j][warp] + __popc(ball[j] & ((1u << lane) - 1u));
        double sum = (double)__uint_as_float(payload[i]);
        for (int64_t q = i + 1; q < n && key[q] == k[j]; ++q) sum += (double)__uint_as_float(payload[q]);
        const float x = (float)sum;
        const int32_t v = (int32_t)(k[j] >> sv);
        atom16[pos] = (uint16_t)((k[j] >> sa) & amask);
        fasc[pos] = (int32_t)(k[j] & fmask);
        if constexpr (sizeof(VT) == 2) {
            valout[pos] = __float2bfloat16_rn(x);
            uval[pos] = x;
        } else {
            valout[pos] = x;
        }
        const int32_t vp = i == 0 ? -1 : (int32_t)(kp[j] >> sv);
        for (int32_t q = vp + 1; q <= v; ++q) vox_ptr[q] = pos;
        if (pos == m - 1)
            for (int32_t q = v + 1; q <= nv; ++q) vox_ptr[q] = m;
    }
}

__global__ void fill_i32_kernel(int32_t* p, int64_t n, int32_t v) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) p[i] = v;
}

static unsigned grid_for(int64_t n, int threads = 256) {
    int64_t b = (n + threads - 1) / threads;
    int64_t cap = (int64_t)device_sm_count() * 32;
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (unsigned)b;
}

life_status build_voxel_layout(life_index_s* ix, const int32_t* atom, const int32_t* voxel, const int32_t* fasc,
                               const float* val, cudaStream_t s) {
    const int64_t n = ix->nnz_raw;
    const int ba = nbits(ix->na), bf = nbits(ix->nf), bv = nbits(ix->nv);
    if (ba + bf + bv > 64) {
        set_error("packed (v,a,f) key needs %d bits (> 64)", ba + bf + bv);
        return LIFE_ERANGE;
    }
    ix->key_bits_a = ba;
    ix->key_bits_f = bf;
    ix->key_bits_v = bv;
    const int sa = bf, sv = bf + ba;
    TmpBuf keys, pay, err;
    LIFE_TRY(keys.alloc(sizeof(uint64_t) * n, s));
    LIFE_TRY(pay.alloc(sizeof(uint32_t) * n, s));
    LIFE_TRY(err.alloc(sizeof(uint32_t), s));
    LIFE_CUDA_TRY(cudaMemsetAsync(err.p, 0, sizeof(uint32_t), s));
    if (n > 0) {
        const uintptr_t al = reinterpret_cast<uintptr_t>(atom) | reinterpret_cast<uintptr_t>(voxel) |
                             reinterpret_cast<uintptr_t>(fasc) | reinterpret_cast<uintptr_t>(val);
        pack_vaf_kernel<<<(unsigned)((n + 1023) / 1024), 256, 0, s>>>(
            atom, voxel, fasc, val, n, ix->na, ix->nv, ix->nf, sa, sv, (al & 15) == 0 ? 1 : 0, keys.as<uint64_t>(),
            pay.as<uint32_t>(), err.as<uint32_t>());
        LIFE_CHECK_LAUNCH();
    }
    uint32_t herr = 0;
    LIFE_CUDA_TRY(cudaMemcpyAsync(&herr, err.p, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    LIFE_CUDA_TRY(cudaStreamSynchronize(s));
    if (herr & DEV_BAD_INDEX) {
        set_error("life_build_index: an atom, voxel or fascicle index is outside its range");
        return LIFE_ERANGE;
    }
    if (herr & DEV_BAD_VALUE) {
        set_error("life_build_index: a Phi value is NaN or infinite");
        return LIFE_EINVAL;
    }
    // The sort is stable, so a list already in fascicle order (Phi written fascicle by
    // fascicle, as tractography writes it) needs only the (v, a) bits sorted.
    LIFE_TRY(radix_sort_pairs(keys, pay, n, (herr & DEV_UNSORTED) ? 0 : sa, ba + bf + bv, s));
    int32_t m = 0;
    TmpBuf count, offset;
    const int64_t nblk = (n + MG_TILE - 1) / MG_TILE;
    if (n > 0) {
        LIFE_TRY(count.alloc(sizeof(int32_t) * (nblk + 1), s));
        LIFE_TRY(offset.alloc(sizeof(int32_t) * (nblk + 1), s));
        LIFE_CUDA_TRY(cudaMemsetAsync(count.as<int32_t>() + nblk, 0, sizeof(int32_t), s));
        head_count_kernel<<<(unsigned)nblk, MG_THREADS, 0, s>>>(keys.as<uint64_t>(), n, count.as<int32_t>());
        LIFE_CHECK_LAUNCH();
        LIFE_TRY(exclusive_scan_i32(count.as<int32_t>(), offset.as<int32_t>(), nblk + 1, s));
        LIFE_CUDA_TRY(cudaMemcpyAsync(&m, offset.as<int32_t>() + nblk, 4, cudaMemcpyDeviceToHost, s));
        LIFE_CUDA_TRY(cudaStreamSynchronize(s));
    }
    ix->nnz = m;
    VoxelLayout& L = ix->vox;
    const bool bf16 = ix->precision == LIFE_BF16;
    if (bf16) LIFE_TRY(ix->uval.alloc(sizeof(float) * (size_t)m));
    LIFE_TRY(L.vox_ptr.alloc(sizeof(int32_t) * ((size_t)ix->nv + 1)));
    LIFE_TRY(L.atom.alloc(sizeof(uint16_t) * (size_t)m));
    LIFE_TRY(L.fasc.alloc(sizeof(int32_t) * (size_t)m));
    LIFE_TRY(L.val.alloc((bf16 ? 2 : 4) * (size_t)m));
    if (m == 0) {
        fill_i32_kernel<<<grid_for(ix->nv + 1), 256, 0, s>>>(L.vox_ptr.as<int32_t>(), ix->nv + 1, 0);
    } else if (bf16) {
        merge_layout_kernel<<<(unsigned)nblk, MG_THREADS, 0, s>>>(
            keys.as<uint64_t>(), pay.as<uint32_t>(), n, offset.as<int32_t>(), m, sa, sv, (1ull << ba) - 1,
            (1ull << bf) - 1, ix->nv, ix->uval.as<float>(), L.atom.as<uint16_t>(),
            L.fasc.as<int32_t>(), L.val.as<__nv_bfloat16>(), L.vox_ptr.as<int32_t>());
    } else {
        merge_layout_kernel<<<(unsigned)nblk, MG_THREADS, 0, s>>>(
            keys.as<uint64_t>(), pay.as<uint32_t>(), n, offset.as<int32_t>(), m, sa, sv, (1ull << ba) - 1,
            (1ull << bf) - 1, ix->nv, nullptr, L.atom.as<uint16_t>(),
            L.fasc.as<int32_t>(), L.val.as<float>(), L.vox_ptr.as<int32_t>());
    }
    LIFE_CHECK_LAUNCH();
    LIFE_CUDA_TRY(cudaStreamSynchronize(s));
    return LIFE_OK;
}

// ------------------------------------------------------------ re-sorting

// The merged list in its own order, the voxel of each entry from the voxels' offsets
// (outputs that are NULL are left out).
__global__ void list_export_kernel(const int32_t* __restrict__ vox_ptr, int32_t nv, const uint16_t* __restrict__ asrc,
                                   const int32_t* __restrict__ fsrc, const float* __restrict__ xsrc, int64_t m,
                                   int32_t* __restrict__ atom, int32_t* __restrict__ voxel,
                                   int32_t* __restrict__ fasc, float* __restrict__ val) {
    for_entry_segments(vox_ptr, nv, m, [&](int64_t i, int64_t v) {
        if (atom) atom[i] = asrc[i];
        if (voxel) voxel[i] = (int32_t)v;
        if (fasc) fasc[i] = fsrc[i];
        if (val) val[i] = xsrc[i];
    });
}

// Re-keys the merged (v, a, f) list in another order; payload = merged position.
__global__ void rekey_kernel(const int32_t* __restrict__ voxel, const uint16_t* __restrict__ atom,
                             const int32_t* __restrict__ fasc, int64_t m, int order, int bv, int ba, int bf,
                             uint64_t* __restrict__ key, uint32_t* __restrict__ payload) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t v = (uint64_t)voxel[i], a = atom[i], f = (uint64_t)fasc[i];
        key[i] = order == LIFE_LAYOUT_FIBER ? (f << (bv + ba)) | (v << ba) | a : (a << (bv + bf)) | (v << bf) | f;
        payload[i] = (uint32_t)i;
    }
}

__global__ void gather_export_kernel(const int32_t* __restrict__ vsrc, const uint16_t* __restrict__ asrc,
                                     const int32_t* __restrict__ fsrc, const float* __restrict__ xsrc,
                                     const uint32_t* __restrict__ perm, int64_t m, int32_t* __restrict__ atom,
                                     int32_t* __restrict__ voxel, int32_t* __restrict__ fasc,
                                     float* __restrict__ val) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t p = perm[i];
        if (atom) atom[i] = asrc[p];
        if (voxel) voxel[i] = vsrc[p];
        if (fasc) fasc[i] = fsrc[p];
        if (val) val[i] = xsrc[p];
    }
}

// Sorted permutation of the merged list for a layout other than its own.
static life_status layout_perm(life_index_s* ix, int layout, const int32_t* voxel, TmpBuf& perm, cudaStream_t s) {
    const int64_t m = ix->nnz;
    TmpBuf keys;
    LIFE_TRY(keys.alloc(sizeof(uint64_t) * m, s));
    LIFE_TRY(perm.alloc(sizeof(uint32_t) * m, s));
    const int bv = ix->key_bits_v, ba = ix->key_bits_a, bf = ix->key_bits_f;
    rekey_kernel<<<grid_for(m), 256, 0, s>>>(voxel, ix->vox.atom.as<uint16_t>(), ix->vox.fasc.as<int32_t>(), m, layout,
                                             bv, ba, bf, keys.as<uint64_t>(), perm.as<uint32_t>());
    LIFE_CHECK_LAUNCH();
    // the list is in (v, a, f) order and the sort stable: only the leading field of the
    // new order, the atom or the fascicle, has to be sorted
    const int low = layout == LIFE_LAYOUT_ATOM ? bv + bf : bv + ba;
    LIFE_TRY(radix_sort_pairs(keys, perm, m, low, bv + ba + bf, s));
    return LIFE_OK;
}

life_status export_layout(life_index_s* ix, int layout, int32_t* atom, int32_t* voxel, int32_t* fasc, float* val,
                          cudaStream_t s) {
    if (layout < LIFE_LAYOUT_VOXEL || layout > LIFE_LAYOUT_ATOM) {
        set_error("life_index_export: unknown layout %d", layout);
        return LIFE_EINVAL;
    }
    const int64_t m = ix->nnz;
    if (m == 0) return LIFE_OK;
    const float* x = ix->precision == LIFE_BF16 ? ix->uval.as<float>() : ix->vox.val.as<float>();
    if (layout == LIFE_LAYOUT_VOXEL) {  // the list's own order
        list_export_kernel<<<entry_segments_grid(m), 256, 0, s>>>(ix->vox.vox_ptr.as<int32_t>(), ix->nv,
                                                                  ix->vox.atom.as<uint16_t>(),
                                                                  ix->vox.fasc.as<int32_t>(), x, m, atom, voxel, fasc,
                                                                  val);
        LIFE_CHECK_LAUNCH();
        LIFE_CUDA_TRY(cudaStreamSynchronize(s));
        return LIFE_OK;
    }
    TmpBuf vox, perm;
    LIFE_TRY(vox.alloc(sizeof(int32_t) * m, s));
    list_export_kernel<<<entry_segments_grid(m), 256, 0, s>>>(ix->vox.vox_ptr.as<int32_t>(), ix->nv, nullptr, nullptr,
                                                              nullptr, m, nullptr, vox.as<int32_t>(), nullptr, nullptr);
    LIFE_CHECK_LAUNCH();
    LIFE_TRY(layout_perm(ix, layout, vox.as<int32_t>(), perm, s));
    gather_export_kernel<<<grid_for(m), 256, 0, s>>>(vox.as<int32_t>(), ix->vox.atom.as<uint16_t>(),
                                                     ix->vox.fasc.as<int32_t>(), x, perm.as<uint32_t>(), m, atom,
                                                     voxel, fasc, val);
    LIFE_CHECK_LAUNCH();
    LIFE_CUDA_TRY(cudaStreamSynchronize(s));
    return LIFE_OK;
}

__global__ void widen_streams_kernel(const uint16_t* __restrict__ a16, const int32_t* __restrict__ f32,
                                     const void* __restrict__ val, int bf16, int64_t m, int32_t* __restrict__ atom,
                                     int32_t* __restrict__ fasc, float* __restrict__ valout) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        if (atom) atom[i] = a16[i];
        if (fasc) fasc[i] = f32[i];
        if (valout)
            valout[i] = bf16 ? __bfloat162float(static_cast<const __nv_bfloat16*>(val)[i])
                             : static_cast<const float*>(val)[i];
    }
}

life_status export_voxel_streams(life_index_s* ix, int32_t* vox_ptr, int32_t* atom, int32_t* fasc, float* val,
                                 cudaStream_t s) {
    if (vox_ptr)
        LIFE_CUDA_TRY(cudaMemcpyAsync(vox_ptr, ix->vox.vox_ptr.p, sizeof(int32_t) * ((size_t)ix->nv + 1),
                                      cudaMemcpyDeviceToDevice, s));
    if (ix->nnz > 0) {
        widen_streams_kernel<<<grid_for(ix->nnz), 256, 0, s>>>(ix->vox.atom.as<uint16_t>(), ix->vox.fasc.as<int32_t>(),
                                                               ix->vox.val.p, ix->precision == LIFE_BF16 ? 1 : 0,
                                                               ix->nnz, atom, fasc, val);
        LIFE_CHECK_LAUNCH();
    }
    LIFE_CUDA_TRY(cudaStreamSynchronize(s));
    return LIFE_OK;
}

// ----------------------------------------------------- atom-sorted chunks

constexpr int ATOM_CHUNK = 256;

__global__ void atom_ptr_kernel(const int32_t* __restrict__ atom_sorted, int64_t m, int32_t na,
                                int32_t* __restrict__ atom_ptr) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t a = atom_sorted[i];
        const int32_t ap = i == 0 ? -1 : atom_sorted[i - 1];
        for (int32_t q = ap + 1; q <= a; ++q) atom_ptr[q] = (int32_t)i;
        if (i == m - 1)
            for (int32_t q = a + 1; q <= na; ++q) atom_ptr[q] = (int32_t)m;
    }
}

life_status build_atom_layout(life_index_s* ix, cudaStream_t s) {
    AtomLayout& A = ix->atoml;
    if (A.built) return LIFE_OK;
    const int64_t m = ix->nnz;
    TmpBuf atom_s;
    LIFE_TRY(atom_s.alloc(sizeof(int32_t) * (m > 0 ? m : 1), s));
    LIFE_TRY(A.voxel.alloc(sizeof(int32_t) * m));
    LIFE_TRY(A.fasc.alloc(sizeof(int32_t) * m));
    LIFE_TRY(A.val.alloc(sizeof(float) * m));
    LIFE_TRY(export_layout(ix, LIFE_LAYOUT_ATOM, atom_s.as<int32_t>(), A.voxel.as<int32_t>(), A.fasc.as<int32_t>(),
                           A.val.as<float>(), s));
    TmpBuf aptr;
    LIFE_TRY(aptr.alloc(sizeof(int32_t) * (ix->na + 1), s));
    if (m == 0) {
        fill_i32_kernel<<<1, 256, 0, s>>>(aptr.as<int32_t>(), ix->na + 1, 0);
    } else {
        atom_ptr_kernel<<<grid_for(m), 256, 0, s>>>(atom_s.as<int32_t>(), m, ix->na, aptr.as<int32_t>());
    }
    LIFE_CHECK_LAUNCH();
    std::vector<int32_t> hptr(ix->na + 1);
    LIFE_CUDA_TRY(cudaMemcpyAsync(hptr.data(), aptr.p, sizeof(int32_t) * (ix->na + 1), cudaMemcpyDeviceToHost, s));
    LIFE_CUDA_TRY(cudaStreamSynchronize(s));
    std::vector<int32_t> cbeg, catom, achunk(ix->na + 1);
    for (int32_t a = 0; a < ix->na; ++a) {
        achunk[a] = (int32_t)catom.size();
        for (int32_t b = hptr[a]; b < hptr[a + 1]; b += ATOM_CHUNK) {
            cbeg.push_back(b);
            catom.push_back(a);
        }
    }
    achunk[ix->na] = (int32_t)catom.size();
    cbeg.push_back((int32_t)m);
    A.n_chunks = (int32_t)catom.size();
    LIFE_TRY(A.chunk_beg.alloc(sizeof(int32_t) * cbeg.size()));
    LIFE_TRY(A.chunk_atom.alloc(sizeof(int32_t) * (catom.size() + 1)));
    LIFE_TRY(A.atom_chunk.alloc(sizeof(int32_t) * achunk.size()));
    LIFE_TRY(A.partial.alloc(sizeof(float) * catom.size() * (size_t)ix->nt));
    LIFE_CUDA_TRY(cudaMemcpyAsync(A.chunk_beg.p, cbeg.data(), sizeof(int32_t) * cbeg.size(), cudaMemcpyHostToDevice, s));
    if (!catom.empty())
        LIFE_CUDA_TRY(cudaMemcpyAsync(A.chunk_atom.p, catom.data(), sizeof(int32_t) * catom.size(),
                                      cudaMemcpyHostToDevice, s));
    LIFE_CUDA_TRY(cudaMemcpyAsync(A.atom_chunk.p, achunk.data(), sizeof(int32_t) * achunk.size(),
                                  cudaMemcpyHostToDevice, s));
    LIFE_CUDA_TRY(cudaStreamSynchronize(s));
    A.built = true;
    return LIFE_OK;
}

}  // namespace life
