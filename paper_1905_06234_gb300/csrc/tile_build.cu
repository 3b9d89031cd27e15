// The tensor-core (brick/tile) layout, built on the device (Sec. 4.1.2): voxels
// grouped into spatial bricks of 128-voxel tiles, a table of the fascicles of each
// brick, and the DSC and WC entry streams.
//
// The merged list is in (v, a, f) order, so a tile's entries are 128 contiguous
// pieces of it and no general sort is needed: one CTA per tile counts its cells
// (atom, row), whose entries are contiguous runs of the list, in shared memory,
// scans the counts in stream order and writes every entry at its place; one CTA
// per brick marks the brick's fascicles in a bitmap whose prefix counts number
// them.  Every entry is read a few times (2 to 6 B each) and written once per
// stream.  Sorting (key, position) pairs instead, as radix passes of 24 B a pair
// with the streams gathered through the positions afterwards, moved about ten
// times as much: for the paper-scale workload (80M entries, BF16 storage) a new index
// with its first DSC and WC took 44.0 ms that way and takes 16.4 ms now (14.1 ms the
// build alone), of which the bricks' tables are 1.3 ms and the streams 3.1 ms (bound by
// the latency of a pass: one 1024-thread CTA an SM, since a pass's cells and entries
// fill its shared memory).  The host's part of the old build (a stable sort of the
// voxels, copies both ways) went with it.  Some shapes are still sooner sorted: see
// sort_is_faster.
#include <algorithm>
#include <cstring>
#include <numeric>
#include <vector>

#include "launch_rules.cuh"
#include "tile_layout.cuh"
#include "tc_ptx.cuh"

namespace life {

static int nbits64(int64_t n) {
    if (n <= 1) return 0;
    uint64_t x = (uint64_t)(n - 1);
    int b = 0;
    while (x) { ++b; x >>= 1; }
    return b;
}

static unsigned grid1d(int64_t n, int threads = 256) {
    int64_t b = (n + threads - 1) / threads;
    int64_t cap = (int64_t)device_sm_count() * 32;
    return (unsigned)std::max<int64_t>(1, std::min(b, cap));
}

// The (atom, row) cells of a 128-atom chunk in DSC stream order: by the cell's place
// in the chunk's S operand (8-row group, 8-atom group, row mod 8, atom mod 8), i.e.
// by its byte offset there.  An 8 x 8 group of cells spans the 32 shared-memory
// banks once, so the run sums that the lanes of a warp store at the same time fall
// on more distinct banks than in (atom, row) order.
__device__ __forceinline__ uint32_t dsc_cell(uint32_t a, uint32_t row) {
    return ((row >> 3) << 10) | (((a >> 3) & 15u) << 6) | ((row & 7u) << 3) | (a & 7u);
}

// ---------------------------------------------------------- bricks and tiles
//
// Groups voxels into bricks (spatial bx x by x bz boxes when coordinates are
// known, else runs of bx*by*bz consecutive voxel ids) and each brick into
// 128-voxel tiles.  shape[3g ..] is the brick shape of group g (one group, or one
// per problem of a batch).  For the combined index of a batch, bricks never mix
// problems: the problem is the leading part of the brick key, and voxel-id runs
// restart at each problem.

struct BrickShape {
    int x, y, z;
};

// Largest coordinate along each axis (at least 0).
__global__ void coord_max_kernel(const int32_t* __restrict__ ijk, int64_t nv, int32_t* __restrict__ mx) {
    int32_t m[3] = {0, 0, 0};
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < nv; v += (int64_t)gridDim.x * blockDim.x)
        for (int d = 0; d < 3; ++d) m[d] = max(m[d], ijk[3 * v + d]);
    for (int d = 0; d < 3; ++d) {
        for (int o = 16; o > 0; o >>= 1) m[d] = max(m[d], __shfl_xor_sync(0xffffffffu, m[d], o));
        if ((threadIdx.x & 31) == 0) atomicMax(mx + d, m[d]);
    }
}

__device__ __forceinline__ int group_of_voxel(const int32_t* __restrict__ off, int n, int64_t v) {
    int lo = 0, hi = n - 1;  // the last group that starts at or before v
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= v) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Brick key of each voxel, and the range of the keys.
__global__ void brick_key_kernel(const int32_t* __restrict__ ijk, int64_t nv, const int32_t* __restrict__ mx,
                                 const int32_t* __restrict__ group_off, int n_groups,
                                 const int32_t* __restrict__ shape, long long* __restrict__ key,
                                 long long* __restrict__ range) {
    long long lo = INT64_MAX, hi = INT64_MIN;
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < nv; v += (int64_t)gridDim.x * blockDim.x) {
        const int g = group_off ? group_of_voxel(group_off, n_groups, v) : 0;
        const int32_t sx = shape[3 * g], sy = shape[3 * g + 1], sz = shape[3 * g + 2];
        long long k;
        if (ijk) {
            const long long nbx = mx[0] / sx + 1, nby = mx[1] / sy + 1;
            k = ((long long)(ijk[3 * v + 2] / sz) * nby + ijk[3 * v + 1] / sy) * nbx + ijk[3 * v] / sx;
        } else {
            k = (group_off ? v - group_off[g] : v) / ((long long)sx * sy * sz);
        }
        if (group_off) k |= (long long)g << 40;
        key[v] = k;
        lo = min(lo, k);
        hi = max(hi, k);
    }
    for (int o = 16; o > 0; o >>= 1) {
        lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMin(range, lo);
        atomicMax(range + 1, hi);
    }
}

__global__ void brick_pair_kernel(const long long* __restrict__ key, int64_t nv, long long lo,
                                  uint64_t* __restrict__ skey, uint32_t* __restrict__ vox) {
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < nv; v += (int64_t)gridDim.x * blockDim.x) {
        skey[v] = (uint64_t)(key[v] - lo);
        vox[v] = (uint32_t)v;
    }
}

__global__ void head_flag_kernel(const uint64_t* __restrict__ key, int64_t m, int32_t* __restrict__ head) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x)
        head[j] = (j == 0 || key[j] != key[j - 1]) ? 1 : 0;
}

// First sorted voxel of each brick (start[n_bricks] = Nv), and the group of each brick.
__global__ void brick_start_kernel(const int32_t* __restrict__ head, const int32_t* __restrict__ bidx,
                                   const uint32_t* __restrict__ vox, int64_t nv, int32_t n_bricks,
                                   const int32_t* __restrict__ group_off, int n_groups,
                                   int32_t* __restrict__ start, int32_t* __restrict__ group) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < nv; j += (int64_t)gridDim.x * blockDim.x) {
        if (!head[j]) continue;
        start[bidx[j]] = (int32_t)j;
        if (group) group[bidx[j]] = group_of_voxel(group_off, n_groups, vox[j]);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) start[n_bricks] = (int32_t)nv;
}

// Tiles of each brick, with a zero after the last for the scan.
__global__ void brick_ntiles_kernel(const int32_t* __restrict__ start, int32_t n_bricks, int32_t* __restrict__ nt) {
    for (int32_t b = blockIdx.x * blockDim.x + threadIdx.x; b <= n_bricks; b += gridDim.x * blockDim.x)
        nt[b] = b < n_bricks ? (start[b + 1] - start[b] + TILE_V - 1) / TILE_V : 0;
}

// tile_vox and tile_brick (tile_vox filled with -1 before).
__global__ void tile_fill_kernel(const uint32_t* __restrict__ vox, const int32_t* __restrict__ head,
                                 const int32_t* __restrict__ bidx, const int32_t* __restrict__ start,
                                 const int32_t* __restrict__ btile, int64_t nv, int32_t* __restrict__ tile_vox,
                                 int32_t* __restrict__ tile_brick) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < nv; j += (int64_t)gridDim.x * blockDim.x) {
        const int32_t b = bidx[j] + head[j] - 1, k = (int32_t)j - start[b], t = btile[b] + k / TILE_V;
        tile_vox[(int64_t)t * TILE_V + k % TILE_V] = (int32_t)vox[j];
        if (k % TILE_V == 0) tile_brick[t] = b;
    }
}

// Entries of each tile (one warp per tile), with a zero after the last for the scan,
// and of its fullest quarter of 32 rows.
__global__ void tile_count_kernel(const int32_t* __restrict__ tile_vox, const int32_t* __restrict__ vox_ptr,
                                  int64_t n_tiles, int32_t* __restrict__ count, int32_t* __restrict__ quarter) {
    const int lane = threadIdx.x & 31;
    const int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (t > n_tiles) return;
    int32_t sum = 0, most = 0;
    if (t < n_tiles)
        for (int r = lane; r < TILE_V; r += 32) {
            const int32_t v = tile_vox[t * TILE_V + r];
            int32_t c = v >= 0 ? vox_ptr[v + 1] - vox_ptr[v] : 0;
            for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
            sum += c;
            most = max(most, c);
        }
    if (lane == 0) {
        count[t] = sum;
        quarter[t] = most;
    }
}

// ------------------------------------------------------ brick fascicle tables

// Calls use(entry, load(entry)) for the entries of the voxels of tiles [t0, t1): each
// warp of the CTA takes 32 tile rows at a time (a lane holds one row's entry range)
// and walks their entries together, 32 at a time, so that short voxels fill the
// lanes too; four such steps' loads are issued before the first is used (one at a
// time left the kernels waiting on memory: the tables of the paper-scale workload
// took 2.2 ms).
template <class L, class U>
__device__ __forceinline__ void for_brick_entries(const int32_t* __restrict__ tile_vox,
                                                  const int32_t* __restrict__ vox_ptr, int t0, int t1, L load, U use) {
    constexpr int B = 4;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int u = 4 * t0 + warp; u < 4 * t1; u += nw) {
        const int32_t v = tile_vox[(int64_t)u * 32 + lane];
        const int beg = v >= 0 ? vox_ptr[v] : 0, len = v >= 0 ? vox_ptr[v + 1] - beg : 0;
        int incl = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const int total = __shfl_sync(0xffffffffu, incl, 31), shift = beg - (incl - len);
        for (int k0 = 0; k0 < total; k0 += 32 * B) {
            int idx[B];
            decltype(load(0)) x[B];
#pragma unroll
            for (int e = 0; e < B; ++e) {
                const int k = k0 + 32 * e + lane;
                int row = 0;  // the first row whose inclusive count is above k
#pragma unroll
                for (int st = 16; st > 0; st >>= 1)
                    if (__shfl_sync(0xffffffffu, incl, row + st - 1) <= k) row += st;
                const int i = __shfl_sync(0xffffffffu, shift, row) + k;
                idx[e] = k < total ? i : -1;
                if (k < total) x[e] = load(i);
            }
#pragma unroll
            for (int e = 0; e < B; ++e)
                if (idx[e] >= 0) use(idx[e], x[e]);
        }
    }
}

constexpr int BT_THREADS = 1024;
constexpr int BT_WINDOW = 1 << 19;  // fascicles of one bitmap pass: 64 KB of bits, 32 KB of prefix counts

// Window of a launch: all fascicles when they are fewer.
static int bt_window(int32_t nf) { return (int)std::min<int64_t>(BT_WINDOW, ((int64_t)nf + 1023) / 1024 * 1024); }

__device__ __forceinline__ void mark_bit(uint32_t* bits, uint32_t f) {
    const uint32_t m = 1u << (f & 31u);
    if (!(*reinterpret_cast<volatile uint32_t*>(bits + (f >> 5)) & m)) atomicOr(bits + (f >> 5), m);
}

// Number of distinct fascicles of each brick, with a zero after the last for the scan.
__global__ void __launch_bounds__(BT_THREADS) brick_count_kernel(const int32_t* __restrict__ tile_vox,
                                                                 const int32_t* __restrict__ vox_ptr,
                                                                 const int32_t* __restrict__ fasc,
                                                                 const int32_t* __restrict__ btile, int32_t nb,
                                                                 int32_t nf, int window, int32_t* __restrict__ count) {
    extern __shared__ uint32_t bits[];
    __shared__ int total;
    const int tid = threadIdx.x, words = window / 32;
    for (int32_t b = blockIdx.x; b < nb; b += gridDim.x) {
        if (tid == 0) total = 0;
        int c = 0;
        for (int64_t w0 = 0; w0 < nf; w0 += window) {
            for (int i = tid; i < words; i += BT_THREADS) bits[i] = 0u;
            __syncthreads();
            for_brick_entries(tile_vox, vox_ptr, btile[b], btile[b + 1],
                              [&](int i) { return __ldg(fasc + i); },
                              [&](int, int32_t id) {
                                  const int64_t f = id - w0;
                                  if (f >= 0 && f < window) mark_bit(bits, (uint32_t)f);
                              });
            __syncthreads();
            for (int i = tid; i < words; i += BT_THREADS) c += __popc(bits[i]);
            __syncthreads();
        }
        for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
        if ((tid & 31) == 0 && c) atomicAdd(&total, c);
        __syncthreads();
        if (tid == 0) count[b] = total;
        __syncthreads();
    }
    if (blockIdx.x == 0 && tid == 0) count[nb] = 0;
}

// Exclusive block scan of one value per thread (BT_THREADS threads); *total gets the sum.
__device__ __forceinline__ int block_excl_scan(int x, int* wsum, int* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    __syncthreads();  // wsum may still be read from an earlier scan
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int t = wsum[lane];
        const int own = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        wsum[lane] = t - own;
        if (lane == 31) *total = t;
    }
    __syncthreads();
    return incl - x + wsum[warp];
}

__device__ __forceinline__ float load_val(const __nv_bfloat16* p) { return __bfloat162float(*p); }
__device__ __forceinline__ float load_val(const float* p) { return *p; }

// Each brick's fascicle table (ascending ids) and, for every entry of the merged
// list, the byte offset 4·(brick-local fascicle) of its slot.  With cv: cv[b] =
// (largest number of entries of one fascicle of brick b) x (largest |val| of the
// brick), rounded up, a bound on Σ|val| over the entries of any of its fascicles
// (integer counts and maxima, so the order of the atomics does not matter).
template <class VT>
__global__ void __launch_bounds__(BT_THREADS) brick_table_kernel(
    const int32_t* __restrict__ tile_vox, const int32_t* __restrict__ vox_ptr, const int32_t* __restrict__ fasc,
    const VT* __restrict__ val, const int32_t* __restrict__ btile, int32_t nb, int32_t nf, int window,
    const int32_t* __restrict__ bptr, int32_t* __restrict__ bfasc, uint16_t* __restrict__ fl, float* __restrict__ cv) {
    extern __shared__ uint32_t bits[];
    __shared__ int wsum[32], total;
    __shared__ uint32_t vmax_bits, cmax;
    const int tid = threadIdx.x, words = window / 32, per = (words + BT_THREADS - 1) / BT_THREADS;
    uint16_t* pre = reinterpret_cast<uint16_t*>(bits + words);  // table slots before each word (< 15872)
    int32_t* cnt = reinterpret_cast<int32_t*>(pre + words);     // entries of each slot (words is a multiple of 32)
    for (int32_t b = blockIdx.x; b < nb; b += gridDim.x) {
        const int32_t o = bptr[b];
        int slot0 = 0;
        uint32_t vm = 0u;
        if (cv) {
            for (int i = tid; i < bptr[b + 1] - o; i += BT_THREADS) cnt[i] = 0;
            if (tid == 0) vmax_bits = cmax = 0u;
        }
        for (int64_t w0 = 0; w0 < nf; w0 += window) {
            for (int i = tid; i < words; i += BT_THREADS) bits[i] = 0u;
            __syncthreads();
            for_brick_entries(tile_vox, vox_ptr, btile[b], btile[b + 1],
                              [&](int i) { return __ldg(fasc + i); },
                              [&](int, int32_t id) {
                                  const int64_t f = id - w0;
                                  if (f >= 0 && f < window) mark_bit(bits, (uint32_t)f);
                              });
            __syncthreads();
            int c = 0;
            for (int e = 0; e < per; ++e)
                if (tid * per + e < words) c += __popc(bits[tid * per + e]);
            int slot = slot0 + block_excl_scan(c, wsum, &total);
            for (int e = 0; e < per; ++e) {
                const int w = tid * per + e;
                if (w >= words) break;
                pre[w] = (uint16_t)slot;
                for (uint32_t x = bits[w]; x; x &= x - 1) bfasc[o + slot++] = (int32_t)(w0 + 32 * w + __ffs(x) - 1);
            }
            __syncthreads();
            struct IdVal {
                int32_t id;
                VT val;
            };
            for_brick_entries(tile_vox, vox_ptr, btile[b], btile[b + 1],
                              [&](int i) { return IdVal{__ldg(fasc + i), cv ? val[i] : VT()}; },
                              [&](int i, const IdVal& x) {
                                  const int64_t f = x.id - w0;
                                  if (f < 0 || f >= window) return;
                                  const uint32_t w = (uint32_t)f >> 5;
                                  const int s = pre[w] + __popc(bits[w] & ((1u << (f & 31)) - 1u));
                                  fl[i] = (uint16_t)(4 * s);
                                  if (cv) {
                                      atomicAdd(cnt + s, 1);
                                      vm = max(vm, __float_as_uint(load_val(&x.val)) & 0x7FFFFFFFu);
                                  }
                              });
            slot0 += total;
            __syncthreads();
        }
        if (!cv) continue;
        uint32_t cm = 0u;
        for (int i = tid; i < slot0; i += BT_THREADS) cm = max(cm, (uint32_t)cnt[i]);
        for (int q = 16; q > 0; q >>= 1) {
            vm = max(vm, __shfl_xor_sync(0xffffffffu, vm, q));
            cm = max(cm, __shfl_xor_sync(0xffffffffu, cm, q));
        }
        if ((tid & 31) == 0) {
            atomicMax(&vmax_bits, vm);
            atomicMax(&cmax, cm);
        }
        __syncthreads();
        if (tid == 0) cv[b] = __fmul_ru((float)cmax, __uint_as_float(vmax_bits));
        __syncthreads();
    }
}

// wb_src[wb_ptr[b] + i] = brick_fasc[brick_fasc_ptr[b] + i], padding slots -1 (one block per brick).
__global__ void wb_src_kernel(const int32_t* __restrict__ bptr, const int32_t* __restrict__ bfasc,
                              const int32_t* __restrict__ wptr, int32_t nb, int32_t* __restrict__ wsrc) {
    for (int32_t b = blockIdx.x; b < nb; b += gridDim.x) {
        const int32_t f0 = bptr[b], n = bptr[b + 1] - f0, o = wptr[b], np = wptr[b + 1] - o;
        for (int32_t i = threadIdx.x; i < np; i += blockDim.x) wsrc[o + i] = i < n ? bfasc[f0 + i] : -1;
    }
}

// -------------------------------------------------------------- entry streams

constexpr int TS_THREADS = 1024;
constexpr int TS_CELLS = TILE_V * DKC;                 // cells of one pass: 16 a thread
constexpr int TS_PER = TS_CELLS / TS_THREADS;
constexpr int TS_BATCH = 2;                            // entries whose loads a thread issues together (4 spill)
constexpr int TS_MAX_C = 4;                            // 128-atom chunks (Na <= 512)
constexpr int TS_STAGE = 19456;                        // entries staged in shared memory before they are written
constexpr size_t TS_SMEM = sizeof(int32_t) * TS_CELLS + sizeof(uint2) * TS_STAGE;

template <class VT>
struct TileStreams {
    const int32_t *tile_vox, *vox_ptr, *tile_base;
    const uint16_t* atom;   // merged list, (v, a, f) order
    const uint16_t* flv;    // its brick-table byte offsets
    const VT* val;          // its values as stored
    uint16_t *soff, *fl;
    VT* out;
    int32_t* chunk_ptr;
    uint16_t *wkey, *wfl;   // WC streams (NULL when the index keeps none)
    VT* wval;
    int32_t* wseg_ptr;
    uint32_t* vmax;         // bits of the largest Σ|val| over one run
    int64_t n_tiles;
    int n_c, n_sub, atom_major;
};

__device__ __forceinline__ uint32_t val_bits(__nv_bfloat16 x) { return __bfloat16_as_ushort(x); }
__device__ __forceinline__ uint32_t val_bits(float x) { return __float_as_uint(x); }
__device__ __forceinline__ void store_bits(__nv_bfloat16* p, uint32_t b) { *p = __ushort_as_bfloat16((uint16_t)b); }
__device__ __forceinline__ void store_bits(float* p, uint32_t b) { *p = __uint_as_float(b); }

// Shared state of a pass: the rows' entry ranges (first entry, prefix counts).
struct TsRows {
    int32_t pre[TILE_V + 1], rbeg[TILE_V];
    int wsum[32], total;
};

// One pass: the entries of a 128-atom chunk of all rows in DSC order (WC = false),
// or of a quarter of the rows with all atoms in WC order, written from stream
// position base on.  Returns the number of entries.
template <class VT, bool WC>
__device__ __forceinline__ int ts_pass(const TileStreams<VT>& A, int32_t* hd, TsRows& R, int base, int last,
                                       int32_t* seg_out, uint32_t& best) {
    const int tid = threadIdx.x, T = R.total;
    int32_t* en = hd + TS_CELLS;                        // end of the cell's run, 0 for an empty cell
    uint2* stage = reinterpret_cast<uint2*>(en);        // (the ends are read before the first entry is staged)
    const uint16_t* __restrict__ atom = A.atom;
    auto locate = [&](int k, int& row) {
        int lo = 0;
#pragma unroll
        for (int st = TILE_V / 2; st > 0; st >>= 1)
            if (R.pre[lo + st] <= k) lo += st;
        row = lo;
        return R.rbeg[lo] + (k - R.pre[lo]);
    };
    auto cell_of = [&](int a, int row) {
        return WC ? (uint32_t)(32 * a + (row & 31)) : dsc_cell((uint32_t)a, (uint32_t)row);
    };
    for (int k0 = tid; k0 < T; k0 += TS_BATCH * TS_THREADS) {
        int idx[TS_BATCH], cell[TS_BATCH];
        bool head[TS_BATCH], tail[TS_BATCH];
#pragma unroll
        for (int e = 0; e < TS_BATCH; ++e) {
            const int k = k0 + e * TS_THREADS;
            idx[e] = -1;
            if (k < T) {
                int row;
                const int i = locate(k, row), a = __ldg(atom + i);
                idx[e] = i;
                // (neighbour indexes stay inside the list where a neighbour is not of this row)
                head[e] = k == R.pre[row] || (int)__ldg(atom + max(i - 1, 0)) != a;
                tail[e] = k + 1 == R.pre[row + 1] || (int)__ldg(atom + min(i + 1, last)) != a;
                cell[e] = (int)cell_of(a, row);
            }
        }
#pragma unroll
        for (int e = 0; e < TS_BATCH; ++e) {
            if (idx[e] < 0) continue;
            if (head[e]) hd[cell[e]] = idx[e];
            if (tail[e]) en[cell[e]] = idx[e] + 1;
        }
    }
    __syncthreads();
    {
        int h[TS_PER], n[TS_PER], sum = 0;
#pragma unroll
        for (int e = 0; e < TS_PER; e += 4) {
            const int4 hv = *reinterpret_cast<const int4*>(hd + TS_PER * tid + e);
            const int4 ev = *reinterpret_cast<const int4*>(en + TS_PER * tid + e);
            h[e] = hv.x; h[e + 1] = hv.y; h[e + 2] = hv.z; h[e + 3] = hv.w;
            n[e] = ev.x ? ev.x - hv.x : 0;
            n[e + 1] = ev.y ? ev.y - hv.y : 0;
            n[e + 2] = ev.z ? ev.z - hv.z : 0;
            n[e + 3] = ev.w ? ev.w - hv.w : 0;
            sum += n[e] + n[e + 1] + n[e + 2] + n[e + 3];
        }
        int run = block_excl_scan(sum, R.wsum, &R.total);  // (the sum of the cells is the number of entries)
        if (WC && tid % (SUB * 32 / TS_PER) == 0) {        // first cell of a 32-atom segment
            const int sg = tid / (SUB * 32 / TS_PER);
            if (sg < A.n_sub) seg_out[sg] = base + run;
        }
#pragma unroll
        for (int e = 0; e < TS_PER; ++e) {
            const int x = run - h[e];
            run += n[e];
            h[e] = x;                                      // place of entry i in the pass: h + i
        }
#pragma unroll
        for (int e = 0; e < TS_PER; e += 4)
            *reinterpret_cast<int4*>(hd + TS_PER * tid + e) = make_int4(h[e], h[e + 1], h[e + 2], h[e + 3]);
    }
    if (!WC && tid == 0) *seg_out = base;
    __syncthreads();
    for (int w0 = 0; w0 < T; w0 += TS_STAGE) {             // one window unless the pass is very large
        for (int k0 = tid; k0 < T; k0 += TS_BATCH * TS_THREADS) {
            int pos[TS_BATCH];
            uint2 rec[TS_BATCH];
#pragma unroll
            for (int e = 0; e < TS_BATCH; ++e) {
                const int k = k0 + e * TS_THREADS;
                pos[e] = -1;
                if (k < T) {
                    int row;
                    const int i = locate(k, row), a = __ldg(atom + i);
                    const VT x = A.val[i];
                    const uint32_t f = __ldg(A.flv + i);
                    const int p = hd[cell_of(a, row)] + i - w0;
                    pos[e] = p < TS_STAGE ? p : -1;
                    uint32_t key;
                    if (WC) {
                        // byte offset of the entry's (row, atom) cell in a scatter warp's Z tile
                        // (row-major, or atom-major for the FP32-storage kernel)
                        const uint32_t r32 = row & 31, a32 = a & 31;
                        key = 4 * (A.atom_major ? a32 * ZW + r32 : r32 * ZW + a32);
                    } else {
                        // byte offset of (row, atom) in an S chunk (< 32768), with the continuation bit
                        const bool cont = k != R.pre[row] && (int)__ldg(atom + max(i - 1, 0)) == a;
                        key = ptx::kmajor_off(row, a & 127u, (128 / 8) * 128) | (cont ? (uint32_t)CONT : 0u);
                        if (!cont && w0 == 0) {
                            // with max |x| the largest Σ|val| over one run bounds every S value of a DSC
                            float sum = fabsf(load_val(&x));
                            const int end = R.rbeg[row] + (R.pre[row + 1] - R.pre[row]);
                            for (int j = i + 1; j < end && (int)__ldg(atom + j) == a; ++j)
                                sum += fabsf(load_val(A.val + j));
                            best = max(best, __float_as_uint(sum));
                        }
                    }
                    // key | byte offset of the fascicle in the brick table (< 15872 fascicles: 16 bits)
                    rec[e] = make_uint2(key | (f << 16), val_bits(x));
                }
            }
#pragma unroll
            for (int e = 0; e < TS_BATCH; ++e)
                if (pos[e] >= 0) stage[pos[e]] = rec[e];
        }
        __syncthreads();
        const int n = min(TS_STAGE, T - w0);
        uint16_t* key_out = (WC ? A.wkey : A.soff) + base + w0;
        uint16_t* fl_out = (WC ? A.wfl : A.fl) + base + w0;
        VT* val_out = (WC ? A.wval : A.out) + base + w0;
#pragma unroll 4
        for (int p = tid; p < n; p += TS_THREADS) {
            const uint2 r = stage[p];
            key_out[p] = (uint16_t)(r.x & 0xFFFFu);
            fl_out[p] = (uint16_t)(r.x >> 16);
            store_bits(val_out + p, r.y);
        }
        __syncthreads();
    }
    return T;
}

// One CTA per tile.  Each pass (a 128-atom chunk of all rows for the DSC stream, a
// quarter of the rows with all atoms for the WC stream) has at most 16384 cells:
// the head and the end of each cell's run are stored in shared memory, the lengths
// scanned in stream order, and each entry then goes to (start of its cell) + (its
// distance from the run's head).  The tile's rows are walked as one list (entry k
// finds its row by a binary search in the rows' prefix counts), so that every
// thread has independent loads in flight whatever the rows' lengths.  A pass's
// entries are put in order in shared memory and written out as they lie: written
// from where they are found, as 2-byte stores that each touch a sector of their
// own, they held the kernel at the rate of those sectors.
template <class VT>
__global__ void __launch_bounds__(TS_THREADS) tile_stream_kernel(const TileStreams<VT> A) {
    extern __shared__ __align__(16) int32_t ts_smem[];
    __shared__ int32_t bound[TS_MAX_C + 1][TILE_V];  // entry range of each row and chunk
    __shared__ TsRows R;
    const int tid = threadIdx.x, lane = tid & 31;
    const int64_t t = blockIdx.x;
    const int n_c = A.n_c;
    for (int u = tid; u < (n_c + 1) * TILE_V; u += TS_THREADS) {
        const int c = u / TILE_V, row = u % TILE_V;
        const int32_t v = A.tile_vox[t * TILE_V + row];
        int lo = 0, hi = 0;
        if (v >= 0) {
            lo = A.vox_ptr[v];
            hi = A.vox_ptr[v + 1];
            if (c == n_c) lo = hi;
            else if (c > 0)  // first entry of the row with an atom of chunk c or later
                while (lo < hi) {
                    const int mid = lo + (hi - lo) / 2;
                    if ((int)A.atom[mid] < DKC * c) lo = mid + 1;
                    else hi = mid;
                }
        }
        bound[c][row] = lo;
    }
    const int last = A.tile_base[A.n_tiles] - 1;  // last entry of the list
    int32_t base = A.tile_base[t];
    if (t == A.n_tiles - 1 && tid == 0) {
        A.chunk_ptr[A.n_tiles * n_c] = last + 1;
        if (A.wkey) A.wseg_ptr[A.n_tiles * 4 * A.n_sub] = last + 1;
    }
    uint32_t best = 0u;
    const int passes = n_c + (A.wkey ? 4 : 0);
    for (int p = 0; p < passes; ++p) {
        const bool wc = p >= n_c;
        const int q = p - n_c;
        if (p == n_c) base = A.tile_base[t];
        for (int i = tid; i < TS_CELLS / 4; i += TS_THREADS)
            reinterpret_cast<int4*>(ts_smem + TS_CELLS)[i] = make_int4(0, 0, 0, 0);
        __syncthreads();  // the bounds are written (first pass)
        int len = 0;
        if (tid < TILE_V) {
            const int c0 = wc ? 0 : p, c1 = wc ? n_c : p + 1;
            len = !wc || (tid >> 5) == q ? bound[c1][tid] - bound[c0][tid] : 0;
            R.rbeg[tid] = bound[c0][tid];
        }
        const int ex = block_excl_scan(len, R.wsum, &R.total);
        if (tid < TILE_V) R.pre[tid] = ex;
        if (tid == 0) R.pre[TILE_V] = R.total;
        __syncthreads();
        base += wc ? ts_pass<VT, true>(A, ts_smem, R, base, last, A.wseg_ptr + (t * 4 + q) * A.n_sub, best)
                   : ts_pass<VT, false>(A, ts_smem, R, base, last, A.chunk_ptr + t * n_c + p, best);
        __syncthreads();
    }
    for (int o = 16; o > 0; o >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, o));
    if (lane == 0 && best) atomicMax(A.vmax, best);
}

// ------------------------------------------------ the same layout by sorting
//
// Counting gives a brick and a tile one CTA each.  That is slower than sorting where
// the entries lie in few, very full tiles (a pass of the streams walks its entries
// once for every TS_STAGE of them), with very many fascicles (the tables walk a
// brick's entries once for every BT_WINDOW ids) and with nearly empty tiles.  There (sort_is_faster) radix sorts of
// (key, entry) pairs over the whole GPU take its place: by (brick, fascicle) for the
// tables, by (tile, cell in stream order) for each stream; the list is in (v, a, f)
// order and the sort stable, so the fascicles of a cell stay in order.  The layout is
// the same, bit for bit.
enum : int { BY_TABLE = 0, BY_DSC = 1, BY_WC = 2 };

// tile · TILE_V + row of each voxel.
__global__ void voxel_slot_kernel(const int32_t* __restrict__ tile_vox, int64_t n, int64_t* __restrict__ slot) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        if (tile_vox[i] >= 0) slot[tile_vox[i]] = i;
}

// Key of each entry of the merged list: brick | fascicle (bf bits), or tile | cell in the
// order of the DSC or the WC stream (16 bits); payload = the entry.
__global__ void entry_key_kernel(const int32_t* __restrict__ vox_ptr, int32_t nv, const int64_t* __restrict__ slot,
                                 const int32_t* __restrict__ tile_brick, const uint16_t* __restrict__ atom,
                                 const int32_t* __restrict__ fasc, int64_t m, int order, int bf,
                                 uint64_t* __restrict__ key, uint32_t* __restrict__ payload) {
    for_entry_segments(vox_ptr, nv, m, [&](int64_t i, int64_t v) {
        const int64_t s = slot[v], t = s / TILE_V;
        const uint32_t row = (uint32_t)(s % TILE_V), a = atom[i];
        key[i] = order == BY_TABLE ? ((uint64_t)tile_brick[t] << bf) | (uint64_t)fasc[i]
                 : order == BY_DSC ? ((uint64_t)t << 16) | ((a >> 7) << 14) | dsc_cell(a, row)
                                   : ((uint64_t)t << 16) | ((row >> 5) << 14) | (a << 5) | (row & 31u);
        payload[i] = (uint32_t)i;
    });
}

// Offsets of the bricks' tables from the sorted (brick, fascicle) keys.
__global__ void sorted_bptr_kernel(const uint64_t* __restrict__ key, int64_t m, int bf, const int32_t* __restrict__ head,
                                   const int32_t* __restrict__ uidx, int32_t nb, int32_t n_unique,
                                   int32_t* __restrict__ bptr) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x) {
        if (!head[j]) continue;
        const int32_t b = (int32_t)(key[j] >> bf), pb = j == 0 ? -1 : (int32_t)(key[j - 1] >> bf);
        for (int32_t q = pb + 1; q <= b; ++q) bptr[q] = uidx[j];
        if (uidx[j] == n_unique - 1)
            for (int32_t q = b + 1; q <= nb; ++q) bptr[q] = n_unique;
    }
}

// The tables' fascicles, the first sorted entry of each slot, and each entry's slot offset.
__global__ void sorted_table_kernel(const uint64_t* __restrict__ key, const uint32_t* __restrict__ pay, int64_t m, int bf,
                                    const int32_t* __restrict__ head, const int32_t* __restrict__ uidx,
                                    const int32_t* __restrict__ bptr, int32_t* __restrict__ bfasc,
                                    int32_t* __restrict__ first, uint16_t* __restrict__ fl) {
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x) {
        const int32_t u = uidx[j] + head[j] - 1;  // (uidx counts the heads before j)
        fl[pay[j]] = (uint16_t)(4 * (u - bptr[key[j] >> bf]));
        if (head[j]) {
            bfasc[u] = (int32_t)(key[j] & ((1ull << bf) - 1));
            first[u] = (int32_t)j;
        }
    }
}

// max into p[b], one atomic where the warp has one b (almost always: the keys are sorted).
__device__ __forceinline__ void brick_max(uint32_t* p, uint32_t b, uint32_t x) {
    if (__all_sync(0xffffffffu, b == __shfl_sync(0xffffffffu, b, 0))) {
        x = __reduce_max_sync(0xffffffffu, x);
        if ((threadIdx.x & 31) == 0) atomicMax(p + b, x);
    } else {
        atomicMax(p + b, x);
    }
}

// Largest entry count of a slot, and largest |val|, of each brick (both zero before).
template <class VT>
__global__ void sorted_cv_max_kernel(const uint64_t* __restrict__ key, const uint32_t* __restrict__ pay, int64_t m, int bf,
                                     const int32_t* __restrict__ head, const int32_t* __restrict__ uidx,
                                     const int32_t* __restrict__ first, int32_t n_unique, const VT* __restrict__ val,
                                     uint32_t* __restrict__ cmax, uint32_t* __restrict__ vmax) {
    const int lane = threadIdx.x & 31;
    for (int64_t j0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) - lane; j0 < m;
         j0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = min(j0 + lane, m - 1);  // (lanes beyond the end repeat the last entry)
        const uint32_t b = (uint32_t)(key[j] >> bf);
        const int32_t u = uidx[j];
        brick_max(cmax, b, head[j] ? (uint32_t)((u + 1 < n_unique ? (int64_t)first[u + 1] : m) - j) : 0u);
        brick_max(vmax, b, __float_as_uint(load_val(val + pay[j])) & 0x7FFFFFFFu);
    }
}

__global__ void sorted_cv_kernel(const uint32_t* __restrict__ cmax, const uint32_t* __restrict__ vmax, int32_t nb,
                                 float* __restrict__ cv) {
    for (int32_t b = blockIdx.x * blockDim.x + threadIdx.x; b < nb; b += gridDim.x * blockDim.x)
        cv[b] = __fmul_ru((float)cmax[b], __uint_as_float(vmax[b]));
}

// A stream from its sorted keys: the DSC's (WC = false: chunk offsets, continuation bits)
// or the WC's (segment offsets); n_seg segments, the offsets one longer.
template <class VT, bool WC>
__global__ void sorted_stream_kernel(const uint64_t* __restrict__ key, const uint32_t* __restrict__ pay, int64_t m,
                                     const uint16_t* __restrict__ flv, const VT* __restrict__ val, int n_c, int n_sub,
                                     int atom_major, int64_t n_seg, uint16_t* __restrict__ okey,
                                     uint16_t* __restrict__ ofl, VT* __restrict__ oval, int32_t* __restrict__ seg_ptr) {
    auto seg_of = [&](uint64_t k) -> int64_t {
        const int64_t t = (int64_t)(k >> 16), part = (int64_t)((k >> 14) & 3u);  // chunk, or row quarter
        return WC ? (t * 4 + part) * n_sub + (int64_t)((k >> 10) & 15u) : t * n_c + part;
    };
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t k = key[j];
        const uint32_t c = (uint32_t)k & 0x3FFFu, i = pay[j];
        if (WC) {
            const uint32_t a32 = (c >> 5) & 31u, r32 = c & 31u;
            okey[j] = (uint16_t)(4 * (atom_major ? a32 * ZW + r32 : r32 * ZW + a32));
        } else {
            const uint32_t row = ((c >> 10) << 3) | ((c >> 3) & 7u), a = (((c >> 6) & 15u) << 3) | (c & 7u);
            okey[j] = (uint16_t)(ptx::kmajor_off(row, a, (128 / 8) * 128) | (j > 0 && key[j - 1] == k ? (uint32_t)CONT : 0u));
        }
        ofl[j] = flv[i];
        oval[j] = val[i];
        const int64_t s = seg_of(k), ps = j == 0 ? -1 : seg_of(key[j - 1]);
        for (int64_t q = ps + 1; q <= s; ++q) seg_ptr[q] = (int32_t)j;
        if (j == m - 1)
            for (int64_t q = s + 1; q <= n_seg; ++q) seg_ptr[q] = (int32_t)m;
    }
}

// Bits of the largest Σ|val| over the entries of one (atom, voxel) run of the DSC stream.
template <class VT>
__global__ void run_vmax_kernel(const uint16_t* __restrict__ soff, const VT* __restrict__ val, int64_t m,
                                uint32_t* __restrict__ out) {
    uint32_t best = 0u;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < m; j += (int64_t)gridDim.x * blockDim.x) {
        if (soff[j] & CONT) continue;
        float sum = fabsf(load_val(val + j));
        for (int64_t k = j + 1; k < m && (soff[k] & CONT); ++k) sum += fabsf(load_val(val + k));
        best = max(best, __float_as_uint(sum));
    }
    for (int o = 16; o > 0; o >>= 1) best = max(best, __shfl_xor_sync(0xffffffffu, best, o));
    if ((threadIdx.x & 31) == 0 && best) atomicMax(out, best);
}

template <class T>
static life_status upload(DevBuf& dst, const std::vector<T>& src, cudaStream_t s) {
    LIFE_TRY(dst.alloc(sizeof(T) * std::max<size_t>(src.size(), 1)));
    if (!src.empty())
        LIFE_CUDA_TRY(cudaMemcpyAsync(dst.p, src.data(), sizeof(T) * src.size(), cudaMemcpyHostToDevice, s));
    return LIFE_OK;
}

template <class T>
static life_status download(std::vector<T>& dst, const void* src, size_t n, cudaStream_t s) {
    dst.resize(n);
    if (n) LIFE_CUDA_TRY(cudaMemcpyAsync(dst.data(), src, sizeof(T) * n, cudaMemcpyDeviceToHost, s));
    return LIFE_OK;
}

// Bricks and tiles of one attempt (device arrays, sizes on the host).
struct TileSet {
    DevBuf tile_vox, tile_brick, brick_tile_ptr, brick_group;
    std::vector<int32_t> btile;  // host copy of brick_tile_ptr
    int64_t n_tiles = 0;
    int32_t n_bricks = 0;
};

static life_status assign_tiles(const life_index_s* ix, const std::vector<BrickShape>& shape, TileSet& H,
                                cudaStream_t s) {
    const int64_t nv = ix->nv;
    const bool grouped = ix->batch.n > 0;
    const int ng = (int)shape.size();
    std::vector<int32_t> hshape;
    for (const BrickShape& b : shape) hshape.insert(hshape.end(), {b.x, b.y, b.z});
    TmpBuf mx, range, dshape, goff, lkey, skey, vox, head, bidx, start, nt;
    LIFE_TRY(mx.alloc(3 * sizeof(int32_t), s));
    LIFE_TRY(range.alloc(2 * sizeof(long long), s));
    LIFE_TRY(dshape.alloc(sizeof(int32_t) * hshape.size(), s));
    LIFE_TRY(lkey.alloc(sizeof(long long) * nv, s));
    LIFE_TRY(skey.alloc(sizeof(uint64_t) * nv, s));
    LIFE_TRY(vox.alloc(sizeof(uint32_t) * nv, s));
    LIFE_TRY(head.alloc(sizeof(int32_t) * nv, s));
    LIFE_TRY(bidx.alloc(sizeof(int32_t) * nv, s));
    LIFE_CUDA_TRY(cudaMemsetAsync(mx.p, 0, 3 * sizeof(int32_t), s));
    const long long range0[2] = {INT64_MAX, INT64_MIN};
    LIFE_CUDA_TRY(cudaMemcpyAsync(range.p, range0, sizeof(range0), cudaMemcpyHostToDevice, s));
    LIFE_CUDA_TRY(cudaMemcpyAsync(dshape.p, hshape.data(), sizeof(int32_t) * hshape.size(), cudaMemcpyHostToDevice, s));
    if (grouped) {
        LIFE_TRY(goff.alloc(sizeof(int32_t) * ix->batch.vox_off.size(), s));
        LIFE_CUDA_TRY(cudaMemcpyAsync(goff.p, ix->batch.vox_off.data(), sizeof(int32_t) * ix->batch.vox_off.size(),
                                      cudaMemcpyHostToDevice, s));
    }
    const int32_t* ijk = ix->voxel_ijk.as<int32_t>();
    if (ijk) {
        coord_max_kernel<<<grid1d(nv), 256, 0, s>>>(ijk, nv, mx.as<int32_t>());
        LIFE_CHECK_LAUNCH();
    }
    brick_key_kernel<<<grid1d(nv), 256, 0, s>>>(ijk, nv, mx.as<int32_t>(), goff.as<int32_t>(), ng,
                                                dshape.as<int32_t>(), lkey.as<long long>(), range.as<long long>());
    LIFE_CHECK_LAUNCH();
    long long hr[2];
    LIFE_CUDA_TRY(cudaMemcpyAsync(hr, range.p, sizeof(hr), cudaMemcpyDeviceToHost, s));
    LIFE_CUDA_TRY(cudaStreamSynchronize(s));
    brick_pair_kernel<<<grid1d(nv), 256, 0, s>>>(lkey.as<long long>(), nv, hr[0], skey.as<uint64_t>(),
                                                 vox.as<uint32_t>());
    LIFE_CHECK_LAUNCH();
    int kb = 0;
    for (uint64_t x = (uint64_t)(hr[1] - hr[0]); x; x >>= 1) ++kb;
    LIFE_TRY(radix_sort_pairs(skey, vox, nv, 0, kb, s));
    head_flag_kernel<<<grid1d(nv), 256, 0, s>>>(skey.as<uint64_t>(), nv, head.as<int32_t>());
    LIFE_CHECK_LAUNCH();
    LIFE_TRY(exclusive_scan_i32(head.as<int32_t>(), bidx.as<int32_t>(), nv, s));
    int32_t last[2];
    LIFE_CUDA_TRY(cudaMemcpyAsync(&last[0], bidx.as<int32_t>() + nv - 1, 4, cudaMemcpyDeviceToHost, s));
    LIFE_CUDA_TRY(cudaMemcpyAsync(&last[1], head.as<int32_t>() + nv - 1, 4, cudaMemcpyDeviceToHost, s));
    LIFE_CUDA_TRY(cudaStreamSynchronize(s));
    H.n_bricks = last[0] + last[1];
    const int32_t nb = H.n_bricks;
    LIFE_TRY(start.alloc(sizeof(int32_t) * ((size_t)nb + 1), s));
    LIFE_TRY(nt.alloc(sizeof(int32_t) * ((size_t)nb + 1), s));
    LIFE_TRY(H.brick_tile_ptr.alloc(sizeof(int32_t) * ((size_t)nb + 1)));
    if (grouped) LIFE_TRY(H.brick_group.alloc(sizeof(int32_t) * (size_t)nb));
    brick_start_kernel<<<grid1d(nv), 256, 0, s>>>(head.as<int32_t>(), bidx.as<int32_t>(), vox.as<uint32_t>(), nv, nb,
                                                  goff.as<int32_t>(), ng, start.as<int32_t>(),
                                                  H.brick_group.as<int32_t>());
    LIFE_CHECK_LAUNCH();
    brick_ntiles_kernel<<<grid1d((int64_t)nb + 1), 256, 0, s>>>(start.as<int32_t>(), nb, nt.as<int32_t>());
    LIFE_CHECK_LAUNCH();
    LIFE_TRY(exclusive_scan_i32(nt.as<int32_t>(), H.brick_tile_ptr.as<int32_t>(), (int64_t)nb + 1, s));
    LIFE_TRY(download(H.btile, H.brick_tile_ptr.p, (size_t)nb + 1, s));
    LIFE_CUDA_TRY(cudaStreamSynchronize(s));
    H.n_tiles = H.btile[nb];
    LIFE_TRY(H.tile_vox.alloc(sizeof(int32_t) * H.n_tiles * TILE_V));
    LIFE_TRY(H.tile_brick.alloc(sizeof(int32_t) * H.n_tiles));
    LIFE_CUDA_TRY(cudaMemsetAsync(H.tile_vox.p, 0xFF, sizeof(int32_t) * H.n_tiles * TILE_V, s));
    tile_fill_kernel<<<grid1d(nv), 256, 0, s>>>(vox.as<uint32_t>(), head.as<int32_t>(), bidx.as<int32_t>(),
                                                start.as<int32_t>(), H.brick_tile_ptr.as<int32_t>(), nv,
                                                H.tile_vox.as<int32_t>(), H.tile_brick.as<int32_t>());
    LIFE_CHECK_LAUNCH();
    return LIFE_OK;
}

// The sorted form of the tables while the bricks are being formed: the entries by
// (brick, fascicle), the heads of equal keys and their ranks.
struct SortedTables {
    TmpBuf slot, key, pay, head, uidx;
    int32_t n_unique = 0;
};

static life_status sort_entries(const life_index_s* ix, const TileSet& H, const TmpBuf& slot, int order, int bits,
                                TmpBuf& key, TmpBuf& pay, cudaStream_t s) {
    const int64_t m = ix->nnz;
    LIFE_TRY(key.alloc(sizeof(uint64_t) * m, s));
    LIFE_TRY(pay.alloc(sizeof(uint32_t) * m, s));
    entry_key_kernel<<<entry_segments_grid(m), 256, 0, s>>>(ix->vox.vox_ptr.as<int32_t>(), ix->nv, slot.as<int64_t>(),
                                               H.tile_brick.as<int32_t>(), ix->vox.atom.as<uint16_t>(),
                                               ix->vox.fasc.as<int32_t>(), m, order, ix->key_bits_f, key.as<uint64_t>(),
                                               pay.as<uint32_t>());
    LIFE_CHECK_LAUNCH();
    return radix_sort_pairs(key, pay, m, 0, bits, s);
}

// Table offsets of the bricks (into L.brick_fasc_ptr) by sorting.
static life_status sort_tables(life_index_s* ix, const TileSet& H, SortedTables& T, cudaStream_t s) {
    const int64_t m = ix->nnz;
    LIFE_TRY(T.slot.alloc(sizeof(int64_t) * ix->nv, s));
    voxel_slot_kernel<<<grid1d(H.n_tiles * TILE_V), 256, 0, s>>>(H.tile_vox.as<int32_t>(), H.n_tiles * TILE_V,
                                                                 T.slot.as<int64_t>());
    LIFE_CHECK_LAUNCH();
    LIFE_TRY(sort_entries(ix, H, T.slot, BY_TABLE, nbits64(H.n_bricks) + ix->key_bits_f, T.key, T.pay, s));
    LIFE_TRY(T.head.alloc(sizeof(int32_t) * m, s));
    LIFE_TRY(T.uidx.alloc(sizeof(int32_t) * m, s));
    head_flag_kernel<<<grid1d(m), 256, 0, s>>>(T.key.as<uint64_t>(), m, T.head.as<int32_t>());
    LIFE_CHECK_LAUNCH();
    LIFE_TRY(exclusive_scan_i32(T.head.as<int32_t>(), T.uidx.as<int32_t>(), m, s));
    int32_t last[2];
    LIFE_CUDA_TRY(cudaMemcpyAsync(&last[0], T.uidx.as<int32_t>() + m - 1, 4, cudaMemcpyDeviceToHost, s));
    LIFE_CUDA_TRY(cudaMemcpyAsync(&last[1], T.head.as<int32_t>() + m - 1, 4, cudaMemcpyDeviceToHost, s));
    LIFE_CUDA_TRY(cudaStreamSynchronize(s));
    T.n_unique = last[0] + last[1];
    sorted_bptr_kernel<<<grid1d(m), 256, 0, s>>>(T.key.as<uint64_t>(), m, ix->key_bits_f, T.head.as<int32_t>(),
                                                 T.uidx.as<int32_t>(), H.n_bricks, T.n_unique,
                                                 ix->tile.brick_fasc_ptr.as<int32_t>());
    LIFE_CHECK_LAUNCH();
    return LIFE_OK;
}

// The rest of the sorted form: the tables and both streams.
template <class VT>
static life_status sort_tables_and_streams(life_index_s* ix, const TileSet& H, SortedTables& T, uint32_t* vmax,
                                           cudaStream_t s) {
    TileLayout& L = ix->tile;
    const VT* val = ix->vox.val.as<VT>();
    const int64_t m = ix->nnz;
    const int bf = ix->key_bits_f, bt = nbits64(H.n_tiles), n_c = L.kp / DKC;
    TmpBuf flv, first;
    LIFE_TRY(flv.alloc(sizeof(uint16_t) * m, s));
    LIFE_TRY(first.alloc(sizeof(int32_t) * T.n_unique, s));
    sorted_table_kernel<<<grid1d(m), 256, 0, s>>>(T.key.as<uint64_t>(), T.pay.as<uint32_t>(), m, bf,
                                                  T.head.as<int32_t>(), T.uidx.as<int32_t>(),
                                                  L.brick_fasc_ptr.as<int32_t>(), L.brick_fasc.as<int32_t>(),
                                                  first.as<int32_t>(), flv.as<uint16_t>());
    LIFE_CHECK_LAUNCH();
    if (L.wc_stream && sizeof(VT) == 2) {  // the FP32 WC sums in FP32 tables
        TmpBuf mx;
        LIFE_TRY(mx.alloc(2 * sizeof(uint32_t) * (size_t)H.n_bricks, s));
        LIFE_CUDA_TRY(cudaMemsetAsync(mx.p, 0, 2 * sizeof(uint32_t) * (size_t)H.n_bricks, s));
        uint32_t* cm = mx.as<uint32_t>();
        sorted_cv_max_kernel<VT><<<grid1d(m), 256, 0, s>>>(T.key.as<uint64_t>(), T.pay.as<uint32_t>(), m, bf,
                                                           T.head.as<int32_t>(), T.uidx.as<int32_t>(),
                                                           first.as<int32_t>(), T.n_unique, val, cm, cm + H.n_bricks);
        LIFE_CHECK_LAUNCH();
        sorted_cv_kernel<<<grid1d(H.n_bricks), 256, 0, s>>>(cm, cm + H.n_bricks, H.n_bricks, L.brick_cv.as<float>());
        LIFE_CHECK_LAUNCH();
    }
    for (TmpBuf* b : {&T.head, &T.uidx, &first}) b->release();
    LIFE_TRY(sort_entries(ix, H, T.slot, BY_DSC, bt + 16, T.key, T.pay, s));
    sorted_stream_kernel<VT, false><<<grid1d(m), 256, 0, s>>>(
        T.key.as<uint64_t>(), T.pay.as<uint32_t>(), m, flv.as<uint16_t>(), val, n_c, L.n_sub, 0, H.n_tiles * n_c,
        L.soff.as<uint16_t>(), L.fl.as<uint16_t>(), L.val.as<VT>(), L.chunk_ptr.as<int32_t>());
    LIFE_CHECK_LAUNCH();
    run_vmax_kernel<VT><<<grid1d(m), 256, 0, s>>>(L.soff.as<uint16_t>(), L.val.as<VT>(), m, vmax);
    LIFE_CHECK_LAUNCH();
    if (!L.wc_stream) return LIFE_OK;
    LIFE_TRY(sort_entries(ix, H, T.slot, BY_WC, bt + 16, T.key, T.pay, s));
    sorted_stream_kernel<VT, true><<<grid1d(m), 256, 0, s>>>(
        T.key.as<uint64_t>(), T.pay.as<uint32_t>(), m, flv.as<uint16_t>(), val, n_c, L.n_sub, sizeof(VT) == 4 ? 1 : 0,
        H.n_tiles * 4 * L.n_sub, L.wkey.as<uint16_t>(), L.wfl.as<uint16_t>(), L.wval.as<VT>(),
        L.wseg_ptr.as<int32_t>());
    LIFE_CHECK_LAUNCH();
    return LIFE_OK;
}

// Whether the layout is sooner there by sorting than by counting, from the entries of
// each tile (base) and of its fullest quarter of 32 rows, in microseconds fitted to builds
// timed both ways on one GB300.  Counting: a stream pass 9 us and 0.5 ns an entry walked,
// the first walk and one more for every TS_STAGE entries of the pass; a window of a brick's
// table 9 us, and three walks at 0.8 ns an entry, or 12 ns where one warp's 32 rows hold
// most of them; the fullest brick and tile, or the SMs' even share if that is more.
// Sorting: 0.5 ms and 0.25 ns an entry, wherever the entries lie.  Whole builds, BF16,
// counted / sorted: 80M entries in 500k voxels 15.7 / 30.0 ms, 10M in 32768 voxels 3.5 /
// 5.3; 3M in 4096 2.9 / 2.9, 6M there 4.6 / 3.8; 1M in 128 25 / 1.8, 10M in 128 1515 /
// 4.8; 50M in 4M voxels with 5M fascicles 29.7 / 22.0, with 50M fascicles 120 / 23.
static bool sort_is_faster(const int32_t* base, const int32_t* quarter, const std::vector<int32_t>& btile, int n_c,
                           bool wc, int64_t nf, int window, int num_sms) {
    constexpr double PASS = 9.0, WALK = 5.0e-4, WINDOW = 9.0, TABLE_WALK = 8.0e-4, ROWS_WALK = 0.012, SORT = 500.0,
                     SORT_ENTRY = 2.5e-4;
    const double sms = std::max(num_sms, 1), windows = (double)((nf + window - 1) / window);
    double tab = 0.0, tab_max = 0.0, str = 0.0, str_max = 0.0;
    for (size_t b = 0; b + 1 < btile.size(); ++b) {
        double most = 0.0;
        for (int32_t t = btile[b]; t < btile[b + 1]; ++t) {
            const double e = base[t + 1] - base[t], q = quarter[t];
            double us = PASS * n_c + WALK * e * (2.0 + e / n_c / TS_STAGE);
            if (wc) us += PASS * 4 + WALK * e * (2.0 + q / TS_STAGE);
            str += us;
            str_max = std::max(str_max, us);
            most = std::max(most, q);
        }
        const double e = base[btile[b + 1]] - base[btile[b]];
        const double us = windows * (WINDOW + 3.0 * std::max(ROWS_WALK * most, TABLE_WALK * e));
        tab += us;
        tab_max = std::max(tab_max, us);
    }
    return std::max(tab_max, tab / sms) + std::max(str_max, str / sms) > SORT + SORT_ENTRY * base[btile.back()];
}

template <class VT>
static life_status build_tables_and_streams(life_index_s* ix, const TileSet& H, const int32_t* tile_base, int window,
                                            SortedTables* sorted, uint32_t* vmax, cudaStream_t s) {
    if (sorted) return sort_tables_and_streams<VT>(ix, H, *sorted, vmax, s);
    TileLayout& L = ix->tile;
    const VoxelLayout& V = ix->vox;
    const int64_t m = ix->nnz;
    TmpBuf flv;
    LIFE_TRY(flv.alloc(sizeof(uint16_t) * std::max<int64_t>(m, 1), s));
    const bool cv = L.wc_stream && sizeof(VT) == 2;  // the FP32 WC sums in FP32 tables
    const size_t bsm = (size_t)window / 32 * 6 + (cv ? sizeof(int32_t) * std::max(L.max_fb, 1) : 0);
    auto bk = brick_table_kernel<VT>;
    LIFE_CUDA_TRY(cudaFuncSetAttribute(bk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bsm));
    bk<<<(unsigned)std::min<int64_t>(H.n_bricks, 65535), BT_THREADS, bsm, s>>>(
        H.tile_vox.as<int32_t>(), V.vox_ptr.as<int32_t>(), V.fasc.as<int32_t>(), V.val.as<VT>(),
        H.brick_tile_ptr.as<int32_t>(), H.n_bricks, ix->nf, window, L.brick_fasc_ptr.as<int32_t>(),
        L.brick_fasc.as<int32_t>(), flv.as<uint16_t>(), cv ? L.brick_cv.as<float>() : nullptr);
    LIFE_CHECK_LAUNCH();
    TileStreams<VT> A{};
    A.tile_vox = H.tile_vox.as<int32_t>();
    A.vox_ptr = V.vox_ptr.as<int32_t>();
    A.tile_base = tile_base;
    A.atom = V.atom.as<uint16_t>();
    A.flv = flv.as<uint16_t>();
    A.val = V.val.as<VT>();
    A.soff = L.soff.as<uint16_t>();
    A.fl = L.fl.as<uint16_t>();
    A.out = L.val.as<VT>();
    A.chunk_ptr = L.chunk_ptr.as<int32_t>();
    A.wkey = L.wc_stream ? L.wkey.as<uint16_t>() : nullptr;
    A.wfl = L.wfl.as<uint16_t>();
    A.wval = L.wval.as<VT>();
    A.wseg_ptr = L.wseg_ptr.as<int32_t>();
    A.vmax = vmax;
    A.n_tiles = H.n_tiles;
    A.n_c = L.kp / DKC;
    A.n_sub = L.n_sub;
    A.atom_major = sizeof(VT) == 4 ? 1 : 0;
    auto tk = tile_stream_kernel<VT>;
    LIFE_CUDA_TRY(cudaFuncSetAttribute(tk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TS_SMEM));
    tk<<<(unsigned)H.n_tiles, TS_THREADS, TS_SMEM, s>>>(A);
    LIFE_CHECK_LAUNCH();
    return LIFE_OK;
}

life_status build_tile_layout(life_index_s* ix, cudaStream_t s) {
    TileLayout& L = ix->tile;
    if (ix->na > 512 || ix->nt > 128) {
        set_error("tensor-core path supports Na <= 512 and Ntheta <= 128 (got %d, %d)", ix->na, ix->nt);
        return LIFE_ENOTSUP;
    }
    if (ix->key_bits_f > 32) {
        set_error("tensor-core path: too many fascicles");
        return LIFE_ENOTSUP;
    }
    if (ix->precision == LIFE_FP32 && ix->na > 384) {
        // D's two FP16 parts (Na/2 columns each) and the 128-column accumulator share
        // the 512 tensor-memory columns of an SM
        set_error("FP32 tensor-core DSC supports Na <= 384 (got %d)", ix->na);
        return LIFE_ENOTSUP;
    }
    if (ix->precision == LIFE_FP32 && ix->sparse_dsc) {
        set_error("the live-entry DSC stream is built for BF16 storage only");
        return LIFE_ENOTSUP;
    }
    const int64_t m = ix->nnz;
    L.vbytes = ix->precision == LIFE_FP32 ? 4 : 2;
    L.np = (ix->nt + 15) / 16 * 16;
    L.kp = (ix->na + 127) / 128 * 128;   // whole 128-atom DSC chunks
    // the FP32-storage WC holds D's FP16 parts (np columns per 128-atom block) and a
    // ring of three 64-column Z slots in tensor memory; beyond that WC runs on the
    // CUDA cores
    L.wc_stream = L.vbytes == 2 || wc32_tmem_cols(L.np, L.kp) <= 512;
    L.n_sub = L.kp / SUB;
    const int bf = ix->key_bits_f;
    TileSet H;
    SortedTables ST;
    std::vector<int32_t> hbptr, hgroup, htile;  // htile: [n_tiles + 1] entry offsets, then the fullest quarters
    TmpBuf count, tcount, tinfo;                // tinfo: htile on the device
    bool ok = false, sorted = false;
    const int window = bt_window(ix->nf);
    const size_t csm = (size_t)window / 8;
    LIFE_CUDA_TRY(cudaFuncSetAttribute(brick_count_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)csm));
    // Every group starts from B0^3 bricks; a group whose largest brick fascicle
    // table overflows halves its brick's largest dimension and the bricks are
    // formed again, until all groups fit (other groups keep their bricks).
    const int B0 = std::max(2, ix->brick_dim);
    const bool grouped = ix->batch.n > 0;
    const int ngroups = grouped ? ix->batch.n : 1;
    std::vector<BrickShape> shape(ngroups, BrickShape{B0, B0, B0});
    for (int attempt = 0; attempt < 32 && !ok; ++attempt) {
        LIFE_TRY(assign_tiles(ix, shape, H, s));
        const int bt = nbits64(H.n_tiles), bb = nbits64(H.n_bricks);
        if (bt + 16 + bf > 64 || bb + bf > 64) {  // (brick, fascicle) is a sort key of the sorted form;
                                                  // the other has been a limit of the layout all along
            set_error("tensor-core layout: sort key too wide");
            return LIFE_ENOTSUP;
        }
        LIFE_TRY(tcount.alloc(sizeof(int32_t) * (H.n_tiles + 1), s));
        LIFE_TRY(tinfo.alloc(2 * sizeof(int32_t) * (H.n_tiles + 1), s));
        tile_count_kernel<<<(unsigned)((H.n_tiles + 8) / 8), 256, 0, s>>>(
            H.tile_vox.as<int32_t>(), ix->vox.vox_ptr.as<int32_t>(), H.n_tiles, tcount.as<int32_t>(),
            tinfo.as<int32_t>() + H.n_tiles + 1);
        LIFE_CHECK_LAUNCH();
        LIFE_TRY(exclusive_scan_i32(tcount.as<int32_t>(), tinfo.as<int32_t>(), H.n_tiles + 1, s));
        LIFE_TRY(download(htile, tinfo.p, 2 * ((size_t)H.n_tiles + 1), s));
        LIFE_CUDA_TRY(cudaStreamSynchronize(s));
        sorted = m > 0 && sort_is_faster(htile.data(), htile.data() + H.n_tiles + 1, H.btile, L.kp / DKC, L.wc_stream,
                                         ix->nf, window, ix->num_sms);
        L.brick_fasc_ptr.release();
        LIFE_TRY(L.brick_fasc_ptr.alloc(sizeof(int32_t) * ((size_t)H.n_bricks + 1)));
        if (sorted) {
            LIFE_TRY(sort_tables(ix, H, ST, s));
        } else {
            LIFE_TRY(count.alloc(sizeof(int32_t) * ((size_t)H.n_bricks + 1), s));
            brick_count_kernel<<<(unsigned)std::min<int64_t>(H.n_bricks, 65535), BT_THREADS, csm, s>>>(
                H.tile_vox.as<int32_t>(), ix->vox.vox_ptr.as<int32_t>(), ix->vox.fasc.as<int32_t>(),
                H.brick_tile_ptr.as<int32_t>(), H.n_bricks, ix->nf, window, count.as<int32_t>());
            LIFE_CHECK_LAUNCH();
            LIFE_TRY(exclusive_scan_i32(count.as<int32_t>(), L.brick_fasc_ptr.as<int32_t>(), (int64_t)H.n_bricks + 1,
                                        s));
        }
        LIFE_TRY(download(hbptr, L.brick_fasc_ptr.p, (size_t)H.n_bricks + 1, s));
        if (grouped) LIFE_TRY(download(hgroup, H.brick_group.p, (size_t)H.n_bricks, s));
        LIFE_CUDA_TRY(cudaStreamSynchronize(s));
        std::vector<int32_t> gmax(ngroups, 0);
        int32_t mx = 0;
        for (int64_t b = 0; b < H.n_bricks; ++b) {
            const int32_t nfb = hbptr[b + 1] - hbptr[b];
            const int g = grouped ? hgroup[b] : 0;
            gmax[g] = std::max(gmax[g], nfb);
            mx = std::max(mx, nfb);
        }
        L.max_fb = mx;
        ok = true;
        bool shrunk = false;
        for (int g = 0; g < ngroups; ++g) {
            if (gmax[g] <= MAX_BRICK_FASC) continue;
            ok = false;
            BrickShape& sh = shape[g];
            int* d = sh.x >= sh.y && sh.x >= sh.z ? &sh.x : (sh.y >= sh.z ? &sh.y : &sh.z);
            if (*d > 1) {
                *d = (*d + 1) / 2;
                shrunk = true;
            }
        }
        if (!ok && !shrunk) break;
    }
    {
        const BrickShape& s0 = shape[0];
        const bool cubic = s0.x == s0.y && s0.y == s0.z;
        L.brick_edge = !ix->voxel_ijk.p ? 0 : (cubic ? s0.x : std::max(s0.x, std::max(s0.y, s0.z)));
        L.brick_b = B0;
    }
    if (!ok) {
        set_error("tensor-core layout: a brick touches %d fascicles (limit %d) even at the smallest brick",
                  L.max_fb, MAX_BRICK_FASC);
        return LIFE_ENOTSUP;
    }
    L.n_tiles = H.n_tiles;
    L.n_bricks = H.n_bricks;
    L.n_nnz = m;
    LIFE_TRY(L.brick_fasc.alloc(sizeof(int32_t) * std::max<int64_t>(hbptr[H.n_bricks], 1)));
    const int n_c = L.kp / DKC;  // 128-atom chunks per tile
    const int64_t n_segs = H.n_tiles * n_c, n_wsegs = H.n_tiles * 4 * L.n_sub;
    // streams padded to whole 8-entry slots (the kernels load 16 bytes at a time)
    const int64_t m_pad = (m + 7) / 8 * 8 + 8;
    auto stream = [&](DevBuf& b, size_t elem) -> life_status {
        LIFE_TRY(b.alloc(elem * m_pad));
        LIFE_CUDA_TRY(cudaMemsetAsync(b.as<char>() + elem * m, 0, elem * (m_pad - m), s));
        return LIFE_OK;
    };
    LIFE_TRY(stream(L.soff, sizeof(uint16_t)));
    LIFE_TRY(stream(L.fl, sizeof(uint16_t)));
    LIFE_TRY(stream(L.val, L.vbytes));
    LIFE_TRY(L.chunk_ptr.alloc(sizeof(int32_t) * (n_segs + 1)));
    if (L.wc_stream) {
        LIFE_TRY(stream(L.wkey, sizeof(uint16_t)));
        LIFE_TRY(stream(L.wfl, sizeof(uint16_t)));
        LIFE_TRY(stream(L.wval, L.vbytes));
        LIFE_TRY(L.wseg_ptr.alloc(sizeof(int32_t) * (n_wsegs + 1)));
    } else {
        L.wkey.release();
        L.wfl.release();
        L.wval.release();
        L.wseg_ptr.release();
    }
    LIFE_TRY(L.brick_cv.alloc(sizeof(float) * std::max<int64_t>(H.n_bricks, 1)));
    LIFE_TRY(L.tile_amax.alloc(sizeof(uint32_t) * 4 * std::max<int64_t>(H.n_tiles, 1)));
    TmpBuf rv;
    LIFE_TRY(rv.alloc(sizeof(uint32_t), s));
    LIFE_CUDA_TRY(cudaMemsetAsync(rv.p, 0, sizeof(uint32_t), s));
    SortedTables* st = sorted ? &ST : nullptr;
    if (L.vbytes == 4)
        LIFE_TRY(build_tables_and_streams<float>(ix, H, tinfo.as<int32_t>(), window, st, rv.as<uint32_t>(), s));
    else
        LIFE_TRY(build_tables_and_streams<__nv_bfloat16>(ix, H, tinfo.as<int32_t>(), window, st, rv.as<uint32_t>(), s));
    std::vector<int32_t> wptr(H.n_bricks + 1, 0);
    {
        // padded, 16-byte aligned per-brick weight slots for the DSC's bulk table loads
        for (int64_t b = 0; b < H.n_bricks; ++b) wptr[b + 1] = wptr[b] + (hbptr[b + 1] - hbptr[b] + 3) / 4 * 4;
        L.wb_total = wptr[H.n_bricks];
        L.n_brick_slots = hbptr[H.n_bricks];
        LIFE_TRY(upload(L.wb_ptr, wptr, s));
        LIFE_TRY(L.wb_src.alloc(sizeof(int32_t) * std::max<int64_t>(L.wb_total, 4)));
        // gathered tables in global memory serve only the live-entry stream (the
        // dense DSC gathers each brick's weights itself)
        if (ix->sparse_dsc != 0 && !grouped)
            LIFE_TRY(L.wb.alloc(sizeof(float) * std::max<int64_t>(L.wb_total, 4)));
        else
            L.wb.release();
        wb_src_kernel<<<(unsigned)std::min<int64_t>(H.n_bricks, 65535), 128, 0, s>>>(
            L.brick_fasc_ptr.as<int32_t>(), L.brick_fasc.as<int32_t>(), L.wb_ptr.as<int32_t>(), H.n_bricks,
            L.wb_src.as<int32_t>());
        LIFE_CHECK_LAUNCH();
    }
    LIFE_TRY(L.x_amax.alloc(sizeof(uint32_t) * (size_t)std::max(ix->num_sms, 1) * 8));
    LIFE_CUDA_TRY(cudaMemsetAsync(L.x_amax.p, 0, sizeof(uint32_t) * (size_t)std::max(ix->num_sms, 1) * 8, s));
    if (L.vbytes == 2) LIFE_TRY(L.d_img.alloc((size_t)2 * L.np * L.kp * 2));
    LIFE_TRY(L.d_info.alloc(sizeof(uint32_t) * (size_t)(1 + L.kp / 8)));
    // live-entry DSC stream: allocated at full size, filled on demand by a DSC call
    L.sparse = ix->sparse_dsc != 0 && !grouped;
    if (L.sparse) {
        LIFE_TRY(L.c_soff.alloc(sizeof(uint16_t) * m_pad));
        LIFE_TRY(L.c_fl.alloc(sizeof(uint16_t) * m_pad));
        LIFE_TRY(L.c_val.alloc(sizeof(__nv_bfloat16) * m_pad));
        LIFE_CUDA_TRY(cudaMemsetAsync(L.c_soff.p, 0, sizeof(uint16_t) * m_pad, s));
        LIFE_CUDA_TRY(cudaMemsetAsync(L.c_fl.p, 0, sizeof(uint16_t) * m_pad, s));
        LIFE_CUDA_TRY(cudaMemsetAsync(L.c_val.p, 0, sizeof(__nv_bfloat16) * m_pad, s));
        const int64_t n_chunks = std::max<int64_t>(H.n_tiles * n_c, 1);
        LIFE_TRY(L.c_chunk_end.alloc(sizeof(int32_t) * n_chunks));
        LIFE_CUDA_TRY(cudaMemsetAsync(L.c_chunk_end.p, 0, sizeof(int32_t) * n_chunks, s));
        LIFE_TRY(L.wb_live.alloc(std::max<int64_t>(L.wb_total, 4)));
        LIFE_CUDA_TRY(cudaMemsetAsync(L.wb_live.p, 0, std::max<int64_t>(L.wb_total, 4), s));
        LIFE_TRY(L.sparse_ctl.alloc(sizeof(SparseCtl)));
        LIFE_CUDA_TRY(cudaMemsetAsync(L.sparse_ctl.p, 0, sizeof(SparseCtl), s));
    } else {
        L.c_soff.release();
        L.c_fl.release();
        L.c_val.release();
        L.c_chunk_end.release();
        L.wb_live.release();
        L.sparse_ctl.release();
        L.tile_brick.release();
    }
    // largest bricks first
    uint32_t vbits = 0u;
    LIFE_CUDA_TRY(cudaMemcpyAsync(&vbits, rv.p, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    LIFE_CUDA_TRY(cudaStreamSynchronize(s));
    std::memcpy(&L.run_vmax, &vbits, sizeof(float));
    std::vector<int64_t> bnnz(H.n_bricks);
    for (int64_t b = 0; b < H.n_bricks; ++b)
        bnnz[b] = (int64_t)htile[H.btile[b + 1]] - htile[H.btile[b]] + 64 * (H.btile[b + 1] - H.btile[b]);
    std::vector<int32_t> order(H.n_bricks);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int32_t x, int32_t y) { return bnnz[x] > bnnz[y]; });
    LIFE_TRY(upload(L.brick_order, order, s));
    const WorkShare W = share_out(order, H.btile, htile, hbptr, ix->num_sms, grouped, L.vbytes == 4);
    L.grid = W.grid();
    L.n_units = (int32_t)W.brick.size();
    std::vector<int32_t> units = W.cta_unit;
    for (const auto* x : {&W.brick, &W.t0, &W.t1}) units.insert(units.end(), x->begin(), x->end());
    LIFE_TRY(upload(L.units, units, s));
    L.tile_vox.swap(H.tile_vox);
    L.brick_tile_ptr.swap(H.brick_tile_ptr);
    if (L.sparse) L.tile_brick.swap(H.tile_brick);
    if (grouped) ix->batch.brick_prob.swap(H.brick_group);
    LIFE_CUDA_TRY(cudaStreamSynchronize(s));  // order and units are host temporaries
    L.built = true;
    return LIFE_OK;
}

}  // namespace life
