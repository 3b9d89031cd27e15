// Tensor-core (tcgen05) SpMVs on the brick/tile layout.
//
// Both SpMVs are split into a sparse part and a dense contraction with the
// dictionary (Eq. 3: M_v = D Phi_v):
//   DSC  y[:,v] = D · S[:,v],   S[a,v] = Σ_f val·w[f]        (S built in shared memory)
//   WC   Z[a,v] = (Dᵀ r[:,v])[a],  g[f] += val·Z[a,v]         (Z read back from TMEM)
// One CTA per SM walks work units: spatial bricks of voxels, or runs of a brick's
// tiles where there are too few bricks to share out evenly.
// A brick's fascicles are renumbered locally so that w is gathered, and g is
// accumulated, in shared memory: each global gather or atomic then serves all of
// a fascicle's entries inside the brick instead of one entry.
//
// The dense contraction runs on tcgen05.mma (kind::f16: BF16 operands, FP32
// accumulation in TMEM), one 128-voxel tile at a time (MMA M = 128).  Operands
// are K-major, no-swizzle core-matrix layouts in shared memory.
#include <algorithm>
#include <cstring>
#include <type_traits>
#include <vector>

#include "launch_rules.cuh"
#include "tile_layout.cuh"
#include "tc_ptx.cuh"

namespace life {

using namespace ptx;

constexpr uint64_t WAIT_LIMIT = 2000000000ull; // ns before a wait gives up

static unsigned grid1d(int64_t n, int threads = 256) {
    int64_t b = (n + threads - 1) / threads;
    int64_t cap = (int64_t)device_sm_count() * 32;
    return (unsigned)std::max<int64_t>(1, std::min(b, cap));
}

__device__ __forceinline__ float gather_slot(const float* __restrict__ w, int32_t id) {
    return id >= 0 ? __ldg(w + id) : 0.0f;
}

__device__ __forceinline__ uint32_t absmax4_bits(const float4& v) {
    return max(max(__float_as_uint(v.x) & 0x7FFFFFFFu, __float_as_uint(v.y) & 0x7FFFFFFFu),
               max(__float_as_uint(v.z) & 0x7FFFFFFFu, __float_as_uint(v.w) & 0x7FFFFFFFu));
}

// Block maximum of the bits of |x| (non-negative floats order as unsigned ints,
// NaN above +inf), written by thread 0 to *out.
__device__ __forceinline__ void block_absmax_out(uint32_t m, uint32_t* out) {
    __shared__ uint32_t wmax[32];
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t t = 0u;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) t = max(t, wmax[i]);
        *out = t;
    }
}

// ------------------------------------------------- live-entry DSC stream
//
// The sparse-w-aware DSC (Sec. 4.2.1: an entry whose weight is zero contributes
// nothing, and SBB-NNLS iterates keep many weights at exactly zero).  Besides the
// full stream, the index keeps a compacted copy holding only the entries of a
// live set L of brick-local fascicles, with the same (tile, 128-atom chunk)
// structure.  Every DSC call checks on the device whether the input's support
// lies inside L ("stale" otherwise); a small decision kernel then picks the full
// or the compacted stream for this call, and may rebuild the compacted stream
// (L := the input's support) when the input is sparse enough and the stored
// copy is stale or has become much larger than needed.  Dropping zero-weight
// entries only removes exact +0 terms from each run sum, so both streams give
// the same S values up to the association of a run's FP32 sum.

enum : uint32_t { DSC_MODE_NONE = 0, DSC_MODE_FULL = 1, DSC_MODE_COMPACT = 2 };

// Thresholds of the decision: the compacted stream is used only while the live
// slots are at most DENSE_FRAC of all slots, and rebuilt once the live count has
// fallen below SHRINK_FRAC of the count it was built for.  A live set that went
// stale may be rebuilt only `gap` decisions after the last rebuild, and each such
// rebuild doubles the gap (up to MAX_GAP): when fascicles keep entering the
// support (SBB-NNLS iterations bring zero weights back to life), the calls fall
// back to the full stream instead of paying a rebuild every time.
constexpr double DENSE_FRAC = 0.92;
constexpr double SHRINK_FRAC = 0.9;
constexpr uint32_t MAX_GAP = 256;
// Who may rebuild: never (the SBB step's DSC of w), with the backoff (the SBB
// step's DSC of the projected gradient), or whenever the live set is stale or
// shrunk (public DSC calls).
enum : int { ALLOW_NONE = 0, ALLOW_BACKOFF = 1, ALLOW_FREE = 2 };

// The decision for this call, taken by the last block of the gather once every
// block's counts are in.
__device__ void dsc_decide(SparseCtl* c, unsigned long long n_slots, int allow, const life_sbb_state* gate,
                           int gate_mode) {
    volatile SparseCtl* vc = c;
    const unsigned long long nl = vc->n_live;
    const bool stale = vc->stale != 0u;
    c->n_live = 0ull;  // the next gather counts from zero
    c->stale = 0u;
    if (gate_skip(gate, gate_mode)) {
        c->mode = DSC_MODE_NONE;
        c->compact_now = 0u;
        return;
    }
    uint32_t mode, cmp = 0u;
    if (c->gap == 0u) c->gap = 1u;
    c->since += 1u;
    const bool shrunk = (double)nl < SHRINK_FRAC * (double)c->n_live_cmp;
    if ((double)nl > DENSE_FRAC * (double)n_slots) {
        mode = DSC_MODE_FULL;
    } else if (allow && (!c->have || (stale && (allow == ALLOW_FREE || c->since >= c->gap)) || (!stale && shrunk))) {
        if (c->have && stale && allow == ALLOW_BACKOFF) c->gap = c->gap * 2u < MAX_GAP ? c->gap * 2u : MAX_GAP;
        cmp = 1u;
        mode = DSC_MODE_COMPACT;
        c->have = 1u;
        c->n_live_cmp = nl;
        c->n_compactions += 1ull;
        c->since = 0u;
    } else {
        mode = stale ? DSC_MODE_FULL : DSC_MODE_COMPACT;
    }
    c->mode = mode;
    c->compact_now = cmp;
    c->n_calls += 1ull;
    if (mode == DSC_MODE_COMPACT) c->n_compact_calls += 1ull;
}

// wb gather plus the liveness bookkeeping: the number of real slots with a
// non-zero value (NaN counts as non-zero) and whether one of them lies outside
// L; the last block to finish takes the call's decision.
constexpr int GATHER_THREADS = 256;

__global__ void __launch_bounds__(GATHER_THREADS, 8) wb_gather_live_kernel(const int32_t* __restrict__ wsrc, int64_t n,
                                                                        const float* __restrict__ w,
                                                                        float* __restrict__ wb,
                                                                        const uint8_t* __restrict__ live,
                                                                        SparseCtl* __restrict__ ctl,
                                                                        unsigned long long n_slots, int allow,
                                                                        const life_sbb_state* gate, int gate_mode,
                                                                        uint32_t* __restrict__ amax) {
    __shared__ unsigned int blk_n, blk_stale, last;
    if (threadIdx.x == 0) blk_n = blk_stale = 0u;
    __syncthreads();
    const int64_t n4 = n >> 2;
    unsigned int cnt = 0u, stale = 0u;
    uint32_t am = 0u;
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n4; j += (int64_t)gridDim.x * blockDim.x) {
        const int4 id = __ldg(reinterpret_cast<const int4*>(wsrc) + j);
        const uchar4 lv = __ldg(reinterpret_cast<const uchar4*>(live) + j);
        float4 v;
        v.x = gather_slot(w, id.x);
        v.y = gather_slot(w, id.y);
        v.z = gather_slot(w, id.z);
        v.w = gather_slot(w, id.w);
        reinterpret_cast<float4*>(wb)[j] = v;
        am = max(am, absmax4_bits(v));
        // padding slots hold 0 and never count
        const bool nx = v.x != 0.0f, ny = v.y != 0.0f, nz = v.z != 0.0f, nw = v.w != 0.0f;
        cnt += (unsigned)nx + (unsigned)ny + (unsigned)nz + (unsigned)nw;
        stale |= (nx && !lv.x) || (ny && !lv.y) || (nz && !lv.z) || (nw && !lv.w);
    }
    for (int o = 16; o > 0; o >>= 1) {
        cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
        stale |= __shfl_xor_sync(0xffffffffu, stale, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&blk_n, cnt);
        atomicOr(&blk_stale, stale);
    }
    block_absmax_out(am, amax + blockIdx.x);   // (its barrier also orders the block counts above)
    if (threadIdx.x == 0) {
        if (blk_n) atomicAdd(&ctl->n_live, (unsigned long long)blk_n);
        if (blk_stale) atomicOr(&ctl->stale, 1u);
        __threadfence();
        last = atomicAdd(&ctl->gather_done, 1u) == gridDim.x - 1 ? 1u : 0u;
        if (last) {
            __threadfence();
            dsc_decide(ctl, n_slots, allow, gate, gate_mode);
            ctl->gather_done = 0u;
        }
    }
}

struct CompactArgs {
    const int32_t* chunk_ptr;
    const int32_t* tile_brick;
    const int32_t* wb_ptr;
    const float* wb;
    const uint16_t* soff;
    const uint16_t* fl;
    const __nv_bfloat16* val;
    uint8_t* wb_live;
    uint16_t* c_soff;
    uint16_t* c_fl;
    __nv_bfloat16* c_val;
    int32_t* c_chunk_end;   // [n_tiles * chunks per tile] end of each chunk's live entries
    SparseCtl* ctl;
    int n_c;                // 128-atom chunks per tile
    int64_t n_chunks, wb_total;
};

constexpr int CMP_THREADS = 256;

__device__ __forceinline__ uint32_t u16_of(const uint4& v, int e) {
    const uint32_t w = e < 2 ? v.x : e < 4 ? v.y : e < 6 ? v.z : v.w;
    return (e & 1) ? (w >> 16) : (w & 0xFFFFu);
}

// Live flags (bit e) of the 8 entries of the slot at `base` inside [beg, end).
__device__ __forceinline__ uint32_t slot_live(const uint4& flv, int base, int beg, int end, const float* wbb) {
    uint32_t m = 0u;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const int j = base + e;
        if (j >= beg && j < end &&
            *reinterpret_cast<const float*>(reinterpret_cast<const char*>(wbb) + u16_of(flv, e)) != 0.0f)
            m |= 1u << e;
    }
    return m;
}

// Rebuild of the live-entry stream, one warp per 128-atom chunk (8 entries per
// lane per step).  A chunk's live entries are written in order to the start of
// the chunk's own range [beg, end) of the compacted arrays, and its end is
// recorded: no scan is needed and the DSC reads [beg, c_chunk_end).  An entry
// continues a run when the previous LIVE entry of the chunk has the same S offset
// (the same (atom, row)): runs are contiguous in the sorted stream, so that is
// the run it belonged to.  L := the slots whose gathered value is non-zero.
__global__ void __launch_bounds__(CMP_THREADS) cmp_rebuild_kernel(CompactArgs C) {
    if (!C.ctl->compact_now) return;
    for (int64_t j = blockIdx.x * (int64_t)CMP_THREADS + threadIdx.x; j < C.wb_total; j += (int64_t)gridDim.x * CMP_THREADS)
        C.wb_live[j] = C.wb[j] != 0.0f ? 1 : 0;
    const int lane = threadIdx.x & 31;
    const uint32_t below = (1u << lane) - 1u;
    const int64_t warps = (int64_t)gridDim.x * (CMP_THREADS / 32);
    for (int64_t ch = blockIdx.x * (int64_t)(CMP_THREADS / 32) + (threadIdx.x >> 5); ch < C.n_chunks; ch += warps) {
        const int64_t t = ch / C.n_c;
        const float* wbb = C.wb + C.wb_ptr[C.tile_brick[t]];
        const int beg = C.chunk_ptr[ch], end = C.chunk_ptr[ch + 1];
        int out = beg;
        uint32_t prev = 0xFFFFFFFFu;  // S offset of the last live entry so far (none)
        for (int base = (beg & ~7) + lane * 8; __any_sync(0xffffffffu, base < end); base += 256) {
            uint4 flv = make_uint4(0u, 0u, 0u, 0u), sov = flv, vav = flv;
            uint32_t m = 0u;
            if (base < end) {
                flv = __ldg(reinterpret_cast<const uint4*>(C.fl + base));
                sov = __ldg(reinterpret_cast<const uint4*>(C.soff + base));
                vav = __ldg(reinterpret_cast<const uint4*>(C.val) + (base >> 3));
                m = slot_live(flv, base, beg, end, wbb);
            }
            const int n = __popc(m);
            int pre = n;  // inclusive prefix of the live counts over the lanes
            for (int x = 1; x < 32; x <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, pre, x);
                if (lane >= x) pre += y;
            }
            const int total = __shfl_sync(0xffffffffu, pre, 31);
            // S offset of this lane's last live entry, and the previous live entry before this lane
            const uint32_t last_so = m ? (u16_of(sov, 31 - __clz(m)) & 0x7FFFu) : 0u;
            const uint32_t has = __ballot_sync(0xffffffffu, m != 0u);
            const uint32_t lower = has & below;
            const uint32_t from = __shfl_sync(0xffffffffu, last_so, lower ? 31 - __clz(lower) : lane);
            uint32_t p = lower ? from : prev;
            int q = out + pre - n;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                if (!((m >> e) & 1u)) continue;
                const uint32_t so = u16_of(sov, e) & 0x7FFFu;
                C.c_soff[q] = (uint16_t)(so | (p == so ? CONT : 0u));
                C.c_fl[q] = (uint16_t)u16_of(flv, e);
                reinterpret_cast<uint16_t*>(C.c_val)[q] = (uint16_t)u16_of(vav, e);
                p = so;
                ++q;
            }
            if (has) prev = __shfl_sync(0xffffffffu, last_so, 31 - __clz(has));
            out += total;
        }
        if (lane == 0) C.c_chunk_end[ch] = out;
    }
}

__global__ void widen_bf16_kernel(const __nv_bfloat16* __restrict__ in, int64_t n, float* __restrict__ out) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = __bfloat162float(in[i]);
}

// The exported forms of the DSC stream's fields (either may be left out).  va: row |
// atom << 7, the cell from its S byte offset, the 128-atom chunk from the entry's place in
// chunk_ptr (n_seg chunks, n_c per tile).  fl: the brick-local fascicle (the stream holds
// its byte offset in the weight table) | 0x8000 when the entry continues the previous
// entry's (atom, row) (the stream keeps that bit in soff).
__global__ void export_cells_kernel(const uint16_t* __restrict__ soff, const uint16_t* __restrict__ fl,
                                    const int32_t* __restrict__ chunk_ptr, int64_t n_seg, int n_c, int64_t n,
                                    uint16_t* __restrict__ va_out, uint16_t* __restrict__ fl_out) {
    for_entry_segments(chunk_ptr, n_seg, n, [&](int64_t i, int64_t s) {
        const uint32_t k = soff[i], so = k & 0x7FFFu;
        const uint32_t row = (so >> 11) * 8 + ((so >> 4) & 7u), a = ((so >> 7) & 15u) * 8 + ((so >> 1) & 7u);
        if (va_out) va_out[i] = (uint16_t)(row | ((a + (uint32_t)s % (uint32_t)n_c * DKC) << 7));
        if (fl_out) fl_out[i] = (uint16_t)((fl[i] >> 2) | (k & CONT));
    });
}

life_status export_tiles(life_index_s* ix, int32_t* tile_vox, int32_t* chunk_ptr, int32_t* brick_tile_ptr,
                         int32_t* brick_fasc_ptr, int32_t* brick_fasc, int32_t* brick_order, uint16_t* va,
                         uint16_t* fl, float* val, cudaStream_t s) {
    TileLayout& L = ix->tile;
    auto cp = [&](void* dst, const DevBuf& src, size_t bytes) -> life_status {
        if (dst && bytes) LIFE_CUDA_TRY(cudaMemcpyAsync(dst, src.p, bytes, cudaMemcpyDeviceToDevice, s));
        return LIFE_OK;
    };
    LIFE_TRY(cp(tile_vox, L.tile_vox, sizeof(int32_t) * L.n_tiles * TILE_V));
    LIFE_TRY(cp(chunk_ptr, L.chunk_ptr, sizeof(int32_t) * (L.n_tiles * (L.kp / DKC) + 1)));
    LIFE_TRY(cp(brick_tile_ptr, L.brick_tile_ptr, sizeof(int32_t) * (L.n_bricks + 1)));
    LIFE_TRY(cp(brick_fasc_ptr, L.brick_fasc_ptr, sizeof(int32_t) * (L.n_bricks + 1)));
    LIFE_TRY(cp(brick_fasc, L.brick_fasc, L.brick_fasc.bytes));
    LIFE_TRY(cp(brick_order, L.brick_order, sizeof(int32_t) * L.n_bricks));
    if ((va || fl) && L.n_nnz > 0) {
        export_cells_kernel<<<entry_segments_grid(L.n_nnz), 256, 0, s>>>(
            L.soff.as<uint16_t>(), L.fl.as<uint16_t>(), L.chunk_ptr.as<int32_t>(), L.n_tiles * (L.kp / DKC), L.kp / DKC,
            L.n_nnz, va, fl);
        LIFE_CHECK_LAUNCH();
    }
    if (val && L.n_nnz > 0) {
        if (L.vbytes == 4) {
            LIFE_TRY(cp(val, L.val, sizeof(float) * L.n_nnz));
        } else {
            widen_bf16_kernel<<<grid1d(L.n_nnz), 256, 0, s>>>(L.val.as<__nv_bfloat16>(), L.n_nnz, val);
            LIFE_CHECK_LAUNCH();
        }
    }
    LIFE_CUDA_TRY(cudaStreamSynchronize(s));
    return LIFE_OK;
}

// ================================================================ kernels

struct TcArgs {
    const int32_t* tile_vox;
    const int32_t* chunk_ptr;  // DSC stream: entries of (tile t, chunk c) from chunk_ptr[t·n_c + c]
    const int32_t* brick_tile_ptr;
    const int32_t* brick_fasc_ptr;
    const int32_t* brick_fasc;
    const int32_t* cta_unit;   // [grid + 1] work units of each CTA
    const int32_t *u_brick, *u_t0, *u_t1;  // per unit: its brick and its tiles [t0, t1) of it
    const uint16_t* soff;
    const uint16_t* fl;
    const __nv_bfloat16* val;
    const uint16_t* wkey;
    const uint16_t* wfl;
    const __nv_bfloat16* wval;
    const int32_t* wseg_ptr;
    const float* D;
    const float* x;      // DSC: w [Nf];   WC: r [Nθ·Nv]
    const float* b;      // DSC residual or NULL
    float* out;          // DSC: y (or NULL);   WC: g (zeroed by the launch before)
    double* partial;     // DSC: per-CTA FP64 Σ out²
    const float* val32;  // DSC on an FP32-storage index: the stream's values (val is then unused)
    const float* wval32; // WC on an FP32-storage index: the WC stream's values (wval is then unused)
    const float* wb;     // DSC on the live-entry stream: brick weight tables gathered before the launch
    const int32_t* wb_src;  // DSC: global fascicle of each brick-table slot (-1 for padding)
    int gather_w;        // DSC: 1 = the producers gather each brick's table from x themselves
    const int32_t* wb_ptr;
    const float* brick_cv;    // WC: per-brick bound on Σ|val| of one fascicle
    uint32_t* tile_amax;      // bits of |r| maxima, 4 slots per tile (their max is the tile's): DSC writes, WC reads
    const life_sbb_state* gate;
    int gate_mode;
    const unsigned char* d_img;  // BF16 storage: D as this kernel's FP16 MMA operand (np x kp, K-major)
    const uint32_t* d_info;      // [0] kD, the operand's scale exponent; [1 ..] column sums of |D| (n_dblk maxima)
    int n_dblk;
    const uint32_t* x_amax;    // DSC: bits of max |x| per block of the pass that looked for it
    int n_xamax;
    float run_vmax;            // DSC: largest Σ|val| over the entries of one (atom, voxel) run
    const int32_t* chunk_end;  // DSC on the live-entry stream: end of each chunk's entries (else NULL:
                               // a chunk ends where the next begins)
    const SparseCtl* ctl;  // DSC: when set, the launch runs only if ctl->mode == want_mode
    uint32_t want_mode;
    uint32_t* status;
    int nt, na, np, kp, n_sub, n_bricks, max_fb;
    int vec4;            // y / b / r pointers 16-byte aligned and Nθ % 4 == 0
    int dstage;          // DSC, small-table form: S stages
    int y_tile;          // DSC: the small-table form, b and Y pass through a tile in shared memory (needs vec4)
    int wgroups;         // WC: scatter warps per TMEM lane quarter (4, or 2 when shared memory is short)
    int rbufs;           // WC: R tile buffers (2 when shared memory allows: the loader runs a tile ahead)
    BatchGate bg;        // batched launch: bricks of problems that are not live are skipped, and DSC
                         // partial sums go to partial[(p * grid + cta) * DSC_EPI_WARPS + epilogue warp]
};

// The first work unit of this CTA at round >= r whose problem is live (r is advanced
// to its round); -1 when none is left.  Every role of a CTA walks the same
// sequence, since the problem states do not change during a launch.
__device__ __forceinline__ int live_unit(const TcArgs& A, int cta, int& r) {
    for (;; ++r) {
        const int u = A.cta_unit[cta] + r;
        if (u >= A.cta_unit[cta + 1]) return -1;
        if (!A.bg.live || batch_live(A.bg, A.bg.brick_prob[A.u_brick[u]], A.gate_mode)) return u;
    }
}

__device__ __forceinline__ uint32_t align_up(uint32_t x, uint32_t a) { return (x + a - 1) / a * a; }

// Bits of |x|: they order non-negative floats, with +inf above every finite value
// and NaN above +inf.
__device__ __forceinline__ uint32_t abs_bits(float x) { return __float_as_uint(x) & 0x7FFFFFFFu; }

// Lane 0 waits (bounded) and the verdict is broadcast to the warp.
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, volatile int* abort) {
    int ok = 1;
    if ((threadIdx.x & 31) == 0) ok = mbar_wait(bar, parity, abort, WAIT_LIMIT) ? 1 : 0;
    return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

// ------------------------------------------------------------ entry slots
// Producer and scatter threads read the entry streams 8 entries at a time with
// 16-byte loads (the streams are padded to a multiple of 8 entries) and load
// their next slot before working on the current one.

constexpr int SLOT = 8;

struct EntrySlot {
    uint4 key, fl, val;   // key: S offset (DSC), Z offset or (row, atom) (WC)
};

__device__ __forceinline__ void load_slot(const uint16_t* key, const TcArgs& A, int base, EntrySlot& s) {
    s.key = __ldg(reinterpret_cast<const uint4*>(key + base));
    s.fl = __ldg(reinterpret_cast<const uint4*>(A.fl + base));
    s.val = __ldg(reinterpret_cast<const uint4*>(A.val) + (base >> 3));
}

__device__ __forceinline__ uint32_t u16_at(const uint4& v, int e) {
    const uint32_t w = e < 2 ? v.x : e < 4 ? v.y : e < 6 ? v.z : v.w;
    return (e & 1) ? (w >> 16) : (w & 0xFFFFu);
}

__device__ __forceinline__ float bf16_at(const uint4& v, int e) { return __uint_as_float(u16_at(v, e) << 16); }

// FP32-storage DSC stream: a slot's 8 values take two 16-byte loads.
struct EntrySlot32 {
    uint4 key, fl, val, val2;
};

__device__ __forceinline__ void load_slot(const uint16_t* key, const TcArgs& A, int base, EntrySlot32& s) {
    s.key = __ldg(reinterpret_cast<const uint4*>(key + base));
    s.fl = __ldg(reinterpret_cast<const uint4*>(A.fl + base));
    const uint4* v = reinterpret_cast<const uint4*>(A.val32) + (base >> 2);
    s.val = __ldg(v);
    s.val2 = __ldg(v + 1);
}

__device__ __forceinline__ float slot_val(const EntrySlot& s, int e) { return bf16_at(s.val, e); }

__device__ __forceinline__ float slot_val(const EntrySlot32& s, int e) {
    const uint4& v = e < 4 ? s.val : s.val2;
    const int i = e & 3;
    return __uint_as_float(i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w);
}

// Value of stream entry j, read from memory (the tail of a run that leaves the warp).
__device__ __forceinline__ float stream_val(const TcArgs& A, const EntrySlot&, int j) {
    return __bfloat162float(A.val[j]);
}

__device__ __forceinline__ float stream_val(const TcArgs& A, const EntrySlot32&, int j) { return A.val32[j]; }

__device__ __forceinline__ int chunk_beg(const TcArgs& A, int t, int c, int n_c) {
    return A.chunk_ptr[(int64_t)t * n_c + c];
}

__device__ __forceinline__ int chunk_end(const TcArgs& A, int t, int c, int n_c) {
    return A.chunk_end ? A.chunk_end[(int64_t)t * n_c + c] : A.chunk_ptr[(int64_t)t * n_c + c + 1];
}

// Advances (r, unit, t, c) to the CTA's next chunk; false when none is left.
__device__ __forceinline__ bool next_chunk(const TcArgs& A, int cta, int n_c, int& r, int& unit, int& t, int& c,
                                           bool& new_unit) {
    new_unit = false;
    if (++c < n_c) return true;
    c = 0;
    if (++t < A.u_t1[unit]) return true;
    ++r;
    const int nu = live_unit(A, cta, r);
    if (nu < 0) return false;
    unit = nu;
    t = A.u_t0[unit];
    new_unit = true;
    return true;
}

// dst[idx[i]] += tab[i] for every non-zero tab[i], i < n (one atomic per fascicle).
// With inv != 0 the table holds int32 values in units of inv.
__device__ __forceinline__ void flush_table(float* dst, const float* tab, const int32_t* __restrict__ idx, int n,
                                            int tid, int nthr, float inv = 0.0f) {
    constexpr int U = 16;  // index loads in flight per thread
    for (int b0 = 0; b0 < n; b0 += U * nthr) {
        int id[U];
        float v[U];
#pragma unroll
        for (int e = 0; e < U; ++e) {
            const int i = b0 + e * nthr + tid;
            v[e] = i < n ? tab[i] : 0.0f;
            if (inv != 0.0f) v[e] = (float)__float_as_int(v[e]) * inv;
            id[e] = (i < n && v[e] != 0.0f) ? __ldg(idx + i) : -1;
        }
#pragma unroll
        for (int e = 0; e < U; ++e)
            if (id[e] >= 0) red_add_global_f32(dst + id[e], v[e]);
    }
}

// ---------------------------------------------------------------------- DSC

constexpr int DSC_PROD_WARPS = 23;   // 28 warps in all: 7 per SM sub-partition fit 72 registers
constexpr int DSC_EPI_WARPS = 4;
constexpr int DSC_MMA_WARP = DSC_PROD_WARPS + DSC_EPI_WARPS;
constexpr int DSC_THREADS = (DSC_MMA_WARP + 1) * 32;
constexpr int DSC_PROD_THREADS = DSC_PROD_WARPS * 32;
constexpr uint32_t DS_BYTES = TILE_V * DKC * 2;           // one S chunk: 128 rows x 128 atoms, bf16
constexpr uint32_t DS_SBO = (DKC / 8) * 128;              // 8-row group stride of an S chunk

// All-zero source of the bulk copies that clear an S stage (zero-initialised
// device memory, read through L2).
static __device__ __align__(128) uint4 g_zero_chunk[DS_BYTES / 16];

// FP32 storage: each epilogue warp transposes its 32 x 32 blocks of Y through a
// padded shared-memory tile.
constexpr uint32_t DSC_TW = 33;  // row stride (floats) of an epilogue warp's transpose tile

// Shared memory of a DSC CTA: D as an MMA operand (BF16 storage only: with FP32
// storage D's two FP16 parts sit in tensor memory), the S stages (FP32 storage:
// hi and lo parts), the brick weight table, and (FP32) the epilogue's transpose tiles.
// (y_tile: a whole tile of Y instead, rows of dsc_y_stride bytes).
__host__ __device__ inline uint32_t dsc_y_stride(int nt) { return (uint32_t)((nt + 31) / 32 * 32 + 4) * 4u; }

__host__ __device__ inline uint32_t dsc_smem_bytes(int np, int kp, int nt, int max_fb, bool f32, int stages,
                                                   bool y_tile) {
    uint32_t d = f32 ? 0u : (uint32_t)np * kp * 2;
    d = (d + 1023) / 1024 * 1024;
    return d + (uint32_t)stages * DS_BYTES * (f32 ? 2u : 1u) + 4u * (uint32_t)((max_fb + 3) / 4 * 4 + 4) +
           (y_tile ? TILE_V * dsc_y_stride(nt) : f32 ? 4u * DSC_EPI_WARPS * 32u * DSC_TW : 0u) + 1024;
}

// Tensor-memory columns of a DSC CTA: two 128-column accumulators (BF16 storage),
// or D's FP16 hi and lo parts (kp/2 columns each) and one accumulator (FP32).
__host__ __device__ inline uint32_t dsc_tmem_cols(int kp, bool f32) {
    return (!f32 || kp + 128 <= 256) ? 256u : 512u;
}

// The FP16 remainder of x after its FP16 rounding h (hi + lo carries 22 bits);
// zero where h is infinite, so that an infinite x stays infinite, not NaN.
__device__ __forceinline__ float f16_rest(float x, __half h) {
    const float hf = __half2float(h);
    return isinf(hf) ? 0.0f : x - hf;
}

// hi = FP16(a), lo = FP16 of the remainder, for a pair (a, b).
__device__ __forceinline__ void split_f16x2(float a, float b, uint32_t& hi, uint32_t& lo) {
    const __half ha = __float2half_rn(a), hb = __float2half_rn(b);
    const __half2 h2 = __halves2half2(ha, hb);
    const __half2 l2 = __floats2half2_rn(f16_rest(a, ha), f16_rest(b, hb));
    hi = *reinterpret_cast<const uint32_t*>(&h2);
    lo = *reinterpret_cast<const uint32_t*>(&l2);
}

// S[so] = s·ss as FP16; SPLIT (FP32 storage) also stores the FP16 rounding of
// the remainder in the stage's second half.
template <bool SPLIT>
__device__ __forceinline__ void store_s(unsigned char* S, uint32_t so, float s, float ss) {
    // so: byte offset of the run's (row, atom) in the chunk (a run head: no CONT bit)
    const float x = s * ss;
    const __half h = __float2half_rn(x);
    *reinterpret_cast<__half*>(S + so) = h;
    if (SPLIT) *reinterpret_cast<__half*>(S + DS_BYTES + so) = __float2half_rn(f16_rest(x, h));
}

// S[a, row] for the runs that start inside this slot (a run = entries with the
// same (atom, row)).  All 32 lanes of the warp call this together; lane i+1
// holds the next 8 entries, so a run that goes on past lane i's slot is finished
// with lane i+1's leading continuation sum (one shuffle).  Only runs that also
// cross lane i+1's slot, or leave the warp, are finished from memory.
struct RunState {
    bool have, head_seen;
    uint32_t so;
    float cs, lead;
};

template <bool CHECK, bool SPLIT, class SlotT>
__device__ __forceinline__ void dsc_runs(const SlotT& s, int base, int beg, int end, const float* wl,
                                         unsigned char* S, RunState& st, float ss) {
    // straight-line code: every lane does the same work for every entry
#pragma unroll
    for (int e = 0; e < SLOT; ++e) {
        bool in = true;
        if (CHECK) {
            const int idx = base + e;
            in = idx >= beg && idx < end;
        }
        const uint32_t k = u16_at(s.key, e);  // S byte offset | CONT
        const float t = in ? slot_val(s, e) * *reinterpret_cast<const float*>(
                                 reinterpret_cast<const char*>(wl) + u16_at(s.fl, e)) : 0.0f;
        const bool head = in && !(k & CONT);
        if (head && st.have) store_s<SPLIT>(S, st.so, st.cs, ss);   // the previous run ends here
        st.lead += (!st.have && !head) ? t : 0.0f;       // continuation of a run owned by the lane before
        st.cs = head ? t : st.cs + t;
        st.so = head ? k : st.so;
        st.have = st.have || head;
    }
    st.head_seen = st.have;
}

template <bool SPLIT, class SlotT>
__device__ __forceinline__ void dsc_slot(const TcArgs& A, const SlotT& s, int base, int beg, int end,
                                         const float* wl, unsigned char* S, int lane, float ss) {
    RunState st{false, false, 0u, 0.0f, 0.0f};
    if (base >= beg && base + SLOT <= end) dsc_runs<false, SPLIT>(s, base, beg, end, wl, S, st, ss);
    else dsc_runs<true, SPLIT>(s, base, beg, end, wl, S, st, ss);
    // a run may pass through this whole slot into the one after it
    const int through = (!st.head_seen && base + SLOT < end) ? 1 : 0;
    const float nlead = __shfl_down_sync(0xffffffffu, st.lead, 1);
    const int nthrough = __shfl_down_sync(0xffffffffu, through, 1);
    if (st.have) {
        const int j0 = base + SLOT;
        if (j0 < end) {
            if (lane < 31 && !nthrough) {
                st.cs += nlead;
            } else {
                for (int j = j0; j < end; ++j) {
                    if (!(A.soff[j] & CONT)) break;
                    st.cs += stream_val(A, s, j) * *reinterpret_cast<const float*>(
                                                       reinterpret_cast<const char*>(wl) + A.fl[j]);
                }
            }
        }
        store_s<SPLIT>(S, st.so, st.cs, ss);
    }
}

// Batched launch: adds this epilogue warp's Σ out² for problem p to its own slot
// (one writer per slot, so the sum is deterministic) and restarts the sum.
__device__ __forceinline__ void dsc_flush_sq(const TcArgs& A, double& sq, int p, int G, int cta, int q, int lane) {
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if (lane == 0 && A.partial) A.partial[((int64_t)p * G + cta) * DSC_EPI_WARPS + q] += sq;
    sq = 0.0;
}

// ------------------------------------------------------ FP16 MMA operands
// The stored precision stays BF16 (Phi values, D); the operands the tensor cores
// read are FP16 (11 significand bits) under exact power-of-two scales, so that
// the per-call roundings of S (DSC) and of the r tile (WC) cost 2^-11 instead
// of the 2^-8 of BF16 (BF16 D values convert to FP16 exactly once scaled into
// FP16's normal range).

// Largest k with bound·2^k < 2^15 (FP16 holds up to 65504), for bound < 2^e;
// 0 for a zero or non-finite bound (NaN and inf then propagate as such).
__device__ __forceinline__ int f16_scale_exp(uint32_t bound_bits) {
    const float b = __uint_as_float(bound_bits);
    if (bound_bits == 0u || !(b <= 3.0e38f)) return 0;
    int e = 0;
    (void)frexpf(b, &e);
    return max(-120, min(120, 15 - e));
}

__device__ __forceinline__ uint32_t warp_max_u32(uint32_t v) {
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Largest of n words, by every warp for itself.
__device__ __forceinline__ uint32_t max_of_parts(const uint32_t* p, int n) {
    uint32_t m = 0u;
    for (int i = threadIdx.x & 31; i < n; i += 32) m = max(m, p[i]);
    return warp_max_u32(m);
}

// ------------------------------------------------- a call's small preparations
//
// One launch before the DSC, or before a WC whose r no DSC of this index wrote,
// does what every CTA of those kernels would otherwise do for itself:
//  - D as the MMA operands the CTAs copy into shared memory with one bulk copy each
//    (BF16 storage: D's BF16 values as FP16 times 2^kD, K-major, once with rows θ for
//    the DSC and once with rows = atoms for the WC), its scale exponent kD, and per
//    block of atoms the largest column sum of |D| (WC's fixed-point bound);
//  - DSC: per block, the bits of max |x| over the finite values of x, the scale of
//    the FP16 S operand (a NaN or inf weight makes its run sums non-finite whatever
//    the scale; leaving it out keeps every other S value scaled into FP16's range);
//  - the zeroes of the g that the next WC adds into.
// Staged by each CTA from the float32 D (a pass to round and store it, one for its
// maximum, one to scale it), D took the first 12 us of every DSC launch and 17 us
// of every WC launch; a copy of the finished operand takes 2 to 3 us, and in the
// kernels only the thread that issues the MMAs waits for it.
// Each block of atoms looks for the maximum of all of D itself, so the blocks are
// large: 1024 threads read the 138 KB of a 96 x 360 D in one round of 16-byte loads
// (256 threads took the launch 3 us longer).
constexpr int PREP_THREADS = 1024;

struct PrepArgs {
    const float* D;
    unsigned char *img_dsc, *img_wc;  // NULL: FP32 storage (the kernels keep D's parts in tensor memory)
    uint32_t* info;                   // [0] kD, [1 ..] column-sum maxima per block of atoms
    const float* x;                   // DSC input, or NULL
    int64_t n_x;
    uint32_t* x_amax;
    float* zero;                      // cleared, or NULL
    int64_t n_zero;
    int nt, na, np, kp, n_dblk, n_xblk;
};

// Part blk of the D work, in blocks of THREADS threads (one atom a warp).
template <int THREADS>
__device__ __forceinline__ void prep_d(const PrepArgs& P, int blk) {
    __shared__ uint32_t dmax_bits, sum_bits;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) dmax_bits = sum_bits = 0u;
    __syncthreads();
    uint32_t m = 0u;
    const int n = P.nt * P.na;
    if ((reinterpret_cast<uintptr_t>(P.D) & 15) == 0) {
#pragma unroll 8
        for (int i = tid; i < n / 4; i += THREADS) m = max(m, absmax4_bits(__ldg(reinterpret_cast<const float4*>(P.D) + i)));
        for (int i = n / 4 * 4 + tid; i < n; i += THREADS) m = max(m, abs_bits(__ldg(P.D + i)));
    } else {
#pragma unroll 8
        for (int i = tid; i < n; i += THREADS) m = max(m, abs_bits(__ldg(P.D + i)));
    }
    m = warp_max_u32(m);
    if (lane == 0) atomicMax(&dmax_bits, m);
    __syncthreads();
    if (!P.img_dsc) {
        if (blk == 0 && tid == 0) P.info[0] = (uint32_t)f16_scale_exp(dmax_bits);
        return;
    }
    // the largest BF16 |D| is the BF16 rounding of the largest |D|
    const float dmax = __bfloat162float(__float2bfloat16_rn(__uint_as_float(dmax_bits)));
    const int kD = f16_scale_exp(abs_bits(dmax));
    if (blk == 0 && tid == 0) P.info[0] = (uint32_t)kD;
    const float sc = ldexpf(1.0f, kD);
    const uint32_t sbo_d = (uint32_t)(P.kp / 8) * 128u, sbo_k = (uint32_t)(P.np / 8) * 128u;
    const int a = blk * (THREADS / 32) + warp;
    float sum = 0.0f;
    for (int t = lane; t < P.np; t += 32) {
        const float d = a < P.na && t < P.nt ? __bfloat162float(__float2bfloat16_rn(__ldg(P.D + (int64_t)P.nt * a + t))) : 0.0f;
        const __half h = __float2half_rn(d * sc);
        *reinterpret_cast<__half*>(P.img_dsc + kmajor_off(t, a, sbo_d)) = h;
        *reinterpret_cast<__half*>(P.img_wc + kmajor_off(a, t, sbo_k)) = h;
        sum += fabsf(d);
    }
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    // (a NaN column sum gives bits above those of +inf)
    if (lane == 0) atomicMax(&sum_bits, abs_bits(sum));
    __syncthreads();
    if (tid == 0) P.info[1 + blk] = sum_bits;
}

__device__ __forceinline__ void prep_zero(const PrepArgs& P, int64_t i0, int64_t n_thr) {
    if (!P.zero) return;
    if ((reinterpret_cast<uintptr_t>(P.zero) & 15) == 0) {
        for (int64_t i = i0; i < P.n_zero / 4; i += n_thr) reinterpret_cast<float4*>(P.zero)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int64_t i = P.n_zero / 4 * 4 + i0; i < P.n_zero; i += n_thr) P.zero[i] = 0.0f;
    } else {
        for (int64_t i = i0; i < P.n_zero; i += n_thr) P.zero[i] = 0.0f;
    }
}

// Blocks [0, n_dblk) prepare D, the n_xblk after them x and the zeroes.
__global__ void __launch_bounds__(PREP_THREADS) tc_prep_kernel(PrepArgs P) {
    if ((int)blockIdx.x < P.n_dblk) {
        prep_d<PREP_THREADS>(P, blockIdx.x);
        return;
    }
    const int blk = blockIdx.x - P.n_dblk;
    const int64_t i0 = blk * (int64_t)PREP_THREADS + threadIdx.x, n_thr = (int64_t)P.n_xblk * PREP_THREADS;
    prep_zero(P, i0, n_thr);
    if (!P.x) return;
    uint32_t m = 0u;
    auto take = [&](float x) {
        const uint32_t bits = abs_bits(x);
        if (bits < 0x7F800000u) m = max(m, bits);
    };
    if ((reinterpret_cast<uintptr_t>(P.x) & 15) == 0) {
#pragma unroll 4
        for (int64_t i = i0; i < P.n_x / 4; i += n_thr) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(P.x) + i);
            take(v.x);
            take(v.y);
            take(v.z);
            take(v.w);
        }
        for (int64_t i = P.n_x / 4 * 4 + i0; i < P.n_x; i += n_thr) take(__ldg(P.x + i));
    } else {
        for (int64_t i = i0; i < P.n_x; i += n_thr) take(__ldg(P.x + i));
    }
    block_absmax_out(m, P.x_amax + blk);
}

// F32 = false: BF16 storage; S (A operand, 128 tile rows x K) and D (B operand)
// in shared memory, Yᵀ[rows x θ] in one of two tensor-memory accumulators.
// F32 = true: FP32 storage; D = D_hi + D_lo (FP16 parts of D·2^kD) is the A
// operand in tensor memory (lane θ), S = S_hi + S_lo the B operand in shared
// memory, Y[θ x rows] = D_hi·S_hi + D_hi·S_lo + D_lo·S_hi in one accumulator
// (the dropped D_lo·S_lo is ~2^-22 of the product).
//
// SMALL (BF16 storage): the form for small brick tables, i.e. sparse tiles (17 entries a
// voxel on the 64^3 workload, where a 128-atom chunk is three 256-entry blocks).  There
// a chunk's cost is its latency, and the table leaves shared memory for more:
//  - the tile's rows of b are bulk-copied into shared memory while its S is formed, b
//    is subtracted from Y in place there and Y bulk-copied out: the epilogue's reads of
//    b, a few 16-byte loads a thread at a time, took 7 us of the 8 us a tile had;
//  - up to four S stages, and the warp that takes a chunk's first block
//    moves on by DSC_ROT from chunk to chunk (the same three of the 23 producers had
//    all the work).
// 64^3 workload: 130 -> 108 us with b, an iteration 418 -> 367 us.  Where it is taken, and
// with how many stages, is dsc_form's rule (with tables of the paper's size it does not
// fit).  FP32 storage, whose accumulator has θ along the lanes, lost by it (64^3: 176 ->
// 306 us).
constexpr int DSC_ROT = 7;

template <bool F32, bool SMALL>
__global__ void __maxnreg__(72) dsc_tc_kernel(TcArgs A) {
    using SlotT = typename std::conditional<F32, EntrySlot32, EntrySlot>::type;
    constexpr uint32_t STG = F32 ? 2 * DS_BYTES : DS_BYTES;  // bytes of one S stage
    constexpr uint32_t NACC = F32 ? 1 : 2;                    // accumulators in flight
    extern __shared__ unsigned char smem_raw[];
    constexpr int NST = SMALL ? DSTAGE_MAX : DSTAGE;
    const int dst = SMALL ? A.dstage : DSTAGE;
    __shared__ uint64_t full_bar[NST], empty_bar[NST], zero_bar[NST], acc_full[2], acc_empty[2], fin_bar, tab_bar,
        d_ready, b_full[DSC_EPI_WARPS];
    __shared__ uint32_t tmem_base;
    __shared__ int abort_flag, never;
    __shared__ int chunk_next[NST];  // next dynamically handed-out 256-entry block of the stage's chunk
    __shared__ double red[DSC_EPI_WARPS];
    if (!A.bg.live && gate_skip(A.gate, A.gate_mode)) return;
    // full or compacted stream: of the two launches of a call, the one not chosen returns here
    if (A.ctl && A.ctl->mode != A.want_mode) return;
    const bool write_y = A.out != nullptr && (A.bg.live || !(A.gate && A.gate_mode == GATE_ACTIVE_Y_EQ8 &&
                                                               A.gate->eq != 8));
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    unsigned char* smem = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t d_bytes = F32 ? 0u : align_up((uint32_t)A.np * A.kp * 2, 1024);
    unsigned char* Ds = smem;
    unsigned char* Ss = smem + d_bytes;
    float* wl = reinterpret_cast<float*>(Ss + dst * STG);
    // the epilogue warps' transpose tiles (F32), or the tile of Y (SMALL)
    float* Ts = wl + ((A.max_fb + 3) / 4 * 4 + 4);
    const uint32_t SBO_D = (uint32_t)(A.kp / 8) * 128u;
    const uint32_t d_copy = (uint32_t)A.np * A.kp * 2;
    if (tid == 0) {
        for (int s = 0; s < dst; ++s) {
            mbar_init(&full_bar[s], DSC_PROD_WARPS);
            mbar_init(&empty_bar[s], 1);
            mbar_init(&zero_bar[s], 1);
            chunk_next[s] = DSC_PROD_WARPS;
        }
        mbar_init(&tab_bar, 1);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], DSC_EPI_WARPS);
        }
        for (int w = 0; w < DSC_EPI_WARPS; ++w) mbar_init(&b_full[w], 1);
        mbar_init(&fin_bar, 1);
        // BF16 storage: one bulk copy; FP32: every producer and epilogue warp stores part of D
        mbar_init(&d_ready, F32 ? DSC_MMA_WARP : 1);
        abort_flag = 0;
        never = 0;
        fence_barrier_init();
        if (!F32) {
            // D as the B operand: rows θ (N), K = atoms, FP16 times 2^kD
            mbar_arrive_expect_tx(&d_ready, d_copy);
            bulk_copy_g2s(Ds, A.d_img, d_copy, &d_ready);
        }
    }
    const int kD = (int)A.d_info[0];
    // S = Σ_run val·x is stored as FP16 times 2^kS, with |S| <= run_vmax · max|x|
    int kS = 0;
    {
        const uint32_t xmax_bits = max_of_parts(A.x_amax, A.n_xamax);
        const float xmax = __uint_as_float(xmax_bits);
        if (xmax_bits != 0u && xmax <= 3.0e38f && A.run_vmax > 0.0f) {
            int ex = 0, er = 0;
            (void)frexpf(xmax, &ex);
            (void)frexpf(A.run_vmax, &er);
            kS = max(-120, min(120, 15 - ex - er));
        }
    }
    const float s_scale = ldexpf(1.0f, kS), y_unscale = ldexpf(1.0f, -kS - kD);
    const uint32_t tmem_cols = dsc_tmem_cols(A.kp, F32);
    if (warp == DSC_MMA_WARP) {
        tmem_alloc(&tmem_base, tmem_cols);
        tmem_relinquish();
    }
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tb = tmem_base;
    const int G = gridDim.x, cta = blockIdx.x;
    const int n_c = A.kp / DKC;
    double sq = 0.0;

    if (F32 && warp < DSC_MMA_WARP) {
        // D·2^kD as FP16 hi and lo parts into tensor memory (lane θ, atom pairs along
        // the columns, hi in [0, kp/2), lo in [kp/2, kp), zero-padded), shared by the
        // producer and epilogue warps: each writes its lane quarter warp % 4, taking
        // every n-th group of 16 columns among the warps of that quarter
        const int q4 = warp & 3, rank = warp >> 2, nwq = (DSC_MMA_WARP - 1 - q4) / 4 + 1;
        const int th = 32 * q4 + lane, half = A.kp / 2;
        const float sc = ldexpf(1.0f, kD);
        const uint32_t ta = tb + ((uint32_t)(32 * q4) << 16);
        for (int c0 = 16 * rank; c0 < half; c0 += 16 * nwq) {
            float d[32];  // loads first: the stores below stay ordered with memory accesses
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                const int a0 = 2 * c0 + j;
                d[j] = (th < A.nt && a0 < A.na) ? __ldg(A.D + (int64_t)A.nt * a0 + th) * sc : 0.0f;
            }
            uint32_t rh[16], rl[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) split_f16x2(d[2 * j], d[2 * j + 1], rh[j], rl[j]);
            tmem_st16(ta + (uint32_t)c0, rh);
            tmem_st16(ta + (uint32_t)(half + c0), rl);
        }
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&d_ready);
    }
    if (warp < DSC_PROD_WARPS) {
        // ---------------- producers: S[a, row] = Σ val·w for one 128-atom chunk
        int r = 0;
        const int u0 = live_unit(A, cta, r);
        if (u0 >= 0) {
            int unit = u0, t = A.u_t0[unit], c = 0;
            int beg = chunk_beg(A, t, 0, n_c), end = chunk_end(A, t, 0, n_c);
            int vw = warp;  // the warp's place in the chunk: it takes block vw first
            uint32_t st = 0, ph = 0;
            int base = (beg & ~7) + tid * SLOT;
            SlotT cur{};
            if (base < end) load_slot(A.soff, A, base, cur);
            bool new_brick = true, dead = false;
            uint32_t tab_ph = 0, tab_n = 0;
            for (;;) {
                if (new_brick) {
                    // every producer is done with the previous brick's weights (and
                    // all take the same abort decision) before the table is replaced
                    if (named_bar_or(1, DSC_PROD_THREADS, dead || abort_flag != 0)) {
                        abort_flag = 1;
                        break;
                    }
                    if (A.gather_w) {
                        // the brick's weights straight from x: slot i holds x[wb_src[o + i]]
                        // (0 for padding); GW slots a round, loads first
                        constexpr int GW = 8;
                        const int o = A.wb_ptr[A.u_brick[unit]], nb4 = A.wb_ptr[A.u_brick[unit] + 1] - o;
                        for (int i0 = tid; i0 < nb4; i0 += GW * DSC_PROD_THREADS) {
                            int32_t id[GW];
#pragma unroll
                            for (int k = 0; k < GW; ++k) {
                                const int i = i0 + k * DSC_PROD_THREADS;
                                id[k] = i < nb4 ? __ldg(A.wb_src + o + i) : -1;
                            }
                            float xv[GW];
#pragma unroll
                            for (int k = 0; k < GW; ++k) xv[k] = id[k] >= 0 ? __ldg(A.x + id[k]) : 0.0f;
#pragma unroll
                            for (int k = 0; k < GW; ++k)
                                if (i0 + k * DSC_PROD_THREADS < nb4) wl[i0 + k * DSC_PROD_THREADS] = xv[k];
                        }
                        // the next brick's slot indices into L2 (they come from DRAM)
                        int rn = r + 1;
                        const int un = live_unit(A, cta, rn);
                        if (un >= 0) {
                            const int o2 = A.wb_ptr[A.u_brick[un]], n2 = A.wb_ptr[A.u_brick[un] + 1] - o2;
                            for (int i = 32 * tid; i < n2; i += 32 * DSC_PROD_THREADS) prefetch_l2(A.wb_src + o2 + i);
                        }
                        named_bar_sync(1, DSC_PROD_THREADS);  // the table is complete
                    } else {
                        if (tid == 0) {  // one bulk copy of the brick's gathered weights
                            const int o = A.wb_ptr[A.u_brick[unit]], nb4 = A.wb_ptr[A.u_brick[unit] + 1] - o;
                            mbar_arrive_expect_tx(&tab_bar, 4u * (uint32_t)nb4);
                            if (nb4 > 0) bulk_copy_g2s(wl, A.wb + o, 4u * (uint32_t)nb4, &tab_bar);
                        }
                        if (!warp_wait(&tab_bar, tab_ph, &abort_flag)) {
                            abort_flag = 1;
                            dead = true;
                        }
                        tab_ph ^= 1u;
                        ++tab_n;
                    }
                }
                unsigned char* S = Ss + st * STG;
                // the stage is free and cleared once the MMA thread's bulk zero copy lands
                if (!dead && !warp_wait(&zero_bar[st], ph, &abort_flag)) {
                    abort_flag = 1;
                    dead = true;
                }
                int nr = r, nunit = unit, nt = t, nc = c;
                bool nnew = false;
                const bool nvalid = next_chunk(A, cta, n_c, nr, nunit, nt, nc, nnew);
                int nbeg = 0, nend = 0;
                if (nvalid) {
                    nbeg = chunk_beg(A, nt, nc, n_c);
                    nend = chunk_end(A, nt, nc, n_c);
                }
                const int nvw = !SMALL ? warp : vw >= DSC_ROT ? vw - DSC_ROT : vw + DSC_PROD_WARPS - DSC_ROT;
                const int nbase = (nbeg & ~7) + (32 * nvw + lane) * SLOT;
                const bool nhave = nvalid && nbase < nend;
                SlotT nxt{};
                bool pf = false;
                // The chunk is cut into 256-entry blocks (one slot per lane): warp w
                // takes block w, then blocks handed out by the stage's counter, so
                // the warps finish a chunk together.  Every lane of a warp runs the
                // same number of slot steps, so dsc_slot can shuffle.
                const int bb = beg & ~7;
                int blk = vw;
                while (!dead && bb + blk * (32 * SLOT) < end) {
                    int nb = 0;
                    if (lane == 0) nb = atomicAdd(&chunk_next[st], 1);
                    nb = __shfl_sync(0xffffffffu, nb, 0);
                    const int b2 = bb + nb * (32 * SLOT) + lane * SLOT;
                    const bool more = bb + nb * (32 * SLOT) < end;  // warp-uniform
                    if (more) {
                        if (b2 < end) load_slot(A.soff, A, b2, nxt);
                        else nxt = SlotT{};
                    } else if (nhave) {
                        load_slot(A.soff, A, nbase, nxt);
                        pf = true;
                    }
                    dsc_slot<F32>(A, cur, base, beg, end, wl, S, lane, s_scale);
                    if (!more) break;
                    cur = nxt;
                    base = b2;
                    blk = nb;
                }
                if (!pf && nhave) load_slot(A.soff, A, nbase, nxt);
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0 && !dead) mbar_arrive(&full_bar[st]);
                if (++st == (uint32_t)dst) {
                    st = 0;
                    ph ^= 1u;
                }
                if (!nvalid) break;
                vw = nvw;
                r = nr;
                unit = nunit;
                t = nt;
                c = nc;
                beg = nbeg;
                end = nend;
                new_brick = nnew;
                base = nbase;
                cur = nxt;  // an empty slot when this lane has none in the next chunk
            }
            // no bulk table copy may still be writing shared memory when the CTA exits
            if (tid == 0 && tab_n > 0 && !mbar_wait(&tab_bar, (tab_n - 1) & 1u, &never, WAIT_LIMIT)) abort_flag = 1;
        }
    } else if (warp < DSC_MMA_WARP) {
        // ---------------- epilogue: TMEM -> y (− b), Σ y² (FP32 per row and tile, FP64 across)
        const int q = warp & 3;  // TMEM lanes 32q .. 32q+31
        const int row = 32 * q + lane;
        const bool vec = A.vec4 != 0;
        uint32_t tcount = 0;
        bool stop = false;
        // SMALL: this thread's row of the tile of Y, and the phase of its warp's b copies
        unsigned char* yrow = reinterpret_cast<unsigned char*>(Ts) + (uint32_t)row * dsc_y_stride(A.nt);
        uint32_t bph = 0;
        int cur_p = -1;  // batched launch: problem whose Σ out² is being accumulated
        if (A.bg.live && lane == 0 && A.partial)
            for (int p = 0; p < A.bg.n; ++p) A.partial[((int64_t)p * G + cta) * DSC_EPI_WARPS + q] = 0.0;
        for (int r = 0; !stop; ++r) {
            const int unit = live_unit(A, cta, r);
            if (unit < 0) break;
            bool wy = write_y;
            if (A.bg.live) {
                const int p = A.bg.brick_prob[A.u_brick[unit]];
                wy = write_y && batch_writes_y(A.bg, p, A.gate_mode);
                if (p != cur_p) {
                    if (cur_p >= 0) dsc_flush_sq(A, sq, cur_p, G, cta, q, lane);
                    cur_p = p;
                }
            }
            for (int t = A.u_t0[unit]; t < A.u_t1[unit]; ++t) {
                const uint32_t ab = tcount % NACC, aph = (tcount / NACC) & 1u;
                int vj[4];     // F32: voxel of tile row 32·g + lane
                int vrow = -1; // SMALL: voxel of this thread's row
                if (SMALL) {
                    vrow = A.tile_vox[(int64_t)t * TILE_V + row];
                    bulk_wait_all<true>();  // this lane's row of the tile before has been read out
                    fence_proxy_async_smem();
                    __syncwarp();
                    if (A.b) {
                        const uint32_t nv = __popc(__ballot_sync(0xffffffffu, vrow >= 0));
                        if (lane == 0) mbar_arrive_expect_tx(&b_full[q], nv * 4u * (uint32_t)A.nt);
                        __syncwarp();
                        if (vrow >= 0) bulk_copy_g2s(yrow, A.b + (int64_t)A.nt * vrow, 4u * (uint32_t)A.nt, &b_full[q]);
                    }
                } else if constexpr (F32) {
                    // before the accumulator is ready: the tile's voxels, and its rows of b
                    // into L2 (this thread's row), so that the loads below hit L2
#pragma unroll
                    for (int g4 = 0; g4 < 4; ++g4) vj[g4] = A.tile_vox[(int64_t)t * TILE_V + 32 * g4 + lane];
                    const int vr = A.tile_vox[(int64_t)t * TILE_V + row];
                    if (A.b && vr >= 0)
                        for (int k = 0; k < A.nt; k += 32) prefetch_l2(A.b + (int64_t)A.nt * vr + k);
                }
                bool ok = warp_wait(&acc_full[ab], aph, &abort_flag);
                if (SMALL && A.b) {  // (also before giving up: the copies are into this CTA)
                    ok = warp_wait(&b_full[q], bph, &never) && ok;
                    bph ^= 1u;
                }
                if (!ok) {
                    abort_flag = 1;
                    stop = true;
                    break;
                }
                tc_fence_after();
                if (SMALL) {
                    __syncwarp();
                    const uint32_t taddr = tb + ((uint32_t)(32 * q) << 16) + ab * 128u;
                    float sqf = 0.0f;
                    uint32_t am = 0u;  // bits of max |y| over this warp's rows (for a WC of y)
                    for (int j = 0; j < A.np; j += 16) {
                        uint32_t rr[16];
                        tmem_ld16(taddr + j, rr);
                        tmem_ld_wait();
#pragma unroll
                        for (int e = 0; e < 16; e += 4) {
                            if (vrow < 0 || j + e >= A.nt) continue;
                            float4 yv = make_float4(__uint_as_float(rr[e]) * y_unscale, __uint_as_float(rr[e + 1]) * y_unscale,
                                                    __uint_as_float(rr[e + 2]) * y_unscale, __uint_as_float(rr[e + 3]) * y_unscale);
                            float4* cell = reinterpret_cast<float4*>(yrow) + (j + e) / 4;
                            if (A.b) {
                                const float4 bv = *cell;
                                yv.x -= bv.x;
                                yv.y -= bv.y;
                                yv.z -= bv.z;
                                yv.w -= bv.w;
                            }
                            if (wy) *cell = yv;
                            sqf += yv.x * yv.x + yv.y * yv.y + yv.z * yv.z + yv.w * yv.w;
                            am = max(max(am, max(abs_bits(yv.x), abs_bits(yv.y))), max(abs_bits(yv.z), abs_bits(yv.w)));
                        }
                        __syncwarp();
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&acc_empty[ab]);
                    if (wy) {
                        fence_proxy_async_smem();
                        if (vrow >= 0) bulk_copy_s2g(A.out + (int64_t)A.nt * vrow, yrow, 4u * (uint32_t)A.nt);
                        bulk_commit();
                        am = warp_max_u32(am);
                        if (lane == 0) A.tile_amax[(int64_t)t * 4 + q] = am;
                    }
                    sq += (double)sqf;
                    ++tcount;
                    continue;
                }
                if constexpr (F32) {
                    // Y[θ, tile row]: each 32 x 32 block (this warp's θ quarter, 32 tile
                    // rows) goes through the warp's shared-memory tile, transposed, so that
                    // lane i then owns tile row 32·g4 + i and reads b / writes y for its 32
                    // θ values with 16-byte accesses.  The accumulator is handed back to the
                    // MMA thread as soon as its last block is in registers.
                    float* Tw = Ts + q * (32 * DSC_TW);
                    const uint32_t taddr = tb + ((uint32_t)(32 * q) << 16) + (uint32_t)A.kp;
                    const int th0 = 32 * q, nth = min(32, A.nt - th0);  // θ of this warp
                    const bool vec = A.vec4 != 0;
                    float sqf = 0.0f;
                    uint32_t am = 0u;  // bits of max |y| over this warp's θ and the tile's rows
                    bool released = false;
#pragma unroll
                    for (int g4 = 0; g4 < 4; ++g4) {
                        if (nth <= 0) break;  // a θ quarter beyond Nθ (warp-uniform)
                        const int v = vj[g4];
                        const int64_t o = (int64_t)A.nt * (v >= 0 ? v : 0) + th0;
#pragma unroll
                        for (int h2 = 0; h2 < 2; ++h2) {  // 16 tile rows per load
                            uint32_t rr[16];
                            tmem_ld16(taddr + (uint32_t)(32 * g4 + 16 * h2), rr);
                            tmem_ld_wait();
#pragma unroll
                            for (int e = 0; e < 16; ++e) Tw[(16 * h2 + e) * DSC_TW + lane] = __uint_as_float(rr[e]);
                        }
                        if (g4 == 3) {
                            tc_fence_before();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(&acc_empty[ab]);
                            released = true;
                        }
                        __syncwarp();
                        if (v >= 0) {
                            const float* trow = Tw + lane * DSC_TW;
                            if (vec) {
                                // the row's b values, all loads issued before their first use
                                float4 bv[8];
#pragma unroll
                                for (int m = 0; m < 8; ++m)
                                    bv[m] = (A.b && 4 * m < nth) ? __ldg(reinterpret_cast<const float4*>(A.b + o) + m)
                                                                 : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
                                for (int m = 0; m < 8; ++m) {
                                    if (4 * m >= nth) break;
                                    float4 yv = make_float4(trow[4 * m] * y_unscale - bv[m].x,
                                                            trow[4 * m + 1] * y_unscale - bv[m].y,
                                                            trow[4 * m + 2] * y_unscale - bv[m].z,
                                                            trow[4 * m + 3] * y_unscale - bv[m].w);
                                    if (wy) reinterpret_cast<float4*>(A.out + o)[m] = yv;
                                    sqf += yv.x * yv.x + yv.y * yv.y + yv.z * yv.z + yv.w * yv.w;
                                    am = max(max(am, max(abs_bits(yv.x), abs_bits(yv.y))),
                                             max(abs_bits(yv.z), abs_bits(yv.w)));
                                }
                            } else {
                                // (eight b values on their way at a time, not each waited for:
                                // 64000 voxels of 15 entries, Nθ = 33: 107 -> 55 us a DSC with b)
                                for (int k0 = 0; k0 < nth; k0 += 8) {
                                    float bk[8];
#pragma unroll
                                    for (int e = 0; e < 8; ++e)
                                        bk[e] = (A.b && k0 + e < nth) ? __ldg(A.b + o + k0 + e) : 0.0f;
#pragma unroll
                                    for (int e = 0; e < 8; ++e) {
                                        if (k0 + e >= nth) break;
                                        const float y = trow[k0 + e] * y_unscale - bk[e];
                                        if (wy) A.out[o + k0 + e] = y;
                                        sqf += y * y;
                                        am = max(am, abs_bits(y));
                                    }
                                }
                            }
                        }
                        __syncwarp();  // the tile is rewritten by the next block
                    }
                    sq += (double)sqf;
                    if (wy) {
                        // slot q of the tile: max |y| over θ quarter q (the four slots of a
                        // tile together hold its max, which is what a WC of y reads)
                        am = warp_max_u32(am);
                        if (lane == 0) A.tile_amax[(int64_t)t * 4 + q] = am;
                    }
                    if (!released) {  // a warp with no θ of its own
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&acc_empty[ab]);
                    }
                    ++tcount;
                    continue;
                }
                const int v = A.tile_vox[(int64_t)t * TILE_V + row];
                const uint32_t taddr = tb + ((uint32_t)(32 * q) << 16) + ab * 128u;
                float sqf = 0.0f;
                uint32_t am = 0u;  // bits of max |y| over this warp's rows (for a WC of y)
                for (int j = 0; j < A.np; j += 32) {
                    uint32_t rr[32];
                    int cnt = 32;
                    if (A.np - j >= 32) {
                        tmem_ld32(taddr + j, rr);
                    } else {
                        uint32_t r16[16];
                        tmem_ld16(taddr + j, r16);
#pragma unroll
                        for (int e = 0; e < 16; ++e) rr[e] = r16[e];
                        cnt = 16;
                    }
                    tmem_ld_wait();
                    if (v < 0) continue;
                    const int64_t o = (int64_t)A.nt * v + j;
                    if (vec && j + cnt <= A.nt) {
                        for (int e = 0; e < cnt; e += 4) {
                            float4 yv = make_float4(__uint_as_float(rr[e]) * y_unscale,
                                                    __uint_as_float(rr[e + 1]) * y_unscale,
                                                    __uint_as_float(rr[e + 2]) * y_unscale,
                                                    __uint_as_float(rr[e + 3]) * y_unscale);
                            if (A.b) {
                                const float4 bv = __ldg(reinterpret_cast<const float4*>(A.b + o + e));
                                yv.x -= bv.x;
                                yv.y -= bv.y;
                                yv.z -= bv.z;
                                yv.w -= bv.w;
                            }
                            if (wy) *reinterpret_cast<float4*>(A.out + o + e) = yv;
                            sqf += yv.x * yv.x + yv.y * yv.y + yv.z * yv.z + yv.w * yv.w;
                            am = max(max(am, max(abs_bits(yv.x), abs_bits(yv.y))), max(abs_bits(yv.z), abs_bits(yv.w)));
                        }
                    } else {
                        for (int e = 0; e < cnt; ++e) {
                            if (j + e < A.nt) {
                                float y = __uint_as_float(rr[e]) * y_unscale;
                                if (A.b) y -= A.b[o + e];
                                if (wy) A.out[o + e] = y;
                                sqf += y * y;
                                am = max(am, abs_bits(y));
                            }
                        }
                    }
                }
                sq += (double)sqf;
                if (wy) {
                    for (int o = 16; o > 0; o >>= 1) am = max(am, __shfl_xor_sync(0xffffffffu, am, o));
                    if (lane == 0) A.tile_amax[(int64_t)t * 4 + q] = am;
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&acc_empty[ab]);
                ++tcount;
            }
        }
        if (SMALL) bulk_wait_all<false>();
        if (A.bg.live) {
            if (cur_p >= 0) dsc_flush_sq(A, sq, cur_p, G, cta, q, lane);
        } else {
            for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
            if (lane == 0) red[q] = sq;
        }
    } else if (F32 && lane == 0) {
        // ---------------- MMA issuer: Y[128 x 128] = D[θ x kp] · S (FP16 hi/lo operands)
        const uint32_t idesc = idesc_f16_f32(128, TILE_V);
        const uint32_t sS = smem_u32(Ss), half = (uint32_t)A.kp / 2, acc = tb + (uint32_t)A.kp;
        uint32_t st = 0, ph = 0, tcount = 0;
        uint32_t zlast = 0;  // bit z: parity of the last zero-copy phase issued on stage z
        bool stop = false;
        for (int z = 0; z < dst; ++z) {  // clear both stages (hi and lo parts) for their first use
            mbar_arrive_expect_tx(&zero_bar[z], STG);
            bulk_copy_g2s(Ss + z * STG, g_zero_chunk, DS_BYTES, &zero_bar[z]);
            bulk_copy_g2s(Ss + z * STG + DS_BYTES, g_zero_chunk, DS_BYTES, &zero_bar[z]);
        }
        // D's parts are in tensor memory once every producer and epilogue warp has stored its share
        if (!mbar_wait(&d_ready, 0, &abort_flag, WAIT_LIMIT)) {
            abort_flag = 1;
            stop = true;
        }
        tc_fence_after();
        for (int r = 0; !stop; ++r) {
            const int unit = live_unit(A, cta, r);
            if (unit < 0) break;
            for (int t = A.u_t0[unit]; t < A.u_t1[unit] && !stop; ++t) {
                if (!mbar_wait(&acc_empty[0], (tcount & 1u) ^ 1u, &abort_flag, WAIT_LIMIT)) {
                    abort_flag = 1;
                    stop = true;
                    break;
                }
                tc_fence_after();
                for (int c = 0; c < n_c; ++c) {
                    if (!mbar_wait(&full_bar[st], ph, &abort_flag, WAIT_LIMIT)) { abort_flag = 1; stop = true; break; }
                    tc_fence_after();
                    const uint32_t sb = sS + st * STG;
#pragma unroll
                    for (int kk = 0; kk < DKC / 16; ++kk) {
                        const uint32_t ah = tb + (uint32_t)c * (DKC / 2) + kk * 8u;  // 16 atoms = 8 columns
                        const uint64_t bh = smem_desc(sb + kk * 256u, 128u, DS_SBO);
                        const uint64_t bl = smem_desc(sb + DS_BYTES + kk * 256u, 128u, DS_SBO);
                        mma_f16_tmem_a(acc, ah, bh, idesc, (c | kk) != 0 ? 1u : 0u);
                        mma_f16_tmem_a(acc, ah, bl, idesc, 1u);
                        mma_f16_tmem_a(acc, ah + half, bh, idesc, 1u);
                    }
                    mma_commit(&empty_bar[st]);
                    // once these MMAs have read the stage, clear it for its next use
                    if (!mbar_wait(&empty_bar[st], ph, &abort_flag, WAIT_LIMIT)) { abort_flag = 1; stop = true; break; }
                    chunk_next[st] = DSC_PROD_WARPS;  // published by the arrive below
                    mbar_arrive_expect_tx(&zero_bar[st], STG);
                    bulk_copy_g2s(Ss + st * STG, g_zero_chunk, DS_BYTES, &zero_bar[st]);
                    bulk_copy_g2s(Ss + st * STG + DS_BYTES, g_zero_chunk, DS_BYTES, &zero_bar[st]);
                    zlast ^= 1u << st;
                    if (++st == (uint32_t)dst) {
                        st = 0;
                        ph ^= 1u;
                    }
                }
                if (stop) break;
                mma_commit(&acc_full[0]);
                ++tcount;
            }
        }
        mma_commit(&fin_bar);
        if (!mbar_wait(&fin_bar, 0, &never, WAIT_LIMIT)) abort_flag = 1;
        for (int z = 0; z < dst; ++z)
            if (!mbar_wait(&zero_bar[z], (zlast >> z) & 1u, &never, WAIT_LIMIT)) abort_flag = 1;
    } else if (!F32 && lane == 0) {
        // ---------------- MMA issuer: Yᵀ[128 x np] = S[128 x kp] · Dᵀ (FP16 operands)
        const uint32_t idesc = idesc_f16_f32(128, (uint32_t)A.np);
        const uint32_t sS = smem_u32(Ss), sD = smem_u32(Ds);
        uint32_t st = 0, ph = 0, tcount = 0;
        uint32_t zlast = 0;  // bit z: parity of the last zero-copy phase issued on stage z
        bool stop = false;
        for (int z = 0; z < dst; ++z) {  // clear both stages for their first use
            mbar_arrive_expect_tx(&zero_bar[z], DS_BYTES);
            bulk_copy_g2s(Ss + z * DS_BYTES, g_zero_chunk, DS_BYTES, &zero_bar[z]);
        }
        if (!mbar_wait(&d_ready, 0, &never, WAIT_LIMIT)) {  // D has arrived (also before the CTA may exit)
            abort_flag = 1;
            stop = true;
        }
        for (int r = 0; !stop; ++r) {
            const int unit = live_unit(A, cta, r);
            if (unit < 0) break;
            for (int t = A.u_t0[unit]; t < A.u_t1[unit] && !stop; ++t) {
                const uint32_t ab = tcount & 1u, aph = (tcount >> 1) & 1u;
                if (!mbar_wait(&acc_empty[ab], aph ^ 1u, &abort_flag, WAIT_LIMIT)) { abort_flag = 1; stop = true; break; }
                tc_fence_after();
                const uint32_t d = tb + ab * 128u;
                for (int c = 0; c < n_c; ++c) {
                    if (!mbar_wait(&full_bar[st], ph, &abort_flag, WAIT_LIMIT)) { abort_flag = 1; stop = true; break; }
                    tc_fence_after();
#pragma unroll
                    for (int kk = 0; kk < DKC / 16; ++kk) {
                        const uint64_t ad = smem_desc(sS + st * DS_BYTES + kk * 256u, 128u, DS_SBO);
                        const uint64_t bd = smem_desc(sD + (uint32_t)c * (DKC / 8) * 128u + kk * 256u, 128u, SBO_D);
                        mma_f16(d, ad, bd, idesc, (c | kk) != 0 ? 1u : 0u);
                    }
                    mma_commit(&empty_bar[st]);
                    // once these MMAs have read the stage, clear it for its next use
                    if (!mbar_wait(&empty_bar[st], ph, &abort_flag, WAIT_LIMIT)) { abort_flag = 1; stop = true; break; }
                    chunk_next[st] = DSC_PROD_WARPS;  // published by the arrive below
                    mbar_arrive_expect_tx(&zero_bar[st], DS_BYTES);
                    bulk_copy_g2s(Ss + st * DS_BYTES, g_zero_chunk, DS_BYTES, &zero_bar[st]);
                    zlast ^= 1u << st;
                    if (++st == (uint32_t)dst) {
                        st = 0;
                        ph ^= 1u;
                    }
                }
                if (stop) break;
                mma_commit(&acc_full[ab]);
                ++tcount;
            }
        }
        mma_commit(&fin_bar);
        // a wait that gives up marks the call failed (the host sees LIFE_ETIMEOUT)
        if (!mbar_wait(&fin_bar, 0, &never, WAIT_LIMIT)) abort_flag = 1;
        // no bulk copy may still be writing shared memory when the CTA exits
        for (int z = 0; z < dst; ++z)
            if (!mbar_wait(&zero_bar[z], (zlast >> z) & 1u, &never, WAIT_LIMIT)) abort_flag = 1;
    }
    tc_fence_before();
    __syncthreads();
    // every role's abort decision is visible after the barrier
    if (abort_flag && tid == 0) atomicOr(A.status, DEV_TIMEOUT);
    if (warp == DSC_MMA_WARP) {
        tc_fence_after();
        tmem_dealloc(tb, tmem_cols);
    }
    if (tid == 0 && A.partial && !A.bg.live && !abort_flag) {
        double tot = 0.0;
        for (int e = 0; e < DSC_EPI_WARPS; ++e) tot += red[e];
        A.partial[blockIdx.x] = tot;
    }
}

// ----------------------------------------------------------------------- WC
//
// Scatter warps work independently: warp w owns TMEM lane quarter q = w % 4
// (tile rows 32q .. 32q+31) and every wgroups-th 32-atom sub-chunk, copies that
// 32x32 block of Z into its own shared-memory tile, and adds val·Z into the
// brick's fascicle table for the entries of those rows and atoms (the WC stream
// is ordered by (tile, row quarter, atom, row, fascicle) for exactly this).

constexpr int WC_SCAT_WARPS = 16;
constexpr int WC_LOAD_WARPS = 3;     // 20 warps in all: at 96 registers an SM sub-partition (16K registers) holds 5
constexpr int WC_MMA_WARP = WC_SCAT_WARPS + WC_LOAD_WARPS;
constexpr int WC_THREADS = (WC_MMA_WARP + 1) * 32;
constexpr int WC_SCAT_THREADS = WC_SCAT_WARPS * 32;
constexpr int WC_LOAD_THREADS = WC_LOAD_WARPS * 32;
// Z goes through tensor memory in 128-atom chunks: a ring of ZSLOTS slots of 128
// columns (all 512), so the tensor cores can fill the next chunks while the
// scatter warps still work on earlier ones
constexpr int ZSLOTS = 4;
constexpr uint32_t ZW_BYTES = 32 * ZW * 4;

// Shared memory of a WC CTA: D as an MMA operand (BF16 storage; with FP32 storage
// D's parts sit in tensor memory), the R tile buffers (FP32: hi and lo parts),
// the scatter warps' Z tiles, the brick table.
__host__ __device__ inline uint32_t wc_smem_bytes(int np, int kp, int max_fb, int wgroups, int rbufs = 1,
                                                  bool f32 = false) {
    uint32_t d = f32 ? 0u : (uint32_t)kp * np * 2;
    d = (d + 1023) / 1024 * 1024;
    uint32_t r = (uint32_t)TILE_V * np * 2;
    r = (r + 1023) / 1024 * 1024 * (f32 ? 2u : 1u);
    return d + (uint32_t)rbufs * r + 4u * wgroups * ZW_BYTES + 4u * (uint32_t)(max_fb > 1 ? max_fb : 1) + 1024;
}

// FIXED: the table holds 32-bit integers in units of 1/sc' (sc' a power of two chosen
// so that no partial sum can leave the int32 range); otherwise FP32.  The Z tile
// holds Z·sc, sc also removing the operand scales from Z, so x = val·Z·sc is in
// table units.  The stream's key and fascicle are byte offsets into the Z tile and
// the table.
template <bool CHECK, bool FIXED>
__device__ __forceinline__ void wc_slot_t(const EntrySlot& s, int base, int beg, int end, const float* Zw,
                                          float* gl, uint32_t gl_s) {
    // all reads of Z before the first add: a read is not moved up past an add to the
    // table (they could overlap for all the compiler knows), and one after the other
    // they are a chain of eight round trips to shared memory
    float x[SLOT];
#pragma unroll
    for (int e = 0; e < SLOT; ++e)
        x[e] = bf16_at(s.val, e) * *reinterpret_cast<const float*>(reinterpret_cast<const char*>(Zw) + u16_at(s.key, e));
#pragma unroll
    for (int e = 0; e < SLOT; ++e) {
        if (CHECK) {
            const int idx = base + e;
            if (idx < beg || idx >= end) continue;
        }
        if (FIXED) atomicAdd(reinterpret_cast<int*>(reinterpret_cast<char*>(gl) + u16_at(s.fl, e)), __float2int_rn(x[e]));
        else red_add_shared_f32(gl_s + u16_at(s.fl, e), x[e]);
    }
}

template <bool FIXED>
__device__ __forceinline__ void wc_slot(const EntrySlot& s, int base, int beg, int end, const float* Zw, float* gl,
                                        uint32_t gl_s) {
    if (base >= beg && base + SLOT <= end) wc_slot_t<false, FIXED>(s, base, beg, end, Zw, gl, gl_s);
    else wc_slot_t<true, FIXED>(s, base, beg, end, Zw, gl, gl_s);
}

__device__ __forceinline__ void wc_load_slot(const TcArgs& A, int base, EntrySlot& s) {
    s.key = __ldg(reinterpret_cast<const uint4*>(A.wkey + base));
    s.fl = __ldg(reinterpret_cast<const uint4*>(A.wfl + base));
    s.val = __ldg(reinterpret_cast<const uint4*>(A.wval) + (base >> 3));
}

// A thin segment (at most WC_THIN entries; 45 on the 64^3 workload, 575 at the paper's
// density) is taken one entry a lane, up to four times, instead of eight consecutive
// entries a lane: with 45 entries that kept six lanes busy for eight entries each.
// Lane i's entries beg + i, beg + 32 + i, ... sit in the four words of each field.
// The kernels come with this path (THIN) and without: it takes WC from 135 to 114 us
// (FP32 storage 188 to 154) on the 64^3 workload, and at the paper's density, where no
// segment is thin, costs 5 % (294 to 309 us).  A launch takes it when its segments hold
// at most WC_THIN_MEAN entries on average (64^3 grids: at 91 a segment 122 against 138
// us, FP32 166 against 199; at 136, where most are no longer thin, 160 against 154).
constexpr int WC_THIN = 128;
constexpr int WC_THIN_MEAN = 96;

__device__ __forceinline__ void wc_load_thin(const TcArgs& A, int beg, int end, int lane, uint32_t (&key)[4],
                                             uint32_t (&fl)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int j = beg + 32 * i + lane;
        key[i] = j < end ? (uint32_t)__ldg(A.wkey + j) : 0u;
        fl[i] = j < end ? (uint32_t)__ldg(A.wfl + j) : 0u;
    }
}

template <bool FIXED>
__device__ __forceinline__ void wc_thin(const uint32_t (&key)[4], const uint32_t (&fl)[4], const float (&val)[4], int beg,
                                        int end, int lane, const float* Zw, float* gl, uint32_t gl_s) {
    float x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
        if (beg + 32 * i < end) x[i] = val[i] * *reinterpret_cast<const float*>(reinterpret_cast<const char*>(Zw) + key[i]);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        if (beg + 32 * i + lane >= end) continue;
        if (FIXED) atomicAdd(reinterpret_cast<int*>(reinterpret_cast<char*>(gl) + fl[i]), __float2int_rn(x[i]));
        else red_add_shared_f32(gl_s + fl[i], x[i]);
    }
}

// The first entries of a segment: a thin one's all, else the first two blocks' slots.
template <bool THIN>
__device__ __forceinline__ void wc_load_first(const TcArgs& A, int beg, int end, int lane, EntrySlot& s0, EntrySlot& s1) {
    if (THIN && end - beg <= WC_THIN) {
        uint32_t k[4], f[4];
        wc_load_thin(A, beg, end, lane, k, f);
        s0.key = make_uint4(k[0], k[1], k[2], k[3]);
        s0.fl = make_uint4(f[0], f[1], f[2], f[3]);
        const uint16_t* wv = reinterpret_cast<const uint16_t*>(A.wval) + beg + lane;
        s0.val.x = beg + lane < end ? (uint32_t)__ldg(wv) << 16 : 0u;
        s0.val.y = beg + 32 + lane < end ? (uint32_t)__ldg(wv + 32) << 16 : 0u;
        s0.val.z = beg + 64 + lane < end ? (uint32_t)__ldg(wv + 64) << 16 : 0u;
        s0.val.w = beg + 96 + lane < end ? (uint32_t)__ldg(wv + 96) << 16 : 0u;
        return;
    }
    const int base = (beg & ~7) + lane * SLOT;
    if (base < end) wc_load_slot(A, base, s0);
    if (base + 32 * SLOT < end) wc_load_slot(A, base + 32 * SLOT, s1);
}

__device__ __forceinline__ int wseg(const TcArgs& A, int t, int q, int s) {
    return A.wseg_ptr[((int64_t)t * 4 + q) * A.n_sub + s];
}

// tile_amax[4t .. 4t+3] = (bits of max |r[θ, v]| over the voxels v of tile t, 0, 0,
// 0), for the tiles of the bricks the WC launch works on (a DSC that stores y
// writes the same slots, one per row quarter).  One block per tile; the row voxel ids are staged in shared
// memory so that the loads of r are independent of one another.
constexpr int AMAX_THREADS = 256;

// Blocks [0, P.n_dblk) prepare D for the WC, the others take the tiles and clear g.
__global__ void __launch_bounds__(AMAX_THREADS) wc_amax_kernel(TcArgs A, PrepArgs P) {
    __shared__ int32_t tv[TILE_V];
    __shared__ uint32_t wmax[AMAX_THREADS / 32];
    const int tid = threadIdx.x;
    if ((int)blockIdx.x < P.n_dblk) {
        prep_d<AMAX_THREADS>(P, blockIdx.x);
        return;
    }
    const int blk = blockIdx.x - P.n_dblk, n_blk = gridDim.x - P.n_dblk;
    prep_zero(P, blk * (int64_t)AMAX_THREADS + tid, (int64_t)n_blk * AMAX_THREADS);
    if (!A.bg.live && gate_skip(A.gate, A.gate_mode)) return;
    const int n_tiles = A.brick_tile_ptr[A.n_bricks];
    for (int t = blk; t < n_tiles; t += n_blk) {
        if (A.bg.live) {
            int lo = 0, hi = A.n_bricks - 1;  // the brick of tile t: last brick starting at or before t
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (A.brick_tile_ptr[mid] <= t) lo = mid;
                else hi = mid - 1;
            }
            if (!batch_live(A.bg, A.bg.brick_prob[lo], A.gate_mode)) continue;
        }
        if (tid < TILE_V) tv[tid] = A.tile_vox[(int64_t)t * TILE_V + tid];
        __syncthreads();
        uint32_t m = 0u;
        if (A.vec4) {
            const int q4 = A.nt >> 2, n = TILE_V * q4;
#pragma unroll 4
            for (int i = tid; i < n; i += AMAX_THREADS) {
                const int row = i / q4, c = i - row * q4, v = tv[row];
                if (v >= 0) {
                    const float4 x = __ldg(reinterpret_cast<const float4*>(A.x + (int64_t)A.nt * v) + c);
                    m = max(max(m, max(abs_bits(x.x), abs_bits(x.y))), max(abs_bits(x.z), abs_bits(x.w)));
                }
            }
        } else {
            const int n = TILE_V * A.nt;
#pragma unroll 4
            for (int i = tid; i < n; i += AMAX_THREADS) {
                const int row = i / A.nt, c = i - row * A.nt, v = tv[row];
                if (v >= 0) m = max(m, abs_bits(__ldg(A.x + (int64_t)A.nt * v + c)));
            }
        }
        for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
        if ((tid & 31) == 0) wmax[tid >> 5] = m;
        __syncthreads();
        if (tid == 0) {
            uint32_t x = wmax[0];
            for (int i = 1; i < AMAX_THREADS / 32; ++i) x = max(x, wmax[i]);
            *reinterpret_cast<uint4*>(A.tile_amax + (int64_t)t * 4) = make_uint4(x, 0u, 0u, 0u);
        }
    }
}

// The loader warps take a tile of r in units of 8 values of θ of one row: thread lt
// takes units lt, lt + WC_LOAD_THREADS, ... in batches of UB, each batch's loads
// issued together.  ngrp = np / 8 units a row; unit / ngrp by a multiplication
// (units < 4096, ngrp <= 16: exact).
struct RUnits {
    int ngrp;
    uint32_t magic;
    __device__ __forceinline__ explicit RUnits(int np) : ngrp(np / 8), magic((65536u + np / 8 - 1) / (np / 8)) {}
    __device__ __forceinline__ int row(int u) const { return (int)(((uint32_t)u * magic) >> 16); }
};

// The voxels (-1 for none) of the rows of this thread's UB units from unit u0 on.
template <int UB>
__device__ __forceinline__ void load_r_voxels(const TcArgs& A, int t, int u0, const RUnits& R, int (&v)[UB]) {
#pragma unroll
    for (int s = 0; s < UB; ++s) {
        const int row = R.row(u0 + s * WC_LOAD_THREADS);
        v[s] = row < TILE_V ? __ldg(A.tile_vox + (int64_t)t * TILE_V + row) : -1;
    }
}

// Loads one tile of r for the loader warps and hands each unit to emit(row, θ / 8,
// values).  v holds the voxels of the first batch on entry; each later batch's are
// read while the batch before it is on its way, so that a batch costs one round
// trip to memory, not two.  (Looked up before each unit's load, they made a tile of
// the medium workload 9 us of loading, in a kernel that needs 6 us a tile for the
// rest.  Handed out by shuffles from a register of each lane they did worse at the
// paper's density: the scatter warps keep the shuffles' pipe busy.)
template <int UB, class Emit>
__device__ __forceinline__ void load_r_tile(const TcArgs& A, int t, const RUnits& R, int (&v)[UB], int lt, bool vec,
                                            Emit emit) {
    const int total = TILE_V * R.ngrp;
    for (int u0 = lt; u0 < total; u0 += UB * WC_LOAD_THREADS) {
        float4 lo[UB], hi[UB];
#pragma unroll
        for (int s = 0; s < UB; ++s) {
            const int u = u0 + s * WC_LOAD_THREADS, g = u - R.row(u) * R.ngrp;
            const float* src = A.x + (int64_t)A.nt * v[s] + 8 * g;
            const int n = v[s] >= 0 ? A.nt - 8 * g : 0;  // values of this unit inside the row
            lo[s] = hi[s] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (vec) {
                if (n >= 4) lo[s] = __ldg(reinterpret_cast<const float4*>(src));
                if (n >= 8) hi[s] = __ldg(reinterpret_cast<const float4*>(src) + 1);
            } else {
                if (n > 0) lo[s].x = __ldg(src);
                if (n > 1) lo[s].y = __ldg(src + 1);
                if (n > 2) lo[s].z = __ldg(src + 2);
                if (n > 3) lo[s].w = __ldg(src + 3);
                if (n > 4) hi[s].x = __ldg(src + 4);
                if (n > 5) hi[s].y = __ldg(src + 5);
                if (n > 6) hi[s].z = __ldg(src + 6);
                if (n > 7) hi[s].w = __ldg(src + 7);
            }
        }
        load_r_voxels(A, t, u0 + UB * WC_LOAD_THREADS, R, v);
#pragma unroll
        for (int s = 0; s < UB; ++s) {
            const int u = u0 + s * WC_LOAD_THREADS, row = R.row(u);
            if (u < total) emit(row, u - row * R.ngrp, lo[s], hi[s]);
        }
    }
}

template <bool THIN>
__global__ void __maxnreg__(96) wc_tc_kernel(TcArgs A) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ uint64_t r_full[2], r_empty[2], z_full[ZSLOTS], z_empty[ZSLOTS], fin_bar, d_ready;
    __shared__ uint32_t tmem_base;
    __shared__ int abort_flag, never;
    if (!A.bg.live && gate_skip(A.gate, A.gate_mode)) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    unsigned char* smem = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t d_bytes = align_up((uint32_t)A.kp * A.np * 2, 1024);
    const uint32_t r_bytes = align_up((uint32_t)TILE_V * A.np * 2, 1024);
    const int wg = A.wgroups;
    unsigned char* Dw = smem;
    unsigned char* Rs = smem + d_bytes;  // A.rbufs tiles of r_bytes
    float* Zc = reinterpret_cast<float*>(Rs + A.rbufs * r_bytes);
    float* gl = Zc + 4 * wg * (ZW_BYTES / 4);
    const uint32_t SBO_K = (uint32_t)(A.np / 8) * 128u;  // 8-row groups of both operands (K = θ)

    if (tid == 0) {
        for (int b = 0; b < 2; ++b) {
            mbar_init(&r_full[b], WC_LOAD_WARPS);
            mbar_init(&r_empty[b], 1);
        }
        for (int z = 0; z < ZSLOTS; ++z) {
            mbar_init(&z_full[z], 1);
            mbar_init(&z_empty[z], WC_SCAT_WARPS);
        }
        mbar_init(&fin_bar, 1);
        mbar_init(&d_ready, 1);
        abort_flag = 0;
        never = 0;
        fence_barrier_init();
        // D as the B operand: rows = atoms (N), K = θ, FP16 times 2^kD
        const uint32_t d_copy = (uint32_t)A.kp * A.np * 2;
        mbar_arrive_expect_tx(&d_ready, d_copy);
        bulk_copy_g2s(Dw, A.d_img, d_copy, &d_ready);
    }
    if (warp == WC_MMA_WARP) {
        tmem_alloc(&tmem_base, 512);
        tmem_relinquish();
    }
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tb = tmem_base;
    const int G = gridDim.x, cta = blockIdx.x;
    // the MMA reads D as FP16 times 2^kD (the BF16 values, exactly); each tile's R
    // as FP16 times 2^kR of its brick, so that Z in tensor memory is 2^(kR+kD) Z
    const int kD = (int)A.d_info[0];

    if (warp < WC_SCAT_WARPS) {
        const int q = warp & 3, h = warp >> 2;
        const bool active = h < wg;               // warps beyond wgroups groups only keep step
        float* Zw = Zc + (active ? (h * 4 + q) : 0) * (ZW_BYTES / 4);
        const uint32_t gl_s = smem_u32(gl);
        const int kc = A.kp / 128;  // 128-atom chunks per tile
        uint32_t kcount = 0;        // chunks handed over so far (ring position)
        bool dead = false;
        // max over atoms of Σθ |D[θ, a]| of the BF16 D (NaN above +inf)
        const float d1 = __uint_as_float(max_of_parts(A.d_info + 1, A.n_dblk));
        for (int r = 0;; ++r) {
            const int unit = live_unit(A, cta, r);
            if (unit < 0) break;
            const int brick = A.u_brick[unit];
            const int fb0 = A.brick_fasc_ptr[brick], nfb = A.brick_fasc_ptr[brick + 1] - fb0;
            // (The maximum is the whole brick's in every unit of it, so that the table's unit,
            // and with it the rounding, does not depend on how bricks are shared out.)
            // Fixed point: every entry adds val·Z with |val·Z| <= max|val|·max_a Σθ|D|·max|r|
            // (up to the BF16 roundings of r and D, < 1 %), and a fascicle has at most
            // cnt entries in the brick, so |any partial sum| <= cv·d1·rmax = bnd.  With
            // sc = 2^(29 - e), bnd < 2^e, a table word stays below 2^29·1.01 + cnt/2 < 2^31.
            // Non-finite or tiny bounds keep the FP32 table.
            uint32_t am = 0u;
            for (int i = 4 * A.brick_tile_ptr[brick] + lane; i < 4 * A.brick_tile_ptr[brick + 1]; i += 32)
                am = max(am, A.tile_amax[i]);
            for (int o = 16; o > 0; o >>= 1) am = max(am, __shfl_xor_sync(0xffffffffu, am, o));
            const float bnd = A.brick_cv[brick] * d1 * __uint_as_float(am);
            int bexp = 0;
            (void)frexpf(bnd, &bexp);
            // (Z·sc < 2^29 / cv must also stay finite: cv >= 1e-28)
            const bool fixed = bnd <= 3.0e38f && bnd >= 1.0e-27f && A.brick_cv[brick] >= 1.0e-28f;
            // Z in tensor memory carries the operand scales 2^(kR + kD); the table
            // unit 2^(bexp - 29) is in true units (sc folds both in, exactly)
            const int kZ = f16_scale_exp(am) + kD;
            const float sc = fixed ? ldexpf(1.0f, 29 - bexp - kZ) : ldexpf(1.0f, -kZ),
                        inv = fixed ? ldexpf(1.0f, bexp - 29) : 0.0f;
            // the table's global fascicle ids, read by the flush at the brick's end
            for (int i = 32 * tid; i < nfb; i += 32 * WC_SCAT_THREADS) prefetch_l2(A.brick_fasc + fb0 + i);
            if (named_bar_or(2, WC_SCAT_THREADS, dead || abort_flag != 0)) break;
            for (int i = tid; i < nfb; i += WC_SCAT_THREADS) gl[i] = 0.0f;
            named_bar_sync(2, WC_SCAT_THREADS);
            const int t0 = A.u_t0[unit], t1 = A.u_t1[unit];
            // this warp's segments in order: (t, s) for t in the brick, s = h, h + wg, ...;
            // a warp step covers two 256-entry blocks (lane i: entries 8i.. of each),
            // and the step after it (or the next segment's first) is loaded while the
            // current one is processed
            const EntrySlot zero{make_uint4(0, 0, 0, 0), make_uint4(0, 0, 0, 0), make_uint4(0, 0, 0, 0)};
            constexpr int BLK = 32 * SLOT;
            // segment bounds of this tile and the next, lane i holding wseg(t, q, i) for i <= n_sub
            int bnd_cur = (active && lane <= A.n_sub) ? wseg(A, t0, q, lane) : 0;
            int bnd_nxt = (active && lane <= A.n_sub && t0 + 1 < t1) ? wseg(A, t0 + 1, q, lane) : 0;
            int beg = __shfl_sync(0xffffffffu, bnd_cur, h), end = __shfl_sync(0xffffffffu, bnd_cur, h + 1);
            if (!active) beg = end = 0;
            int base = (beg & ~7) + lane * SLOT;
            EntrySlot cur0 = zero, cur1 = zero;
            if (active) wc_load_first<THIN>(A, beg, end, lane, cur0, cur1);
            for (int t = t0; t < t1 && !dead; ++t) {
                for (int j = 0; j < kc && !dead; ++j, ++kcount) {
                    // chunk j (atoms 128j ..) of tile t sits in slot zs of the ring
                    const uint32_t zs = kcount % ZSLOTS, zu = (kcount / ZSLOTS) & 1u;
                    if (!warp_wait(&z_full[zs], zu, &abort_flag)) {
                        abort_flag = 1;
                        dead = true;
                        break;
                    }
                    tc_fence_after();
                    if (active) {
                        for (int s = 4 * j + h; s < 4 * j + 4; s += wg) {
                            int ns = s + wg, nt = t;
                            if (ns >= A.n_sub) {
                                ns = h;
                                ++nt;
                            }
                            const bool nvalid = nt < t1;
                            const int nb_src = nt == t ? bnd_cur : bnd_nxt;
                            const int nbeg0 = __shfl_sync(0xffffffffu, nb_src, ns), nend0 = __shfl_sync(0xffffffffu, nb_src, ns + 1);
                            const int nbeg = nvalid ? nbeg0 : 0, nend = nvalid ? nend0 : 0;
                            const int nbase = (nbeg & ~7) + lane * SLOT;
                            EntrySlot nxt0 = zero, nxt1 = zero;
                            if (beg < end) {  // an empty segment needs neither Z nor a pass
                                uint32_t rr[32];
                                tmem_ld32(tb + ((uint32_t)(32 * q) << 16) + zs * 128u + (uint32_t)(32 * (s - 4 * j)), rr);
                                tmem_ld_wait();
                                float* zrow = Zw + lane * ZW;
#pragma unroll
                                for (int e = 0; e < 32; ++e) zrow[e] = __uint_as_float(rr[e]) * sc;
                                __syncwarp();
                                if (THIN && end - beg <= WC_THIN) {
                                    wc_load_first<THIN>(A, nbeg, nend, lane, nxt0, nxt1);
                                    const uint32_t k[4] = {cur0.key.x, cur0.key.y, cur0.key.z, cur0.key.w},
                                                   f[4] = {cur0.fl.x, cur0.fl.y, cur0.fl.z, cur0.fl.w};
                                    const float x[4] = {__uint_as_float(cur0.val.x), __uint_as_float(cur0.val.y),
                                                        __uint_as_float(cur0.val.z), __uint_as_float(cur0.val.w)};
                                    if (fixed) wc_thin<true>(k, f, x, beg, end, lane, Zw, gl, gl_s);
                                    else wc_thin<false>(k, f, x, beg, end, lane, Zw, gl, gl_s);
                                } else
                                for (;;) {
                                    const int b2 = base + 2 * BLK;
                                    const bool more = __shfl_sync(0xffffffffu, b2, 0) < end;
                                    if (more) {
                                        if (b2 < end) wc_load_slot(A, b2, nxt0);
                                        if (b2 + BLK < end) wc_load_slot(A, b2 + BLK, nxt1);
                                    } else {
                                        wc_load_first<THIN>(A, nbeg, nend, lane, nxt0, nxt1);
                                    }
                                    if (fixed) {
                                        wc_slot<true>(cur0, base, beg, end, Zw, gl, gl_s);
                                        wc_slot<true>(cur1, base + BLK, beg, end, Zw, gl, gl_s);
                                    } else {
                                        wc_slot<false>(cur0, base, beg, end, Zw, gl, gl_s);
                                        wc_slot<false>(cur1, base + BLK, beg, end, Zw, gl, gl_s);
                                    }
                                    if (!more) break;
                                    cur0 = nxt0;
                                    cur1 = nxt1;
                                    nxt0 = zero;
                                    nxt1 = zero;
                                    base = b2;
                                }
                                __syncwarp();
                            } else {
                                wc_load_first<THIN>(A, nbeg, nend, lane, nxt0, nxt1);
                            }
                            cur0 = nxt0;
                            cur1 = nxt1;
                            base = nbase;
                            beg = nbeg;
                            end = nend;
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&z_empty[zs]);  // this warp is done with the slot
                }
                if (active) {
                    bnd_cur = bnd_nxt;
                    bnd_nxt = (lane <= A.n_sub && t + 2 < t1) ? wseg(A, t + 2, q, lane) : 0;
                }
            }
            if (named_bar_or(2, WC_SCAT_THREADS, dead || abort_flag != 0)) break;
            flush_table(A.out, gl, A.brick_fasc + fb0, nfb, tid, WC_SCAT_THREADS, inv);
        }
    } else if (warp < WC_MMA_WARP) {
        // ---------------- R tile loader: r[:, v] -> FP16 A operand times 2^kR of the
        // brick (rows = voxels, K = θ); kR from the brick's max |r|, as the scatter warps compute it
        const int lt = tid - WC_SCAT_THREADS;
        const bool vec = A.vec4 != 0;
        const RUnits RU(A.np);
        int vv[4], tv = -1;  // the first batch's voxels of tile tv
        uint32_t tcount = 0;
        bool stop = false;
        for (int r = 0; !stop; ++r) {
            const int unit = live_unit(A, cta, r);
            if (unit < 0) break;
            int r_next = r + 1;
            const int next_unit = live_unit(A, cta, r_next), brick = A.u_brick[unit];
            uint32_t am = 0u;
            for (int i = 4 * A.brick_tile_ptr[brick] + lane; i < 4 * A.brick_tile_ptr[brick + 1]; i += 32)
                am = max(am, A.tile_amax[i]);
            const float rs = ldexpf(1.0f, f16_scale_exp(warp_max_u32(am)));
            for (int t = A.u_t0[unit]; t < A.u_t1[unit]; ++t) {
                // R buffer rb, used for the k-th time (tiles go round the buffers)
                const uint32_t rb = A.rbufs == 2 ? (tcount & 1u) : 0u, rk = A.rbufs == 2 ? (tcount >> 1) : tcount;
                unsigned char* Rb = Rs + rb * r_bytes;
                if (tv != t) load_r_voxels(A, t, lt, RU, vv);
                if (!warp_wait(&r_empty[rb], (rk & 1u) ^ 1u, &abort_flag)) {
                    abort_flag = 1;
                    stop = true;
                    break;
                }
                load_r_tile(A, t, RU, vv, lt, vec, [&](int row, int g8, const float4& lo, const float4& hi) {
                    const __half2 p0 = __floats2half2_rn(lo.x * rs, lo.y * rs), p1 = __floats2half2_rn(lo.z * rs, lo.w * rs);
                    const __half2 p2 = __floats2half2_rn(hi.x * rs, hi.y * rs), p3 = __floats2half2_rn(hi.z * rs, hi.w * rs);
                    uint4 pk;
                    pk.x = *reinterpret_cast<const uint32_t*>(&p0);
                    pk.y = *reinterpret_cast<const uint32_t*>(&p1);
                    pk.z = *reinterpret_cast<const uint32_t*>(&p2);
                    pk.w = *reinterpret_cast<const uint32_t*>(&p3);
                    *reinterpret_cast<uint4*>(Rb + kmajor_off(row, 8 * g8, SBO_K)) = pk;
                });
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&r_full[rb]);
                ++tcount;
                tv = t + 1 < A.u_t1[unit] ? t + 1 : next_unit >= 0 ? A.u_t0[next_unit] : t;
                load_r_voxels(A, tv, lt, RU, vv);  // of the tile after this one
                // pull the voxel rows of r of the tile A.rbufs ahead into L2 (the
                // loader runs A.rbufs - 1 tiles ahead of the tensor cores), so that
                // loading it later is not a chain of DRAM round trips
                int tn = t + A.rbufs;
                if (tn >= A.u_t1[unit]) {
                    tn -= A.u_t1[unit];
                    tn = (next_unit >= 0 && A.u_t0[next_unit] + tn < A.u_t1[next_unit])
                             ? A.u_t0[next_unit] + tn : -1;
                }
                if (tn >= 0) {
                    const int32_t* tvn = A.tile_vox + (int64_t)tn * TILE_V;
                    for (int row = lt; row < TILE_V; row += WC_LOAD_THREADS) {
                        const int v = __ldg(tvn + row);
                        if (v < 0) continue;
                        const char* a = reinterpret_cast<const char*>(A.x + (int64_t)A.nt * v);
                        const char* e = a + 4 * A.nt - 1;
                        for (const char* c = a; c < e; c += 128) prefetch_l2(c);
                        prefetch_l2(e);
                    }
                }
            }
        }
    } else if (lane == 0) {
        // ---------------- MMA issuer: Zᵀ[128 x kp] = R[128 x np] · Dᵀ, one 128-atom chunk
        // (N = 128) at a time into the next slot of the tensor-memory ring (FP16 operands)
        const uint32_t idesc = idesc_f16_f32(128, 128u);
        const uint32_t sR0 = smem_u32(Rs), sD = smem_u32(Dw);
        const int kc = A.kp / 128;
        uint32_t tcount = 0, kcount = 0;
        bool stop = false;
        if (!mbar_wait(&d_ready, 0, &never, WAIT_LIMIT)) {  // D has arrived (also before the CTA may exit)
            abort_flag = 1;
            stop = true;
        }
        for (int r = 0; !stop; ++r) {
            const int unit = live_unit(A, cta, r);
            if (unit < 0) break;
            for (int t = A.u_t0[unit]; t < A.u_t1[unit] && !stop; ++t) {
                const uint32_t rb = A.rbufs == 2 ? (tcount & 1u) : 0u, rk = A.rbufs == 2 ? (tcount >> 1) : tcount;
                const uint32_t sR = sR0 + rb * r_bytes;
                if (!mbar_wait(&r_full[rb], rk & 1u, &abort_flag, WAIT_LIMIT)) {
                    abort_flag = 1;
                    stop = true;
                    break;
                }
                for (int j = 0; j < kc; ++j, ++kcount) {
                    const uint32_t zs = kcount % ZSLOTS, zu = (kcount / ZSLOTS) & 1u;
                    if (!mbar_wait(&z_empty[zs], zu ^ 1u, &abort_flag, WAIT_LIMIT)) {  // the slot's last chunk is read
                        abort_flag = 1;
                        stop = true;
                        break;
                    }
                    tc_fence_after();
                    for (int kk = 0; kk < A.np / 16; ++kk) {
                        const uint64_t ad = smem_desc(sR + kk * 256u, 128u, SBO_K);
                        const uint64_t bd = smem_desc(sD + (uint32_t)(16 * j) * SBO_K + kk * 256u, 128u, SBO_K);
                        mma_f16(tb + zs * 128u, ad, bd, idesc, kk != 0 ? 1u : 0u);
                    }
                    mma_commit(&z_full[zs]);
                }
                if (stop) break;
                mma_commit(&r_empty[rb]);
                ++tcount;
            }
        }
        mma_commit(&fin_bar);
        if (!mbar_wait(&fin_bar, 0, &never, WAIT_LIMIT)) abort_flag = 1;
    }
    tc_fence_before();
    __syncthreads();
    if (abort_flag && tid == 0) atomicOr(A.status, DEV_TIMEOUT);
    if (warp == WC_MMA_WARP) {
        tc_fence_after();
        tmem_dealloc(tb, 512);
    }
}

// ------------------------------------------------------------ FP32-storage WC
//
// Z is computed transposed, Z[a, row] = Σθ D[θ, a]·r[θ, row] for each 128-atom
// block of a tile: D = D_hi + D_lo (FP16 parts of D·2^kD) is the A operand in
// tensor memory (lane = atom of the block, np/2 columns per part), the R tile
// R_hi + R_lo (FP16 parts of r·2^kR) the B operand in shared memory, one half
// tile (64 rows, N = 64) at a time: Z = D_hi·R_hi + D_hi·R_lo + D_lo·R_hi into
// the next of three 64-column slots.  Scatter warp w reads tensor-memory lane
// quarter w % 4, i.e. atoms 32·(w % 4) .. of every block, for the row quarters
// h, h + wgroups, ... (h = w / 4), and adds val·Z into FP32 brick tables.

constexpr int Z32_SLOTS = 3;

template <bool CHECK>
__device__ __forceinline__ void wc32_slot_t(const EntrySlot32& s, int base, int beg, int end, const float* Zw,
                                            uint32_t gl_s) {
    // (reads before adds, as in wc_slot_t)
    float x[SLOT];
#pragma unroll
    for (int e = 0; e < SLOT; ++e)
        // key: byte offset of (atom, row) in the atom-major Z tile, which holds Z·sc
        x[e] = slot_val(s, e) * *reinterpret_cast<const float*>(reinterpret_cast<const char*>(Zw) + u16_at(s.key, e));
#pragma unroll
    for (int e = 0; e < SLOT; ++e) {
        if (CHECK) {
            const int idx = base + e;
            if (idx < beg || idx >= end) continue;
        }
        red_add_shared_f32(gl_s + u16_at(s.fl, e), x[e]);
    }
}

__device__ __forceinline__ void wc32_load_slot(const TcArgs& A, int base, EntrySlot32& s) {
    s.key = __ldg(reinterpret_cast<const uint4*>(A.wkey + base));
    s.fl = __ldg(reinterpret_cast<const uint4*>(A.wfl + base));
    const uint4* v = reinterpret_cast<const uint4*>(A.wval32) + (base >> 2);
    s.val = __ldg(v);
    s.val2 = __ldg(v + 1);
}

// Adds val·Z·sc for the entries [beg, end) of one WC segment (Zw[atom][row] holds
// the segment's 32 x 32 block of Z·sc); lane i takes entries 8i .. of each
// 256-entry block, the next block loaded while the current one is processed.
__device__ __forceinline__ void wc32_segment(const TcArgs& A, int beg, int end, const float* Zw, uint32_t gl_s,
                                             int lane) {
    int base = (beg & ~7) + lane * SLOT;
    EntrySlot32 cur{};
    if (base < end) wc32_load_slot(A, base, cur);
    for (;;) {
        const int nb = base + 32 * SLOT;
        const bool more = __shfl_sync(0xffffffffu, nb, 0) < end;  // warp-uniform
        EntrySlot32 nxt{};
        if (more && nb < end) wc32_load_slot(A, nb, nxt);
        if (base >= beg && base + SLOT <= end) wc32_slot_t<false>(cur, base, beg, end, Zw, gl_s);
        else wc32_slot_t<true>(cur, base, beg, end, Zw, gl_s);
        if (!more) break;
        cur = nxt;
        base = nb;
    }
}

template <bool THIN>
__global__ void __maxnreg__(96) wc_tc32_kernel(TcArgs A) {
    extern __shared__ unsigned char smem_raw[];
    __shared__ uint64_t r_full[2], r_empty[2], z_full[Z32_SLOTS], z_empty[Z32_SLOTS], fin_bar, d_ready;
    __shared__ uint32_t tmem_base;
    __shared__ int abort_flag, never;
    if (!A.bg.live && gate_skip(A.gate, A.gate_mode)) return;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    unsigned char* smem = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t r_part = align_up((uint32_t)TILE_V * A.np * 2, 1024), r_bytes = 2 * r_part;  // hi, lo
    const int wg = A.wgroups, kc = A.kp / 128;
    unsigned char* Rs = smem;  // A.rbufs tiles of r_bytes
    float* Zc = reinterpret_cast<float*>(Rs + A.rbufs * r_bytes);
    float* gl = Zc + 4 * wg * (ZW_BYTES / 4);
    const uint32_t SBO_K = (uint32_t)(A.np / 8) * 128u;  // 8-row groups of the R tile (K = θ)
    const uint32_t zb = (uint32_t)(kc * A.np);           // first column of the Z slots
    if (tid == 0) {
        for (int b = 0; b < 2; ++b) {
            mbar_init(&r_full[b], WC_LOAD_WARPS);
            mbar_init(&r_empty[b], 1);
        }
        for (int z = 0; z < Z32_SLOTS; ++z) {
            mbar_init(&z_full[z], 1);
            mbar_init(&z_empty[z], WC_SCAT_WARPS);
        }
        mbar_init(&fin_bar, 1);
        mbar_init(&d_ready, 4 * kc);  // the warps that store D's blocks
        abort_flag = 0;
        never = 0;
        fence_barrier_init();
    }
    if (warp == WC_MMA_WARP) {
        tmem_alloc(&tmem_base, 512);
        tmem_relinquish();
    }
    fence_proxy_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tb = tmem_base;
    const int G = gridDim.x, cta = blockIdx.x;
    const int kD = (int)A.d_info[0];

    if (warp < WC_SCAT_WARPS) {
        const int q = warp & 3, h = warp >> 2;  // atoms 32q .. of each block; row quarters h, h + wg, ...
        const bool active = h < wg;             // warps beyond wgroups groups only keep step
        float* Zw = Zc + (active ? warp : 0) * (ZW_BYTES / 4);
        const uint32_t gl_s = smem_u32(gl);
        if (h < kc) {
            // D·2^kD of block h (atoms 128h + 32q + lane) as FP16 hi and lo parts into
            // this warp's lanes: θ pairs along the columns, zero-padded
            const float sc = ldexpf(1.0f, kD);
            const int a = 128 * h + 32 * q + lane, half = A.np / 2;
            const uint32_t ta = tb + ((uint32_t)(32 * q) << 16) + (uint32_t)(h * A.np);
            for (int c0 = 0; c0 < half; c0 += 8) {
                uint32_t rh[8], rl[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int t0 = 2 * (c0 + j);
                    float d0 = 0.0f, d1 = 0.0f;
                    if (a < A.na) {
                        if (t0 < A.nt) d0 = __ldg(A.D + (int64_t)A.nt * a + t0) * sc;
                        if (t0 + 1 < A.nt) d1 = __ldg(A.D + (int64_t)A.nt * a + t0 + 1) * sc;
                    }
                    split_f16x2(d0, d1, rh[j], rl[j]);
                }
                tmem_st8(ta + (uint32_t)c0, rh);
                tmem_st8(ta + (uint32_t)(half + c0), rl);
            }
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&d_ready);
        }
        uint32_t kcount = 0;  // Z slots handed over so far (ring position)
        bool dead = false;
        for (int r = 0;; ++r) {
            const int unit = live_unit(A, cta, r);
            if (unit < 0) break;
            const int brick = A.u_brick[unit];
            const int fb0 = A.brick_fasc_ptr[brick], nfb = A.brick_fasc_ptr[brick + 1] - fb0;
            uint32_t am = 0u;
            for (int i = 4 * A.brick_tile_ptr[brick] + lane; i < 4 * A.brick_tile_ptr[brick + 1]; i += 32)
                am = max(am, A.tile_amax[i]);
            am = warp_max_u32(am);
            // Z in tensor memory is 2^(kR + kD)·Z (kR from the brick's max |r|, as the loader scales R)
            const float sc = ldexpf(1.0f, -(f16_scale_exp(am) + kD));
            for (int i = 32 * tid; i < nfb; i += 32 * WC_SCAT_THREADS) prefetch_l2(A.brick_fasc + fb0 + i);
            if (named_bar_or(2, WC_SCAT_THREADS, dead || abort_flag != 0)) break;
            for (int i = tid; i < nfb; i += WC_SCAT_THREADS) gl[i] = 0.0f;
            named_bar_sync(2, WC_SCAT_THREADS);
            const int t0 = A.u_t0[unit], t1 = A.u_t1[unit];
            for (int t = t0; t < t1 && !dead; ++t) {
                // segment bounds of the tile: lane i holds wseg(t, rq, i) for this warp's k-th row quarter rq
                int bq[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const int rq = h + k * wg;
                    bq[k] = (active && rq < 4 && lane <= A.n_sub) ? wseg(A, t, rq, lane) : 0;
                }
                for (int j = 0; j < kc && !dead; ++j) {
                    for (int hh = 0; hh < 2 && !dead; ++hh, ++kcount) {
                        // rows 64hh .. of atom block j sit in slot zs of the ring
                        const uint32_t zs = kcount % Z32_SLOTS, zu = (kcount / Z32_SLOTS) & 1u;
                        // a thin segment's entries are on their way while its Z is waited for
                        // (with four scatter groups a warp has one row quarter, h)
                        uint32_t tk[4], tf[4];
                        float tx[4];
                        bool thin = false;
                        if (THIN) {
                            const int tb0 = __shfl_sync(0xffffffffu, bq[0], 4 * j + q);
                            const int te0 = __shfl_sync(0xffffffffu, bq[0], 4 * j + q + 1);
                            thin = (h >> 1) == hh && te0 - tb0 <= WC_THIN;  // (no entries: te0 = tb0)
                            if (thin) {
                                wc_load_thin(A, tb0, te0, lane, tk, tf);
#pragma unroll
                                for (int i = 0; i < 4; ++i)
                                    tx[i] = tb0 + 32 * i + lane < te0 ? __ldg(A.wval32 + tb0 + 32 * i + lane) : 0.0f;
                            }
                        }
                        if (!warp_wait(&z_full[zs], zu, &abort_flag)) {
                            abort_flag = 1;
                            dead = true;
                            break;
                        }
                        tc_fence_after();
                        if (active) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) {
                                const int rq = h + k * wg;
                                if (rq >= 4 || (rq >> 1) != hh) continue;
                                const int sub = 4 * j + q;
                                const int beg = __shfl_sync(0xffffffffu, bq[k], sub);
                                const int end = __shfl_sync(0xffffffffu, bq[k], sub + 1);
                                if (beg >= end) continue;  // an empty segment needs no Z
                                uint32_t rr[32];
                                tmem_ld32(tb + ((uint32_t)(32 * q) << 16) + zb + zs * 64u + 32u * (uint32_t)(rq & 1),
                                          rr);
                                tmem_ld_wait();
                                float* zrow = Zw + lane * ZW;  // this lane's atom, the row quarter's 32 rows
#pragma unroll
                                for (int e = 0; e < 32; ++e) zrow[e] = __uint_as_float(rr[e]) * sc;
                                __syncwarp();
                                if (THIN && k == 0 && thin) wc_thin<false>(tk, tf, tx, beg, end, lane, Zw, gl, gl_s);
                                else wc32_segment(A, beg, end, Zw, gl_s, lane);
                                __syncwarp();
                            }
                        }
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&z_empty[zs]);  // this warp is done with the slot
                    }
                }
            }
            if (named_bar_or(2, WC_SCAT_THREADS, dead || abort_flag != 0)) break;
            flush_table(A.out, gl, A.brick_fasc + fb0, nfb, tid, WC_SCAT_THREADS);
        }
    } else if (warp < WC_MMA_WARP) {
        // ---------------- R tile loader: r[:, v]·2^kR of the brick as FP16 hi and lo
        // parts (rows = voxels, K = θ), kR as the scatter warps compute it
        const int lt = tid - WC_SCAT_THREADS;
        const bool vec = A.vec4 != 0;
        const RUnits RU(A.np);
        int vv[2], tv = -1;  // the first batch's voxels of tile tv
        uint32_t tcount = 0;
        bool stop = false;
        for (int r = 0; !stop; ++r) {
            const int unit = live_unit(A, cta, r);
            if (unit < 0) break;
            int r_next = r + 1;
            const int next_unit = live_unit(A, cta, r_next), brick = A.u_brick[unit];
            uint32_t am = 0u;
            for (int i = 4 * A.brick_tile_ptr[brick] + lane; i < 4 * A.brick_tile_ptr[brick + 1]; i += 32)
                am = max(am, A.tile_amax[i]);
            const float rs = ldexpf(1.0f, f16_scale_exp(warp_max_u32(am)));
            for (int t = A.u_t0[unit]; t < A.u_t1[unit]; ++t) {
                const uint32_t rb = A.rbufs == 2 ? (tcount & 1u) : 0u, rk = A.rbufs == 2 ? (tcount >> 1) : tcount;
                unsigned char* Rb = Rs + rb * r_bytes;
                if (tv != t) load_r_voxels(A, t, lt, RU, vv);
                if (!warp_wait(&r_empty[rb], (rk & 1u) ^ 1u, &abort_flag)) {
                    abort_flag = 1;
                    stop = true;
                    break;
                }
                load_r_tile(A, t, RU, vv, lt, vec, [&](int row, int g8, const float4& lo, const float4& hi) {
                    uint4 ph, pl;
                    split_f16x2(lo.x * rs, lo.y * rs, ph.x, pl.x);
                    split_f16x2(lo.z * rs, lo.w * rs, ph.y, pl.y);
                    split_f16x2(hi.x * rs, hi.y * rs, ph.z, pl.z);
                    split_f16x2(hi.z * rs, hi.w * rs, ph.w, pl.w);
                    const uint32_t off = kmajor_off(row, 8 * g8, SBO_K);
                    *reinterpret_cast<uint4*>(Rb + off) = ph;
                    *reinterpret_cast<uint4*>(Rb + r_part + off) = pl;
                });
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) mbar_arrive(&r_full[rb]);
                ++tcount;
                tv = t + 1 < A.u_t1[unit] ? t + 1 : next_unit >= 0 ? A.u_t0[next_unit] : t;
                load_r_voxels(A, tv, lt, RU, vv);  // of the tile after this one
                // pull the voxel rows of r of the tile A.rbufs ahead into L2
                int tn = t + A.rbufs;
                if (tn >= A.u_t1[unit]) {
                    tn -= A.u_t1[unit];
                    tn = (next_unit >= 0 && A.u_t0[next_unit] + tn < A.u_t1[next_unit])
                             ? A.u_t0[next_unit] + tn : -1;
                }
                if (tn >= 0) {
                    const int32_t* tvn = A.tile_vox + (int64_t)tn * TILE_V;
                    for (int row = lt; row < TILE_V; row += WC_LOAD_THREADS) {
                        const int v = __ldg(tvn + row);
                        if (v < 0) continue;
                        const char* a = reinterpret_cast<const char*>(A.x + (int64_t)A.nt * v);
                        const char* e = a + 4 * A.nt - 1;
                        for (const char* c = a; c < e; c += 128) prefetch_l2(c);
                        prefetch_l2(e);
                    }
                }
            }
        }
    } else if (lane == 0) {
        // ---------------- MMA issuer: Z[128 atoms x 64 rows] = D_blk · R_half for each
        // 128-atom block and half tile, into the next slot of the tensor-memory ring
        const uint32_t idesc = idesc_f16_f32(128, 64);
        const uint32_t sR0 = smem_u32(Rs), half = (uint32_t)A.np / 2;
        uint32_t tcount = 0, kcount = 0;
        bool stop = false;
        // D's parts are in tensor memory once the warps that store them have arrived
        if (!mbar_wait(&d_ready, 0, &abort_flag, WAIT_LIMIT)) {
            abort_flag = 1;
            stop = true;
        }
        tc_fence_after();
        for (int r = 0; !stop; ++r) {
            const int unit = live_unit(A, cta, r);
            if (unit < 0) break;
            for (int t = A.u_t0[unit]; t < A.u_t1[unit] && !stop; ++t) {
                const uint32_t rb = A.rbufs == 2 ? (tcount & 1u) : 0u, rk = A.rbufs == 2 ? (tcount >> 1) : tcount;
                const uint32_t sR = sR0 + rb * r_bytes;
                if (!mbar_wait(&r_full[rb], rk & 1u, &abort_flag, WAIT_LIMIT)) {
                    abort_flag = 1;
                    stop = true;
                    break;
                }
                for (int j = 0; j < kc && !stop; ++j) {
                    for (int hh = 0; hh < 2; ++hh, ++kcount) {
                        const uint32_t zs = kcount % Z32_SLOTS, zu = (kcount / Z32_SLOTS) & 1u;
                        if (!mbar_wait(&z_empty[zs], zu ^ 1u, &abort_flag, WAIT_LIMIT)) {  // the slot was read
                            abort_flag = 1;
                            stop = true;
                            break;
                        }
                        tc_fence_after();
                        const uint32_t zt = tb + zb + zs * 64u;
                        const uint32_t sb = sR + (uint32_t)(8 * hh) * SBO_K;  // rows 64hh .. 64hh + 63
                        for (int kk = 0; kk < A.np / 16; ++kk) {
                            const uint32_t ah = tb + (uint32_t)(j * A.np) + kk * 8u;  // 16 θ = 8 columns
                            const uint64_t bh = smem_desc(sb + kk * 256u, 128u, SBO_K);
                            const uint64_t bl = smem_desc(sb + r_part + kk * 256u, 128u, SBO_K);
                            mma_f16_tmem_a(zt, ah, bh, idesc, kk != 0 ? 1u : 0u);
                            mma_f16_tmem_a(zt, ah, bl, idesc, 1u);
                            mma_f16_tmem_a(zt, ah + half, bh, idesc, 1u);
                        }
                        mma_commit(&z_full[zs]);
                    }
                }
                if (stop) break;
                mma_commit(&r_empty[rb]);
                ++tcount;
            }
        }
        mma_commit(&fin_bar);
        if (!mbar_wait(&fin_bar, 0, &never, WAIT_LIMIT)) abort_flag = 1;
    }
    tc_fence_before();
    __syncthreads();
    if (abort_flag && tid == 0) atomicOr(A.status, DEV_TIMEOUT);
    if (warp == WC_MMA_WARP) {
        tc_fence_after();
        tmem_dealloc(tb, 512);
    }
}

// ============================================================== launchers

// WC scatter groups for the next launch: the requested number (4 by default),
// halved while the kernel's shared memory would not fit; 0 if even 1 does not.
int wc_effective_groups(const life_index_s* ix) {
    int optin = 0;
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, ix->device) != cudaSuccess) return 0;
    const TileLayout& L = ix->tile;
    int wg = ix->wc_groups > 0 ? ix->wc_groups : 4;
    while (wg >= 1 && wc_smem_bytes(L.np, L.kp, L.max_fb, wg, 1, L.vbytes == 4) + 256 > (uint32_t)optin) wg /= 2;
    return wg;
}

// R tile buffers of the WC kernel with wg scatter groups: two when they fit.
static int wc_r_buffers(const life_index_s* ix, int wg) {
    int optin = 0;
    if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, ix->device) != cudaSuccess) return 1;
    const TileLayout& L = ix->tile;
    return wc_smem_bytes(L.np, L.kp, L.max_fb, wg, 2, L.vbytes == 4) + 256 <= (uint32_t)optin ? 2 : 1;
}

static TcArgs make_args(life_index_s* ix) {
    TileLayout& L = ix->tile;
    TcArgs A{};
    A.tile_vox = L.tile_vox.as<int32_t>();
    A.chunk_ptr = L.chunk_ptr.as<int32_t>();
    A.brick_tile_ptr = L.brick_tile_ptr.as<int32_t>();
    A.brick_fasc_ptr = L.brick_fasc_ptr.as<int32_t>();
    A.brick_fasc = L.brick_fasc.as<int32_t>();
    const int32_t* u = L.units.as<int32_t>();
    A.cta_unit = u;
    A.u_brick = u + L.grid + 1;
    A.u_t0 = A.u_brick + L.n_units;
    A.u_t1 = A.u_t0 + L.n_units;
    A.soff = L.soff.as<uint16_t>();
    A.wkey = L.wkey.as<uint16_t>();
    A.wfl = L.wfl.as<uint16_t>();
    A.wval = L.wval.as<__nv_bfloat16>();
    A.wseg_ptr = L.wseg_ptr.as<int32_t>();
    A.fl = L.fl.as<uint16_t>();
    A.val = L.val.as<__nv_bfloat16>();
    A.wb = L.wb.as<float>();
    A.wb_ptr = L.wb_ptr.as<int32_t>();
    A.brick_cv = L.brick_cv.as<float>();
    A.tile_amax = L.tile_amax.as<uint32_t>();
    A.run_vmax = L.run_vmax;
    A.nt = ix->nt;
    A.na = ix->na;
    A.np = L.np;
    A.kp = L.kp;
    A.n_sub = L.n_sub;
    A.n_bricks = (int)L.n_bricks;
    A.max_fb = L.max_fb;
    A.status = dev_status_word();
    return A;
}

// What the kernels of one call read besides the layout: D's operands and scale, and
// (for a DSC) max |x|; zero (nf floats, or NULL) is cleared on the way.
static PrepArgs prep_args(life_index_s* ix, const float* D, float* zero, int threads) {
    TileLayout& L = ix->tile;
    PrepArgs P{};
    P.D = D;
    if (L.vbytes == 2) {
        P.img_dsc = L.d_img.as<unsigned char>();
        P.img_wc = P.img_dsc + (size_t)L.np * L.kp * 2;
    }
    P.info = L.d_info.as<uint32_t>();
    P.zero = zero;
    P.n_zero = zero ? ix->nf : 0;
    P.nt = ix->nt;
    P.na = ix->na;
    P.np = L.np;
    P.kp = L.kp;
    P.n_dblk = L.vbytes == 2 ? L.kp / (threads / 32) : 1;
    return P;
}

life_status dsc_tc(life_index_s* ix, const float* D, const float* w, const float* b, float* y, double* partial,
                   int* n_partial, const life_sbb_state* gate, int gate_mode, cudaStream_t s, const BatchGate& bg,
                   float* zero) {
    TcArgs A = make_args(ix);
    A.bg = bg;
    if (!A.status) {
        set_error("dsc_tc: no device status word");
        return LIFE_ENOMEM;
    }
    A.D = D;
    A.x = w;
    A.b = b;
    A.out = y;
    A.partial = partial;
    A.gate = gate;
    A.gate_mode = gate_mode;
    A.vec4 = (ix->nt % 4 == 0 && ((reinterpret_cast<uintptr_t>(y) | reinterpret_cast<uintptr_t>(b)) & 15) == 0) ? 1 : 0;
    TileLayout& L = ix->tile;
    const bool f32 = L.vbytes == 4;
    if (f32) {
        A.val = nullptr;
        A.val32 = L.val.as<float>();
    }
    int optin = 0;
    LIFE_CUDA_TRY(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, ix->device));
    const DscForm form = dsc_form(L.n_nnz, L.n_tiles, L.n_bricks, A.kp / DKC, !f32 && A.vec4, [&](int stages) {
        return dsc_smem_bytes(A.np, A.kp, A.nt, A.max_fb, f32, stages, true) + 512 <= (uint32_t)optin;
    });
    A.y_tile = form.y_tile ? 1 : 0;
    A.dstage = form.stages;
    const uint32_t smem = dsc_smem_bytes(A.np, A.kp, A.nt, A.max_fb, f32, A.dstage, A.y_tile != 0);
    const bool sparse = L.sparse && !bg.live && L.wb_total > 0 && L.n_nnz > 0;
    if (sparse) {
        // the last block decides: full or compacted stream, rebuild or not (the
        // SBB step's DSC of w never rebuilds: its support lies inside that of the
        // previous projected gradient; the DSC of the projected gradient rebuilds
        // with the backoff; a public call whenever its input needs it)
        wb_gather_live_kernel<<<ix->num_sms * 8, GATHER_THREADS, 0, s>>>(
            L.wb_src.as<int32_t>(), L.wb_total, w, L.wb.as<float>(), L.wb_live.as<uint8_t>(),
            L.sparse_ctl.as<SparseCtl>(), (unsigned long long)L.n_brick_slots,
            !gate ? ALLOW_FREE : (gate_mode == GATE_ACTIVE ? ALLOW_NONE : ALLOW_BACKOFF), gate, gate_mode,
            L.x_amax.as<uint32_t>());
        LIFE_CHECK_LAUNCH();
    }
    PrepArgs P = prep_args(ix, D, zero, PREP_THREADS);
    if (!sparse) {  // the DSC gathers each brick's weights itself: this pass finds max |w|
        P.x = w;
        P.n_x = ix->nf;
        P.x_amax = L.x_amax.as<uint32_t>();
    }
    P.n_xblk = ix->num_sms;
    tc_prep_kernel<<<P.n_dblk + P.n_xblk, PREP_THREADS, 0, s>>>(P);
    LIFE_CHECK_LAUNCH();
    A.x_amax = L.x_amax.as<uint32_t>();
    A.n_xamax = sparse ? ix->num_sms * 8 : P.n_xblk;
    A.gather_w = sparse ? 0 : 1;
    A.wb_src = L.wb_src.as<int32_t>();
    A.d_img = P.img_dsc;
    A.d_info = P.info;
    A.n_dblk = P.n_dblk;
    auto kern = f32 ? dsc_tc_kernel<true, false> : A.y_tile ? dsc_tc_kernel<false, true> : dsc_tc_kernel<false, false>;
    LIFE_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int grid = L.grid;
    if (n_partial) *n_partial = grid;
    if (!sparse) {
        kern<<<grid, DSC_THREADS, smem, s>>>(A);
        LIFE_CHECK_LAUNCH();
        return LIFE_OK;
    }
    SparseCtl* ctl = L.sparse_ctl.as<SparseCtl>();
    if (!(gate && gate_mode == GATE_ACTIVE)) {
        CompactArgs C{};
        C.chunk_ptr = L.chunk_ptr.as<int32_t>();
        C.tile_brick = L.tile_brick.as<int32_t>();
        C.wb_ptr = L.wb_ptr.as<int32_t>();
        C.wb = L.wb.as<float>();
        C.soff = L.soff.as<uint16_t>();
        C.fl = L.fl.as<uint16_t>();
        C.val = L.val.as<__nv_bfloat16>();
        C.wb_live = L.wb_live.as<uint8_t>();
        C.c_soff = L.c_soff.as<uint16_t>();
        C.c_fl = L.c_fl.as<uint16_t>();
        C.c_val = L.c_val.as<__nv_bfloat16>();
        C.c_chunk_end = L.c_chunk_end.as<int32_t>();
        C.ctl = ctl;
        C.n_c = L.kp / DKC;
        C.n_chunks = L.n_tiles * C.n_c;
        C.wb_total = L.wb_total;
        const unsigned cg = (unsigned)std::max<int64_t>(
            1, std::min<int64_t>((C.n_chunks + CMP_THREADS / 32 - 1) / (CMP_THREADS / 32), (int64_t)ix->num_sms * 16));
        cmp_rebuild_kernel<<<cg, CMP_THREADS, 0, s>>>(C);
        LIFE_CHECK_LAUNCH();
    }
    A.ctl = ctl;
    A.want_mode = DSC_MODE_FULL;
    kern<<<grid, DSC_THREADS, smem, s>>>(A);
    LIFE_CHECK_LAUNCH();
    A.want_mode = DSC_MODE_COMPACT;
    A.soff = L.c_soff.as<uint16_t>();
    A.fl = L.c_fl.as<uint16_t>();
    A.val = L.c_val.as<__nv_bfloat16>();
    A.chunk_end = L.c_chunk_end.as<int32_t>();
    kern<<<grid, DSC_THREADS, smem, s>>>(A);
    LIFE_CHECK_LAUNCH();
    return LIFE_OK;
}

life_status wc_tc(life_index_s* ix, const float* D, const float* r, float* g, const life_sbb_state* gate, int gate_mode,
                  cudaStream_t s, const BatchGate& bg, bool r_is_dsc_out) {
    TcArgs A = make_args(ix);
    A.bg = bg;
    if (!A.status) {
        set_error("wc_tc: no device status word");
        return LIFE_ENOMEM;
    }
    A.D = D;
    A.x = r;
    A.out = g;
    A.gate = gate;
    A.gate_mode = gate_mode;
    A.vec4 = (ix->nt % 4 == 0 && (reinterpret_cast<uintptr_t>(r) & 15) == 0) ? 1 : 0;
    A.wgroups = wc_effective_groups(ix);
    if (A.wgroups < 1) {
        set_error("wc_tc: %u bytes of shared memory needed even with one scatter group",
                  wc_smem_bytes(A.np, A.kp, A.max_fb, 1, 1, ix->tile.vbytes == 4));
        return LIFE_ENOTSUP;
    }
    A.rbufs = wc_r_buffers(ix, A.wgroups);
    const bool f32 = ix->tile.vbytes == 4;
    if (f32) {
        A.wval = nullptr;
        A.wval32 = ix->tile.wval.as<float>();
    }
    const uint32_t smem = wc_smem_bytes(A.np, A.kp, A.max_fb, A.wgroups, A.rbufs, f32);
    const bool thin = ix->nnz <= (int64_t)WC_THIN_MEAN * ix->tile.n_tiles * 4 * A.n_sub;
    auto kern = f32 ? (thin ? wc_tc32_kernel<true> : wc_tc32_kernel<false>) : thin ? wc_tc_kernel<true> : wc_tc_kernel<false>;
    LIFE_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    // (blocks as in the launch that wrote d_info: the DSC's, or this call's own)
    const PrepArgs P = prep_args(ix, D, g, r_is_dsc_out ? PREP_THREADS : AMAX_THREADS);
    A.d_img = P.img_wc;
    A.d_info = P.info;
    A.n_dblk = P.n_dblk;
    if (!r_is_dsc_out) {
        // (after a DSC of this index that wrote r, its epilogue left the tiles' maxima and
        // its preparations D's operands and the zeroed g)
        const int64_t blk = std::min<int64_t>(std::max<int64_t>(ix->tile.n_tiles, 1), (int64_t)ix->num_sms * 8);
        wc_amax_kernel<<<(unsigned)(P.n_dblk + blk), AMAX_THREADS, 0, s>>>(A, P);
        LIFE_CHECK_LAUNCH();
    }
    kern<<<ix->tile.grid, WC_THREADS, smem, s>>>(A);
    LIFE_CHECK_LAUNCH();
    return LIFE_OK;
}

life_status sparse_stats(life_index_s* ix, int64_t* out, cudaStream_t s) {
    for (int i = 0; i < 6; ++i) out[i] = 0;
    TileLayout& L = ix->tile;
    if (!L.built || !L.sparse) return LIFE_OK;
    SparseCtl c{};
    const int n_c = L.kp / DKC;
    std::vector<int32_t> ends((size_t)(L.n_tiles * n_c)), sp((size_t)(L.n_tiles * n_c + 1));
    LIFE_CUDA_TRY(cudaMemcpyAsync(&c, L.sparse_ctl.p, sizeof(SparseCtl), cudaMemcpyDeviceToHost, s));
    if (!ends.empty()) {
        LIFE_CUDA_TRY(cudaMemcpyAsync(ends.data(), L.c_chunk_end.p, sizeof(int32_t) * ends.size(),
                                      cudaMemcpyDeviceToHost, s));
        LIFE_CUDA_TRY(cudaMemcpyAsync(sp.data(), L.chunk_ptr.p, sizeof(int32_t) * sp.size(), cudaMemcpyDeviceToHost, s));
    }
    LIFE_CUDA_TRY(cudaStreamSynchronize(s));
    int64_t ncmp = 0;
    for (int64_t t = 0; t < L.n_tiles; ++t)
        for (int c2 = 0; c2 < n_c; ++c2) ncmp += ends[t * n_c + c2] - sp[t * n_c + c2];
    out[0] = (int64_t)c.n_calls;
    out[1] = (int64_t)c.n_compact_calls;
    out[2] = (int64_t)c.n_compactions;
    out[3] = c.have ? ncmp : 0;
    out[4] = L.n_nnz;
    out[5] = (int64_t)c.n_live_cmp;
    return LIFE_OK;
}

}  // namespace life
