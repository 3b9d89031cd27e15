// CUDA-core FP32 SpMVs on the voxel-sorted layout.
//
// DSC (y = M w) and WC (g = M^T r) as in Sec. 4.2.2 (GPU-specific optimizations):
// voxel-based restructuring and partitioning, one warp per voxel segment, the
// Nθ loop spread over the 32 lanes (Nθ padded to a multiple of 32 inside the
// kernel), the dictionary D staged in shared memory, and zero val·w products
// skipped (Sec. 4.2.1, "BLAS call for DSC").  WC reduces each warp's 32 dot
// products with a transpose-reduction of shuffles and adds val·dot into g[f]
// with one atomic per nonzero (the paper's coefficient-based WC also uses atomics).
//
// Hybrid restructuring (Sec. 4.1.2: the voxel-restructured Phi with each voxel's
// entries reordered by atom) is what the voxel layout stores, (v, a, f); the
// RUNS variants use it: a run of equal atoms inside a voxel costs one pass over
// D's column (DSC: D[:,a]·Σ val·w; WC: one dot <D[:,a], r[:,v]> shared by the
// run's entries) instead of one per entry.  Which variant runs is chosen at
// build time or, as the paper chooses its restructuring, by timing both
// (life_index_autotune).
#include "life_internal.cuh"
#include "tc_ptx.cuh"

namespace life {

constexpr int SIMT_THREADS = 1024;
constexpr size_t SIMT_SMEM_LIMIT = 200 * 1024;

__device__ __forceinline__ double block_sum_f64(double v, double* sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) sh[warp] = v;
    __syncthreads();
    double t = 0.0;
    if (warp == 0) {
        t = lane < nw ? sh[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    }
    return t;  // valid in thread 0
}

// D into shared memory, columns padded to NTW·32 floats; by 16-byte accesses where D
// allows, eight a thread in flight (one float at a time, the 138 KB of a 96 x 360 D
// were a third of a small call's time).
template <int NTW>
__device__ __forceinline__ void stage_D(float* Ds, const float* __restrict__ D, int nt, int na) {
    constexpr int ntp = NTW * 32;
    if ((nt & 3) == 0 && (reinterpret_cast<uintptr_t>(D) & 15) == 0) {
        constexpr int q = ntp / 4;
#pragma unroll 8
        for (int i = threadIdx.x; i < na * q; i += SIMT_THREADS) {
            const int a = i / q, t = 4 * (i - a * q);
            reinterpret_cast<float4*>(Ds)[i] = t < nt ? __ldg(reinterpret_cast<const float4*>(D + (int64_t)nt * a + t))
                                                      : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        }
        return;
    }
#pragma unroll 8
    for (int i = threadIdx.x; i < na * ntp; i += SIMT_THREADS) {
        const int a = i / ntp, t = i - a * ntp;
        Ds[i] = t < nt ? __ldg(D + t + (int64_t)nt * a) : 0.0f;
    }
}

template <class VT>
__device__ __forceinline__ float ldval(const VT* p, int64_t k);
template <>
__device__ __forceinline__ float ldval<float>(const float* p, int64_t k) { return __ldg(p + k); }
template <>
__device__ __forceinline__ float ldval<__nv_bfloat16>(const __nv_bfloat16* p, int64_t k) {
    return __bfloat162float(p[k]);
}

// y[:,v] = Σ_k D[:,a_k] val_k w[f_k]  (− b[:,v]), entry by entry;  per-block FP64 Σ out².
template <int NTW, bool SMEM_D, class VT>
__global__ void __launch_bounds__(SIMT_THREADS)
dsc_simt_kernel(const int32_t* __restrict__ vox_ptr, const uint16_t* __restrict__ atom,
                const int32_t* __restrict__ fasc, const VT* __restrict__ val, const float* __restrict__ D,
                int nt, int na, int nv, const float* __restrict__ w, const float* __restrict__ b,
                float* __restrict__ y, double* __restrict__ partial, const life_sbb_state* gate, int gate_mode,
                const BatchGate bg) {
    extern __shared__ __align__(16) float Ds[];
    __shared__ double red[32];
    bool write_y = y != nullptr;
    if (!bg.live) {
        if (gate_skip(gate, gate_mode)) return;
        if (gate && gate_mode == GATE_ACTIVE_Y_EQ8 && gate->eq != 8) write_y = false;
    }
    constexpr int NTP = NTW * 32;
    if (SMEM_D) {
        stage_D<NTW>(Ds, D, nt, na);
        __syncthreads();
    }
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    const int wid = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    double sq = 0.0;
    // Batched launch: the warps stride over the voxels of all problems and jump
    // over those of problems that are not live, so the live ones always get the
    // whole grid; Σ out² goes to a slot per (problem, warp).
    int p = 0, cur_p = -1;
    bool live = true, wy = write_y;
    if (bg.live && partial && lane == 0)
        for (int q = 0; q < bg.n; ++q) partial[(int64_t)q * warps + wid] = 0.0;
    for (int v = wid; v < nv; v += warps) {
        if (bg.live) {
            if (v >= bg.vox_off[p + 1] || cur_p < 0) {
                while (v >= bg.vox_off[p + 1]) ++p;
                live = batch_live(bg, p, gate_mode);
                wy = write_y && batch_writes_y(bg, p, gate_mode);
            }
            if (!live) {
                // first voxel of this warp's sequence at or after the problem's end
                const int end = bg.vox_off[p + 1];
                v += ((end - v + warps - 1) / warps - 1) * warps;
                continue;
            }
            if (p != cur_p) {
                if (cur_p >= 0 && lane == 0 && partial) partial[(int64_t)cur_p * warps + wid] += sq;
                sq = 0.0;
                cur_p = p;
            }
        }
        float acc[NTW];
#pragma unroll
        for (int q = 0; q < NTW; ++q) acc[q] = 0.0f;
        const int beg = vox_ptr[v], end = vox_ptr[v + 1];
        for (int base = beg; base < end; base += 32) {
            const int k = base + lane;
            int a_l = 0;
            float s_l = 0.0f;
            if (k < end) {
                a_l = atom[k];
                s_l = ldval<VT>(val, k) * __ldg(w + fasc[k]);
            }
            const int cnt = min(32, end - base);
#pragma unroll 4
            for (int j = 0; j < cnt; ++j) {
                const float s = __shfl_sync(0xffffffffu, s_l, j);
                const int a = __shfl_sync(0xffffffffu, a_l, j);
                if (s != 0.0f) {
                    if (SMEM_D) {
                        const float* d = Ds + a * NTP + lane;
#pragma unroll
                        for (int q = 0; q < NTW; ++q) acc[q] = fmaf(d[q * 32], s, acc[q]);
                    } else {
                        const float* d = D + (int64_t)nt * a;
#pragma unroll
                        for (int q = 0; q < NTW; ++q) {
                            const int t = q * 32 + lane;
                            acc[q] = fmaf(t < nt ? __ldg(d + t) : 0.0f, s, acc[q]);
                        }
                    }
                }
            }
        }
        float sqv = 0.0f;  // this voxel's Σ out² in FP32, promoted to FP64 once per voxel
#pragma unroll
        for (int q = 0; q < NTW; ++q) {
            const int t = q * 32 + lane;
            if (t < nt) {
                const int64_t o = t + (int64_t)nt * v;
                float out = acc[q];
                if (b) out -= b[o];
                if (wy) y[o] = out;
                sqv = fmaf(out, out, sqv);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) sqv += __shfl_xor_sync(0xffffffffu, sqv, o);
        if (lane == 0) sq += (double)sqv;
    }
    if (bg.live) {
        if (cur_p >= 0 && lane == 0 && partial) partial[(int64_t)cur_p * warps + wid] += sq;
        return;
    }
    const double tot = block_sum_f64(sq, red);
    if (threadIdx.x == 0 && partial) partial[blockIdx.x] = tot;
}

// Lane j of the warp ends with Σ over lanes of x[j] (31 shuffles for 32 sums).
__device__ __forceinline__ float transpose_reduce32(float (&x)[32], int lane) {
#pragma unroll
    for (int s = 16; s >= 1; s >>= 1) {
        const bool upper = (lane & s) != 0;
#pragma unroll
        for (int i = 0; i < s; ++i) {
            const float send = upper ? x[i] : x[i + s];
            const float keep = upper ? x[i + s] : x[i];
            x[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
        }
    }
    return x[0];
}

// g[f] += val_k <D[:,a_k], r[:,v_k]> for every nonzero (g zeroed by the caller), with D
// too large for shared memory.
template <int NTW, class VT>
__global__ void __launch_bounds__(SIMT_THREADS)
wc_simt_kernel(const int32_t* __restrict__ vox_ptr, const uint16_t* __restrict__ atom,
               const int32_t* __restrict__ fasc, const VT* __restrict__ val, const float* __restrict__ D, int nt,
               int na, int nv, const float* __restrict__ r, float* __restrict__ g, const life_sbb_state* gate,
               int gate_mode, const BatchGate bg) {
    if (!bg.live && gate_skip(gate, gate_mode)) return;
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    int p = 0;
    bool live = true, first = true;
    for (int v = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < nv; v += warps) {
        if (bg.live) {
            // batched launch: skip the voxels of problems that are not live
            if (first || v >= bg.vox_off[p + 1]) {
                while (v >= bg.vox_off[p + 1]) ++p;
                live = batch_live(bg, p, gate_mode);
                first = false;
            }
            if (!live) {
                const int end = bg.vox_off[p + 1];
                v += ((end - v + warps - 1) / warps - 1) * warps;
                continue;
            }
        }
        const int beg = vox_ptr[v], end = vox_ptr[v + 1];
        if (beg == end) continue;
        float rr[NTW];
#pragma unroll
        for (int q = 0; q < NTW; ++q) {
            const int t = q * 32 + lane;
            rr[q] = t < nt ? r[t + (int64_t)nt * v] : 0.0f;
        }
        for (int base = beg; base < end; base += 32) {
            const int k = base + lane;
            int a_l = 0;
            if (k < end) a_l = atom[k];
            float part[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                const int a = __shfl_sync(0xffffffffu, a_l, j);
                float p = 0.0f;
                const float* d = D + (int64_t)nt * a;
#pragma unroll
                for (int q = 0; q < NTW; ++q) {
                    const int t = q * 32 + lane;
                    p = fmaf(t < nt ? __ldg(d + t) : 0.0f, rr[q], p);
                }
                part[j] = p;
            }
            const float dot = transpose_reduce32(part, lane);
            if (k < end) ptx::red_add_global_f32(g + fasc[k], ldval<VT>(val, k) * dot);
        }
    }
}

// ------------------------------------------------- D in shared memory, pipelined
//
// A warp walks its voxels' entries in windows of 32 (the last of a voxel may be
// shorter, an empty voxel has one empty window).  The loads of a window (voxel
// bounds, then atom, fascicle and value, then the gather of w) depend on one
// another; each is issued one window ahead of the next stage, so that while a
// window is worked on the w of the next and the entries of the one after are on
// their way.  Without that, a sparse voxel (17 entries on the medium workload) is
// a chain of four round trips to memory and the kernels wait for latency, not for
// shared memory: 201 us a DSC and 204 us a WC there, now 107 and 130.

// Windows of a warp in order: voxels v, v + warps, ... (of live problems only, in a
// batched launch).
struct SimtWalk {
    int v, base, end;    // the window [base, min(base + 32, end)) of voxel v; v >= nv: none left
    int nv2, nbeg, nend; // the next voxel and its bounds
    int p;               // batched launch: problem of nv2

    // first voxel at or after v (in steps of `warps`) that is worked on
    __device__ __forceinline__ int skip(int v, int nv, int warps, const BatchGate& bg, int mode) {
        if (!bg.live) return v;
        while (v < nv) {
            while (v >= bg.vox_off[p + 1]) ++p;
            if (batch_live(bg, p, mode)) break;
            const int e = bg.vox_off[p + 1];
            v += (e - v + warps - 1) / warps * warps;
        }
        return v;
    }
    __device__ __forceinline__ void look(const int32_t* __restrict__ vox_ptr, int v2, int nv, int warps,
                                         const BatchGate& bg, int mode) {
        nv2 = skip(v2, nv, warps, bg, mode);
        nbeg = nend = 0;
        if (nv2 < nv) {
            nbeg = __ldg(vox_ptr + nv2);
            nend = __ldg(vox_ptr + nv2 + 1);
        }
    }
    __device__ __forceinline__ void next(const int32_t* __restrict__ vox_ptr, int nv, int warps, const BatchGate& bg,
                                         int mode) {
        if (base + 32 < end) {
            base += 32;
            return;
        }
        v = nv2;
        base = nbeg;
        end = nend;
        look(vox_ptr, nv2 < nv ? nv2 + warps : nv2, nv, warps, bg, mode);
    }
};

// Hybrid order: inside a voxel the entries are sorted by atom, so a run of equal
// atoms is summed first (segmented scan over the lanes) and D's column is applied
// once per run: y[:,v] += D[:,a] · Σ_run val·w.  The window's runs (their sum and
// the place of their column) are compacted into the warp's shared buffer and read
// back as broadcasts, two a 16-byte load: handed round by shuffles, two a run, they
// cost the load/store pipe almost as much as the column's own 3 reads (Nθ = 96).
// That pipe bounds the kernel at the paper's density (23.8M entries, 1.36 a run:
// 415 -> 292 us, 4.0 cycles a run and SM, of which the columns' bytes are 3).
template <int NTW, class VT>
__global__ void __launch_bounds__(SIMT_THREADS)
dsc_runs_kernel(const int32_t* __restrict__ vox_ptr, const uint16_t* __restrict__ atom,
                const int32_t* __restrict__ fasc, const VT* __restrict__ val, const float* __restrict__ D, int nt,
                int na, int nv, const float* __restrict__ w, const float* __restrict__ b, float* __restrict__ y,
                double* __restrict__ partial, const life_sbb_state* gate, int gate_mode, const BatchGate bg) {
    extern __shared__ __align__(16) float Ds[];
    __shared__ double red[32];
    bool write_y = y != nullptr;
    if (!bg.live) {
        if (gate_skip(gate, gate_mode)) return;
        if (gate && gate_mode == GATE_ACTIVE_Y_EQ8 && gate->eq != 8) write_y = false;
    }
    constexpr int NTP = NTW * 32;
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    const int wid = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    // 16 bytes hold two runs: (sum, column offset) twice
    float2* buf = reinterpret_cast<float2*>(Ds + (size_t)na * NTP) + 32 * (threadIdx.x >> 5);
    SimtWalk it;   // the window whose entries are being loaded
    it.p = 0;
    it.look(vox_ptr, wid, nv, warps, bg, gate_mode);
    it.v = it.nv2;
    it.base = it.nbeg;
    it.end = it.nend;
    it.look(vox_ptr, it.v < nv ? it.v + warps : it.v, nv, warps, bg, gate_mode);
    if (bg.live && partial && lane == 0)
        for (int q = 0; q < bg.n; ++q) partial[(int64_t)q * warps + wid] = 0.0;
    struct Win {
        int v, a;
        bool last;
        float x;
    };
    auto load = [&](Win& n, int& f) {
        const int k = it.base + lane;
        n.v = it.v;
        n.last = it.base + 32 >= it.end;
        n.a = -1 - lane;   // lanes beyond the end form runs of their own
        n.x = 0.0f;
        f = -1;
        if (it.v < nv && k < it.end) {
            n.a = __ldg(atom + k);
            n.x = ldval<VT>(val, k);
            f = __ldg(fasc + k);
        }
    };
    Win w0, w1;   // w0: x holds val·w; w1: x holds val
    int f1, f2;
    load(w0, f1);
    const float g0 = f1 >= 0 ? __ldg(w + f1) : 0.0f;
    it.next(vox_ptr, nv, warps, bg, gate_mode);
    load(w1, f1);
    stage_D<NTW>(Ds, D, nt, na);
    __syncthreads();
    w0.x *= g0;
    double sq = 0.0;
    int p = 0, cur_p = -1;
    bool wy = write_y;
    float acc[NTW];
#pragma unroll
    for (int q = 0; q < NTW; ++q) acc[q] = 0.0f;
    while (w0.v < nv) {
        it.next(vox_ptr, nv, warps, bg, gate_mode);
        Win w2;
        load(w2, f2);
        const float g1 = f1 >= 0 ? __ldg(w + f1) : 0.0f;
        float bv[NTW];
#pragma unroll
        for (int q = 0; q < NTW; ++q) {
            const int t = q * 32 + lane;
            bv[q] = (b && w0.last && t < nt) ? __ldg(b + t + (int64_t)nt * w0.v) : 0.0f;
        }
        // run sums of the window, compacted
        const int a_up = __shfl_up_sync(0xffffffffu, w0.a, 1), a_dn = __shfl_down_sync(0xffffffffu, w0.a, 1);
        const uint32_t heads = __ballot_sync(0xffffffffu, lane == 0 || a_up != w0.a);
        const int start = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));
        float rs = w0.x;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const float y2 = __shfl_up_sync(0xffffffffu, rs, o);
            if (lane - o >= start) rs += y2;
        }
        const bool tail = w0.a >= 0 && (lane == 31 || a_dn != w0.a) && rs != 0.0f;
        const uint32_t m = __ballot_sync(0xffffffffu, tail);
        if (tail) buf[__popc(m & ((1u << lane) - 1u))] = make_float2(rs, __int_as_float(w0.a * NTP));
        __syncwarp();
        const int n = __popc(m);
        int j = 0;
        for (; j + 4 <= n; j += 4) {
            const float4 u0 = *reinterpret_cast<const float4*>(buf + j), u1 = *reinterpret_cast<const float4*>(buf + j + 2);
            const float *d0 = Ds + __float_as_int(u0.y) + lane, *d1 = Ds + __float_as_int(u0.w) + lane,
                        *d2 = Ds + __float_as_int(u1.y) + lane, *d3 = Ds + __float_as_int(u1.w) + lane;
#pragma unroll
            for (int q = 0; q < NTW; ++q) {
                acc[q] = fmaf(d0[q * 32], u0.x, acc[q]);
                acc[q] = fmaf(d1[q * 32], u0.z, acc[q]);
                acc[q] = fmaf(d2[q * 32], u1.x, acc[q]);
                acc[q] = fmaf(d3[q * 32], u1.z, acc[q]);
            }
        }
        for (; j < n; ++j) {
            const float2 u = buf[j];
            const float* d = Ds + __float_as_int(u.y) + lane;
#pragma unroll
            for (int q = 0; q < NTW; ++q) acc[q] = fmaf(d[q * 32], u.x, acc[q]);
        }
        __syncwarp();  // the buffer is rewritten by the next window
        if (w0.last) {
            if (bg.live) {
                while (w0.v >= bg.vox_off[p + 1]) ++p;
                if (p != cur_p) {
                    if (cur_p >= 0 && lane == 0 && partial) partial[(int64_t)cur_p * warps + wid] += sq;
                    sq = 0.0;
                    cur_p = p;
                    wy = write_y && batch_writes_y(bg, p, gate_mode);
                }
            }
            float sqv = 0.0f;  // this voxel's Σ out² in FP32, promoted to FP64 once per voxel
#pragma unroll
            for (int q = 0; q < NTW; ++q) {
                const int t = q * 32 + lane;
                if (t < nt) {
                    const float out = acc[q] - bv[q];
                    if (wy) y[t + (int64_t)nt * w0.v] = out;
                    sqv = fmaf(out, out, sqv);
                }
                acc[q] = 0.0f;
            }
            if (partial) {
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) sqv += __shfl_xor_sync(0xffffffffu, sqv, o);
                if (lane == 0) sq += (double)sqv;
            }
        }
        w0 = w1;
        w0.x *= g1;
        w1 = w2;
        f1 = f2;
    }
    if (bg.live) {
        if (cur_p >= 0 && lane == 0 && partial) partial[(int64_t)cur_p * warps + wid] += sq;
        return;
    }
    const double tot = block_sum_f64(sq, red);
    if (threadIdx.x == 0 && partial) partial[blockIdx.x] = tot;
}

// Lane j % 16 of each half warp ends with Σ over the half's lanes of x[j % 16].
__device__ __forceinline__ float transpose_reduce16(float (&x)[16], int lane) {
#pragma unroll
    for (int s = 8; s >= 1; s >>= 1) {
        const bool upper = (lane & s) != 0;
#pragma unroll
        for (int i = 0; i < s; ++i) {
            const float send = upper ? x[i] : x[i + s];
            const float keep = upper ? x[i + s] : x[i];
            x[i] = keep + __shfl_xor_sync(0xffffffffu, send, s);
        }
    }
    return x[0];
}

// One dot <D[:,a], r[:,v]> per run of equal atoms of a window (RUNS) or per entry,
// the lanes over θ; the dots of 16 are reduced across the lanes together, and every
// entry adds val · (its run's dot) to g[f] (zeroed by the caller).  The columns'
// places go through the warp's shared buffer, four a 16-byte load, instead of one
// shuffle each, and dots beyond the window's last (in eights) are left out.  The
// load/store pipe bounds it (23.8M entries: 528 -> 459 us, 5.6 cycles an entry and
// SM: 3 for the column, 1 for the reduction, 1 for the scattered add).
template <int NTW, class VT, bool RUNS>
__global__ void __launch_bounds__(SIMT_THREADS)
wc_window_kernel(const int32_t* __restrict__ vox_ptr, const uint16_t* __restrict__ atom,
                 const int32_t* __restrict__ fasc, const VT* __restrict__ val, const float* __restrict__ D, int nt,
                 int na, int nv, const float* __restrict__ r, float* __restrict__ g, const life_sbb_state* gate,
                 int gate_mode, const BatchGate bg) {
    extern __shared__ __align__(16) float Ds[];
    if (!bg.live && gate_skip(gate, gate_mode)) return;
    constexpr int NTP = NTW * 32;
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    const int wid = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    int32_t* buf = reinterpret_cast<int32_t*>(Ds + (size_t)na * NTP) + 32 * (threadIdx.x >> 5);
    SimtWalk it;
    it.p = 0;
    it.look(vox_ptr, wid, nv, warps, bg, gate_mode);
    it.v = it.nv2;
    it.base = it.nbeg;
    it.end = it.nend;
    it.look(vox_ptr, it.v < nv ? it.v + warps : it.v, nv, warps, bg, gate_mode);
    int v0, n0, a0, f0, v1, n1, a1, f1;   // window being worked on, and the one after
    float x0, x1, rr[NTW], rn[NTW];
    auto load = [&](int& v, int& n, int& a, int& f, float& x) {
        const int k = it.base + lane;
        v = it.v;
        n = it.v < nv ? min(32, it.end - it.base) : 0;
        a = 0;
        f = 0;
        x = 0.0f;
        if (lane < n) {
            a = __ldg(atom + k);
            f = __ldg(fasc + k);
            x = ldval<VT>(val, k);
        }
    };
    auto load_r = [&](int v, float (&d)[NTW]) {
#pragma unroll
        for (int q = 0; q < NTW; ++q) {
            const int t = q * 32 + lane;
            d[q] = v < nv && t < nt ? __ldg(r + t + (int64_t)nt * v) : 0.0f;
        }
    };
    load(v0, n0, a0, f0, x0);
    load_r(v0, rr);
    stage_D<NTW>(Ds, D, nt, na);
    __syncthreads();
    while (v0 < nv) {
        it.next(vox_ptr, nv, warps, bg, gate_mode);
        load(v1, n1, a1, f1, x1);
        if (v1 != v0) load_r(v1, rn);
        if (n0 > 0) {
            // the window's distinct columns, in order (RUNS), or every entry's
            int slot = lane, nd = n0;
            if (RUNS) {
                const int a_up = __shfl_up_sync(0xffffffffu, a0, 1);
                const uint32_t heads = __ballot_sync(0xffffffffu, lane < n0 && (lane == 0 || a_up != a0));
                slot = __popc(heads & (0xffffffffu >> (31 - lane))) - 1;
                nd = __popc(heads);
            }
            buf[lane] = 0;
            __syncwarp();
            if (lane < n0) buf[slot] = a0 * NTP;
            __syncwarp();
            float half[2] = {0.0f, 0.0f};
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (16 * h >= nd) continue;
                float part[16];
#pragma unroll
                for (int j = 8; j < 16; ++j) part[j] = 0.0f;
#pragma unroll
                for (int g8 = 0; g8 < 2; ++g8) {
                    if (g8 == 1 && 16 * h + 8 >= nd) continue;
#pragma unroll
                    for (int j4 = 0; j4 < 2; ++j4) {
                        const int4 o = *reinterpret_cast<const int4*>(buf + 16 * h + 8 * g8 + 4 * j4);
                        const float *d0 = Ds + o.x + lane, *d1 = Ds + o.y + lane, *d2 = Ds + o.z + lane,
                                    *d3 = Ds + o.w + lane;
                        float p0 = 0.0f, p1 = 0.0f, p2 = 0.0f, p3 = 0.0f;
#pragma unroll
                        for (int q = 0; q < NTW; ++q) {
                            p0 = fmaf(d0[q * 32], rr[q], p0);
                            p1 = fmaf(d1[q * 32], rr[q], p1);
                            p2 = fmaf(d2[q * 32], rr[q], p2);
                            p3 = fmaf(d3[q * 32], rr[q], p3);
                        }
                        part[8 * g8 + 4 * j4] = p0;
                        part[8 * g8 + 4 * j4 + 1] = p1;
                        part[8 * g8 + 4 * j4 + 2] = p2;
                        part[8 * g8 + 4 * j4 + 3] = p3;
                    }
                }
                half[h] = transpose_reduce16(part, lane);
            }
            // lane j ends with dot j: its own half's sum plus the other half's
            const bool up = lane >= 16;
            float dot = (up ? half[1] : half[0]) + __shfl_xor_sync(0xffffffffu, up ? half[0] : half[1], 16);
            if (RUNS) dot = __shfl_sync(0xffffffffu, dot, slot & 31);
            if (lane < n0) ptx::red_add_global_f32(g + f0, x0 * dot);
        }
        if (v1 != v0) {
#pragma unroll
            for (int q = 0; q < NTW; ++q) rr[q] = rn[q];
        }
        v0 = v1;
        n0 = n1;
        a0 = a1;
        f0 = f1;
        x0 = x1;
    }
}

// dL/dD on the atom-sorted chunks: partial[c][θ] = Σ_{k∈c} val_k w[f_k] gy[θ, v_k].
// One warp per chunk, the lanes over θ.  A window of 32 entries is read with one
// entry a lane (and the next window's entries while this one is worked on); entries
// of one voxel are adjacent, so their val·w are summed first and gy's column is read
// once per voxel, eight columns' loads issued together: one entry at a time, each
// waiting for its own voxel, weight and column, a chunk was 256 chains of loads.
// What bounds it now is the columns' traffic from L2 (4 Nθ bytes a voxel run).
// Medium workload (4.5M entries, Nθ = 96): both launches 211 -> 162 us.
constexpr int GRAD_THREADS = 256;

template <int NTW>
__global__ void __launch_bounds__(GRAD_THREADS)
graddD_chunk_kernel(const int32_t* __restrict__ chunk_beg, int n_chunks, const int32_t* __restrict__ voxel,
                    const int32_t* __restrict__ fasc, const float* __restrict__ val, const float* __restrict__ w,
                    const float* __restrict__ gy, int nt, float* __restrict__ partial) {
    constexpr int U = NTW <= 4 ? 8 : 4;  // columns in flight
    __shared__ __align__(16) float2 runs[GRAD_THREADS / 32][32];
    float2* buf = runs[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    for (int c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; c < n_chunks; c += warps) {
        float acc[NTW];
#pragma unroll
        for (int q = 0; q < NTW; ++q) acc[q] = 0.0f;
        const int beg = chunk_beg[c], end = chunk_beg[c + 1];
        int v1 = -1 - lane;   // lanes beyond the end form runs of their own
        float s1 = 0.0f;
        if (beg + lane < end) {
            v1 = __ldg(voxel + beg + lane);
            s1 = __ldg(val + beg + lane) * __ldg(w + __ldg(fasc + beg + lane));
        }
        for (int base = beg; base < end; base += 32) {
            const int v = v1, k2 = base + 32 + lane;
            const float s0 = s1;
            float rs = s0;
            v1 = -1 - lane;
            s1 = 0.0f;
            if (k2 < end) {
                v1 = __ldg(voxel + k2);
                s1 = __ldg(val + k2) * __ldg(w + __ldg(fasc + k2));
            }
            const int v_up = __shfl_up_sync(0xffffffffu, v, 1), v_dn = __shfl_down_sync(0xffffffffu, v, 1);
            const uint32_t heads = __ballot_sync(0xffffffffu, lane == 0 || v_up != v);
            const int start = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const float y2 = __shfl_up_sync(0xffffffffu, rs, o);
                if (lane - o >= start) rs += y2;
            }
            // A NaN or inf in gy must reach dL/dD as in the oracle's sum over the entries: no
            // skip on a zero sum, and a run whose terms would differ in sign for an infinite
            // gy (inf - inf, inf * 0) is marked by the voxel's sign bit
            const uint32_t pos = __ballot_sync(0xffffffffu, s0 > 0.0f), neg = __ballot_sync(0xffffffffu, s0 < 0.0f),
                           zer = __ballot_sync(0xffffffffu, s0 == 0.0f),
                           run = (0xffffffffu >> (31 - lane)) & (0xffffffffu << start);
            const bool mixed = ((pos & run) != 0u) + ((neg & run) != 0u) + ((zer & run) != 0u) > 1;
            const bool tail = v >= 0 && (lane == 31 || v_dn != v);
            const uint32_t m = __ballot_sync(0xffffffffu, tail);
            if (tail)
                buf[__popc(m & ((1u << lane) - 1u))] = make_float2(rs, __uint_as_float((uint32_t)v | (mixed ? 0x80000000u : 0u)));
            __syncwarp();
            const int n = __popc(m);
            for (int j0 = 0; j0 < n; j0 += U) {
                float e[U][NTW], sj[U];
                bool mx[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const float2 x = j0 + u < n ? buf[j0 + u] : make_float2(0.0f, 0.0f);
                    sj[u] = x.x;
                    mx[u] = __float_as_int(x.y) < 0;
                    const float* col = gy + (int64_t)nt * (__float_as_int(x.y) & 0x7FFFFFFF);
#pragma unroll
                    for (int q = 0; q < NTW; ++q) {
                        const int t = q * 32 + lane;
                        e[u][q] = j0 + u < n && t < nt ? __ldg(col + t) : 0.0f;
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u) {
#pragma unroll
                    for (int q = 0; q < NTW; ++q) {
                        acc[q] = fmaf(e[u][q], sj[u], acc[q]);
                        if (mx[u]) acc[q] = fmaf(e[u][q], 0.0f, acc[q]);  // nothing but for an infinite gy: NaN
                    }
                }
            }
            __syncwarp();  // the buffer is rewritten by the next window
        }
#pragma unroll
        for (int q = 0; q < NTW; ++q) {
            const int t = q * 32 + lane;
            if (t < nt) partial[(int64_t)c * nt + t] = acc[q];
        }
    }
}

// gD[θ, a] = Σ over the chunks of atom a: one block per (atom, 32 θ), its warps
// taking every n-th chunk, their sums added in warp order (so the result does not
// depend on timing).  One thread per (θ, a) walked all chunks of its atom alone.
constexpr int GRAD_RED_WARPS = 8;

__global__ void __launch_bounds__(32 * GRAD_RED_WARPS)
graddD_reduce_kernel(const int32_t* __restrict__ atom_chunk, int nt, const float* __restrict__ partial,
                     float* __restrict__ gD) {
    __shared__ float part[GRAD_RED_WARPS][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int a = blockIdx.x, t = 32 * blockIdx.y + lane;
    const int c1 = atom_chunk[a + 1];
    float s = 0.0f;
    if (t < nt) {
#pragma unroll 4
        for (int c = atom_chunk[a] + warp; c < c1; c += GRAD_RED_WARPS) s += __ldg(partial + (int64_t)c * nt + t);
    }
    part[warp][lane] = s;
    __syncthreads();
    if (warp == 0 && t < nt) {
        float sum = part[0][lane];
#pragma unroll
        for (int i = 1; i < GRAD_RED_WARPS; ++i) sum += part[i][lane];
        gD[(int64_t)a * nt + t] = sum;
    }
}

// ----------------------------------------------------------- dispatchers

#define LIFE_NTW_SWITCH(ntw, ...)                              \
    switch (ntw) {                                             \
        case 1: { constexpr int NTW = 1; __VA_ARGS__; } break; \
        case 2: { constexpr int NTW = 2; __VA_ARGS__; } break; \
        case 3: { constexpr int NTW = 3; __VA_ARGS__; } break; \
        case 4: { constexpr int NTW = 4; __VA_ARGS__; } break; \
        case 5: { constexpr int NTW = 5; __VA_ARGS__; } break; \
        case 6: { constexpr int NTW = 6; __VA_ARGS__; } break; \
        case 7: { constexpr int NTW = 7; __VA_ARGS__; } break; \
        case 8: { constexpr int NTW = 8; __VA_ARGS__; } break; \
        default: set_error("Ntheta > 256 is not supported"); return LIFE_ENOTSUP; \
    }

template <int NTW, bool SMEM, class VT>
static life_status launch_dsc(life_index_s* ix, const float* D, const float* w, const float* b, float* y,
                              double* partial, int* n_partial, const life_sbb_state* gate, int gate_mode,
                              cudaStream_t s, const BatchGate& bg) {
    // by runs only with D in shared memory (and a buffer of 32 runs a warp behind it)
    const bool runs = SMEM && (ix->simt_runs & SIMT_RUNS_DSC);
    const size_t smem = (SMEM ? (size_t)ix->na * NTW * 32 * sizeof(float) : 0) + (runs ? SIMT_THREADS * sizeof(float2) : 0);
    auto kern = runs ? dsc_runs_kernel<NTW, VT> : dsc_simt_kernel<NTW, SMEM, VT>;
    if (SMEM) LIFE_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int grid = ix->num_sms;
    kern<<<grid, SIMT_THREADS, smem, s>>>(ix->vox.vox_ptr.as<int32_t>(), ix->vox.atom.as<uint16_t>(),
                                          ix->vox.fasc.as<int32_t>(), static_cast<const VT*>(ix->vox.val.p), D,
                                          ix->nt, ix->na, ix->nv, w, b, y, partial, gate, gate_mode, bg);
    LIFE_CHECK_LAUNCH();
    if (n_partial) *n_partial = grid;
    return LIFE_OK;
}

template <int NTW, bool SMEM, class VT>
static life_status launch_wc(life_index_s* ix, const float* D, const float* r, float* g, const life_sbb_state* gate,
                             int gate_mode, cudaStream_t s, const BatchGate& bg) {
    const size_t smem = SMEM ? (size_t)ix->na * NTW * 32 * sizeof(float) + SIMT_THREADS * sizeof(int32_t) : 0;
    auto kern = !SMEM ? wc_simt_kernel<NTW, VT>
                      : (ix->simt_runs & SIMT_RUNS_WC) ? wc_window_kernel<NTW, VT, true> : wc_window_kernel<NTW, VT, false>;
    if (SMEM) LIFE_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int grid = ix->num_sms;
    kern<<<grid, SIMT_THREADS, smem, s>>>(ix->vox.vox_ptr.as<int32_t>(), ix->vox.atom.as<uint16_t>(),
                                          ix->vox.fasc.as<int32_t>(), static_cast<const VT*>(ix->vox.val.p), D,
                                          ix->nt, ix->na, ix->nv, r, g, gate, gate_mode, bg);
    LIFE_CHECK_LAUNCH();
    return LIFE_OK;
}

int simt_total_warps(const life_index_s* ix) { return ix->num_sms * (SIMT_THREADS / 32); }

life_status dsc_simt(life_index_s* ix, const float* D, const float* w, const float* b, float* y, double* partial,
                     int* n_partial, const life_sbb_state* gate, int gate_mode, cudaStream_t s, const BatchGate& bg) {
    const int ntw = (ix->nt + 31) / 32;
    const bool smem = (size_t)ix->na * ntw * 32 * sizeof(float) <= SIMT_SMEM_LIMIT;
    const bool bf = ix->precision == LIFE_BF16;
    LIFE_NTW_SWITCH(ntw, {
        if (smem && bf) return launch_dsc<NTW, true, __nv_bfloat16>(ix, D, w, b, y, partial, n_partial, gate, gate_mode, s, bg);
        if (smem) return launch_dsc<NTW, true, float>(ix, D, w, b, y, partial, n_partial, gate, gate_mode, s, bg);
        if (bf) return launch_dsc<NTW, false, __nv_bfloat16>(ix, D, w, b, y, partial, n_partial, gate, gate_mode, s, bg);
        return launch_dsc<NTW, false, float>(ix, D, w, b, y, partial, n_partial, gate, gate_mode, s, bg);
    });
    return LIFE_OK;
}

life_status wc_simt(life_index_s* ix, const float* D, const float* r, float* g, const life_sbb_state* gate,
                    int gate_mode, cudaStream_t s, const BatchGate& bg) {
    const int ntw = (ix->nt + 31) / 32;
    const bool smem = (size_t)ix->na * ntw * 32 * sizeof(float) <= SIMT_SMEM_LIMIT;
    const bool bf = ix->precision == LIFE_BF16;
    LIFE_NTW_SWITCH(ntw, {
        if (smem && bf) return launch_wc<NTW, true, __nv_bfloat16>(ix, D, r, g, gate, gate_mode, s, bg);
        if (smem) return launch_wc<NTW, true, float>(ix, D, r, g, gate, gate_mode, s, bg);
        if (bf) return launch_wc<NTW, false, __nv_bfloat16>(ix, D, r, g, gate, gate_mode, s, bg);
        return launch_wc<NTW, false, float>(ix, D, r, g, gate, gate_mode, s, bg);
    });
    return LIFE_OK;
}

// The two launches of dL/dD, with the split-K partial sums in `partial` (chunks x Nθ).
static life_status launch_grad_D(const life_index_s* ix, const float* gy, const float* w, float* gD, float* partial,
                                 cudaStream_t s) {
    const AtomLayout& A = ix->atoml;
    const int ntw = (ix->nt + 31) / 32;
    if (A.n_chunks > 0) {
        const int64_t blocks = std::min<int64_t>(((int64_t)A.n_chunks * 32 + GRAD_THREADS - 1) / GRAD_THREADS,
                                                 (int64_t)ix->num_sms * 16);
        LIFE_NTW_SWITCH(ntw, {
            graddD_chunk_kernel<NTW><<<(unsigned)blocks, GRAD_THREADS, 0, s>>>(
                A.chunk_beg.as<int32_t>(), A.n_chunks, A.voxel.as<int32_t>(), A.fasc.as<int32_t>(),
                A.val.as<float>(), w, gy, ix->nt, partial);
        });
        LIFE_CHECK_LAUNCH();
    }
    graddD_reduce_kernel<<<dim3(ix->na, ntw), 32 * GRAD_RED_WARPS, 0, s>>>(A.atom_chunk.as<int32_t>(), ix->nt, partial,
                                                                          gD);
    LIFE_CHECK_LAUNCH();
    return LIFE_OK;
}

life_status grad_D_simt(life_index_s* ix, const float* gy, const float* w, float* gD, cudaStream_t s) {
    LIFE_TRY(build_atom_layout(ix, s));
    return launch_grad_D(ix, gy, w, gD, ix->atoml.partial.as<float>(), s);
}

}  // namespace life

// ------------------------------------------- dL/dD without device allocation
//
// life_dsc_grad_D_noalloc: the same two kernels as life_dsc_grad_D, with the
// split-K partial sums in a fixed device array compiled into this library
// instead of memory of the index (nnz / 256 · Nθ floats, about 120 MB at the
// paper's scale, which life_dsc_grad_D's first call allocates and the index keeps).
// It serves callers that may not allocate device memory while they run (for
// example code being captured into a CUDA graph, or an allocation-free real-time
// loop).

#include <mutex>

namespace life {

constexpr int64_t GRAD_D_NOALLOC_MAX_FLOATS = int64_t(1) << 20;  // 4 MiB on every device

// Device array for the partial sums.  In host code this name is only a stand-in;
// its device address comes from cudaGetSymbolAddress (see noalloc_scratch()).
static __device__ __align__(256) float g_grad_d_scratch[GRAD_D_NOALLOC_MAX_FLOATS];

// Per-device address of g_grad_d_scratch, looked up once with that device current.
static life_status noalloc_scratch(float** out) {
    static std::mutex mu;
    static float* addr[64] = {nullptr};
    int dev = 0;
    LIFE_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) {
        set_error("life_dsc_grad_D_noalloc: device ordinal %d out of range", dev);
        return LIFE_ERANGE;
    }
    std::lock_guard<std::mutex> lock(mu);
    if (!addr[dev]) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_grad_d_scratch);
        if (e != cudaSuccess || !p) {
            set_error("life_dsc_grad_D_noalloc: cudaGetSymbolAddress failed: %s", cudaGetErrorString(e));
            return LIFE_ECUDA;
        }
        addr[dev] = static_cast<float*>(p);
    }
    *out = addr[dev];
    return LIFE_OK;
}

}  // namespace life

extern "C" life_status life_dsc_grad_D_noalloc(life_index idx, const float* gy, const float* w, float* gD,
                                               void* stream) {
    using namespace life;
    if (!idx || !gy || !w || !gD) {
        set_error("life_dsc_grad_D_noalloc: null argument");
        return LIFE_EINVAL;
    }
    AtomLayout& A = idx->atoml;
    if (!A.built) {
        set_error("life_dsc_grad_D_noalloc: the atom-sorted layout is missing; call life_dsc_grad_D once "
                  "on this index during set-up (that call builds it)");
        return LIFE_EINVAL;
    }
    const int64_t need = (int64_t)A.n_chunks * idx->nt;
    if (need > GRAD_D_NOALLOC_MAX_FLOATS) {
        set_error("life_dsc_grad_D_noalloc: needs %lld floats of scratch (atom chunks x Ntheta), the fixed "
                  "array holds %lld; use life_dsc_grad_D", (long long)need, (long long)GRAD_D_NOALLOC_MAX_FLOATS);
        return LIFE_ERANGE;
    }
    float* partial = nullptr;
    LIFE_TRY(noalloc_scratch(&partial));
    return launch_grad_D(idx, gy, w, gD, partial, (cudaStream_t)stream);
}
