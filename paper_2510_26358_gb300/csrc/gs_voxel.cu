// Voxel-hash insertion of fused points (Sec. III-B, Eq. 5) and the LRU active
// set of the incremental map ("Memory Management").
//
// Keys: k = floor(x/v) P1 + floor(y/v) P2 + floor(z/v) P3 in unsigned 64-bit
// arithmetic (wrap-around), P = Teschner et al.'s primes, x/v divided in
// float32 (IEEE) before the floor.  The all-ones key is folded onto its
// predecessor so that it can mark empty hash slots.
//
// Insertion of a batch of points at frame f uses one open-addressing table
// over the batch's point keys (capacity a power of two >= 2 points, linear
// probing; each slot keeps the smallest point index that carries its key):
//   1. every point inserts its key (atomicCAS) and records its slot;
//   2. every device splat probes its key: found -> last_used = f and the
//      voxel is marked known; every host-resident key likewise -> reload flag;
//   3. the points that are the first of an unknown voxel create new splats,
//      compacted in point order (deterministic): mean = the point, isotropic
//      log-scale ln(s_init), identity rotation, opacity o_init, SH DC =
//      (rgb - 1/2) / Y00, higher coefficients 0.
// LRU selection: with n > tau splats, the (n - tau) smallest (last_used,
// index) pairs are flagged, by an exact radix select of the last_used value
// (three passes of 11, 11 and 10 bits) and an ordered count of the ties.
// Partition: a stable split of the splat rows by a flag array into a kept and
// a moved set; either side may live in host-mapped memory (offload, reload).
#include "gs_internal.cuh"
#include "gs_rows.cuh"
#include "gs_scan.cuh"

#include <cmath>

namespace {
constexpr unsigned long long kEmpty = ~0ull;
constexpr int kSelBins = 2048;  // 11-bit digits: three passes over the 32 bits
}

struct gs_voxel {
    int64_t max_points = 0, max_items = 0;
    uint64_t cap = 0;
    int cap_bits = 0;
    unsigned long long *tkey = nullptr;  // [cap]
    int32_t *tmin = nullptr;             // [cap]
    int32_t *tknown = nullptr;           // [cap]
    uint32_t *pslot = nullptr;           // [max_points]
    uint32_t *block_sum = nullptr, *block_off = nullptr;  // [nblocks]
    uint32_t *hist = nullptr;            // [kSelBins]
    uint32_t *sel = nullptr;             // [4] prefix, mask, remaining rank, finished blocks
    int64_t *state = nullptr;            // [0] new splats needed, [1] capacity flag, [2] kept, [3] moved
    int64_t kernel_launches = 0;
};

namespace gs {
namespace {

constexpr int VT = 256;
constexpr int VCHUNK = kRowChunk;  // items of a block of the ordered kernels
static_assert(VCHUNK == 2 * VT, "two items a thread");
constexpr unsigned long long kP1 = 73856093ull, kP2 = 19349663ull, kP3 = 83492791ull;
constexpr float kY00 = 0.28209479177387814f;

__device__ __forceinline__ unsigned long long voxel_key(float x, float y, float z, float v) {
    const long long cx = (long long)floorf(__fdiv_rn(x, v));
    const long long cy = (long long)floorf(__fdiv_rn(y, v));
    const long long cz = (long long)floorf(__fdiv_rn(z, v));
    const unsigned long long k = (unsigned long long)cx * kP1 + (unsigned long long)cy * kP2 +
                                 (unsigned long long)cz * kP3;
    return k == kEmpty ? kEmpty - 1 : k;
}

__device__ __forceinline__ uint32_t slot_of(unsigned long long k, int bits) {
    return (uint32_t)((k * 0x9E3779B97F4A7C15ull) >> (64 - bits));
}

__global__ void __launch_bounds__(VT) k_voxel_keys(const float *xyz, int64_t n, int32_t stride, float v,
                                                   unsigned long long *keys) {
    for (int64_t i = (int64_t)blockIdx.x * VT + threadIdx.x; i < n; i += (int64_t)gridDim.x * VT) {
        const float *p = xyz + i * stride;
        keys[i] = voxel_key(p[0], p[1], p[2], v);
    }
}

__global__ void __launch_bounds__(VT) k_table_insert(const float *pts, int64_t n, float v, unsigned long long *tkey,
                                                     int32_t *tmin, uint32_t *pslot, int bits) {
    const uint32_t mask = (1u << bits) - 1u;
    for (int64_t i = (int64_t)blockIdx.x * VT + threadIdx.x; i < n; i += (int64_t)gridDim.x * VT) {
        const float *p = pts + 6 * i;
        const unsigned long long k = voxel_key(p[0], p[1], p[2], v);
        uint32_t s = slot_of(k, bits);
        // at most n distinct keys in a table of >= 2n slots: a free or
        // matching slot exists, so the probe ends within (mask + 1) steps
        for (uint32_t probe = 0; probe <= mask; ++probe) {
            const unsigned long long cur = atomicCAS(tkey + s, kEmpty, k);
            if (cur == kEmpty || cur == k) {
                atomicMin(tmin + s, (int32_t)i);
                pslot[i] = s;
                break;
            }
            s = (s + 1u) & mask;
        }
    }
}

// Empties the table: keys all ones, smallest point index at its largest, no
// voxel known (one launch, 16-byte stores; the capacity is a multiple of 16).
__global__ void __launch_bounds__(VT) k_table_clear(unsigned long long *tkey, int32_t *tmin, int32_t *tknown,
                                                    int64_t cap) {
    const int64_t stride = (int64_t)gridDim.x * VT;
    const uint4 ones = make_uint4(~0u, ~0u, ~0u, ~0u), zero = make_uint4(0u, 0u, 0u, 0u);
    const uint4 large = make_uint4(0x7F7F7F7Fu, 0x7F7F7F7Fu, 0x7F7F7F7Fu, 0x7F7F7F7Fu);
    for (int64_t i = (int64_t)blockIdx.x * VT + threadIdx.x; i < cap / 4; i += stride) {
        reinterpret_cast<uint4 *>(tkey)[2 * i] = ones;
        reinterpret_cast<uint4 *>(tkey)[2 * i + 1] = ones;
        reinterpret_cast<uint4 *>(tmin)[i] = large;
        reinterpret_cast<uint4 *>(tknown)[i] = zero;
    }
}

// Probes the keys of the device splats (found -> last_used = frame) and of the
// host-resident ones (reload = found) in one launch, and marks their voxels known.
__global__ void __launch_bounds__(VT) k_table_probe(const unsigned long long *splat_keys, int64_t n_splats,
                                                    int32_t *last_used, int32_t frame,
                                                    const unsigned long long *host_keys, int64_t n_host, int32_t *reload,
                                                    const unsigned long long *tkey, int32_t *tknown, int bits) {
    const uint32_t mask = (1u << bits) - 1u;
    for (int64_t j = (int64_t)blockIdx.x * VT + threadIdx.x; j < n_splats + n_host; j += (int64_t)gridDim.x * VT) {
        const bool host = j >= n_splats;
        unsigned long long k = host ? host_keys[j - n_splats] : splat_keys[j];
        if (k == kEmpty) k = kEmpty - 1;
        uint32_t s = slot_of(k, bits);
        bool found = false;
        for (uint32_t probe = 0; probe <= mask; ++probe) {
            const unsigned long long cur = tkey[s];
            if (cur == kEmpty) break;
            if (cur == k) {
                found = true;
                tknown[s] = 1;
                break;
            }
            s = (s + 1u) & mask;
        }
        if (host) reload[j - n_splats] = found ? 1 : 0;
        else if (found) last_used[j] = frame;
    }
}

__device__ __forceinline__ uint32_t is_creator(int64_t i, int64_t n, const uint32_t *pslot, const int32_t *tmin,
                                               const int32_t *tknown) {
    if (i >= n) return 0u;
    const uint32_t s = pslot[i];
    return (tknown[s] == 0 && tmin[s] == (int32_t)i) ? 1u : 0u;
}

// Called by every thread after the block's results are written: true in the
// one block that finishes last, which then sees the others' (and puts the
// counter back to 0).
__device__ __forceinline__ bool last_block(uint32_t *done) {
    __shared__ bool s_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        s_last = atomicAdd(done, 1u) == gridDim.x - 1;
        if (s_last) *done = 0u;
    }
    __syncthreads();
    if (s_last) __threadfence();
    return s_last;
}

// Where a chunk count's exclusive scan goes: total -> state[0] (and *total),
// total > capacity -> state[1], (items - total, total) -> split[0, 1].
struct ScanOut {
    uint32_t *block_sum, *block_off, *done;
    int64_t capacity;
    int64_t *state, *total, *split;
};

// Writes the block's count; the last block scans all of them (eight a thread
// at a time: a scan of its own cost a launch of 2-4 us).
__device__ __forceinline__ void count_and_scan(uint32_t c, const ScanOut &S, int64_t items) {
    __shared__ uint32_t sm[VT / 32];
    const uint32_t t = block_sum_u32<VT>(c, sm);
    if (threadIdx.x == 0) S.block_sum[blockIdx.x] = t;
    if (!last_block(S.done)) return;
    const int nblocks = (int)gridDim.x;
    uint32_t carry = 0;
    for (int b0 = 0; b0 < nblocks; b0 += 8 * VT) {
        const int b = b0 + 8 * threadIdx.x;
        uint32_t v[8], sum = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            v[k] = b + k < nblocks ? __ldcg(S.block_sum + b + k) : 0u;
            sum += v[k];
        }
        uint32_t tot, ex = carry + block_scan_u32<VT>(sum, sm, tot);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (b + k < nblocks) S.block_off[b + k] = ex;
            ex += v[k];
        }
        carry += tot;
    }
    if (threadIdx.x == 0) {
        S.state[0] = carry;
        S.state[1] = (int64_t)carry > S.capacity ? 1 : 0;
        if (S.total) *S.total = carry;
        if (S.split) {
            S.split[0] = items - carry;
            S.split[1] = carry;
        }
    }
}

__global__ void __launch_bounds__(VT) k_creator_count(int64_t n, const uint32_t *pslot, const int32_t *tmin,
                                                      const int32_t *tknown, ScanOut S) {
    const int64_t i = (int64_t)blockIdx.x * VCHUNK + threadIdx.x;
    count_and_scan(is_creator(i, n, pslot, tmin, tknown) + is_creator(i + VT, n, pslot, tmin, tknown), S, n);
}

struct EmitArgs {
    const float *pts;
    int64_t n;
    float v, log_s, omega;
    const uint32_t *pslot;
    const int32_t *tmin, *tknown;
    const uint32_t *block_off;
    const int64_t *state;
    float *means, *log_scales, *quats, *opacity, *sh;
    unsigned long long *keys;
};

// The new splats of a chunk of points are consecutive: their rows are written
// element by element, neighbouring threads on neighbouring words (a thread a
// row, 48 words apart, took 47 us for 0.2M splats of SH degree 3, 11 us).
template <int NSH>
__global__ void __launch_bounds__(VT) k_creator_emit(EmitArgs A) {
    __shared__ uint32_t sm[VT / 32];
    __shared__ uint16_t rows[VCHUNK];
    if (A.state[1]) return;
    const int64_t i0 = (int64_t)blockIdx.x * VCHUNK, o0 = A.block_off[blockIdx.x];
    const int64_t i = i0 + 2 * threadIdx.x;
    const uint32_t c0 = is_creator(i, A.n, A.pslot, A.tmin, A.tknown);
    const uint32_t c1 = is_creator(i + 1, A.n, A.pslot, A.tmin, A.tknown);
    uint32_t tot;
    uint32_t o = block_scan_u32<VT>(c0 + c1, sm, tot);
    if (c0) rows[o++] = (uint16_t)(2 * threadIdx.x);
    if (c1) rows[o] = (uint16_t)(2 * threadIdx.x + 1);
    __syncthreads();
    const int n = (int)tot;
    const float *pts = A.pts + 6 * i0;
    for (int e = threadIdx.x; e < 3 * n; e += VT) {
        const int r = e / 3, ch = e - 3 * r;
        A.means[3 * o0 + e] = pts[6 * rows[r] + ch];
        A.log_scales[3 * o0 + e] = A.log_s;
    }
    for (int e = threadIdx.x; e < 4 * n; e += VT) A.quats[4 * o0 + e] = (e & 3) == 0 ? 1.f : 0.f;
    for (int r = threadIdx.x; r < n; r += VT) {
        const float *p = pts + 6 * rows[r];
        A.opacity[o0 + r] = A.omega;
        A.keys[o0 + r] = voxel_key(p[0], p[1], p[2], A.v);
    }
    float *sh = A.sh + o0 * NSH;
    auto dc = [&](int r, int ch) { return (pts[6 * rows[r] + 3 + ch] - 0.5f) / kY00; };
    if (NSH % 4 == 0 && ((uintptr_t)sh & 15) == 0) {
        constexpr int W = NSH / 4 > 0 ? NSH / 4 : 1;
        for (int e = threadIdx.x; e < W * n; e += VT) {
            const int r = e / W;
            reinterpret_cast<float4 *>(sh)[e] =
                e - r * W == 0 ? make_float4(dc(r, 0), dc(r, 1), dc(r, 2), 0.f) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    } else {
        for (int e = threadIdx.x; e < NSH * n; e += VT) {
            const int r = e / NSH, k = e - r * NSH;
            sh[e] = k < 3 ? dc(r, k) : 0.f;
        }
    }
}

// ---------------------------------------------------------------------------
// LRU selection
// ---------------------------------------------------------------------------

__device__ __forceinline__ uint32_t lru_bits(int32_t v) { return (uint32_t)v ^ 0x80000000u; }

// One pass of the radix select over an 11-bit digit (the first: prefix and
// mask 0, rank `rank`): the last block to finish takes the digit in which the
// remaining rank falls and clears the histogram for the next pass.  (A
// launch each for the start, every pass and every choice of a digit took 12
// launches a selection of 2-5 us each; this takes five.)  Values are mostly
// alike (recent frames), so a warp that agrees on its digit adds once.
__global__ void __launch_bounds__(VT) k_sel_pass(const int32_t *lu, int64_t n, uint32_t *sel, int shift, int bits,
                                                 bool first, uint32_t rank, uint32_t *hist) {
    __shared__ uint32_t h[kSelBins];
    __shared__ uint32_t sm[VT / 32];
    for (int i = threadIdx.x; i < kSelBins; i += VT) h[i] = 0;
    __syncthreads();
    const uint32_t prefix = first ? 0u : sel[0], mask = first ? 0u : sel[1], left = first ? rank : sel[2];
    const uint32_t dmask = (1u << bits) - 1u;
    const int64_t stride = (int64_t)gridDim.x * VT;
    const int64_t whole = n / VT * VT;  // whole warps take part in the vote
    for (int64_t i0 = (int64_t)blockIdx.x * VT + threadIdx.x; i0 < whole; i0 += 4 * stride) {
        uint32_t u[4];  // four loads in flight; the strides past the end are warp-uniform
#pragma unroll
        for (int k = 0; k < 4; ++k) u[k] = i0 + k * stride < whole ? lru_bits(lu[i0 + k * stride]) : 0u;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if (i0 + k * stride >= whole) break;
            const uint32_t d = (u[k] & mask) == prefix ? (u[k] >> shift) & dmask : ~0u;
            if (__all_sync(0xffffffffu, d == __shfl_sync(0xffffffffu, d, 0))) {
                if ((threadIdx.x & 31) == 0 && d != ~0u) atomicAdd(h + d, 32u);
            } else if (d != ~0u) {
                atomicAdd(h + d, 1u);
            }
        }
    }
    if (blockIdx.x == 0 && whole + threadIdx.x < n) {
        const uint32_t u = lru_bits(lu[whole + threadIdx.x]);
        if ((u & mask) == prefix) atomicAdd(h + ((u >> shift) & dmask), 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kSelBins; i += VT)
        if (h[i]) atomicAdd(hist + i, h[i]);
    if (!last_block(sel + 3)) return;
    constexpr int PER = kSelBins / VT;
    uint32_t c[PER], sum = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        c[k] = __ldcg(hist + PER * threadIdx.x + k);
        sum += c[k];
    }
    uint32_t tot, before = block_scan_u32<VT>(sum, sm, tot);
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        if (before < left && before + c[k] >= left) {
            sel[0] = prefix | (uint32_t)(PER * threadIdx.x + k) << shift;
            sel[1] = mask | dmask << shift;
            sel[2] = left - before;
        }
        before += c[k];
        hist[PER * threadIdx.x + k] = 0;
    }
}

__global__ void __launch_bounds__(VT) k_sel_eqcount(const int32_t *lu, int64_t n, const uint32_t *sel, ScanOut S) {
    const int64_t j = (int64_t)blockIdx.x * VCHUNK + threadIdx.x;
    const uint32_t f = sel[0];
    uint32_t c = 0;
#pragma unroll
    for (int i = 0; i < 2; ++i) c += j + i * VT < n && lru_bits(lu[j + i * VT]) == f;
    count_and_scan(c, S, n);
}

__global__ void __launch_bounds__(VT) k_sel_mark(const int32_t *lu, int64_t n, const uint32_t *sel,
                                                 const uint32_t *block_off, int32_t *flags) {
    __shared__ uint32_t sm[VT / 32];
    const int64_t j = (int64_t)blockIdx.x * VCHUNK + 2 * threadIdx.x;
    const uint32_t f = sel[0], r = sel[2];
    uint32_t u[2], eq[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        u[i] = j + i < n ? lru_bits(lu[j + i]) : 0xFFFFFFFFu;
        eq[i] = j + i < n && u[i] == f;
    }
    uint32_t tot;
    uint32_t rank = block_off[blockIdx.x] + block_scan_u32<VT>(eq[0] + eq[1], sm, tot);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        if (j + i < n) flags[j + i] = (u[i] < f || (eq[i] && rank < r)) ? 1 : 0;
        rank += eq[i];
    }
}

__global__ void k_fill_i32(int32_t *p, int64_t n, int32_t v) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        p[i] = v;
}

// ---------------------------------------------------------------------------
// stable partition
// ---------------------------------------------------------------------------

__global__ void __launch_bounds__(VT) k_flag_count(const int32_t *flags, int64_t n, ScanOut S) {
    const int64_t j = (int64_t)blockIdx.x * VCHUNK + threadIdx.x;
    uint32_t c = 0;
#pragma unroll
    for (int i = 0; i < 2; ++i) c += j + i * VT < n && flags[j + i * VT] != 0;
    count_and_scan(c, S, n);
}

struct PartArgs {
    const int32_t *flags;
    int64_t n;
    const uint32_t *block_off;
    const float *in[5];
    float *kept[5], *moved[5];
    const unsigned long long *in_keys;
    unsigned long long *kept_keys, *moved_keys;
    const int32_t *in_lu;
    int32_t *kept_lu, *moved_lu;
};

// One side's rows of a block's chunk (consecutive there): the arrays one
// after the other, neighbouring threads on neighbouring words, which also
// makes whole-line writes of the rows that go to host memory.
template <int NSH>
__device__ __forceinline__ void copy_side(const PartArgs &A, int64_t j0, int64_t o0, const uint16_t *rows, int n,
                                          float *const dst[5], unsigned long long *keys, int32_t *lu) {
    copy_rows<VT, NSH, ROWS_COPY>(A.in[4] + j0 * NSH, dst[4] + o0 * NSH, rows, n);
    copy_rows<VT, 3, ROWS_COPY>(A.in[0] + 3 * j0, dst[0] + 3 * o0, rows, n);
    copy_rows<VT, 3, ROWS_COPY>(A.in[1] + 3 * j0, dst[1] + 3 * o0, rows, n);
    copy_rows<VT, 4, ROWS_COPY>(A.in[2] + 4 * j0, dst[2] + 4 * o0, rows, n);
    copy_rows<VT, 1, ROWS_COPY>(A.in[3] + j0, dst[3] + o0, rows, n);
    if (A.in_keys) copy_elements<VT, 1, ROWS_COPY>(A.in_keys + j0, keys + o0, rows, n);
    if (A.in_lu) copy_elements<VT, 1, ROWS_COPY>(A.in_lu + j0, lu + o0, rows, n);
}

template <int NSH>
__global__ void __launch_bounds__(VT) k_partition(PartArgs A) {
    __shared__ uint32_t sm[VT / 32];
    __shared__ uint16_t rows[VCHUNK];  // kept rows from the front, moved rows after them
    const int64_t j0 = (int64_t)blockIdx.x * VCHUNK;
    const int64_t moved0 = A.block_off[blockIdx.x], kept0 = j0 - moved0;
    const int n = (int)(A.n - j0 < VCHUNK ? A.n - j0 : VCHUNK);
    const int i = 2 * threadIdx.x;
    const uint32_t f0 = i < n && A.flags[j0 + i], f1 = i + 1 < n && A.flags[j0 + i + 1];
    uint32_t moved;
    uint32_t m = block_scan_u32<VT>(f0 + f1, sm, moved);  // moved rows before this thread's
    const int kept = n - (int)moved;
    if (i < n) rows[f0 ? kept + m : i - m] = (uint16_t)i;
    m += f0;
    if (i + 1 < n) rows[f1 ? kept + m : i + 1 - m] = (uint16_t)(i + 1);
    __syncthreads();
    copy_side<NSH>(A, j0, moved0, rows + kept, (int)moved, A.moved, A.moved_keys, A.moved_lu);
    copy_side<NSH>(A, j0, kept0, rows, kept, A.kept, A.kept_keys, A.kept_lu);
}

int grid_for(int64_t n) { return (int)std::max<int64_t>(1, std::min<int64_t>((n + VT - 1) / VT, 152 * 16)); }
int nblocks_for(int64_t n) { return (int)std::max<int64_t>(1, (n + VCHUNK - 1) / VCHUNK); }

ScanOut scan_out(gs_voxel *vx, int64_t capacity, int64_t *state, int64_t *total, int64_t *split) {
    return {vx->block_sum, vx->block_off, vx->sel + 3, capacity, state, total, split};
}

bool params_set(const gs_param_arrays *a) {
    return a && a->means && a->log_scales && a->quats && a->opacity_logits && a->sh;
}

}  // namespace
}  // namespace gs

using namespace gs;

extern "C" {

gs_status gs_voxel_keys(const float *xyz, int64_t n, int32_t stride, float voxel, uint64_t *keys, void *stream) {
    if (n < 0 || stride < 3 || !(voxel > 0.f) || (n > 0 && (!xyz || !keys))) {
        set_last_error("gs_voxel_keys: bad arguments");
        return GS_ERR_INVALID_ARG;
    }
    if (n == 0) return GS_OK;
    k_voxel_keys<<<grid_for(n), VT, 0, (cudaStream_t)stream>>>(xyz, n, stride, voxel,
                                                                 reinterpret_cast<unsigned long long *>(keys));
    return check_launch("voxel_keys");
}

gs_status gs_voxel_create(int64_t max_points, int64_t max_items, gs_voxel **out) {
    if (!out || max_points < 0 || max_items < 0 || max_points > (1ll << 29) || max_items > (1ll << 30)) {
        set_last_error("gs_voxel_create: bad arguments");
        return GS_ERR_INVALID_ARG;
    }
    gs_voxel *vx = new gs_voxel();
    vx->max_points = max_points;
    vx->max_items = max_items;
    vx->cap_bits = 4;
    while ((1ll << vx->cap_bits) < 2 * std::max<int64_t>(1, max_points)) ++vx->cap_bits;
    vx->cap = 1ull << vx->cap_bits;
    const int nb = nblocks_for(std::max(max_points, max_items));
    cudaError_t e = cudaMalloc(&vx->tkey, sizeof(unsigned long long) * vx->cap);
    if (e == cudaSuccess) e = cudaMalloc(&vx->tmin, sizeof(int32_t) * vx->cap);
    if (e == cudaSuccess) e = cudaMalloc(&vx->tknown, sizeof(int32_t) * vx->cap);
    if (e == cudaSuccess) e = cudaMalloc(&vx->pslot, sizeof(uint32_t) * std::max<int64_t>(1, max_points));
    if (e == cudaSuccess) e = cudaMalloc(&vx->block_sum, sizeof(uint32_t) * nb);
    if (e == cudaSuccess) e = cudaMalloc(&vx->block_off, sizeof(uint32_t) * nb);
    if (e == cudaSuccess) e = cudaMalloc(&vx->hist, sizeof(uint32_t) * kSelBins);
    if (e == cudaSuccess) e = cudaMalloc(&vx->sel, sizeof(uint32_t) * 4);
    if (e == cudaSuccess) e = cudaMalloc(&vx->state, sizeof(int64_t) * 4);
    if (e == cudaSuccess) e = cudaMemset(vx->state, 0, sizeof(int64_t) * 4);
    if (e == cudaSuccess) e = cudaMemset(vx->hist, 0, sizeof(uint32_t) * kSelBins);
    if (e == cudaSuccess) e = cudaMemset(vx->sel, 0, sizeof(uint32_t) * 4);
    if (e != cudaSuccess) {
        set_last_error(std::string("gs_voxel_create: ") + cudaGetErrorString(e));
        gs_voxel_destroy(vx);
        return GS_ERR_CUDA;
    }
    *out = vx;
    return GS_OK;
}

void gs_voxel_destroy(gs_voxel *vx) {
    if (!vx) return;
    void *ptrs[] = {vx->tkey, vx->tmin, vx->tknown, vx->pslot, vx->block_sum, vx->block_off, vx->hist, vx->sel,
                    vx->state};
    for (void *p : ptrs)
        if (p) cudaFree(p);
    delete vx;
}

gs_status gs_voxel_insert(gs_voxel *vx, const gs_insert_params *p, const float *points, int64_t n_points,
                          const uint64_t *splat_keys, int32_t *last_used, int64_t n_splats, const uint64_t *host_keys,
                          int32_t *reload, int64_t n_host, int32_t sh_degree, const gs_param_arrays *new_splats,
                          uint64_t *new_keys, int64_t new_capacity, int64_t *n_new, void *stream) {
    if (!vx || !p || n_points < 0 || n_points > vx->max_points || n_splats < 0 || n_host < 0 || sh_degree < 0 ||
        sh_degree > 3 || new_capacity < 0 || new_capacity > 0x7FFFFFFFll || !(p->voxel > 0.f) ||
        !(p->s_init > 0.f) || !(p->o_init > 0.f && p->o_init < 1.f)) {
        set_last_error("gs_voxel_insert: bad arguments");
        return GS_ERR_INVALID_ARG;
    }
    if ((n_points > 0 && !points) || (n_splats > 0 && (!splat_keys || !last_used)) ||
        (n_host > 0 && (!host_keys || !reload)) || (new_capacity > 0 && (!params_set(new_splats) || !new_keys))) {
        set_last_error("gs_voxel_insert: NULL array");
        return GS_ERR_INVALID_ARG;
    }
    cudaStream_t s = (cudaStream_t)stream;
    const unsigned long long *sk = reinterpret_cast<const unsigned long long *>(splat_keys);
    const unsigned long long *hk = reinterpret_cast<const unsigned long long *>(host_keys);
    ++vx->kernel_launches;
    k_table_clear<<<grid_for((int64_t)vx->cap / 4), VT, 0, s>>>(vx->tkey, vx->tmin, vx->tknown, (int64_t)vx->cap);
    if (n_points > 0) {
        ++vx->kernel_launches;
        k_table_insert<<<grid_for(n_points), VT, 0, s>>>(points, n_points, p->voxel, vx->tkey, vx->tmin, vx->pslot,
                                                         vx->cap_bits);
    }
    if (n_splats + n_host > 0) {
        ++vx->kernel_launches;
        k_table_probe<<<grid_for(n_splats + n_host), VT, 0, s>>>(sk, n_splats, last_used, p->frame, hk, n_host, reload,
                                                                 vx->tkey, vx->tknown, vx->cap_bits);
    }
    const int nb = nblocks_for(n_points);
    ++vx->kernel_launches;
    k_creator_count<<<nb, VT, 0, s>>>(n_points, vx->pslot, vx->tmin, vx->tknown,
                                      scan_out(vx, new_capacity, vx->state, n_new, nullptr));
    gs_status r = check_launch("voxel_insert");
    if (r != GS_OK || n_points == 0) return r;
    EmitArgs A{};
    A.pts = points;
    A.n = n_points;
    A.v = p->voxel;
    A.log_s = (float)std::log((double)p->s_init);
    A.omega = (float)std::log((double)p->o_init / (1.0 - (double)p->o_init));
    A.pslot = vx->pslot;
    A.tmin = vx->tmin;
    A.tknown = vx->tknown;
    A.block_off = vx->block_off;
    A.state = vx->state;
    if (new_capacity > 0) {
        A.means = new_splats->means;
        A.log_scales = new_splats->log_scales;
        A.quats = new_splats->quats;
        A.opacity = new_splats->opacity_logits;
        A.sh = new_splats->sh;
        A.keys = reinterpret_cast<unsigned long long *>(new_keys);
    }
    if (new_capacity > 0) {
        ++vx->kernel_launches;
        switch (sh_degree) {
            case 0: k_creator_emit<3><<<nb, VT, 0, s>>>(A); break;
            case 1: k_creator_emit<12><<<nb, VT, 0, s>>>(A); break;
            case 2: k_creator_emit<27><<<nb, VT, 0, s>>>(A); break;
            default: k_creator_emit<48><<<nb, VT, 0, s>>>(A);
        }
    }
    return check_launch("voxel_emit");
}

gs_status gs_voxel_status(gs_voxel *vx, void *stream, int64_t *n_new) {
    if (!vx) {
        set_last_error("gs_voxel_status: NULL argument");
        return GS_ERR_INVALID_ARG;
    }
    int64_t h[4] = {0, 0, 0, 0};
    cudaError_t e = cudaStreamSynchronize((cudaStream_t)stream);
    if (e == cudaSuccess) e = cudaMemcpy(h, vx->state, sizeof h, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) {
        set_last_error(std::string("gs_voxel_status: ") + cudaGetErrorString(e));
        return GS_ERR_CUDA;
    }
    if (n_new) *n_new = h[0];
    return h[1] ? GS_ERR_CAPACITY : GS_OK;
}

gs_status gs_active_select(gs_voxel *vx, const int32_t *last_used, int64_t n, int64_t tau, int32_t *flags,
                           void *stream) {
    if (!vx || n < 0 || n > vx->max_items || tau < 0 || (n > 0 && (!last_used || !flags))) {
        set_last_error("gs_active_select: bad arguments");
        return GS_ERR_INVALID_ARG;
    }
    if (n == 0) return GS_OK;
    cudaStream_t s = (cudaStream_t)stream;
    const int64_t m = n - tau;
    if (m <= 0 || m >= n) {
        ++vx->kernel_launches;
        k_fill_i32<<<grid_for(n), VT, 0, s>>>(flags, n, m <= 0 ? 0 : 1);
        return check_launch("active_select");
    }
    vx->kernel_launches += 5;
    const int shift[3] = {21, 10, 0}, bits[3] = {11, 11, 10};
    for (int p = 0; p < 3; ++p)
        k_sel_pass<<<grid_for(n / 4), VT, 0, s>>>(last_used, n, vx->sel, shift[p], bits[p], p == 0, (uint32_t)m, vx->hist);
    const int nb = nblocks_for(n);
    k_sel_eqcount<<<nb, VT, 0, s>>>(last_used, n, vx->sel, scan_out(vx, INT64_MAX, vx->state + 2, nullptr, nullptr));
    k_sel_mark<<<nb, VT, 0, s>>>(last_used, n, vx->sel, vx->block_off, flags);
    return check_launch("active_select");
}

gs_status gs_partition(gs_voxel *vx, const int32_t *flags, int64_t n, int32_t sh_degree, const gs_param_arrays *in,
                       const uint64_t *in_keys, const int32_t *in_last_used, const gs_param_arrays *kept,
                       uint64_t *kept_keys, int32_t *kept_last_used, const gs_param_arrays *moved, uint64_t *moved_keys,
                       int32_t *moved_last_used, int64_t *counts, void *stream) {
    if (!vx || n < 0 || n > vx->max_items || sh_degree < 0 || sh_degree > 3 ||
        (n > 0 && (!flags || !params_set(in) || !params_set(kept) || !params_set(moved))) ||
        (in_keys && (!kept_keys || !moved_keys)) || (in_last_used && (!kept_last_used || !moved_last_used))) {
        set_last_error("gs_partition: bad arguments");
        return GS_ERR_INVALID_ARG;
    }
    cudaStream_t s = (cudaStream_t)stream;
    const int nb = nblocks_for(n);
    ++vx->kernel_launches;
    k_flag_count<<<nb, VT, 0, s>>>(flags, n, scan_out(vx, INT64_MAX, vx->state + 2, nullptr, counts));
    if (n == 0) return check_launch("partition");
    PartArgs A{};
    A.flags = flags;
    A.n = n;
    A.block_off = vx->block_off;
    const float *ins[5] = {in->means, in->log_scales, in->quats, in->opacity_logits, in->sh};
    float *ks[5] = {kept->means, kept->log_scales, kept->quats, kept->opacity_logits, kept->sh};
    float *ms[5] = {moved->means, moved->log_scales, moved->quats, moved->opacity_logits, moved->sh};
    for (int i = 0; i < 5; ++i) {
        A.in[i] = ins[i];
        A.kept[i] = ks[i];
        A.moved[i] = ms[i];
    }
    A.in_keys = reinterpret_cast<const unsigned long long *>(in_keys);
    A.kept_keys = reinterpret_cast<unsigned long long *>(kept_keys);
    A.moved_keys = reinterpret_cast<unsigned long long *>(moved_keys);
    A.in_lu = in_last_used;
    A.kept_lu = kept_last_used;
    A.moved_lu = moved_last_used;
    ++vx->kernel_launches;
    switch (sh_degree) {
        case 0: k_partition<3><<<nb, VT, 0, s>>>(A); break;
        case 1: k_partition<12><<<nb, VT, 0, s>>>(A); break;
        case 2: k_partition<27><<<nb, VT, 0, s>>>(A); break;
        default: k_partition<48><<<nb, VT, 0, s>>>(A);
    }
    return check_launch("partition");
}

}  // extern "C"
