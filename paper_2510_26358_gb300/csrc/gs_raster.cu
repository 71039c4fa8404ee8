// Tile rasteriser: forward alpha compositing and its adjoint.
//
// One CTA owns one tile at a time and pulls tiles of every view from a global
// work counter, so a single persistent launch covers all cameras of the
// batch, whatever their sizes.  Gaussians of the tile's depth-sorted list are
// staged `batch_depth` at a time in shared memory; each thread walks them for
// its pixels.
//
// Forward (front to back):  alpha = min(alpha_max, o e^{pw}); skip alpha <
// alpha_min; a fragment that would take T below t_min ends the pixel before it
// is blended; C += alpha T c, D += alpha T z, T *= (1 - alpha).  The CTA leaves
// a tile as soon as every pixel has ended.  Per pixel it keeps the list count
// up to the last blended fragment and the final T.
//
// Backward (back to front from that count): alpha is recomputed with the same
// instructions, T is recovered by division, and with h = gC.c + gD z + gA
//   dL/dalpha_j = T_j h_j - (sum_{k>j} w_k h_k) / (1 - alpha_j).
// The 10 image-space gradient components of each Gaussian are summed over the
// lane's pixels and then over the warp before they are added to its row by
// float atomics.
//
// The forward, and the backward of renders with few tiles, divide a tile into
// quadrants of 8x8 pixels, two a lane, and a warp holds one, two or four
// quadrants.  Of each entry it works only the quadrants that the Gaussian's
// ellipse reaches and that still have a pixel to blend: the passes are bound by
// instruction issue (FP32, selects and compares), and of the pixel slots of a
// walk over whole 16x16 tiles only 43 % blend (4M orchard, six 1920x1200 views;
// of the quadrants an entry meets 2.55 of 4 blend, 2.99 are reached).  The
// backward of larger renders takes a column of pixels a thread (see
// k_raster_bwd for why).  Pixel updates run without branches: a pixel
// that a fragment does not reach takes alpha = 0, for which each update is
// exactly the identity.
//
// The VAR variants also render each pixel's depth distribution under the
// weights w: its mean mu = sum w z / W and variance var = sum w (z - mu)^2 / W,
// W = sum w.  They are accumulated front to back by the weighted Welford
// update, in depths relative to the first blended fragment's, c:
//   W += w;  y = z - c;  d = y - m;  m += d w / W;  M2 += w d (y - m),
// so that rounding scales with the spread of the depths, not with the depth
// itself (mu = D / A in float loses ~sqrt(n) ulps of a 5 m depth, which a
// centimetre-scale variance term magnifies).  mu = c + m and var = M2 / W are
// kept per pixel (with 1/W) for the backward, and alpha is written as W
// (1 - T in exact arithmetic).  With sum w (z - mu) = 0 the adjoints are
//   dmu/dw_k = (z_k - mu) / W,                dmu/dz_k = w_k / W,
//   dvar/dw_k = ((z_k - mu)^2 - var) / W,     dvar/dz_k = 2 w_k (z_k - mu) / W,
// so with a = gmu / W and b = gvar / W, h gains a dz + b (dz^2 - var) and
// dL/dz gains w (a + 2 b dz), dz = z - mu.
#include "gs_internal.cuh"

namespace gs {
namespace {

// Paddings of the quadrant test (see quad_mask).
constexpr float kQuadRelPad = 1e-3f, kQuadAbsPad = 1e-2f;

// Entries staged at a time, at most (the configuration's batch depth below
// it): with 64 the staged entries of 20 one-warp CTAs of the forward fit an SM.
// The backward in pairs of entries takes all of kPairsDepth where few tiles leave
// the SMs idle anyway, and less where more CTAs an SM are worth more (128, 64, 32
// entries, us): 300 tiles of 16x16 54, 68, 71; 3600 127, 118, 120; 8x8: 4270 380, 409,
// 410.  (The backward by columns takes the configuration's depth.)
constexpr int kFwdDepth = 64, kPairsDepth = 128;

// How many quadrants a warp of the forward takes, by the number of 16x16 tiles
// (or as many pixels), in multiples of the measured GPU's 152 SMs.  Whole tiles share the most work between quadrants but make the
// fewest warps: with few tiles the time is the longest list's chain of
// entries, which is shorter the less a warp does for each.  Measured (one,
// two, four quadrants a warp, us).  The whole step: 300 tiles (320x240,
// box of 10k) 288, 298, -; 1200 (orchard of 200k, as below) 247, 258, -; 2400
// 318, 319, -; 3600 249, 247, -; the kernel: 7200 87, 64, 75; 24,480 (1M) -, 391,
// 406; 54,000 (4M) -, 971, 936.  With the variance (one, two; more do not fit the
// registers) 2400 tiles 73, 97; 7200 139, 107.
constexpr int kFwdHalfTiles = 152 * 16, kFwdWholeTiles = 152 * 256, kVarHalfTiles = 152 * 24;
// The backward works pairs of entries below kColumnTiles (16x16 tiles, or as many
// pixels), where that takes half of the time, and columns of pixels from there
// on, where the sums' order must stay (see k_raster_bwd).  8x8 tiles take columns
// from kColumnTiles8 of them on, where those are the faster ones.  Pairs, columns,
// us, orchard of 200k, one to three 640x480 views, without and with the variance:
// 16x16 1200 tiles 55, 145 and 57, 102; 2400 84, 184 and 88, 139; 3600 172, 354 and 184, 276;
// 8x8 4800 39, 66 and 41, 66; 9600 104, 96 and 113, 100; 14,400 203, 178 and 219, 188.
// (8x8 with long lists: 800k, 4800 tiles 164, 209; 6300 154, 183; of 1.3M in 2135 to 6405
// tiles one list's walk sets the time, 395 to 420 either way.)
// kDeepTiles counts tiles of any size, as CTAs: see kPairsDepth.
constexpr int kColumnTiles = 152 * 24, kColumnTiles8 = 152 * 48, kDeepTiles = 152 * 3;

// Resident warps an SM that each variant's registers are bounded for, as CTAs
// (4M orchard: 20 warps of whole tiles 0.94 ms, with 24 bytes spilled, 24 0.99 ms
// with more, 16 1.23 ms; 32-pixel tiles spill up to 28 bytes with one or two).
constexpr int fwd_blocks(int warps, int q, bool var) {
    return (var ? (q == 4 ? 16 : 20) : (q == 4 ? 20 : q == 2 ? 28 : 40)) / warps;
}

constexpr int bwd_blocks(int warps) { return 16 / warps; }  // 128 registers a thread

// One step of the weighted Welford update (the VAR variants), for one pixel and
// for a packed pair; both round alike.  The first fragment (W == 0: every
// weight is positive) sets zc.  The pair takes its weights and depths negated
// (as the forward stages them) and keeps zc negated; a pixel with weight 0
// keeps its values (before its first fragment zc changes, m and M2 stay 0).
__device__ __forceinline__ void welford(float w, float z, float &W, float &zc, float &m, float &M2) {
    if (W == 0.f) zc = z;
    W = __fadd_rn(W, w);
    const float y = z - zc;
    const float d = y - m;
    m = __fmaf_rn(d, __fmul_rn(w, rcp_approx(fmaxf(W, 1e-30f))), m);
    M2 = __fmaf_rn(__fmul_rn(w, d), y - m, M2);
}
__device__ __forceinline__ void welford2(f2 nw, f2 nz, f2 &W, f2 &nzc, f2 &m, f2 &M2) {
    float w0, w1, c0, c1;
    f2_unpack(W, w0, w1);
    f2_unpack(nzc, c0, c1);
    const float z = f2_lo(nz);
    nzc = f2_pack(w0 == 0.f ? z : c0, w1 == 0.f ? z : c1);
    W = f2_sub(W, nw);
    f2_unpack(W, w0, w1);
    const f2 r = f2_pack(rcp_approx(fmaxf(w0, 1e-30f)), rcp_approx(fmaxf(w1, 1e-30f)));
    const f2 y = f2_sub(nzc, nz), nd = f2_sub(m, y);
    m = f2_fma(nd, f2_mul(nw, r), m);
    M2 = f2_fma(f2_mul(nw, nd), f2_sub(y, m), M2);
}

struct RasterArgs {
    const ViewInfo *views;
    int32_t n_views, n_tiles, depth;
    Consts c;
    const float4 *rec;
    const uint32_t *vals;
    const uint2 *ranges;
    const uint32_t *order;  // tiles in work order
    uint32_t *counter;
    uint32_t *last;
    float *tfin;
    // forward outputs
    float *rgb, *depth_out, *alpha_out;
    float *mean_out, *var_out;  // VAR variants: depth mean and variance per pixel
    float4 *vstat;              // VAR variants: (mean, var, 1/W, 0) per pixel, for the backward
    // backward inputs / outputs
    const float *dL_drgb, *dL_ddepth, *dL_dalpha;
    const float *dL_dmean, *dL_dvar;  // VAR variant
    float *g2d;
    uint8_t *state;  // pair states: touched pairs are marked
};

// A tile is divided into quadrants of 8x8 pixels, two a lane: lane l holds
// column l % 8 and rows l / 8 and l / 8 + 4 of each of its quadrants, packed
// in one f32x2 pair.  A warp holds Q quadrants (4: a 16x16 tile; 2: a 16x8
// half; 1), which share the row and the column terms of every exponent.
template <int TW, int TH, int Q>
struct Share {
    static constexpr int QX = Q >= 2 ? 2 : 1, QY = Q == 4 ? 2 : 1;
    static constexpr int NWX = TW / (8 * QX);            // warps across
    static constexpr int NW = NWX * (TH / (8 * QY));     // warps a tile
    static constexpr int NT = 32 * NW;
    static_assert(TW % (8 * QX) == 0 && TH % (8 * QY) == 0 && NW * Q <= 16, "whole warps a tile");
    // first pixel of warp w's share, relative to the tile
    __device__ static constexpr int wx(int w) { return (w % NWX) * 8 * QX; }
    __device__ static constexpr int wy(int w) { return (w / NWX) * 8 * QY; }
};

// The next tile in work order, or -1.  Every CTA draws one number past the
// tiles; the last of these puts the counter back for the next launch (a clearing
// launch before each pass cost 1-2 us).
__device__ __forceinline__ int next_tile(const RasterArgs &A) {
    const uint32_t w = atomicAdd(A.counter, 1u);
    if (w < (uint32_t)A.n_tiles) return (int)A.order[w];
    if (w == (uint32_t)A.n_tiles + gridDim.x - 1u) *A.counter = 0u;
    return -1;
}

// Which quadrants a staged Gaussian can reach, bit w * Q + q for quadrant q
// of warp w: the tile test of the binning on the quadrant's box of pixel
// centres, with fixed paddings (0.1 % and 0.01 px) that exceed the rounding of
// the exponents below, so an unset bit is a quadrant without a fragment to
// keep.  kExactPath marks an entry whose fragments must take every branch:
// one whose alpha may need the clamp at alpha_max, or with a value that is
// not finite (0 x inf would leak into pixels that it does not reach).
constexpr uint32_t kExactPath = 0x80000000u;
template <int TW, int TH, int Q>
__device__ __forceinline__ uint32_t quad_mask(const float4 r0, const float4 r1, const float4 r2, int x0, int y0,
                                              const Consts &k) {
    using S = Share<TW, TH, Q>;
    float f = r0.x * 0.f + r0.y * 0.f + r0.z * 0.f + r0.w * 0.f;
    f += r1.x * 0.f + r1.y * 0.f + r1.z * 0.f + r1.w * 0.f;
    f += r2.x * 0.f + r2.y * 0.f + r2.z * 0.f + r2.w * 0.f;
    if (!(f == 0.f)) return ~0u;
    const float4 t = reach_terms(r1, k.log2_alpha_min, 1.f + kQuadRelPad);
    uint32_t m = r1.w < k.log2_alpha_noclamp ? 0u : kExactPath;
#pragma unroll
    for (int w = 0; w < S::NW; ++w)
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int x = x0 + S::wx(w) + 8 * (q % S::QX), y = y0 + S::wy(w) + 8 * (q / S::QX);
            if (tile_reached(r0, r1, t, x, x + 7, y, y + 7, kQuadAbsPad)) m |= 1u << (w * Q + q);
        }
    return m;
}

// One staged list entry of the forward: what the packed arithmetic multiplies
// a pair of pixels by is stored twice, side by side, so that one 16-byte
// shared load gives two packed operands (broadcasting a register into a pair
// costs an instruction for every operand).
struct FwdEntry {
    float4 u;    // U, l11, k1
    float4 row;  // V, V, k2, k2
    float4 l;    // l12, l12, l22, l22
    float4 or_;  // -log2 o twice, -r twice
    float4 gb;   // -g twice, -b twice
    float4 z;    // -z twice
};
struct F2x2 {
    f2 a, b;
};
__device__ __forceinline__ F2x2 load_f2x2(const float4 &v) {
    const ulonglong2 x = *reinterpret_cast<const ulonglong2 *>(&v);
    return {{x.x}, {x.y}};
}

// One CTA works a tile at a time (persistent, tiles taken in the work order).
// Each warp walks, of every 32 staged entries, those that reach one of its
// quadrants that still has a live pixel (one ballot a quadrant), and of such an
// entry only the quadrants it reaches: of the pixel slots of a 16x16 tile's
// walk 45 % blend, of those worked here 60 %.  A pixel stops at the first
// fragment that would take its transmittance below t_min (its threshold thr
// then admits nothing), the warp when all of its pixels have, the CTA when all
// warps have.
//
// Within a quadrant the two pixels of a lane are worked without branches: a
// pixel that the fragment does not reach takes alpha = 0, for which T - T
// alpha and C + T alpha c are exactly T and C.  alpha is carried negated, as
// packed instructions cannot negate, and so is the staged colour.  Decisions
// and sums round exactly as e = log2 o - t1^2 - t2^2, alpha = min(alpha_max,
// 2^e), T' = fma(-T, alpha, T), C' = fma(T alpha, c, C) taken one by one.
// (Against two warps a tile, four pixels a thread with a branch each: 4M
// orchard, six 1920x1200 views, 1151 -> 936 us; three 1280x720 views of 500k
// 194 -> 172; 161x119, 3k 52 -> 28.)
template <int TW, int TH, int Q, bool VAR>
__global__ void __launch_bounds__(Share<TW, TH, Q>::NT, fwd_blocks(Share<TW, TH, Q>::NW, Q, VAR))
    k_raster_fwd(RasterArgs A) {
    using S = Share<TW, TH, Q>;
    constexpr int QX = S::QX, QY = S::QY, NW = S::NW, NT = S::NT;
    extern __shared__ float4 smem[];
    FwdEntry *sE = reinterpret_cast<FwdEntry *>(smem);
    uint32_t *sM = reinterpret_cast<uint32_t *>(sE + A.depth);
    __shared__ int s_tile;
    const int tid = threadIdx.x, lane = tid & 31, wid = NW > 1 ? tid >> 5 : 0;
    const float amax = A.c.alpha_max, tmin = A.c.t_min, l2amin = A.c.log2_alpha_min;
    for (;;) {
        __syncthreads();
        if (tid == 0) {
            s_tile = next_tile(A);
        }
        __syncthreads();
        const int tile = s_tile;
        if (tile < 0) break;
        const int v = view_of_tile(A.views, A.n_views, tile);
        const ViewInfo vi = A.views[v];
        const int lt = tile - vi.tile_off;
        const int tx0 = (lt % vi.ntx) * TW, ty0 = (lt / vi.ntx) * TH;
        const int px0 = tx0 + S::wx(wid) + (lane & 7), py0 = ty0 + S::wy(wid) + (lane >> 3);
        const uint2 rg = A.ranges[tile];
        f2 T[Q], Cr[Q], Cg[Q], Cb[Q], D[Q];
        float thr[Q][2];  // -log2 alpha_min while the pixel lives, then -inf
        uint32_t cnt[Q][2];
        f2 Wsum[Q], nzc[Q], mr[Q], M2[Q];  // nzc = -zc
        uint32_t live = 0;  // bit q: quadrant q has a live pixel
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            T[q] = f2_bcast(1.f);
            Cr[q] = Cg[q] = Cb[q] = D[q] = f2_bcast(0.f);
            Wsum[q] = nzc[q] = mr[q] = M2[q] = f2_bcast(0.f);
            const int px = px0 + 8 * (q % QX), py = py0 + 8 * (q / QX);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                cnt[q][h] = 0;
                thr[q][h] = px < vi.W && py + 4 * h < vi.H ? -l2amin : -INFINITY;
            }
            if (__any_sync(0xffffffffu, fmaxf(thr[q][0], thr[q][1]) > -INFINITY)) live |= 1u << q;
        }
        // entries worked since the quadrants were last looked at: counted across
        // batches, so that a warp which few entries of each reach leaves too
        int since = 0;
        for (uint32_t b0 = rg.x; b0 < rg.y; b0 += A.depth) {
            if (__syncthreads_and(live == 0)) break;
            const int nb = min((int)(rg.y - b0), A.depth);
            for (int j = tid; j < nb; j += NT) {
                const uint32_t pair = A.vals[b0 + j];
                const float4 r0 = A.rec[3 * (size_t)pair], r1 = A.rec[3 * (size_t)pair + 1];
                const float4 r2 = A.rec[3 * (size_t)pair + 2];
                float4 a, b;
                stage_record(r0, r1, a, b);
                sE[j].u = make_float4(a.x, b.x, a.z, 0.f);
                sE[j].row = make_float4(a.y, a.y, a.w, a.w);
                sE[j].l = make_float4(b.y, b.y, b.z, b.z);
                sE[j].or_ = make_float4(-b.w, -b.w, -r2.x, -r2.x);
                sE[j].gb = make_float4(-r2.y, -r2.y, -r2.z, -r2.z);
                sE[j].z = make_float4(-r2.w, -r2.w, 0.f, 0.f);
                sM[j] = quad_mask<TW, TH, Q>(r0, r1, r2, tx0, ty0, A.c);
            }
            __syncthreads();
            for (int jb = 0; jb < nb && live; jb += 32) {
                const uint32_t mine = jb + lane < nb ? sM[jb + lane] : 0u;
                uint32_t E[Q], todo = 0, all = ~0u;
                const uint32_t exact = __ballot_sync(0xffffffffu, mine & kExactPath);
#pragma unroll
                for (int q = 0; q < Q; ++q) {
                    E[q] = __ballot_sync(0xffffffffu, (mine >> (wid * Q + q)) & 1u);
                    if (!(live >> q & 1u)) E[q] = 0;
                    todo |= E[q];
                    all &= E[q];
                }
                while (todo) {
                    const int j = __ffs(todo) - 1;
                    todo &= todo - 1;
                    const FwdEntry &e = sE[jb + j];
                    const uint32_t j1 = b0 + jb + j - rg.x + 1;
                    const float4 u = e.u;
                    const F2x2 row = load_f2x2(e.row), l = load_f2x2(e.l), o = load_f2x2(e.or_);
                    f2 U1[QX], DY[QY], IN[QY];
#pragma unroll
                    for (int x = 0; x < QX; ++x)
                        U1[x] = f2_bcast(__fmaf_rn(u.y, __fsub_rn((float)(px0 + 8 * x), u.x), u.z));
#pragma unroll
                    for (int y = 0; y < QY; ++y) {
                        DY[y] = f2_sub(f2_pack((float)(py0 + 8 * y), (float)(py0 + 8 * y + 4)), row.a);
                        const f2 t2 = f2_fma(l.b, DY[y], row.b);
                        IN[y] = f2_fma(t2, t2, o.a);
                    }
                    if (!(exact >> j & 1u)) {
                        const F2x2 gb = load_f2x2(e.gb), z = load_f2x2(e.z);
                        float al[Q][2], tn[Q][2];  // -alpha, the transmittance after
                        bool in[Q][2];
                        auto decide = [&](int q) {
                            const f2 t1 = f2_fma(l.a, DY[q / QX], U1[q % QX]);
                            float n[2];  // -e
                            f2_unpack(f2_fma(t1, t1, IN[q / QX]), n[0], n[1]);
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                in[q][h] = n[h] <= thr[q][h];
                                al[q][h] = in[q][h] ? -ex2_approx(-n[h]) : 0.f;
                            }
                            f2_unpack(f2_fma(T[q], f2_pack(al[q][0], al[q][1]), T[q]), tn[q][0], tn[q][1]);
                        };
                        auto stop = [&](int q) {
#pragma unroll
                            for (int h = 0; h < 2; ++h)
                                if (tn[q][h] < tmin) {
                                    thr[q][h] = -INFINITY;
                                    al[q][h] = 0.f;
                                    in[q][h] = false;
                                }
                        };
                        auto blend = [&](int q) {
                            const f2 nal = f2_pack(al[q][0], al[q][1]);
                            const f2 nw = f2_mul(nal, T[q]);
                            T[q] = f2_fma(T[q], nal, T[q]);
                            Cr[q] = f2_fma(nw, o.b, Cr[q]);
                            Cg[q] = f2_fma(nw, gb.a, Cg[q]);
                            Cb[q] = f2_fma(nw, gb.b, Cb[q]);
                            D[q] = f2_fma(nw, z.a, D[q]);
                            if (VAR) welford2(nw, z.a, Wsum[q], nzc[q], mr[q], M2[q]);
#pragma unroll
                            for (int h = 0; h < 2; ++h)
                                if (in[q][h]) cnt[q][h] = j1;
                        };
                        if (Q > 1 && (all >> j & 1u)) {
                            // every quadrant, interleaved and with one test for
                            // pixels that end (972 -> 936 us, 4M orchard)
                            float low = 1.f;
#pragma unroll
                            for (int q = 0; q < Q; ++q) {
                                decide(q);
                                low = fminf(low, fminf(tn[q][0], tn[q][1]));
                            }
                            if (low < tmin) {
#pragma unroll
                                for (int q = 0; q < Q; ++q) stop(q);
                            }
#pragma unroll
                            for (int q = 0; q < Q; ++q) blend(q);
                        } else {
#pragma unroll
                            for (int q = 0; q < Q; ++q)
                                if (E[q] >> j & 1u) {
                                    decide(q);
                                    if (fminf(tn[q][0], tn[q][1]) < tmin) stop(q);
                                    blend(q);
                                }
                        }
                    } else {
                        const float cx = e.or_.z, cy = e.gb.x, cz = e.gb.z, cw = e.z.x;
#pragma unroll
                        for (int q = 0; q < Q; ++q) {
                            if (!(E[q] >> j & 1u)) continue;
                            const f2 t1 = f2_fma(l.a, DY[q / QX], U1[q % QX]);
                            float n[2];
                            f2_unpack(f2_fma(t1, t1, IN[q / QX]), n[0], n[1]);
                            float t[2], cr[2], cg[2], cb[2], d[2];
                            f2_unpack(T[q], t[0], t[1]);
                            f2_unpack(Cr[q], cr[0], cr[1]);
                            f2_unpack(Cg[q], cg[0], cg[1]);
                            f2_unpack(Cb[q], cb[0], cb[1]);
                            f2_unpack(D[q], d[0], d[1]);
                            float W[2], zc[2], m[2], v[2];
                            f2_unpack(Wsum[q], W[0], W[1]);
                            f2_unpack(nzc[q], zc[0], zc[1]);
                            f2_unpack(mr[q], m[0], m[1]);
                            f2_unpack(M2[q], v[0], v[1]);
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                // (an exponent that is not a number is not below the threshold)
                                if (!(thr[q][h] > -INFINITY) || -n[h] < l2amin) continue;
                                const float alpha = fminf(amax, ex2_approx(-n[h]));
                                const float tn = __fmaf_rn(-t[h], alpha, t[h]);
                                if (tn < tmin) {
                                    thr[q][h] = -INFINITY;
                                    continue;
                                }
                                const float w = __fmul_rn(alpha, t[h]);
                                cr[h] = __fmaf_rn(w, -cx, cr[h]);
                                cg[h] = __fmaf_rn(w, -cy, cg[h]);
                                cb[h] = __fmaf_rn(w, -cz, cb[h]);
                                d[h] = __fmaf_rn(w, -cw, d[h]);
                                if (VAR) {
                                    zc[h] = -zc[h];
                                    welford(w, -cw, W[h], zc[h], m[h], v[h]);
                                    zc[h] = -zc[h];
                                }
                                t[h] = tn;
                                cnt[q][h] = j1;
                            }
                            T[q] = f2_pack(t[0], t[1]);
                            Cr[q] = f2_pack(cr[0], cr[1]);
                            Cg[q] = f2_pack(cg[0], cg[1]);
                            Cb[q] = f2_pack(cb[0], cb[1]);
                            D[q] = f2_pack(d[0], d[1]);
                            Wsum[q] = f2_pack(W[0], W[1]);
                            nzc[q] = f2_pack(zc[0], zc[1]);
                            mr[q] = f2_pack(m[0], m[1]);
                            M2[q] = f2_pack(v[0], v[1]);
                        }
                    }
                    // every eight entries, quadrants whose pixels have all ended leave the walk
                    if (++since == 8) {
                        since = 0;
                        uint32_t left = 0;
#pragma unroll
                        for (int q = 0; q < Q; ++q) {
                            if (!__any_sync(0xffffffffu, fmaxf(thr[q][0], thr[q][1]) > -INFINITY)) {
                                E[q] = 0;
                                live &= ~(1u << q);
                            }
                            left |= E[q];
                            all &= E[q];
                        }
                        todo &= left;
                    }
                }
            }
        }
        const int64_t hw = (int64_t)vi.W * vi.H;
        float *rgb = A.rgb + 3 * (int64_t)vi.pix_off;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int px = px0 + 8 * (q % QX);
            float t[2], cr[2], cg[2], cb[2], d[2];
            f2_unpack(T[q], t[0], t[1]);
            f2_unpack(Cr[q], cr[0], cr[1]);
            f2_unpack(Cg[q], cg[0], cg[1]);
            f2_unpack(Cb[q], cb[0], cb[1]);
            f2_unpack(D[q], d[0], d[1]);
            float W[2], zc[2], m[2], v[2];
            f2_unpack(Wsum[q], W[0], W[1]);
            f2_unpack(nzc[q], zc[0], zc[1]);
            f2_unpack(mr[q], m[0], m[1]);
            f2_unpack(M2[q], v[0], v[1]);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int py = py0 + 8 * (q / QX) + 4 * h;
                if (px >= vi.W || py >= vi.H) continue;
                const int64_t pl = (int64_t)py * vi.W + px;
                const int64_t pix = vi.pix_off + pl;
                rgb[pl] = cr[h];
                rgb[hw + pl] = cg[h];
                rgb[2 * hw + pl] = cb[h];
                A.depth_out[pix] = d[h];
                // 1 - T loses the relative precision of a small alpha (T near 1);
                // the variance variant has the direct sum of the weights at hand,
                // which keeps it, as the normalised depth D / alpha needs
                A.alpha_out[pix] = VAR ? W[h] : 1.f - t[h];
                A.last[pix] = cnt[q][h];
                A.tfin[pix] = t[h];
                if (VAR) {
                    // (zc stands negated; 0 where nothing blended)
                    const float mean = W[h] > 0.f ? m[h] - zc[h] : 0.f;
                    const float iw = W[h] > 0.f ? 1.f / W[h] : 0.f;
                    const float var = v[h] * iw;
                    A.mean_out[pix] = mean;
                    A.var_out[pix] = var;
                    A.vstat[pix] = make_float4(mean, var, iw, 0.f);
                }
            }
        }
    }
}

// The forward of an 8x8 tile, which is one quadrant: its list holds what
// reaches it already, so there is nothing to skip, and two pixels a lane
// with a branch each are cheaper than the packed pairs of k_raster_fwd (three
// 1280x720 views of a 500k orchard: 0.169 ms here, 0.217 there; with the
// variance 0.266 and 0.332).  A thread holds PF vertically adjacent pixels of one column, which share the
// shared-memory reads and the column part of every fragment's exponent.  A
// pixel stops at the first fragment that would take its transmittance below
// t_min, the thread when all of its pixels have, the CTA when all threads have.
// The VAR variant holds four more values a pixel: at least 640 resident
// threads an SM keeps it at 96 registers without spills (0: no minimum).
template <int TW, int TH, int PF, bool VAR>
__global__ void __launch_bounds__(TW * TH / PF, VAR ? 640 / (TW * TH / PF) : 0) k_raster_fwd_columns(RasterArgs A) {
    constexpr int NT = TW * TH / PF;
    static_assert(NT % 32 == 0, "the forward needs whole warps");
    extern __shared__ float4 smem[];
    float4 *sA = smem, *sB = smem + A.depth, *sC = smem + 2 * A.depth;
    __shared__ int s_tile;
    const int tid = threadIdx.x;
    const float amax = A.c.alpha_max, tmin = A.c.t_min, l2amin = A.c.log2_alpha_min;
    for (;;) {
        __syncthreads();
        if (tid == 0) {
            s_tile = next_tile(A);
        }
        __syncthreads();
        const int tile = s_tile;
        if (tile < 0) break;
        const int v = view_of_tile(A.views, A.n_views, tile);
        const ViewInfo vi = A.views[v];
        const int lt = tile - vi.tile_off;
        const int px = (lt % vi.ntx) * TW + tid % TW;
        const int py0 = (lt / vi.ntx) * TH + (tid / TW) * PF;
        const float pxf = (float)px;
        const uint2 rg = A.ranges[tile];
        float T[PF], Cr[PF], Cg[PF], Cb[PF], D[PF];
        float Wsum[PF], zc[PF], mr[PF], M2[PF];
        uint32_t cnt[PF];
        bool live[PF];
        int nlive = 0;
#pragma unroll
        for (int i = 0; i < PF; ++i) {
            T[i] = 1.f;
            Cr[i] = Cg[i] = Cb[i] = D[i] = 0.f;
            Wsum[i] = zc[i] = mr[i] = M2[i] = 0.f;
            cnt[i] = 0;
            live[i] = px < vi.W && py0 + i < vi.H;
            nlive += live[i];
        }
        for (uint32_t b0 = rg.x; b0 < rg.y; b0 += A.depth) {
            if (__syncthreads_and(nlive == 0)) break;
            const int nb = min((int)(rg.y - b0), A.depth);
            for (int j = tid; j < nb; j += NT) {
                uint32_t pair = A.vals[b0 + j];
                float4 r0 = A.rec[3 * (size_t)pair], r1 = A.rec[3 * (size_t)pair + 1];
                float4 a, bb;
                stage_record(r0, r1, a, bb);
                sA[j] = a;
                sB[j] = bb;
                sC[j] = A.rec[3 * (size_t)pair + 2];
            }
            __syncthreads();
            for (int j = 0; j < nb && nlive > 0; ++j) {
                const float4 a = sA[j], b = sB[j];
                float dxi, u1;
                frag_column(a, b, pxf, dxi, u1);
#pragma unroll
                for (int i = 0; i < PF; ++i) {
                    float t1, t2, dyi;
                    const float e = frag_pixel(a, b, u1, (float)(py0 + i), t1, t2, dyi);
                    if (!live[i] || e < l2amin) continue;
                    const float al = fminf(amax, ex2_approx(e));
                    const float Tn = __fmaf_rn(-T[i], al, T[i]);
                    if (Tn < tmin) {
                        live[i] = false;
                        --nlive;
                        continue;
                    }
                    const float wgt = __fmul_rn(al, T[i]);
                    const float4 c = sC[j];
                    Cr[i] = __fmaf_rn(wgt, c.x, Cr[i]);
                    Cg[i] = __fmaf_rn(wgt, c.y, Cg[i]);
                    Cb[i] = __fmaf_rn(wgt, c.z, Cb[i]);
                    D[i] = __fmaf_rn(wgt, c.w, D[i]);
                    if (VAR) welford(wgt, c.w, Wsum[i], zc[i], mr[i], M2[i]);
                    T[i] = Tn;
                    cnt[i] = b0 + j - rg.x + 1;
                }
            }
        }
#pragma unroll
        for (int i = 0; i < PF; ++i) {
            const int py = py0 + i;
            if (px >= vi.W || py >= vi.H) continue;
            const int64_t pl = (int64_t)py * vi.W + px;
            const int64_t pix = vi.pix_off + pl;
            const int64_t hw = (int64_t)vi.W * vi.H;
            float *rgb = A.rgb + 3 * (int64_t)vi.pix_off;
            rgb[pl] = Cr[i];
            rgb[hw + pl] = Cg[i];
            rgb[2 * hw + pl] = Cb[i];
            A.depth_out[pix] = D[i];
            // 1 - T loses the relative precision of a small alpha (T near 1);
            // the variance variant has the direct sum of the weights at hand,
            // which keeps it, as the normalised depth D / alpha needs
            A.alpha_out[pix] = VAR ? Wsum[i] : 1.f - T[i];
            A.last[pix] = cnt[i];
            A.tfin[pix] = T[i];
            if (VAR) {
                const float mean = zc[i] + mr[i];
                const float iw = Wsum[i] > 0.f ? 1.f / Wsum[i] : 0.f;
                const float var = M2[i] * iw;
                A.mean_out[pix] = mean;
                A.var_out[pix] = var;
                A.vstat[pix] = make_float4(mean, var, iw, 0.f);
            }
        }
    }
}

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// One staged list entry of the backward in pairs (see FwdEntry).
struct BwdEntry {
    float4 u;    // U, l11, k1, hx
    float4 row;  // V, V, k2, k2
    float4 l;    // l12, l12, l22, l22
    float4 or_;  // -log2 o twice, r twice
    float4 gb;   // g twice, b twice
    float4 z;    // z twice, hy, pair (bits)
};

// Warp sums of the ten image-space components go through shared memory: each
// lane stores its ten values of an entry as one row of kSumRow floats, and
// once kSumSlots entries are pending the warp sums them together, a lane adding
// one 16-byte column over half of the rows.  (Against a butterfly of
// shuffles an entry at a time, 12 shuffles and some 35 selects and adds, an
// entry takes 3 shared stores, 4 loads and 8 packed adds.)  The row stride of
// 12 floats and the rotated row order below keep stores and loads free of
// bank conflicts.
constexpr int kSumSlots = 4, kSumRow = 12;
constexpr int kSumBytes = kSumSlots * 32 * kSumRow * (int)sizeof(float);

__device__ __forceinline__ void red_add2(float *p, float a, float b) {
    asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(a), "f"(b) : "memory");
}

// Component pair c of an entry's raw sums (u, v), (qa, qb), (qc, ln o), (r, g) or
// (b, z) turned into gradients and added to its pair's row.  The raw sums are
// negated (dpw and the weights are carried negated); dL/dQ = -1/2 sum gpw d
// d^T; dpw/du = (Q d)_x = l11 t1 / s^2, dpw/dv = (l12 t1 + l22 t2) / s^2 with 1/s^2
// = 2 ln 2.
__device__ __forceinline__ void add_gradients(const BwdEntry &e, int c, float x, float y, float *g2d, uint8_t *state) {
    const uint32_t pair = __float_as_uint(e.z.w);
    if (c == 0) {
        state[pair] = kPairTouched;
        y = -kTwoLn2 * __fmaf_rn(e.l.x, x, e.l.z * y);
        x = -kTwoLn2 * (e.u.y * x);
    } else {
        x *= c <= 2 ? 0.5f : -1.f;
        y = c == 1 ? y : -y;
    }
    red_add2(g2d + (size_t)pair * kGrad + 2 * c, x, y);
}

// Sums the n pending entries' rows; byte k of `which` is the staged index of
// slot k.  Where one warp works the tile they go to the pairs' gradient rows;
// else to the warp's part of tile_sums, from which the CTA adds them once a
// batch (one atomic a tile and component instead of one a warp, in a fixed
// order inside the tile).
template <bool ONE_WARP>
__device__ __forceinline__ void flush_sums(const float *sum, const BwdEntry *sE, int n, uint32_t which, int lane,
                                           float *tile_sums, float *g2d, uint8_t *state) {
    __syncwarp();
    // lane = 8 f + 2 slot + half: column f (components 4f .. 4f + 3) of a slot's rows 16 half .. 16 half + 15
    const int f = lane >> 3, turn = lane & 7, slot = turn >> 1, half = lane & 1;
    const bool active = f < 3 && slot < n;
    f2 v[4][2];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k][0] = v[k][1] = f2_bcast(0.f);
    if (active) {
        const float *col = sum + (slot * 32 + 16 * half) * kSumRow + 4 * f;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const F2x2 x = load_f2x2(*reinterpret_cast<const float4 *>(col + ((i + turn) & 15) * kSumRow));
            v[i & 3][0] = i < 4 ? x.a : f2_add(v[i & 3][0], x.a);
            v[i & 3][1] = i < 4 ? x.b : f2_add(v[i & 3][1], x.b);
        }
    }
    float4 t;
    f2_unpack(f2_add(f2_add(v[0][0], v[1][0]), f2_add(v[2][0], v[3][0])), t.x, t.y);
    f2_unpack(f2_add(f2_add(v[0][1], v[1][1]), f2_add(v[2][1], v[3][1])), t.z, t.w);
    t.x += __shfl_xor_sync(0xffffffffu, t.x, 1);
    t.y += __shfl_xor_sync(0xffffffffu, t.y, 1);
    t.z += __shfl_xor_sync(0xffffffffu, t.z, 1);
    t.w += __shfl_xor_sync(0xffffffffu, t.w, 1);
    if (active && 2 * f + half < kGrad / 2) {
        const int j = which >> (8 * slot) & 255u, c = 2 * f + half;
        const float x = half ? t.z : t.x, y = half ? t.w : t.y;
        if (ONE_WARP) add_gradients(sE[j], c, x, y, g2d, state);
        else *reinterpret_cast<float2 *>(tile_sums + j * kGrad + 2 * c) = make_float2(x, y);
    }
    __syncwarp();
}

// The backward with few tiles (below kColumnTiles): one quadrant a warp, back to
// front over the tile's list with the forward's masks.  A warp's walk is then
// a chain that little else on the SM hides.  Two entries are worked together
// (only T and the suffix sum go from one to the next), and the next batch's
// records are copied in while this one is worked, their pair ids read a batch
// earlier still.  A pixel that a fragment does not reach takes alpha = 0 and runs
// the same instructions, which are then exactly the identity (T * 1, acc + 0 * h,
// sums + 0; the reciprocal approximation returns 1 for 1 on sm_103, measured).
// The alpha decision is taken on -e = fma(t1, t1, fma(t2, t2, -log2 o)), which is
// exactly the negation of e = fma(-t1, t1, fma(-t2, t2, log2 o)) (round to nearest
// is symmetric), so both passes take the same decisions bit for bit.  Measured
// against one entry at a time with loads at the head of a batch of 64: 300 tiles
// of 16x16 (box of 10k) 83 -> 55 us; 3600 (orchard of 300k, variance) 129 -> 116; 8x8
// tiles: 4270 with long lists (orchard of 1.3M, 481x280) 517 -> 394.
template <int TW, int TH, bool VAR>
__global__ void __launch_bounds__(Share<TW, TH, 1>::NT, bwd_blocks(Share<TW, TH, 1>::NW))
    k_raster_bwd_pairs(RasterArgs A) {
    using S = Share<TW, TH, 1>;
    constexpr int NW = S::NW, NT = S::NT;
    constexpr int PT = (kPairsDepth + NT - 1) / NT;  // staged entries a thread
    extern __shared__ float4 smem[];
    BwdEntry *sE = reinterpret_cast<BwdEntry *>(smem);
    float4 *sR = reinterpret_cast<float4 *>(sE + A.depth);  // records copied ahead
    uint32_t *sM = reinterpret_cast<uint32_t *>(sR + 3 * A.depth);
    const int tid = threadIdx.x, lane = tid & 31, wid = NW > 1 ? tid >> 5 : 0;
    float *sums = reinterpret_cast<float *>(sM + A.depth) + wid * (kSumBytes / 4);
    float *all_sums = reinterpret_cast<float *>(sM + A.depth) + NW * (kSumBytes / 4);
    float *tile_sums = all_sums + wid * A.depth * kGrad;
    __shared__ uint32_t s_worked[NW][kPairsDepth / 32];
    __shared__ int s_tile;
    __shared__ uint32_t s_max[NW];
    const float amax = A.c.alpha_max, nl2amin = -A.c.log2_alpha_min;
    const f2 ONE = f2_bcast(1.f), ZERO = f2_bcast(0.f);
    for (;;) {
        __syncthreads();
        if (tid == 0) s_tile = next_tile(A);
        __syncthreads();
        const int tile = s_tile;
        if (tile < 0) break;
        const int v = view_of_tile(A.views, A.n_views, tile);
        const ViewInfo vi = A.views[v];
        const int lt = tile - vi.tile_off;
        const int tx0 = (lt % vi.ntx) * TW, ty0 = (lt / vi.ntx) * TH;
        const int px = tx0 + S::wx(wid) + (lane & 7), py0 = ty0 + S::wy(wid) + (lane >> 3);
        const uint2 rg = A.ranges[tile];
        const int64_t hw = (int64_t)vi.W * vi.H;
        const float *grgb = A.dL_drgb + 3 * (int64_t)vi.pix_off;
        uint32_t cnt[2];
        float t_[2], r_[2], g_[2], b_[2], d_[2], a_[2], z_[2], ma_[2], mb_[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int py = py0 + 4 * h;
            cnt[h] = 0;
            t_[h] = 1.f;
            r_[h] = g_[h] = b_[h] = d_[h] = a_[h] = z_[h] = ma_[h] = mb_[h] = 0.f;
            if (px < vi.W && py < vi.H) {
                const int64_t pl = (int64_t)py * vi.W + px;
                const int64_t pix = vi.pix_off + pl;
                cnt[h] = A.last[pix];
                t_[h] = A.tfin[pix];
                r_[h] = grgb[pl];
                g_[h] = grgb[hw + pl];
                b_[h] = grgb[2 * hw + pl];
                d_[h] = A.dL_ddepth ? A.dL_ddepth[pix] : 0.f;
                a_[h] = A.dL_dalpha ? A.dL_dalpha[pix] : 0.f;
                if (VAR) {
                    const float4 vs = A.vstat[pix];
                    z_[h] = vs.x;
                    ma_[h] = A.dL_dmean ? A.dL_dmean[pix] * vs.z : 0.f;
                    mb_[h] = A.dL_dvar ? A.dL_dvar[pix] * vs.z : 0.f;
                    a_[h] = __fmaf_rn(-mb_[h], vs.y, a_[h]);  // the -b var part of every h
                }
            }
        }
        const uint32_t wmax = __reduce_max_sync(0xffffffffu, max(cnt[0], cnt[1]));
        f2 T = f2_pack(t_[0], t_[1]), nacc = ZERO;  // nacc = -acc
        const f2 gR = f2_pack(r_[0], r_[1]), gG = f2_pack(g_[0], g_[1]), gB = f2_pack(b_[0], b_[1]);
        const f2 gD = f2_pack(d_[0], d_[1]), gA = f2_pack(a_[0], a_[1]);
        const f2 zmu = f2_pack(z_[0], z_[1]), ga = f2_pack(ma_[0], ma_[1]), gb = f2_pack(mb_[0], mb_[1]);
        uint32_t maxcnt = wmax;
        if constexpr (NW > 1) {
            if (lane == 0) s_max[wid] = wmax;
            __syncthreads();
#pragma unroll
            for (int w = 0; w < NW; ++w) maxcnt = max(maxcnt, s_max[w]);
        }
        struct Work {
            int j, count;
            float4 u, ez;
            F2x2 row, l, o, gbc;
            float dxi, u1;
            f2 DY, IN;
            f2 sR, sG, sB, sZ;  // -wgt dL/dc
            f2 ng;              // -dL/dpw of each pixel
        };
        auto begin = [&](Work &w, const BwdEntry &e) {
            w.u = e.u;
            w.row = load_f2x2(e.row);
            w.l = load_f2x2(e.l);
            w.o = load_f2x2(e.or_);
            w.gbc = load_f2x2(e.gb);
            w.ez = e.z;
            w.dxi = __fsub_rn((float)px, w.u.x);
            w.u1 = __fmaf_rn(w.u.y, w.dxi, w.u.z);
            w.DY = f2_sub(f2_pack((float)py0, (float)(py0 + 4)), w.row.a);
            const f2 t2 = f2_fma(w.l.b, w.DY, w.row.b);
            w.IN = f2_fma(t2, t2, w.o.a);
        };
        auto work = [&](Work &w, uint32_t rel0) {
            const f2 CW = load_f2x2(w.ez).a;
            const f2 t1 = f2_fma(w.l.a, w.DY, f2_bcast(w.u1));
            float n[2], al[2], ag[2];  // -e, -alpha, the -alpha that has a gradient through pw
            f2_unpack(f2_fma(t1, t1, w.IN), n[0], n[1]);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const bool in = rel0 + w.j < cnt[h] && n[h] <= nl2amin && w.count;
                al[h] = in ? -ex2_approx(-n[h]) : 0.f;
                ag[h] = al[h] >= -amax ? al[h] : 0.f;
                al[h] = fmaxf(-amax, al[h]);
            }
            const f2 nal = f2_pack(al[0], al[1]);
            float om[2];
            f2_unpack(f2_add(ONE, nal), om[0], om[1]);
            const f2 r1m = f2_pack(rcp_approx(om[0]), rcp_approx(om[1]));  // 1 / (1 - alpha)
            T = f2_mul(T, r1m);  // transmittance before this fragment
            const f2 nwgt = f2_mul(nal, T);
            f2 hh = f2_fma(gR, w.o.b, f2_fma(gG, w.gbc.a, f2_fma(gB, w.gbc.b, f2_fma(gD, CW, gA))));
            f2 gz = gD;
            if (VAR) {
                const f2 dz = f2_sub(CW, zmu);
                const f2 t = f2_fma(gb, dz, ga);  // a + b dz
                hh = f2_fma(t, dz, hh);
                gz = f2_add(gz, f2_fma(gb, dz, t));  // a + 2 b dz
            }
            // dL/dalpha = T h - acc / (1 - alpha)
            const f2 dLda = f2_fma(T, hh, f2_mul(nacc, r1m));
            nacc = f2_fma(nwgt, hh, nacc);
            w.ng = f2_mul(dLda, f2_pack(ag[0], ag[1]));
            w.sR = f2_mul(nwgt, gR);
            w.sG = f2_mul(nwgt, gG);
            w.sB = f2_mul(nwgt, gB);
            w.sZ = f2_mul(nwgt, gz);
        };
        // Moments of the lane's two pixels about the middle of its rows, which lie
        // at -2 and 2 from there: with S_k = sum of row^k (-gpw), t1 and t2 affine in
        // the row, dy = dym + row.  (About the first row the terms are up to twice
        // as large and cancel.)
        auto finish = [&](const Work &w, float *mine_sum) {
            const float l12 = f2_lo(w.l.a), l22 = f2_lo(w.l.b);
            const float dyi = f2_lo(w.DY) + 2.f, dym = dyi + w.ez.z;
            const float t2_m = __fmaf_rn(l22, dyi, f2_lo(w.row.b)), t1_m = __fmaf_rn(l12, dyi, w.u1);
            const float dx = w.dxi + w.u.w;
            float a0, a1;
            f2_unpack(w.ng, a0, a1);
            const float S0 = a0 + a1, S1 = 2.f * (a1 - a0), S2 = 4.f * S0;
            // (u, v, qa, qb), (qc, ln o, r, g), (b, z)
            *reinterpret_cast<float4 *>(mine_sum) =
                make_float4(__fmaf_rn(l12, S1, t1_m * S0), __fmaf_rn(t2_m, S0, l22 * S1), dx * dx * S0,
                            dx * __fmaf_rn(dym, S0, S1));
            *reinterpret_cast<float4 *>(mine_sum + 4) =
                make_float4(__fmaf_rn(dym, __fmaf_rn(dym, S0, S1), __fmaf_rn(dym, S1, S2)), S0,
                            f2_lo(w.sR) + f2_hi(w.sR), f2_lo(w.sG) + f2_hi(w.sG));
            *reinterpret_cast<float2 *>(mine_sum + 8) =
                make_float2(f2_lo(w.sB) + f2_hi(w.sB), f2_lo(w.sZ) + f2_hi(w.sZ));
        };
        uint32_t id[PT], id1[PT];
        auto load_ids = [&](int64_t h, uint32_t (&to)[PT]) {  // of the batch that ends at h, if there is one
            const int64_t l = max((int64_t)rg.x, h - A.depth);
#pragma unroll
            for (int k = 0; k < PT; ++k)
                if (l + tid + k * NT < h && tid + k * NT < A.depth) to[k] = A.vals[l + tid + k * NT];
        };
        auto copy_records = [&](int64_t h, const uint32_t (&of)[PT]) {
            const int64_t l = max((int64_t)rg.x, h - A.depth);
#pragma unroll
            for (int k = 0; k < PT; ++k)
                if (l + tid + k * NT < h && tid + k * NT < A.depth) {
#pragma unroll
                    for (int c = 0; c < 3; ++c) cp_async16(sR + 3 * (tid + k * NT) + c, A.rec + 3 * (size_t)of[k] + c);
                }
            cp_async_commit();
        };
        const int64_t top = (int64_t)rg.x + maxcnt;
        load_ids(top, id);
        copy_records(top, id);
        load_ids(top - A.depth, id1);
        for (int64_t hi = top; hi > (int64_t)rg.x; hi -= A.depth) {
            const int64_t lo = max((int64_t)rg.x, hi - A.depth);
            const int nb = (int)(hi - lo);
            __syncthreads();
            cp_async_wait_all();
#pragma unroll
            for (int k = 0; k < PT; ++k) {
                const int j = tid + k * NT;
                if (j < nb) {
                    const float4 r0 = sR[3 * j], r1 = sR[3 * j + 1], r2 = sR[3 * j + 2];
                    float4 a, b;
                    stage_record(r0, r1, a, b);
                    sE[j].u = make_float4(a.x, b.x, a.z, r0.z);
                    sE[j].row = make_float4(a.y, a.y, a.w, a.w);
                    sE[j].l = make_float4(b.y, b.y, b.z, b.z);
                    sE[j].or_ = make_float4(-b.w, -b.w, r2.x, r2.x);
                    sE[j].gb = make_float4(r2.y, r2.y, r2.z, r2.z);
                    sE[j].z = make_float4(r2.w, r2.w, r0.w, __uint_as_float(id[k]));
                    sM[j] = quad_mask<TW, TH, 1>(r0, r1, r2, tx0, ty0, A.c);
                }
                id[k] = id1[k];
            }
            copy_records(hi - A.depth, id);  // (each slot has been read by its own thread)
            load_ids(hi - 2 * (int64_t)A.depth, id1);
            __syncthreads();
            uint32_t which = 0;
            int pending = 0;
            if (NW > 1 && lane < kPairsDepth / 32) s_worked[wid][lane] = 0u;
            __syncwarp();
            for (int jb = (nb - 1) & ~31; jb >= 0; jb -= 32) {
                const uint32_t rel0 = (uint32_t)(lo + jb - rg.x);
                if (rel0 >= wmax) continue;  // no pixel of this warp reached these entries
                const uint32_t mine = jb + lane < nb ? sM[jb + lane] : 0u;
                uint32_t todo = __ballot_sync(0xffffffffu, (mine >> wid & 1u) && rel0 + lane < wmax);
                if (NW > 1 && lane == 0) s_worked[wid][jb / 32] = todo;
                while (todo) {
                    Work w[2];
                    w[0].j = 31 - __clz(todo);
                    w[0].count = 1;
                    todo ^= 1u << w[0].j;
                    // (an odd last one is worked next to itself with alpha = 0)
                    w[1].count = todo != 0;
                    w[1].j = todo ? 31 - __clz(todo) : w[0].j;
                    if (todo) todo ^= 1u << w[1].j;
                    begin(w[0], sE[jb + w[0].j]);
                    begin(w[1], sE[jb + w[1].j]);
                    work(w[0], rel0);
                    work(w[1], rel0);
                    finish(w[0], sums + (pending * 32 + lane) * kSumRow);
                    finish(w[1], sums + ((pending + 1) * 32 + lane) * kSumRow);
                    which = which << 8 | (uint32_t)(jb + w[0].j);
                    if (w[1].count) which = which << 8 | (uint32_t)(jb + w[1].j);
                    pending += 1 + w[1].count;
                    if (pending > kSumSlots - 2) {
                        flush_sums<NW == 1>(sums, sE, pending, __byte_perm(which << 8 * (kSumSlots - pending), 0, 0x0123),
                                            lane, tile_sums, A.g2d, A.state);
                        pending = 0;
                    }
                }
            }
            // (the pending entries' staged records go with this batch)
            if (pending)
                flush_sums<NW == 1>(sums, sE, pending, __byte_perm(which << 8 * (kSumSlots - pending), 0, 0x0123), lane,
                                    tile_sums, A.g2d, A.state);
            if constexpr (NW > 1) {
                __syncthreads();
                for (int i = tid; i < nb * (kGrad / 2); i += NT) {
                    const int j = i / (kGrad / 2), c = i - j * (kGrad / 2);
                    float2 t = make_float2(0.f, 0.f);
                    bool any = false;
#pragma unroll
                    for (int w = 0; w < NW; ++w)
                        if (s_worked[w][j >> 5] >> (j & 31) & 1u) {
                            const float2 x =
                                *reinterpret_cast<const float2 *>(all_sums + (w * A.depth + j) * kGrad + 2 * c);
                            t.x += x.x;
                            t.y += x.y;
                            any = true;
                        }
                    if (any) add_gradients(sE[j], c, t.x, t.y, A.g2d, A.state);
                }
            }
        }
    }
}

// Sums ten per-lane values over the warp by recursive halving: at each of the
// five butterfly levels a lane keeps half of its remaining components and
// sends the other half to its partner, so 12 shuffles replace 50.  Afterwards
// lane l holds the warp total of component
//   comp(l) = 5*b4 + 3*b3 + 2*b2 + b1      (bK = bit K of l),
// valid when (b3 == 0 and not (b2 and b1)) or (b3 == 1 and b2 == 0); lanes l
// and l^1 hold the same total.  reduce10_component gives comp(l) or -1.
__device__ __forceinline__ float warp_reduce_scatter10(const float v[10], int lane) {
    const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4, b1 = lane & 2;
    float a[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        float send = b4 ? v[i] : v[i + 5];
        float keep = b4 ? v[i + 5] : v[i];
        a[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
    float c[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        float hiv = i + 3 < 5 ? a[i + 3] : 0.f;
        float send = b3 ? a[i] : hiv;
        float keep = b3 ? hiv : a[i];
        c[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
    float d[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        float hiv = i + 2 < 3 ? c[i + 2] : 0.f;
        float send = b2 ? c[i] : hiv;
        float keep = b2 ? hiv : c[i];
        d[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    }
    float send = b1 ? d[0] : d[1];
    float keep = b1 ? d[1] : d[0];
    float e = keep + __shfl_xor_sync(0xffffffffu, send, 2);
    return e + __shfl_xor_sync(0xffffffffu, e, 1);
}

__device__ __forceinline__ int reduce10_component(int lane) {
    const int b4 = (lane >> 4) & 1, b3 = (lane >> 3) & 1, b2 = (lane >> 2) & 1, b1 = (lane >> 1) & 1;
    const bool ok = b3 == 0 ? !(b2 && b1) : b2 == 0;
    return ok ? 5 * b4 + 3 * b3 + 2 * b2 + b1 : -1;
}

// The backward of renders of kColumnTiles and more: a thread works PPT pixels of
// a column, a warp's sums go to the rows by one butterfly an entry.  Quadrants
// and sums about their middle, added to rows in double, took 1559 us where this
// takes 1870 (4M orchard, six 1920x1200 views) and come nearer to 64 bits, but
// move results that must stay where they are: the gradients of a long thin
// Gaussian near a camera are sums over thousands of tiles that largely cancel, and
// in another order of the terms the quaternion gradients of that step changed by
// up to 1.6e-4 in norm (240 random maps; repeating the same order changes them by
// 1e-6, 3e-5 at most, and one map in eight passed 2e-5 in norm or 8e-4 at an
// element by more than that).  Below kColumnTiles a Gaussian covers fewer tiles,
// and some 360 gradients in the other order stayed inside.  The terms, their order
// inside a warp, and the float rows are therefore fixed.
//
// At least 512 resident threads per SM (16 warps, 128 registers a thread):
// with eight pixels a thread, measured best on the 500k orchard (16 one-warp
// blocks: 0.435 ms; 14: 0.441 ms).
//
// A thread's PPT pixels are worked in Q = PPT/2 packed pairs (pixel p in the
// low half, pixel p + Q in the high half), so that one f32x2 instruction does
// the arithmetic of two pixels.  The alpha decision is taken on
// -e = fma(t1, t1, fma(t2, t2, -log2 o)), which is exactly the negation of
// the forward's e = fma(-t1, t1, fma(-t2, t2, log2 o)) (round to nearest is
// symmetric), so both passes take the same decisions bit for bit.
template <int TW, int TH, int PPT, bool VAR>
__global__ void __launch_bounds__(TW * TH / PPT, 512 / (TW * TH / PPT)) k_raster_bwd(RasterArgs A) {
    constexpr int NT = TW * TH / PPT;
    static_assert(NT % 32 == 0, "the backward needs whole warps");
    static_assert(PPT % 2 == 0, "the backward works pixels in pairs");
    constexpr int NW = (NT + 31) / 32;
    constexpr int Q = PPT / 2;
    extern __shared__ float4 smem[];
    float4 *sA = smem, *sB = smem + A.depth, *sC = smem + 2 * A.depth;
    float2 *sH = reinterpret_cast<float2 *>(smem + 3 * A.depth);
    uint32_t *sP = reinterpret_cast<uint32_t *>(sH + A.depth);
    __shared__ int s_tile;
    __shared__ uint32_t s_max[NW];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const float amax = A.c.alpha_max, nl2amin = -A.c.log2_alpha_min;
    const f2 ONE = f2_bcast(1.f);
    // component this lane adds after the reduction (even lanes only), and the
    // factors c0 + c11 l11 + c22 l22 that turn its raw sum into the gradient
    // (the colour and depth sums come out negated, see below)
    const int my_comp = (lane & 1) ? -1 : reduce10_component(lane);
    const float sc0 = my_comp == G_QA || my_comp == G_QC ? -0.5f
                      : my_comp == G_QB                  ? -1.f
                      : my_comp == G_U || my_comp == G_V ? 0.f
                      : my_comp == G_LNO                 ? 1.f
                                                         : -1.f;
    const float sc11 = my_comp == G_U ? kTwoLn2 : 0.f;
    const float sc22 = my_comp == G_V ? kTwoLn2 : 0.f;
    for (;;) {
        __syncthreads();
        if (tid == 0) {
            s_tile = next_tile(A);
        }
        __syncthreads();
        const int tile = s_tile;
        if (tile < 0) break;
        const int v = view_of_tile(A.views, A.n_views, tile);
        const ViewInfo vi = A.views[v];
        const int lt = tile - vi.tile_off;
        const int px = (lt % vi.ntx) * TW + tid % TW;
        const int py0 = (lt / vi.ntx) * TH + (tid / TW) * PPT;
        const float pxf = (float)px;
        const f2 PY0 = f2_pack((float)py0, (float)(py0 + Q));
        const uint2 rg = A.ranges[tile];
        const int64_t hw = (int64_t)vi.W * vi.H;
        const float *grgb = A.dL_drgb + 3 * (int64_t)vi.pix_off;
        uint32_t cnt[PPT], mycnt = 0;
        f2 T[Q], gR[Q], gG[Q], gB[Q], gD[Q], gA[Q], nacc[Q];  // nacc = -acc
        f2 zmu[Q], ga[Q], gb[Q];
#pragma unroll
        for (int p = 0; p < Q; ++p) {
            float t_[2], r_[2], g_[2], b_[2], d_[2], a_[2], z_[2], ma_[2], mb_[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int i = p + h * Q, py = py0 + i;
                cnt[i] = 0;
                t_[h] = 1.f;
                r_[h] = g_[h] = b_[h] = d_[h] = a_[h] = z_[h] = ma_[h] = mb_[h] = 0.f;
                if (px < vi.W && py < vi.H) {
                    const int64_t pl = (int64_t)py * vi.W + px;
                    const int64_t pix = vi.pix_off + pl;
                    cnt[i] = A.last[pix];
                    t_[h] = A.tfin[pix];
                    r_[h] = grgb[pl];
                    g_[h] = grgb[hw + pl];
                    b_[h] = grgb[2 * hw + pl];
                    d_[h] = A.dL_ddepth ? A.dL_ddepth[pix] : 0.f;
                    a_[h] = A.dL_dalpha ? A.dL_dalpha[pix] : 0.f;
                    if (VAR) {
                        const float4 vs = A.vstat[pix];
                        z_[h] = vs.x;
                        ma_[h] = A.dL_dmean ? A.dL_dmean[pix] * vs.z : 0.f;
                        mb_[h] = A.dL_dvar ? A.dL_dvar[pix] * vs.z : 0.f;
                        a_[h] = __fmaf_rn(-mb_[h], vs.y, a_[h]);  // the -b var part of every h
                    }
                }
                mycnt = max(mycnt, cnt[i]);
            }
            T[p] = f2_pack(t_[0], t_[1]);
            gR[p] = f2_pack(r_[0], r_[1]);
            gG[p] = f2_pack(g_[0], g_[1]);
            gB[p] = f2_pack(b_[0], b_[1]);
            gD[p] = f2_pack(d_[0], d_[1]);
            gA[p] = f2_pack(a_[0], a_[1]);
            nacc[p] = f2_bcast(0.f);
            if (VAR) {
                zmu[p] = f2_pack(z_[0], z_[1]);
                ga[p] = f2_pack(ma_[0], ma_[1]);
                gb[p] = f2_pack(mb_[0], mb_[1]);
            }
        }
        uint32_t wmax = mycnt;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) wmax = max(wmax, __shfl_xor_sync(0xffffffffu, wmax, o));
        if (lane == 0) s_max[wid] = wmax;
        __syncthreads();
        uint32_t maxcnt = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) maxcnt = max(maxcnt, s_max[w]);
        for (int64_t hi = (int64_t)rg.x + maxcnt; hi > (int64_t)rg.x; hi -= A.depth) {
            const int64_t lo = max((int64_t)rg.x, hi - A.depth);
            const int nb = (int)(hi - lo);
            __syncthreads();
            for (int j = tid; j < nb; j += NT) {
                uint32_t pair = A.vals[lo + j];
                float4 r0 = A.rec[3 * (size_t)pair], r1 = A.rec[3 * (size_t)pair + 1];
                float4 a, bb;
                stage_record(r0, r1, a, bb);
                sA[j] = a;
                sB[j] = bb;
                sC[j] = A.rec[3 * (size_t)pair + 2];
                sH[j] = make_float2(r0.z, r0.w);
                sP[j] = pair;
            }
            __syncthreads();
            for (int j = nb - 1; j >= 0; --j) {
                const uint32_t rel = (uint32_t)(lo + j - rg.x);
                if (rel >= wmax) continue;  // no pixel of this warp reached this entry
                const float4 a = sA[j], b = sB[j];
                float dxi, u1;
                frag_column(a, b, pxf, dxi, u1);
                // the forward's alpha decision for each of the thread's pixels:
                // ar = the unclamped alpha of a pixel the fragment reaches, else 0
                float ar[PPT], t1_0 = 0.f, t2_0 = 0.f, dyi_0 = 0.f;
                bool any = false;
                {
                    const f2 AY = f2_bcast(a.y), L12 = f2_bcast(b.y), L22 = f2_bcast(b.z);
                    const f2 U1 = f2_bcast(u1), K2 = f2_bcast(a.w), NBW = f2_bcast(-b.w);
                    f2 PY = PY0;
#pragma unroll
                    for (int p = 0; p < Q; ++p) {
                        const f2 dy = f2_sub(PY, AY);  // dyi = py - V, exact as in the forward
                        if (p + 1 < Q) PY = f2_add(PY, ONE);
                        const f2 t1 = f2_fma(L12, dy, U1);
                        const f2 t2 = f2_fma(L22, dy, K2);
                        const f2 ne = f2_fma(t1, t1, f2_fma(t2, t2, NBW));  // -e
                        if (p == 0) {
                            t1_0 = f2_lo(t1);
                            t2_0 = f2_lo(t2);
                            dyi_0 = f2_lo(dy);
                        }
                        float n_[2];
                        f2_unpack(ne, n_[0], n_[1]);
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int i = p + h * Q;
                            const bool in = rel < cnt[i] && n_[h] <= nl2amin;
                            ar[i] = in ? ex2_approx(-n_[h]) : 0.f;
                            any |= in;
                        }
                    }
                }
                if (!__any_sync(0xffffffffu, any)) continue;
                // Every pixel runs the same instructions: a pixel this fragment
                // does not reach takes alpha = 0, for which each update below is
                // exactly the identity (T * 1, acc + 0 * h, sums + 0; the
                // reciprocal approximation returns 1 for 1 on sm_103, measured).
                // The blended sums are carried negated (nwgt = -wgt), which
                // saves the negations the packed instructions cannot fold.
                const float4 c = sC[j];
                const f2 CX = f2_bcast(c.x), CY = f2_bcast(c.y), CZ = f2_bcast(c.z), CW = f2_bcast(c.w);
                f2 sR, sG, sB_, sZ;  // sums of -wgt dL/dc
                // R_k = sum over pairs p of p^k gpw (k = 0, 1, 2), gpw = dL/dpw
                f2 R0, R1, R2;
#pragma unroll
                for (int p = 0; p < Q; ++p) {
                    const float a0 = ar[p], a1 = ar[p + Q];
                    const f2 nal = f2_pack(fmaxf(-amax, -a0), fmaxf(-amax, -a1));  // -alpha
                    // alpha of an unclamped pixel, else 0: a clamped alpha has no
                    // gradient through pw
                    const f2 ag = f2_pack(a0 <= amax ? a0 : 0.f, a1 <= amax ? a1 : 0.f);
                    float o_[2];
                    f2_unpack(f2_add(ONE, nal), o_[0], o_[1]);
                    const f2 r1m = f2_pack(rcp_approx(o_[0]), rcp_approx(o_[1]));  // 1 / (1 - alpha)
                    T[p] = f2_mul(T[p], r1m);  // transmittance before this fragment
                    const f2 nwgt = f2_mul(nal, T[p]);
                    f2 h = f2_fma(gR[p], CX, f2_fma(gG[p], CY, f2_fma(gB[p], CZ, f2_fma(gD[p], CW, gA[p]))));
                    f2 gz = gD[p];
                    if (VAR) {
                        const f2 dz = f2_sub(CW, zmu[p]);
                        const f2 t = f2_fma(gb[p], dz, ga[p]);  // a + b dz
                        h = f2_fma(t, dz, h);
                        gz = f2_add(gz, f2_fma(gb[p], dz, t));  // a + 2 b dz
                    }
                    // dL/dalpha = T h - acc / (1 - alpha)
                    const f2 dLda = f2_fma(T[p], h, f2_mul(nacc[p], r1m));
                    nacc[p] = f2_fma(nwgt, h, nacc[p]);
                    const f2 gpw = f2_mul(dLda, ag);
                    if (p == 0) {
                        sR = f2_mul(nwgt, gR[p]);
                        sG = f2_mul(nwgt, gG[p]);
                        sB_ = f2_mul(nwgt, gB[p]);
                        sZ = f2_mul(nwgt, gz);
                        R0 = gpw;
                    } else {
                        sR = f2_fma(nwgt, gR[p], sR);
                        sG = f2_fma(nwgt, gG[p], sG);
                        sB_ = f2_fma(nwgt, gB[p], sB_);
                        sZ = f2_fma(nwgt, gz, sZ);
                        R0 = f2_add(R0, gpw);
                    }
                    if (p == 1) {
                        R1 = gpw;
                        R2 = gpw;
                    } else if (p > 1) {
                        R1 = f2_fma(gpw, f2_bcast((float)p), R1);
                        R2 = f2_fma(gpw, f2_bcast((float)(p * p)), R2);
                    }
                }
                if (Q == 1) R1 = R2 = f2_bcast(0.f);
                // S_k = sum over the column's pixels i of i^k gpw: pixel p + Q
                // sits in the high half of pair p
                float r0l, r0h, r1l, r1h, r2l, r2h;
                f2_unpack(R0, r0l, r0h);
                f2_unpack(R1, r1l, r1h);
                f2_unpack(R2, r2l, r2h);
                const float S0 = r0l + r0h;
                const float S1 = __fmaf_rn((float)Q, r0h, r1l + r1h);
                const float S2 = __fmaf_rn((float)(Q * Q), r0h, __fmaf_rn((float)(2 * Q), r1h, r2l + r2h));
                // per-lane raw moments: the pixel offsets are dx (one per column)
                // and dy_i = dy_0 + i, and t1, t2 are affine in i; the
                // per-Gaussian factors are applied once after the warp reduction
                const float2 hh = sH[j];
                const float dx = dxi + hh.x, dy0 = dyi_0 + hh.y;
                const float sy = __fmaf_rn(dy0, S0, S1);  // sum gpw dy
                float g[kGrad];
                g[G_LNO] = S0;
                g[G_U] = __fmaf_rn(t1_0, S0, b.y * S1);  // sum gpw t1, t1_i = t1_0 + l12 i
                g[G_V] = __fmaf_rn(t2_0, S0, b.z * S1);  // sum gpw t2, t2_i = t2_0 + l22 i
                g[G_QA] = dx * dx * S0;                     // sum gpw dx^2
                g[G_QB] = dx * sy;                          // sum gpw dx dy
                g[G_QC] = __fmaf_rn(dy0, sy, __fmaf_rn(dy0, S1, S2));  // sum gpw dy^2
                g[G_R] = f2_lo(sR) + f2_hi(sR);
                g[G_G] = f2_lo(sG) + f2_hi(sG);
                g[G_B] = f2_lo(sB_) + f2_hi(sB_);
                g[G_Z] = f2_lo(sZ) + f2_hi(sZ);
                const float tot = warp_reduce_scatter10(g, lane);
                if (my_comp >= 0) {
                    // dL/dQ = -1/2 sum gpw d d^T; dpw/du = (Q d)_x = l11 t1 / s^2,
                    // dpw/dv = (l12 t1 + l22 t2) / s^2 with 1/s^2 = 2 ln 2: each lane
                    // scales its sum by c0 + c11 l11 + c22 l22 (constants per lane;
                    // c0 = -1 undoes the negation of the colour and depth sums)
                    float *gp = A.g2d + (size_t)sP[j] * kGrad;
                    atomicAdd(gp + my_comp, tot * __fmaf_rn(sc11, b.x, __fmaf_rn(sc22, b.z, sc0)));
                    if (my_comp == G_U) {
                        atomicAdd(gp + G_V, kTwoLn2 * b.y * tot);
                        A.state[sP[j]] = kPairTouched;
                    }
                }
            }
        }
    }
}

// zero the image-space gradients of the visible pairs (a backward that does
// not follow its projection directly)
__global__ void k_zero_g2d(const uint32_t *vis_pair, const DevState *st, float *g2d) {
    uint32_t n = st->n_vis;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n * kGrad; i += gridDim.x * blockDim.x)
        g2d[(size_t)vis_pair[i / kGrad] * kGrad + i % kGrad] = 0.f;
}

// The kernel of one pass for a tile size, with its launch shape.  The limit on
// a kernel's dynamic shared memory belongs to the function, not to a
// workspace: smem_most is what its largest depth takes, the same for every
// workspace, so that opening one never lowers the limit under another.
struct RasterKernel {
    void (*fn)(RasterArgs);
    int threads, depth;  // depth: entries staged at a time
    size_t smem, smem_most;
};
constexpr int kMostDepth = 256;  // of the configuration (see check_config)

// The forward's quadrants a warp.
template <int TW, int TH, int Q, bool VAR>
RasterKernel fwd_variant(int depth) {
    const int d = std::min(depth, kFwdDepth);
    constexpr size_t entry = sizeof(FwdEntry) + sizeof(uint32_t);
    return {k_raster_fwd<TW, TH, Q, VAR>, Share<TW, TH, Q>::NT, d, d * entry, kFwdDepth * entry};
}
template <int TW, int TH>
RasterKernel fwd_kernel(const gs_workspace *ws, bool var) {
    const int d = ws->cfg.batch_depth;
    if constexpr (TW * TH >= 256) {
        const int64_t tiles = ws->n_tiles * (TW * TH / 256);
        if (!var)
            return tiles >= kFwdWholeTiles ? fwd_variant<TW, TH, 4, false>(d)
                   : tiles >= kFwdHalfTiles ? fwd_variant<TW, TH, 2, false>(d) : fwd_variant<TW, TH, 1, false>(d);
        return tiles >= kVarHalfTiles ? fwd_variant<TW, TH, 2, true>(d) : fwd_variant<TW, TH, 1, true>(d);
    }
    else {
        constexpr size_t entry = 3 * sizeof(float4);
        return {var ? k_raster_fwd_columns<TW, TH, 2, true> : k_raster_fwd_columns<TW, TH, 2, false>, TW * TH / 2, d,
                d * entry, kMostDepth * entry};
    }
}

// The backward's.
template <int TW, int TH, bool VAR>
RasterKernel bwd_pairs_variant(int depth, int64_t n_tiles) {
    const int d = std::min(depth, TW * TH < 256 || n_tiles <= kDeepTiles ? kPairsDepth : kPairsDepth / 2);
    using S = Share<TW, TH, 1>;
    constexpr size_t entry = sizeof(BwdEntry) + 3 * sizeof(float4) + sizeof(uint32_t) +
                             (S::NW > 1 ? S::NW * kGrad * sizeof(float) : 0);
    constexpr size_t sums = S::NW * kSumBytes;
    return {k_raster_bwd_pairs<TW, TH, VAR>, S::NT, d, d * entry + sums, kPairsDepth * entry + sums};
}
// Pixels a thread of the column variant.  More amortise the reduction and the
// shared-memory reads (500k orchard, 16x16 tiles: 4 -> 0.467 ms, 8, one warp a
// tile, 0.435); the VAR variant holds three more values a pixel and keeps 4 (8
// spills); an 8x8 tile keeps 2 so that its CTA is a whole warp.
template <int TW, int TH, bool VAR>
RasterKernel bwd_columns_variant(int depth) {
    constexpr int PPT = TW * TH >= 256 ? (VAR ? 4 : 8) : 2;
    constexpr size_t entry = 3 * sizeof(float4) + sizeof(float2) + sizeof(uint32_t);
    return {k_raster_bwd<TW, TH, PPT, VAR>, TW * TH / PPT, depth, depth * entry, kMostDepth * entry};
}
template <int TW, int TH>
RasterKernel bwd_kernel(const gs_workspace *ws, bool var) {
    const int d = ws->cfg.batch_depth;
    if (TW * TH < 256 ? ws->n_tiles >= kColumnTiles8 : ws->n_tiles * (TW * TH / 256) >= kColumnTiles)
        return var ? bwd_columns_variant<TW, TH, true>(d) : bwd_columns_variant<TW, TH, false>(d);
    return var ? bwd_pairs_variant<TW, TH, true>(d, ws->n_tiles) : bwd_pairs_variant<TW, TH, false>(d, ws->n_tiles);
}

RasterKernel raster_kernel(const gs_workspace *ws, bool forward, bool var) {
    const int tw = ws->cfg.tile_w, th = ws->cfg.tile_h;
    if (tw == 8) return forward ? fwd_kernel<8, 8>(ws, var) : bwd_kernel<8, 8>(ws, var);
    if (tw == 16 && th == 16) return forward ? fwd_kernel<16, 16>(ws, var) : bwd_kernel<16, 16>(ws, var);
    if (tw == 16) return forward ? fwd_kernel<16, 32>(ws, var) : bwd_kernel<16, 32>(ws, var);
    return forward ? fwd_kernel<32, 16>(ws, var) : bwd_kernel<32, 16>(ws, var);
}

RasterArgs make_args(gs_workspace *ws) {
    RasterArgs A{};
    A.views = ws->views;
    A.n_views = ws->n_views;
    A.n_tiles = (int32_t)ws->n_tiles;
    A.c = ws->consts;
    A.rec = ws->rec;
    A.vals = ws->inst_val;
    A.ranges = ws->ranges;
    A.order = ws->tile_order;
    A.last = ws->last;
    A.tfin = ws->tfin;
    return A;
}

gs_status run(gs_workspace *ws, RasterArgs A, bool forward, bool var, cudaStream_t s) {
    StageTimer timer(ws, forward ? GS_STAGE_RASTER_FWD : GS_STAGE_RASTER_BWD, s);
    ++ws->kernel_launches;
    const RasterKernel k = raster_kernel(ws, forward, var);
    A.depth = k.depth;
    const int grid = forward ? (var ? ws->raster_grid_fwd_var : ws->raster_grid_fwd)
                             : (var ? ws->raster_grid_bwd_var : ws->raster_grid_bwd);
    k.fn<<<grid, k.threads, k.smem, s>>>(A);
    return check_launch(forward ? "raster_fwd" : "raster_bwd");
}

}  // namespace

gs_status raster_configure(gs_workspace *ws) {
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < 4 && e == cudaSuccess; ++i) {
        const bool forward = i < 2, var = i & 1;
        const RasterKernel k = raster_kernel(ws, forward, var);
        e = cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k.smem_most);
        int occ = 0;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k.fn, k.threads, k.smem);
        int32_t &grid = forward ? (var ? ws->raster_grid_fwd_var : ws->raster_grid_fwd)
                                : (var ? ws->raster_grid_bwd_var : ws->raster_grid_bwd);
        grid = std::max(1, occ) * ws->num_sms;
    }
    if (e != cudaSuccess) {
        set_last_error(std::string("raster_configure: ") + cudaGetErrorString(e));
        return GS_ERR_CUDA;
    }
    return GS_OK;
}

gs_status launch_raster_fwd(gs_workspace *ws, float *rgb, float *depth, float *alpha, float *mean,
                            float *var, cudaStream_t s) {
    RasterArgs A = make_args(ws);
    A.counter = &ws->st->fwd_counter;
    A.rgb = rgb;
    A.depth_out = depth;
    A.alpha_out = alpha;
    if (mean) {
        A.mean_out = mean;
        A.var_out = var;
        A.vstat = ws->vstat;
    }
    return run(ws, A, true, mean != nullptr, s);
}

gs_status launch_raster_bwd(gs_workspace *ws, const float *dL_drgb, const float *dL_ddepth,
                            const float *dL_dalpha, bool var, const float *dL_dmean, const float *dL_dvar,
                            cudaStream_t s) {
    RasterArgs A = make_args(ws);
    A.counter = &ws->st->bwd_counter;
    A.dL_drgb = dL_drgb;
    A.dL_ddepth = dL_ddepth;
    A.dL_dalpha = dL_dalpha;
    if (var) {
        A.vstat = ws->vstat;
        A.dL_dmean = dL_dmean;
        A.dL_dvar = dL_dvar;
    }
    A.g2d = ws->g2d;
    A.state = ws->pair_state;
    // the projection clears the rows; a second backward of the same
    // projection clears them itself
    if (!ws->g2d_clear) {
        StageTimer timer(ws, GS_STAGE_ZERO_GRAD, s);
        ++ws->kernel_launches;
        k_zero_g2d<<<ws->num_sms * 4, 256, 0, s>>>(ws->vis_pair, ws->st, ws->g2d);
        gs_status r = check_launch("zero_g2d");
        if (r != GS_OK) return r;
    }
    ws->g2d_clear = false;
    return run(ws, A, false, var, s);
}

}  // namespace gs
