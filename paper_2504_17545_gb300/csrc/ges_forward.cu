// Forward render of Gaussian-enhanced Surfels (Sec. 3, Eq. 1-5) for sm_103a.
//
// Per view, on one stream:
//   k_prep_local  each CTA owns a fixed range of surfels or Gaussians: it sets
//                 each primitive up (surfel raster record + colour, or Gaussian
//                 record: projection, conic, exact support, colour), appends
//                 the visible ones to its own segment of the visible list, and
//                 counts tile overlaps in a shared-memory histogram (16-bit
//                 counters packed in pairs), which it writes out as one row.
//   k_colscan     per tile, exclusive scan of those rows over the CTAs (each
//                 CTA's start inside the tile's list), the place of the tile's
//                 list, and the capacity check.
//   k_fill_local  each CTA re-walks its visible segment and places every
//                 (tile, primitive) pair with shared-memory cursors.
//   k_raster      one warp per 8x4 pixel block: it reads its tile's list, culls
//                 the entries by bbox and depth and tests the records of the
//                 rest (short lists: all at once, see raster_short; long ones:
//                 the warps of a CTA share a block).  Pass 1 keeps the
//                 lexicographic min of (depth, surfel id); pass 2 accumulates
//                 the depth-tested Gaussians (Eq. 2-4); the epilogue applies
//                 Eq. 5.  Everything per pixel stays in registers.
// No global atomics per primitive are needed for binning, so hot tiles do not
// serialise.  (Histogram counts added to global per-tile totals by each
// preprocess CTA, instead of rows and a column scan, cost 97 us of a 4K view's
// preprocess and 5 us of every view of a batch.)
// Very large images (more than 32768 tiles) and callers without binning
// scratch use k_prep_atomic / k_fill_atomic instead (global counters).
//
// List order inside a tile is not fixed (shared-memory atomics), but the
// z-buffer min is order independent and the Gaussian sums are accumulated
// exactly in 64-bit fixed point (alpha in units of 2^-30, its products with the
// colours 2^-46, geometry sums 2^-32), so the image is
// bit-identical run to run without any sort and without float atomics.
#include <limits.h>

#include "ges_internal.cuh"

namespace ges {

LocalBins plan_local_bins(int64_t N, int64_t M, int num_sms)
{
    LocalBins b{0, 0, 1, 1};
    const int P = 2 * num_sms;   // two 16-warp CTAs per SM
    if (N > 0 && M > 0) {
        b.Ps = (int)((P * N + (N + M) / 2) / (N + M));
        b.Ps = b.Ps < 1 ? 1 : (b.Ps > P - 1 ? P - 1 : b.Ps);
        b.Pg = P - b.Ps;
    } else if (N > 0) {
        b.Ps = P;
    } else if (M > 0) {
        b.Pg = P;
    }
    // a CTA's count for one tile must fit in 16 bits
    const int64_t cap = 60000;
    if (N > 0 && (N + b.Ps - 1) / b.Ps > cap) b.Ps = (int)((N + cap - 1) / cap);
    if (M > 0 && (M + b.Pg - 1) / b.Pg > cap) b.Pg = (int)((M + cap - 1) / cap);
    if (b.Ps > 0) b.Rs = (N + b.Ps - 1) / b.Ps;
    if (b.Pg > 0) b.Rg = (M + b.Pg - 1) / b.Pg;
    // ranges start on multiples of 4 primitives (keeps vector stores aligned)
    b.Rs = (b.Rs + 3) & ~(int64_t)3;
    b.Rg = (b.Rg + 3) & ~(int64_t)3;
    return b;
}

LocalBins plan_local_bins_per_cta(int64_t N, int64_t M, int64_t prims_per_cta)
{
    const int64_t R = prims_per_cta < 256 ? 256 : (prims_per_cta > 60000 ? 60000 : prims_per_cta);
    LocalBins b{0, 0, 1, 1};
    b.Ps = (int)((N + R - 1) / R);
    b.Pg = (int)((M + R - 1) / R);
    if (b.Ps > 0) b.Rs = ((N + b.Ps - 1) / b.Ps + 3) & ~(int64_t)3;
    if (b.Pg > 0) b.Rg = ((M + b.Pg - 1) / b.Pg + 3) & ~(int64_t)3;
    return b;
}

namespace {

__device__ __forceinline__ unsigned lane_id() { return threadIdx.x & 31u; }

// A 64-byte record as four float4 stores, built from its fields (no
// reinterpretation of the local copy).
__device__ __forceinline__ void store_rec(float4 *dst, const SurfelRec &r)
{
    dst[0] = make_float4(r.ur, r.vr, r.iz0, r.gu);
    dst[1] = make_float4(r.gv, r.au, r.av, r.a0);
    dst[2] = make_float4(r.bu, r.bv, r.b0, __int_as_float(r.id));
    dst[3] = make_float4(r.izmax, __uint_as_float(r.bb_lo), __uint_as_float(r.bb_hi), r.pad);
}

// The first three quarters of a staged Gaussian record (what alpha, the depth
// key and the colour need).
__device__ __forceinline__ GaussRec gauss_rec3(float4 a, float4 b, float4 c)
{
    GaussRec g;
    g.px = a.x; g.py = a.y; g.pxl = a.z; g.pyl = a.w;
    g.la = b.x; g.lb = b.y; g.lc = b.z; g.sigma = b.w;
    g.key = c.x; g.r = c.y; g.g = c.z; g.b = c.w;
    g.id = 0; g.bb_lo = 0u; g.bb_hi = 0u; g.pad = 0.f;
    return g;
}

// Where a set-up's colours (Eq. 1) come from.
enum ColourFrom : int {
    COL_PASS = 0,     // the batch's colour pass (ran before for the Gaussians, surfels need nothing)
    COL_HERE = 1,     // evaluated with the geometry, the SH row read by its thread
    COL_STAGED = 2,   // evaluated later from an SH row staged in shared memory (see sh_stage)
};
// Set up primitive i of the given kind; on success write its record and
// return its pixel bbox and cull key.
// kGd: the scene's Gaussian kind (a template argument, so that each kernel
// carries only its own set-up code).  kCol: ColourFrom.
template <int kGd, bool kTr = false, int kCol = COL_HERE>
__device__ __forceinline__ bool setup_and_store(const SceneView &S, const CamParams &C, const OptParams &O,
                                                const ViewScratch &X, bool surf, int64_t i, int &x0, int &y0,
                                                int &x1, int &y1, unsigned &key)
{
    const int nb = mask_bits(C.tsx, C.tsy);
    if (surf) {
        SurfelOut o;
        // the record goes out before the colour is evaluated: its registers
        // are free again for the SH row
        surfel_geom(S, C, O, i, o, kTr ? X.s_tside + 4 * i : nullptr);
        if (!o.valid_quat) atomicOr(X.status + ST_FLAGS, FLAG_BADQ);
        if (!o.visible) return false;
        store_rec(X.s_rec + 4 * i, o.rec);
        if (kCol == COL_HERE) {
            surfel_colour(S, i, o);
            X.s_rgb[i] = make_float4(o.rgb[0], o.rgb[1], o.rgb[2], 0.f);
        }
        x0 = o.x0; y0 = o.y0; x1 = o.x1; y1 = o.y1;
        // the translucent lists are sorted by the centre's depth instead
        key = kTr ? depth_key(X.s_tside[4 * i].z) : surfel_key_bits(o.rec.izmax, nb);
    } else {
        GaussOut o;
        if (kGd == 2) gauss2d_setup(S, C, O, i, o, kCol == COL_HERE);
        else gauss_geom(S, C, O, i, o);
        if (!o.valid_quat) atomicOr(X.status + ST_FLAGS, FLAG_BADQ);
        if (!o.visible) return false;
        if (kGd == 2) {
            store_rec(X.g_rec + 4 * i, o.drec);
        } else {
            // three quarters of the record before the colour is evaluated
            float4 *dst = X.g_rec + 4 * i;
            dst[0] = make_float4(o.rec.px, o.rec.py, o.rec.pxl, o.rec.pyl);
            dst[1] = make_float4(o.rec.la, o.rec.lb, o.rec.lc, o.rec.sigma);
            dst[3] = make_float4(__int_as_float(o.rec.id), __uint_as_float(o.rec.bb_lo),
                                 __uint_as_float(o.rec.bb_hi), o.rec.pad);
            if (kCol == COL_HERE) {
                gauss_colour(S, i, o);
                dst[2] = make_float4(o.rec.key, colour_q(o.rec.r), colour_q(o.rec.g), colour_q(o.rec.b));
            } else if (kCol == COL_PASS) {
                const float4 c = X.g_col[i];   // the colour pass's colour
                dst[2] = make_float4(o.rec.key, c.x, c.y, c.z);
            } else {
                dst[2].x = o.rec.key;          // the staged colour joins it
            }
        }
        if (kGd == 2 || O.geo) {
            float4 a0 = o.aux[0];
            if (kGd == 2 && kCol == COL_PASS) {
                const float4 c = X.g_col[i];   // the colour pass's colour
                a0.x = c.x; a0.y = c.y; a0.z = c.z;
            }
            X.g_aux[2 * i] = a0;               // (2D: a staged colour joins log2 sigma')
            X.g_aux[2 * i + 1] = o.aux[1];
        }
        x0 = o.x0; y0 = o.y0; x1 = o.x1; y1 = o.y1;
        // 3D: d - eps; 2D: the smallest planar depth less eps
        key = gauss_key_bits(kGd == 2 ? 1.f / o.drec.izmax - o.drec.pad : o.rec.key, nb);
    }
    return true;
}

// Staged SH rows (16 coefficients per channel: 192 bytes in FP32, 96 in 16
// bits).  A warp copies the rows of its visible primitives to its own shared
// space, 16 bytes per lane and consecutive lanes consecutive bytes, while it
// sets up the next 32 primitives, and evaluates the colours afterwards.  A row
// per thread read directly (12 loads of 16 bytes, 192 bytes apart between the
// lanes: 32 cache lines per load) added its whole time to the set-up's: of the
// preprocess of a 1080p view (1M + 300k, FP32) 110 us, 47 were the colours;
// staged it takes 90 (200k + 2.5M: 195 -> 163; 2.25M + 750k in FP16: 217 -> 186).
// The copies must cost few instructions: with the chunk's place worked out one
// by one the set-up issued 84M instead of 56M instructions and gained nothing.
// kChunks 16-byte chunks per row, 12 or 6.  Chunk c of row r lies at c ^ swz(r),
// which spreads equal chunks of eight consecutive rows over all banks.
constexpr int kShRows = 16;     // basis functions of a staged row
template <int kChunks>
__device__ __forceinline__ int sh_swz(int r) { return kChunks == 12 ? r >> 1 & 3 : r >> 2 & 1; }

template <int kChunks>
__device__ __forceinline__ void sh_stage(const void *sh, int64_t i0, unsigned vis, unsigned char *st)
{
    // the lane's chunks: number 32 j + lane of the 32 rows; three of them
    // (j = 0, 1, 2) end on a whole number of rows, then the pattern repeats
    constexpr int kRep = kChunks / 3, kRepRows = 96 / kChunks;
    const unsigned base = (unsigned)__cvta_generic_to_shared(st);
    const int lane = (int)lane_id();
    const unsigned char *src = reinterpret_cast<const unsigned char *>(sh) + (i0 * kChunks + lane) * 16;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const int g = 32 * j + lane, r = kChunks == 12 ? (g * 43) >> 9 : (g * 43) >> 8, c = g - kChunks * r;
        const unsigned dst = base + (unsigned)(16 * (kChunks * r + (c ^ sh_swz<kChunks>(r)))), v = vis >> r;
#pragma unroll
        for (int m = 0; m < kRep; ++m)
            if (v & (1u << (kRepRows * m)))
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                             :: "r"(dst + 16u * kChunks * kRepRows * m), "l"(src + 512 * j + 1536 * m) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// The colour from the lane's staged row, by sh_colour's operations in their order.
template <int kChunks>
__device__ __forceinline__ void sh_staged_colour(const unsigned char *st, bool half, const float *dir, float *rgb)
{
    const int lane = (int)lane_id();
    float Y[kShRows];
    sh_basis(kShRows, dir[0], dir[1], dir[2], Y);
    float v[3] = {0.5f, 0.5f, 0.5f};
    const uint4 *row = reinterpret_cast<const uint4 *>(st) + kChunks * lane;
    const int k0 = sh_swz<kChunks>(lane);
#pragma unroll
    for (int q = 0; q < kChunks; ++q) {
        const uint4 x = row[q ^ k0];
        const unsigned e[4] = {x.x, x.y, x.z, x.w};
        constexpr int kN = kChunks == 12 ? 4 : 8;
#pragma unroll
        for (int k = 0; k < kN; ++k) {
            float c;
            if (kChunks == 12) {
                c = __uint_as_float(e[k]);
            } else {
                const unsigned short h = (unsigned short)(k & 1 ? e[k / 2] >> 16 : e[k / 2] & 0xffffu);
                c = half ? __half2float(__ushort_as_half(h)) : __bfloat162float(__ushort_as_bfloat16(h));
            }
            v[(kN * q + k) % 3] = fmaf(c, Y[(kN * q + k) / 3], v[(kN * q + k) % 3]);
        }
    }
    rgb[0] = fmaxf(v[0], 0.f); rgb[1] = fmaxf(v[1], 0.f); rgb[2] = fmaxf(v[2], 0.f);
}

// ---------------------------------------------------------------------------
// local binning

// Calls f(c, tx, ty) for every tile that the bbox (c.y, c.z) of a lane's entry
// c touches (on: the lane has one).  A lane walks a bbox of up to kLaneTiles
// tiles itself; larger ones the whole warp walks, a tile per lane (a primitive
// right in front of the camera covers every tile of the image: one lane alone
// took 330 us for the 8160 tiles of a 1080p view).  All 32 lanes call it.
constexpr int kLaneTiles = 32;
template <class F>
__device__ __forceinline__ void for_tiles(bool on, const int4 &c, int tsx, int tsy, F f)
{
    const int lane = (int)lane_id();
    const int tx0 = (c.y & 0xffff) >> tsx, tx1 = (c.z & 0xffff) >> tsx;
    const int ty0 = (int)((unsigned)c.y >> 16) >> tsy, ty1 = (int)((unsigned)c.z >> 16) >> tsy;
    const int n = on ? (tx1 - tx0 + 1) * (ty1 - ty0 + 1) : 0;
    if (n <= kLaneTiles) {
        if (n > 0)
            for (int ty = ty0; ty <= ty1; ++ty)
                for (int tx = tx0; tx <= tx1; ++tx) f(c, tx, ty);
    }
    unsigned big = __ballot_sync(0xffffffffu, n > kLaneTiles);
    while (big) {
        const int o = __ffs(big) - 1;
        big &= big - 1;
        const auto from = [&](int x) { return __shfl_sync(0xffffffffu, x, o); };
        const int4 b = make_int4(from(c.x), from(c.y), from(c.z), from(c.w));
        const int bx = from(tx0), by = from(ty0), w = from(tx1 - tx0 + 1), bn = from(n);
        const float iw = 1.f / (float)w;
        for (int k = lane; k < bn; k += 32) {
            const int r = bbox_row(k, w, iw);
            f(b, bx + (k - r * w), by + r);
        }
    }
}

// CTA c of a view: its range of primitives.  hist: ceil(T/2) shared words
// (two 16-bit counters each); vcnt: a shared counter.
// kKind: 1 a surfel range, 2 a Gaussian range (each its own code)
// kCol COL_STAGED: the shared memory after the histogram holds an SH row per
// thread.
template <int kGd, bool kTr, int kKind, int kCol>
__device__ __forceinline__ void prep_local_body(const SceneView &S, const CamParams &C, const OptParams &O,
                                                const ViewScratch &X, const LocalBins &B, int c, unsigned *hist,
                                                unsigned &vcnt)
{
    const int T = C.tiles_x * C.tiles_y, words = (T + 1) >> 1;
    const int row_bytes = 3 * kShRows * (S.sh_dtype == GES_F32 ? 4 : 2);
    unsigned char *stage = reinterpret_cast<unsigned char *>(hist + ((words + 3) & ~3)) +
                           (size_t)(threadIdx.x >> 5) * 32 * row_bytes;
    constexpr bool surf = kKind == 1;
    unsigned pending = 0;   // the lanes whose rows are being staged
    // The colours of round i's staged rows.  Nothing but the mask is carried
    // over from the set-up: the position and the word beside the colour are
    // read again (from L2), which is cheaper than spilling them.
    const auto colour = [&](int64_t i) {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncwarp();
        if (pending >> lane_id() & 1u) {
            const float *pos = surf ? S.s_pos : S.g_pos;
            float dir[3], L, rgb[3];
            view_dir(C, __ldg(pos + 3 * i), __ldg(pos + 3 * i + 1), __ldg(pos + 3 * i + 2), dir, L);
            if (S.sh_dtype == GES_F32) sh_staged_colour<12>(stage, false, dir, rgb);
            else sh_staged_colour<6>(stage, S.sh_dtype == GES_F16, dir, rgb);
            if (surf) {
                X.s_rgb[i] = make_float4(rgb[0], rgb[1], rgb[2], 0.f);
            } else {
                const float r = colour_q(rgb[0]), g = colour_q(rgb[1]), b = colour_q(rgb[2]);
                if (kGd == 2) X.g_aux[2 * i] = make_float4(r, g, b, X.g_aux[2 * i].w);
                else X.g_rec[4 * i + 2] = make_float4(X.g_rec[4 * i + 2].x, r, g, b);
            }
        }
        __syncwarp();       // the rows are read: the space is free
    };
    const int64_t R = surf ? B.Rs : B.Rg, n = surf ? S.N : S.M;
    const int64_t beg = (int64_t)(surf ? c : c - B.Ps) * R;
    const int64_t end = beg + R < n ? beg + R : n;
    for (int w = threadIdx.x; w < words; w += kPrepThreads) hist[w] = 0u;
    if (threadIdx.x == 0) vcnt = 0u;
    __syncthreads();
    // the CTA's segment of visible primitives: (id, bbox lo, bbox hi, key)
    // per entry, so that the fill reads its entries contiguously instead of
    // gathering each record's bbox
    int4 *seg = reinterpret_cast<int4 *>(surf ? X.s_vis : X.g_vis) + beg;
    for (int64_t i0 = beg; i0 < end; i0 += kPrepThreads) {
        const int64_t i = i0 + threadIdx.x;
        int x0 = 0, y0 = 0, x1 = -1, y1 = -1;
        unsigned key = 0;
        const bool vis = i < end && setup_and_store<kGd, kTr, kCol>(S, C, O, X, surf, i, x0, y0, x1, y1, key);
        const int4 entry = make_int4((int)i, (int)pack_xy(x0, y0), (int)pack_xy(x1, y1), (int)key);
        const unsigned m = __ballot_sync(0xffffffffu, vis);
        if (kCol == COL_STAGED) {
            // the rows asked for a round ago are here: their colours, then this round's rows
            if (i0 != beg) colour(i - kPrepThreads);
            pending = m;
            const void *sh = surf ? S.s_sh : S.g_sh;
            if (S.sh_dtype == GES_F32) sh_stage<12>(sh, i - (int64_t)lane_id(), m, stage);
            else sh_stage<6>(sh, i - (int64_t)lane_id(), m, stage);
        }
        if (m) {
            const int leader = __ffs(m) - 1;
            unsigned b = 0;
            if ((int)lane_id() == leader) b = atomicAdd(&vcnt, (unsigned)__popc(m));
            b = __shfl_sync(0xffffffffu, b, leader);
            if (vis) seg[b + __popc(m & ((1u << lane_id()) - 1u))] = entry;
        }
        for_tiles(vis, entry, C.tsx, C.tsy, [&](const int4 &, int tx, int ty) {
            const int t = ty * C.tiles_x + tx;
            atomicAdd(hist + (t >> 1), (t & 1) ? 65536u : 1u);
        });
    }
    if (kCol == COL_STAGED && beg < end)
        colour(beg + (end - beg - 1) / kPrepThreads * kPrepThreads + threadIdx.x);
    __syncthreads();
    unsigned *row = X.hist + (size_t)c * words;
    for (int w = threadIdx.x; w < words; w += kPrepThreads) row[w] = hist[w];
    if (threadIdx.x == 0) {
        X.vcount[c] = vcnt;
        atomicAdd(X.status + (surf ? ST_SVIS : ST_GVIS), vcnt);
    }
}

template <int kGd, bool kTr, int kCol>
__global__ void __launch_bounds__(kPrepThreads, 2) k_prep_local(SceneView S, CamParams C, OptParams O,
                                                                ViewScratch X, LocalBins B)
{
    extern __shared__ __align__(16) unsigned hist[];
    __shared__ unsigned vcnt;
    // the two kinds' code apart, so that neither's registers count for the other
    if ((int)blockIdx.x < B.Ps) prep_local_body<kGd, kTr, 1, kCol>(S, C, O, X, B, blockIdx.x, hist, vcnt);
    else prep_local_body<kGd, kTr, 2, kCol>(S, C, O, X, B, blockIdx.x, hist, vcnt);
}

// Space for the lists of the tiles whose totals a warp holds (n tiles on each
// lane, their sum in tot): one addition to the list space handed out so far,
// so the lists lie in the order the warps arrive in (nothing depends on it).
// Returns the start of the lane's first list.
__device__ __forceinline__ int alloc_lists(const ViewScratch &X, bool surf, int64_t tot)
{
    const int lane = (int)lane_id();
    int64_t incl = tot;                  // 64 bits: lists too large are found, not wrapped
    for (int d = 1; d < 32; d <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += y;
    }
    int64_t at = 0;
    if (lane == 31) {
        unsigned long long *space = reinterpret_cast<unsigned long long *>(X.status + (surf ? ST_SCUR : ST_GCUR));
        at = (int64_t)atomicAdd(space, (unsigned long long)incl);
        atomicAdd(X.status + (surf ? ST_SPAIRS : ST_GPAIRS), (unsigned)incl);
        if (at + incl > (surf ? X.s_cap : X.g_cap)) atomicOr(X.status + ST_FLAGS, surf ? FLAG_SOVF : FLAG_GOVF);
    }
    return (int)(__shfl_sync(0xffffffffu, at, 31) + incl - tot);
}

// Per tile: exclusive scan of the counts over the CTAs of one kind, and a
// place for the tile's list.  Block = 64 tiles x kW warps: a lane takes one
// histogram word (two tiles), warp w the CTAs [w P/kW, (w+1) P/kW).  A single
// view is bound by the latency of the rows' loads, so 32 warps share the CTAs
// of a tile there; in a batch the blocks of the other views hide it, and 8
// warps have fewer barriers and partial sums per row.  Scanning the totals in
// a launch of its own, by one CTA per kind, the two launches took 27.9 us of a
// 1080p view (1M + 300k primitives) and 115.5 us of a 4K one (2.25M + 750k);
// this one takes 10.8 and 23.1 us.
template <int kW>
__device__ __forceinline__ void colscan_body(const ViewScratch &X, int T, const LocalBins &B, int bx, bool surf,
                                             unsigned (*part)[kColTiles + 1])
{
    const int P = surf ? B.Ps : B.Pg, r0 = surf ? 0 : B.Ps;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int words = (T + 1) >> 1, word = bx * 32 + lane;
    const int a = r0 + (int)((int64_t)P * w / kW), b = r0 + (int)((int64_t)P * (w + 1) / kW);
    const unsigned *h = X.hist + word;
    unsigned s0 = 0, s1 = 0;
    if (word < words) {
#pragma unroll 8
        for (int r = a; r < b; ++r) {
            const unsigned v = h[(size_t)r * words];
            s0 += v & 0xffffu;
            s1 += v >> 16;
        }
    }
    part[w][2 * lane] = s0;
    part[w][2 * lane + 1] = s1;
    __syncthreads();
    // the warps' sums of each tile in turn (row kW: the totals); groups of kW
    // lanes, one tile each
    for (int q = threadIdx.x / kW; q < kColTiles; q += 32) {
        const int k = threadIdx.x % kW;
        const unsigned v = part[k][q];
        unsigned incl = v;
        for (int d = 1; d < kW; d <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, incl, d, kW);
            if (k >= d) incl += y;
        }
        part[k][q] = incl - v;
        if (k == kW - 1) part[kW][q] = incl;
    }
    __syncthreads();
    if (w == 0) {
        const int n0 = (int)part[kW][2 * lane], n1 = (int)part[kW][2 * lane + 1];
        const int at = alloc_lists(X, surf, (int64_t)n0 + n1);
        int2 *rng = surf ? X.s_rng : X.g_rng;
        if (2 * word < T) rng[2 * word] = make_int2(at, at + n0);
        if (2 * word + 1 < T) rng[2 * word + 1] = make_int2(at + n0, at + n0 + n1);
    }
    if (word >= words) return;
    unsigned p0 = part[w][2 * lane], p1 = part[w][2 * lane + 1];
    uint2 *out = reinterpret_cast<uint2 *>(X.base) + word;
#pragma unroll 8
    for (int r = a; r < b; ++r) {
        const unsigned v = h[(size_t)r * words];
        out[(size_t)r * words] = make_uint2(p0, p1);
        p0 += v & 0xffffu;
        p1 += v >> 16;
    }
}

__global__ void __launch_bounds__(1024) k_colscan(ViewScratch X, int T, LocalBins B)
{
    __shared__ unsigned part[33][kColTiles + 1];
    colscan_body<32>(X, T, B, blockIdx.x, blockIdx.y == 0, part);
}

// The raster's work items, by one CTA while the others fill.  A tile is
// rastered by a warp per block, or, if its list (both kinds together) is long,
// by all warps of a CTA block after block.  One view: an item per tile, or per
// block of a shared tile (above bit 24 of the word 1 + block), the costly ones
// first in buckets of a quarter octave, so that none starts when the rest is
// done: in the order of the tiles the SMs stood idle for 17 % of a 1080p view's
// raster and 40 % of a 4-sample one's.  A batch: the shared tiles, then the
// others, each longest first, then those with short lists (raster_short; not
// counted one by one: their shared counter would be every thread's).  The
// translucent render: the tiles, longest first.
// Long is above total / kShareSlots entries (total: of all views): such a
// tile's warps would still be at work when all other tiles are done.  At half
// that, ordinary views slow down (a shared block's z-buffers cull less: 1080p
// raster 158 -> 161 us, at a quarter 193 us); at twice that, a 250x200 view of
// 1.2M primitives takes 146 instead of 83 us (580 us with no sharing).  Short
// lists (kShareMin) are not worth the merge.
constexpr unsigned kShareMin = 256u;
// at most this many entries in each of a tile's lists: raster_short's, an entry per lane
constexpr int kShort = 32;
__device__ __forceinline__ bool short_lists(const int2 &sr, const int2 &gr)
{
    return max(sr.y - sr.x, gr.y - gr.x) <= kShort;
}
enum OrderOf : int { ORDER_VIEW, ORDER_TILES, ORDER_BATCH };
// Returns (to all threads) the number of shared (ORDER_BATCH) and short tiles.
template <int kOf>
__device__ __forceinline__ uint2 order_body(const ViewScratch &X, int T, unsigned long long total, unsigned *sh)
{
    unsigned *start = sh;                     // [64] buckets, then the short ones
    const unsigned share = max((unsigned)min(total / kShareSlots, 0x7fffffffull), kShareMin);
    // a tile's bucket, 0..63, costly first (not one view: 0..31 shared, 32..63 not, half octaves; 64 short)
    bool blocks = false;
    const auto bucket = [&](const int2 &s, const int2 &g) {
        blocks = false;
        if (kOf == ORDER_BATCH && short_lists(s, g)) return 64;
        const unsigned n = (unsigned)((s.y - s.x) + (g.y - g.x));
        const bool sh_ = n > share;
        blocks = kOf == ORDER_VIEW && sh_;
        const unsigned b = __float_as_uint((float)(1u + (blocks ? n / 8u : n)));
        return kOf != ORDER_VIEW ? (sh_ ? 31 : 63) - min((int)(b >> 22) - (127 << 1), 31) : 63 - min((int)(b >> 21) - (127 << 2), 63);
    };
    // f(t, tile t's lists) for all tiles, with t >= T for lanes past the end; the
    // lists of kAhead tiles are read at once (this CTA ends last in sparse views)
    constexpr int kAhead = 4;
    const auto each_tile = [&](auto f) {
        for (int t0 = 0; t0 < T; t0 += kAhead * kFillThreads) {
            int2 sr[kAhead], gr[kAhead];
#pragma unroll
            for (int j = 0; j < kAhead; ++j) {
                const int t = min(t0 + j * kFillThreads + (int)threadIdx.x, T - 1);
                sr[j] = X.s_rng[t];
                gr[j] = X.g_rng[t];
            }
#pragma unroll
            for (int j = 0; j < kAhead; ++j)
                if (t0 + j * kFillThreads < T) f(t0 + j * kFillThreads + (int)threadIdx.x, sr[j], gr[j]);
        }
    };
    // takes places in the lane's bucket (on: it has a tile)
    const auto take = [&](bool on, int k) {
        unsigned at = 0;
        if (on && k < 64) at = atomicAdd(start + k, blocks ? (unsigned)kOrderItems : 1u);
        if constexpr (kOf == ORDER_BATCH) {
            const unsigned m = __ballot_sync(0xffffffffu, on && k == 64);
            unsigned first = 0;
            if (lane_id() == 0 && m) first = atomicAdd(start + 64, (unsigned)__popc(m));
            first = __shfl_sync(0xffffffffu, first, 0);
            if (on && k == 64) at = first + __popc(m & ((1u << lane_id()) - 1u));
        }
        return at;
    };
    if (threadIdx.x < 65) start[threadIdx.x] = 0u;
    __syncthreads();
    each_tile([&](int t, const int2 &sr, const int2 &gr) {
        const int k = bucket(sr, gr);
        take(t < T, k);
    });
    __syncthreads();
    if (threadIdx.x < 32) {
        const unsigned a = start[2 * threadIdx.x], b = start[2 * threadIdx.x + 1];
        unsigned incl = a + b;
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned y = __shfl_up_sync(0xffffffffu, incl, d);
            if ((int)threadIdx.x >= d) incl += y;
        }
        start[2 * threadIdx.x] = incl - a - b;
        start[2 * threadIdx.x + 1] = incl - b;
        if (threadIdx.x == 15) start[65] = incl;
        if (threadIdx.x == 31) {
            start[66] = start[64];
            start[64] = incl;
            if (kOf == ORDER_VIEW) X.status[ST_ITEMS] = incl;
        }
    }
    __syncthreads();
    const uint2 counts = make_uint2(start[65], start[66]);
    each_tile([&](int t, const int2 &sr, const int2 &gr) {
        const int b = bucket(sr, gr);
        const unsigned at = take(t < T, b);
        if (t >= T) return;
        if (blocks)
            for (unsigned k = 0; k < kOrderItems; ++k) X.order[at + k] = (unsigned)t | (k + 1u) << 24;
        else
            X.order[at] = (unsigned)t;
    });
    return counts;
}

// sorted (translucent render): the lists hold sort keys (id, depth key)
// instead of (id, cull word)
__device__ __forceinline__ void fill_local_body(const ViewScratch &X, int T, int tiles_x, int tsx, int tsy,
                                                const LocalBins &B, int c, unsigned *cur, bool sorted)
{
    const bool surf = c < B.Ps;
    const int64_t beg = (int64_t)(surf ? c : c - B.Ps) * (surf ? B.Rs : B.Rg);
    const int4 *seg = reinterpret_cast<const int4 *>(surf ? X.s_vis : X.g_vis) + beg;
    // the thread's first entry is read while the cursors are set
    const unsigned n = X.vcount[c];
    int4 e = threadIdx.x < n ? seg[threadIdx.x] : make_int4(0, 0, 0, 0);
    if (X.status[ST_FLAGS] & (FLAG_SOVF | FLAG_GOVF)) return;
    const int2 *rng = surf ? X.s_rng : X.g_rng;
    const unsigned *brow = X.base + (size_t)c * (2 * ((T + 1) >> 1));
#pragma unroll 4
    for (int t = threadIdx.x; t < T; t += kFillThreads) cur[t] = (unsigned)rng[t].x + brow[t];
    __syncthreads();
    uint2 *list = surf ? X.s_list : X.g_list;
    for (unsigned k0 = 0; k0 < n; k0 += kFillThreads) {
        const unsigned k = k0 + threadIdx.x;
        const int4 c = e;
        if (k + kFillThreads < n) e = seg[k + kFillThreads];
        for_tiles(k < n, c, tsx, tsy, [&](const int4 &v, int tx, int ty) {
            unsigned w = (unsigned)v.w;
            if (!sorted)
                w |= row_mask((int)((unsigned)v.y >> 16), (int)((unsigned)v.z >> 16), ty, tsx, tsy) |
                     col_mask(v.y & 0xffff, v.z & 0xffff, tx, tsx);
            list[atomicAdd(cur + ty * tiles_x + tx, 1u)] = make_uint2((unsigned)v.x, w);
        });
    }
}

__global__ void __launch_bounds__(kFillThreads, 2) k_fill_local(ViewScratch X, int T, int tiles_x, int tsx, int tsy,
                                                             LocalBins B)
{
    extern __shared__ unsigned cur[];    // T cursors
    if (blockIdx.x == 0) {
        // (the translucent kernels take whole tiles)
        const unsigned long long total = (unsigned long long)X.status[ST_SPAIRS] + X.status[ST_GPAIRS];
        if (X.s_tside) order_body<ORDER_TILES>(X, T, total, cur);
        else order_body<ORDER_VIEW>(X, T, total, cur);
    }
    else fill_local_body(X, T, tiles_x, tsx, tsy, B, blockIdx.x - 1, cur, X.s_tside != nullptr);
}

// ---------------------------------------------------------------------------
// atomic binning (fallback)

__device__ __forceinline__ void append_visible(bool vis, int64_t i, unsigned *counter, int *list)
{
    const unsigned m = __ballot_sync(0xffffffffu, vis);
    if (m == 0u) return;
    const unsigned lane = lane_id();
    const int leader = __ffs(m) - 1;
    unsigned base = 0;
    if ((int)lane == leader) base = atomicAdd(counter, (unsigned)__popc(m));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (vis) list[base + __popc(m & ((1u << lane) - 1u))] = (int)i;
}

template <int kGd, bool kTr = false>
__global__ void __launch_bounds__(256) k_prep_atomic(SceneView S, CamParams C, OptParams O, ViewScratch X,
                                                     int n_sblocks)
{
    const bool surf = (int)blockIdx.x < n_sblocks;
    const int64_t i = (int64_t)(surf ? blockIdx.x : blockIdx.x - n_sblocks) * 256 + threadIdx.x;
    int x0 = 0, y0 = 0, x1 = -1, y1 = -1;
    unsigned key = 0;
    const bool vis = i < (surf ? S.N : S.M) && setup_and_store<kGd, kTr>(S, C, O, X, surf, i, x0, y0, x1, y1, key);
    int *cnt = surf ? X.s_cnt : X.g_cnt;
    for_tiles(vis, make_int4(0, (int)pack_xy(x0, y0), (int)pack_xy(x1, y1), 0), C.tsx, C.tsy,
              [&](const int4 &, int tx, int ty) { atomicAdd(cnt + ty * C.tiles_x + tx, 1); });
    append_visible(vis, i, X.status + (surf ? ST_SVIS : ST_GVIS), surf ? X.s_vis : X.g_vis);
}

// the list entry of one primitive, from its record (bbox and cull key)
__device__ __forceinline__ int4 record_entry(const ViewScratch &X, bool surf, int gdim, int id, int nb)
{
    const float4 r3 = (surf ? X.s_rec : X.g_rec)[4 * (int64_t)id + 3];
    const unsigned key = X.s_tside ? depth_key(X.s_tside[4 * (int64_t)id].z)
                                   : (surf ? surfel_key_bits(r3.x, nb)
                                           : gauss_key_bits(gdim == 2 ? 1.f / r3.x - r3.w : r3.w, nb));
    return make_int4(id, __float_as_int(r3.y), __float_as_int(r3.z), (int)key);
}

__global__ void __launch_bounds__(256) k_fill_atomic(ViewScratch X, int gdim, int tiles_x, int tsx, int tsy)
{
    if (X.status[ST_FLAGS] & (FLAG_SOVF | FLAG_GOVF)) return;
    const unsigned ns = X.status[ST_SVIS], ng = X.status[ST_GVIS];
    const unsigned stride = gridDim.x * blockDim.x;
    const bool sorted = X.s_tside != nullptr;
    for (unsigned k0 = blockIdx.x * blockDim.x; k0 < ns + ng; k0 += stride) {
        const unsigned k = k0 + threadIdx.x;
        const bool surf = k < ns, on = k < ns + ng;
        int4 e = make_int4(0, 0, 0, 0);
        if (on) e = record_entry(X, surf, gdim, surf ? X.s_vis[k] : X.g_vis[k - ns], mask_bits(tsx, tsy));
        // surfels, then Gaussians: a warp may hold both
        for (int kind = 0; kind < 2; ++kind) {
            int2 *rng = kind == 0 ? X.s_rng : X.g_rng;
            uint2 *list = kind == 0 ? X.s_list : X.g_list;
            for_tiles(on && surf == (kind == 0), e, tsx, tsy, [&](const int4 &v, int tx, int ty) {
                unsigned w = (unsigned)v.w;
                if (!sorted)
                    w |= row_mask((int)((unsigned)v.y >> 16), (int)((unsigned)v.z >> 16), ty, tsx, tsy) |
                         col_mask(v.y & 0xffff, v.z & 0xffff, tx, tsx);
                list[atomicAdd(&rng[ty * tiles_x + tx].y, 1)] = make_uint2((unsigned)v.x, w);
            });
        }
    }
}

// ---------------------------------------------------------------------------
// list allocation (atomic binning; k_colscan does it for local bins)

// Places for the lists from the tiles' totals.  The ends start at the lists'
// starts (the fill moves them), and the counters go back to zero.
__global__ void __launch_bounds__(kAllocTiles) k_alloc(ViewScratch X, int T)
{
    const bool surf = blockIdx.y == 0;
    int *cnt = surf ? X.s_cnt : X.g_cnt;
    const int t = blockIdx.x * kAllocTiles + threadIdx.x;
    const int at = alloc_lists(X, surf, t < T ? cnt[t] : 0);
    if (t < T) {
        (surf ? X.s_rng : X.g_rng)[t] = make_int2(at, at);
        cnt[t] = 0;
    }
}

// ---------------------------------------------------------------------------
// raster

// 16-byte planes of one staged Gaussian: the three quarters of its record that
// alpha, the depth test and the colour need; with geometry the first word of
// its side data; 2D Gaussians take their fourth quarter (eps) and both side
// words
template <int kG, bool kGeo>
__host__ __device__ constexpr int gauss_planes() { return kG == 2 ? 6 : (kGeo ? 4 : 3); }

// Surfel normal from its record, camera space, facing the camera: the record's
// 1/z = iz0 + gu (u - ur) + gv (v - vr) equals (n . ray)/(n . P), so
// m = (gu fx, gv fy, iz0 - gu (ur - cx) - gv (vr - cy)) = n / (n . P).
__device__ __forceinline__ void surfel_normal(const float4 *rec, int id, const CamParams &C, float *nrm)
{
    const float4 r0 = rec[4 * (int64_t)id], r1 = rec[4 * (int64_t)id + 1];
    const float mx = r0.w * C.fx, my = r1.x * C.fy;
    const float mz = r0.z - r0.w * (r0.x - C.cx) - r1.x * (r0.y - C.cy);
    const float inv = -rsqrtf(fmaf(mx, mx, fmaf(my, my, mz * mz)));
    nrm[0] = mx * inv; nrm[1] = my * inv; nrm[2] = mz * inv;
}

// Geometry outputs of a render (Sec. 6.4, Eq. 10-12); any may be null.
struct GeoMaps {
    float *ns;            // [3,H,W] surfel normal (0 where no surfel)
    float *dsm;           // [H,W] D_smooth
    float *nsm;           // [3,H,W] N_smooth
    float *dg;            // [H,W] D_G
    float *ng;            // [3,H,W] N_G
};

// One 8x4 pixel block of a tile, and its lane's pixel.
// kS surfel samples per pixel: 1 (the centre) or 4 (the 2x2 grid at +-0.25
// px, 4x multisampling of Sec. 5; the Gaussians stay at the centre).
template <int kS>
struct WarpBlock {
    int px, py;
    unsigned need;         // the block's column and row bits in a list entry's cull word
    bool wactive, in_img;
    float u, v, us, vs;    // pixel centre; sample k sits at (us + 0.5 (k & 1), vs + 0.5 (k >> 1))
    __device__ __forceinline__ WarpBlock(const CamParams &C, int tile, int block, unsigned lane)
    {
        // the 8x4 blocks fill the tile row by row
        const int tx = tile % C.tiles_x, ty = tile / C.tiles_x;
        const int wpr = 1 << (C.tsx - 3);          // blocks per tile row
        const int bc = block & (wpr - 1), br = block >> (C.tsx - 3);
        need = (1u << bc) | (1u << (wpr + br));
        const int wx0 = (tx << C.tsx) + bc * kWarpW, wy0 = (ty << C.tsy) + br * kWarpH;
        wactive = wx0 < C.W && wy0 < C.H;        // warp-uniform
        px = wx0 + (int)(lane & 7);
        py = wy0 + (int)(lane >> 3);
        in_img = px < C.W && py < C.H;
        u = px + 0.5f;
        v = py + 0.5f;
        us = kS == 4 ? px + 0.25f : u;
        vs = kS == 4 ? py + 0.25f : v;
    }
};

// Pass 1 state of one lane: per sample the 1/z of the nearest hit (0: none)
// and its surfel id; wmin: the smallest 'best' over the warp's samples.
template <int kS>
struct SurfelZ {
    float best[kS];
    int bid[kS];
    float wmin;
    __device__ __forceinline__ void init(bool in_img)
    {
#pragma unroll
        for (int k = 0; k < kS; ++k) { best[k] = in_img ? 0.f : INFINITY; bid[k] = 0x7fffffff; }
        wmin = 0.f;
    }
};

// A test of one surfel record (planes a0..a2) at the lane's samples: the
// lexicographic (depth, id) min does not depend on the order of the tests.
template <int kS>
__device__ __forceinline__ void surfel_test(const float4 &a0, const float4 &a1, const float4 &a2,
                                            const WarpBlock<kS> &B, float izn, SurfelZ<kS> &z)
{
    const int id = __float_as_int(a2.w);
#pragma unroll
    for (int k = 0; k < kS; ++k) {
        const float du = B.us + 0.5f * (k & 1) - a0.x, dv = B.vs + 0.5f * (k >> 1) - a0.y;
        const float iz = fmaf(a0.w, du, fmaf(a1.x, dv, a0.z));
        const float A = fmaf(a1.y, du, fmaf(a1.z, dv, a1.w));
        const float Bq = fmaf(a2.x, du, fmaf(a2.y, dv, a2.z));
        const float q = fmaf(A, A, fmaf(Bq, Bq, -iz * iz));
        if (q <= 0.f && iz < izn && (iz > z.best[k] || (iz == z.best[k] && id < z.bid[k]))) {
            z.best[k] = iz;
            z.bid[k] = id;
        }
    }
}

// *p = v where on (a predicated store: a branch around it would be divergent)
__device__ __forceinline__ void store_if(bool on, float2 *p, float x, float y)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %0, 0;\n\t@q st.shared.v2.f32 [%1], {%2, %3};\n\t}"
                 :: "r"((int)on), "r"((unsigned)__cvta_generic_to_shared(p)), "f"(x), "f"(y) : "memory");
}

// records that are cheaper tested one at a time than as a batch
template <int kS>
__host__ __device__ constexpr int few_surfels() { return kS == 4 ? 12 : 8; }

// Pass 1 over up to 32 queued records (q[0..n)) at once, a record per lane:
// the lanes evaluate their records at one sample after another (two columns
// per packed FP32 instruction; the same operations per sample as
// surfel_test, so the same bits), a warp maximum finds the sample's nearest
// hit, and the lane that holds it writes (1/z, id) to the sample's slot.  A
// sample hit by two records at exactly the same depth is seen by counting the
// writes, and the batch is then tested record by record.
// Why a record per lane: a record read by all lanes from shared memory (48
// bytes each) holds the SM's load path for 12 cycles per test, more than the
// test's arithmetic (2.85 M tests of a 1080p view: 110 us); here each record is
// read once, and the warp maximum costs one instruction per sample.  With
// staged records and a pixel per lane the raster took 201 us of a 1080p view
// (1M surfels + 300k Gaussians), 208 us of a 4-sample one; with this and the
// tiles in order of length 139 and 143 us.
// The rows are not unrolled: the raster's paths share the instruction cache, and
// four unrolled rows (2.6 % faster when there was one path) left warps without
// instructions 1.9 instead of 0.7 cycles per issue; the orbit batch 3740 -> 3555
// us, a 1080p view's raster 162 -> 157, a 4K one's 663 -> 637.
template <int kS>
__device__ __forceinline__ void surfel_batch(const uint2 *q, float2 *slot, int n, const float4 *__restrict__ rec,
                                             const WarpBlock<kS> &B, float izn, unsigned lane, SurfelZ<kS> &z)
{
    float4 a0 = make_float4(0.f, 0.f, 0.f, 0.f), a1 = make_float4(0.f, 0.f, 0.f, 1.f), a2 = a0;   // A = 1: never inside
    if ((int)lane < n) {
        const float4 *rp = rec + 4 * (int64_t)q[lane].x;
        a0 = rp[0]; a1 = rp[1]; a2 = rp[2];
    }
    bool each = n <= few_surfels<kS>();
    if (!each) {
        constexpr int kCols = kS == 4 ? 16 : 8, kRows = kS == 4 ? 8 : 4;
        constexpr float kStep = kS == 4 ? 0.5f : 1.f;
#pragma unroll
        for (int k = 0; k < kS; ++k) slot[32 * k + lane] = make_float2(0.f, __int_as_float(0x7fffffff));
        __syncwarp();
        const float ub = B.us - kStep * (float)((lane & 7) * (kCols / 8)) - a0.x;       // exact: multiples of 1/256
        const float vb = B.vs - kStep * (float)((lane >> 3) * (kRows / 4)) - a0.y;
        const float2 ub2 = make_float2(ub, ub), gu = make_float2(a0.w, a0.w), ng = make_float2(-a0.w, -a0.w);
        const float2 au = make_float2(a1.y, a1.y), bu = make_float2(a2.x, a2.x);
        int writes = 0;
#pragma unroll 1
        for (int r = 0; r < kRows; ++r) {
            const float dv = vb + kStep * (float)r;
            const float tz = fmaf(a1.x, dv, a0.z), ta = fmaf(a1.z, dv, a1.w), tb = fmaf(a2.y, dv, a2.z);
            const float2 tz2 = make_float2(tz, tz), nz2 = make_float2(-tz, -tz);
            const float2 ta2 = make_float2(ta, ta), tb2 = make_float2(tb, tb);
#pragma unroll
            for (int c = 0; c < kCols; c += 2) {
                const float2 du = __fadd2_rn(ub2, make_float2(kStep * (float)c, kStep * (float)(c + 1)));
                const float2 iz = __ffma2_rn(gu, du, tz2), nz = __ffma2_rn(ng, du, nz2);
                const float2 A = __ffma2_rn(au, du, ta2), Bq = __ffma2_rn(bu, du, tb2);
                const float2 qq = __ffma2_rn(A, A, __ffma2_rn(Bq, Bq, __fmul2_rn(nz, iz)));
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float izh = h ? iz.y : iz.x;
                    const bool in = (h ? qq.y : qq.x) <= 0.f && izh < izn;
                    const int key = in ? __float_as_int(izh) : INT_MIN;    // positive floats order as integers
                    const int best = __reduce_max_sync(0xffffffffu, key);
                    const bool wins = in && key == best;
                    store_if(wins, slot + r * kCols + c + h, izh, a2.w);
                    writes += wins;
                }
            }
        }
        __syncwarp();
        int hits = 0;
        float2 s[kS];
#pragma unroll
        for (int k = 0; k < kS; ++k) {
            // the lane's sample k
            s[k] = kS == 4 ? slot[(2 * (lane >> 3) + (k >> 1)) * kCols + 2 * (lane & 7) + (k & 1)] : slot[lane];
            hits += __float_as_int(s[k].y) != 0x7fffffff;
        }
        __syncwarp();
        each = __reduce_add_sync(0xffffffffu, writes - hits) != 0;
        if (!each) {
#pragma unroll
            for (int k = 0; k < kS; ++k) {
                const int id = __float_as_int(s[k].y);
                if (s[k].x > z.best[k] || (s[k].x == z.best[k] && id < z.bid[k])) {
                    z.best[k] = s[k].x;
                    z.bid[k] = id;
                }
            }
        }
    }
    if (each) {
        for (int j = 0; j < n; ++j) {
            const auto from = [&](float x) { return __shfl_sync(0xffffffffu, x, j); };
            const float4 b0 = make_float4(from(a0.x), from(a0.y), from(a0.z), from(a0.w));
            const float4 b1 = make_float4(from(a1.x), from(a1.y), from(a1.z), from(a1.w));
            const float4 b2 = make_float4(from(a2.x), from(a2.y), from(a2.z), from(a2.w));
            surfel_test<kS>(b0, b1, b2, B, izn, z);
        }
    }
    float bmin = z.best[0];
#pragma unroll
    for (int k = 1; k < kS; ++k) bmin = fminf(bmin, z.best[k]);
    z.wmin = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(bmin)));
}

// The entries of one tile list on their way to one warp: kD groups of 32 (an
// entry per lane) are in flight in shared memory at any time, so that a long
// list is not read one L2 round trip per group (the raster of a view with a
// list of thousands of entries took half as long again with one group ahead).
// A lane copies, waits for and reads its own entries only.
template <int kD>
struct ListRing {
    const uint2 *list;
    uint2 *ring;          // [32 kD], this lane's entry of group g at 32 (g % kD)
    int at, end, g, step; // entry of this lane to copy next; groups taken; entries from group to group
    __device__ __forceinline__ void copy(int slot)
    {
        if (at < end)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;"
                         :: "r"((unsigned)__cvta_generic_to_shared(ring + 32 * slot)), "l"(list + at) : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
        at += step;
    }
    // starts the copies of the first kD groups (group k at beg + st k)
    __device__ __forceinline__ void open(const uint2 *l, int beg, int e, int st, uint2 *r, unsigned lane)
    {
        list = l; ring = r + lane; at = beg + (int)lane; end = e; g = 0; step = st;
#pragma unroll
        for (int k = 0; k < kD; ++k) copy(k);
    }
    // the lane's entry of the next group, (0, 0) past the end
    __device__ __forceinline__ uint2 take()
    {
        asm volatile("cp.async.wait_group %0;" :: "n"(kD - 1) : "memory");
        return at - step * kD < end ? ring[32 * (g % kD)] : make_uint2(0u, 0u);
    }
    // copies a later group in its place (once the entry has been used)
    __device__ __forceinline__ void more()
    {
        copy(g % kD);
        ++g;
    }
};
constexpr int kRing = 8;   // groups of list entries in flight per warp

// Pass 1 over one tile list (opened in ring), by one warp for its own 8x4
// block.  The lanes take 32 entries at a time and queue the ones whose bbox
// touches the block and whose largest 1/z over the disc is not below every
// 1/z the block already holds; 32 queued ones are tested as a batch.  No
// other warp is waited for.
template <int kS>
__device__ __forceinline__ void surfel_pass(ListRing<kRing> &ring, const float4 *__restrict__ rec, int n_list,
                                            const WarpBlock<kS> &B, float izn, unsigned lane, uint2 *q, float2 *slot,
                                            SurfelZ<kS> &z)
{
    int n = 0;
    for (int k = 0; k < n_list; k += ring.step) {
        const uint2 c = ring.take();
        const bool keep = (c.y & B.need) == B.need && !(__uint_as_float(c.y) < z.wmin);
        const unsigned mask = __ballot_sync(0xffffffffu, keep);
        ring.more();
        if (keep) q[n + __popc(mask & ((1u << lane) - 1u))] = c;
        n += __popc(mask);
        __syncwarp();
        if (n < 32) continue;
        surfel_batch<kS>(q, slot, 32, rec, B, izn, lane, z);
        // the ones left over, against the depths found meanwhile
        const bool more = 32 + (int)lane < n;
        const uint2 l = more ? q[32 + lane] : make_uint2(0u, 0u);
        const bool left = more && !(__uint_as_float(l.y) < z.wmin);
        const unsigned lm = __ballot_sync(0xffffffffu, left);
        if (left) q[__popc(lm & ((1u << lane) - 1u))] = l;
        n = __popc(lm);
        __syncwarp();
    }
    if (n) surfel_batch<kS>(q, slot, n, rec, B, izn, lane, z);
    __syncwarp();
}

// Resolve of pass 1: C_s is the mean of the samples' colours (background
// where a sample hits nothing), D_s the nearest sample's depth.
template <int kS>
__device__ __forceinline__ void surfel_resolve(const SurfelZ<kS> &z, bool in_img, const float4 *__restrict__ s_rgb,
                                               const float *bg, float &bmax, float &Ds, float *Cs)
{
    bmax = z.best[0];
#pragma unroll
    for (int k = 1; k < kS; ++k) bmax = fmaxf(bmax, z.best[k]);
    Ds = bmax > 0.f ? 1.f / bmax : INFINITY;
    if (kS == 1) {
        Cs[0] = bg[0]; Cs[1] = bg[1]; Cs[2] = bg[2];
        if (z.bid[0] != 0x7fffffff) {
            const float4 c = s_rgb[z.bid[0]];
            Cs[0] = c.x; Cs[1] = c.y; Cs[2] = c.z;
        }
    } else {
        float sr = 0.f, sgc = 0.f, sb = 0.f;
#pragma unroll
        for (int k = 0; k < kS; ++k) {
            float4 c = make_float4(bg[0], bg[1], bg[2], 0.f);
            if (in_img && z.bid[k] != 0x7fffffff) c = s_rgb[z.bid[k]];
            sr += c.x; sgc += c.y; sb += c.z;
        }
        Cs[0] = sr * (1.f / kS); Cs[1] = sgc * (1.f / kS); Cs[2] = sb * (1.f / kS);
    }
}

// Pass 2 sums of one lane, in 64-bit fixed point: W_G in units of 2^-30
// (each alpha rounded once to that grid), the colour sums in units of 2^-46
// (that alpha times the record colour in 2^-16 units, an exact integer
// product), the geometry sums in units of 2^-32.
struct GaussAcc {
    long long r = 0, g = 0, b = 0, w = 0;
    long long d = 0, nx = 0, ny = 0, nz = 0;   // D_G, N_G (geometry maps)
};

// One Gaussian (its staged planes s) at the lane's pixel (Eq. 2-4).
template <int kS, int kG, bool kGeo>
__device__ __forceinline__ void gauss_test(const float4 *s, const WarpBlock<kS> &B, float Ds, float amin32, float izn,
                                           GaussAcc &acc)
{
    float a, depth, ok;
    unsigned cr, cg, cb;   // record colours, 2^-16 units
    float4 sd = make_float4(0.f, 0.f, 0.f, 0.f);
    if (kG == 2) {
        const float4 r0 = s[0], r1 = s[1], r2 = s[2], x0 = s[4];
        sd = s[5];
        const float du = B.u - r0.x, dv = B.v - r0.y;
        const float iz = fmaf(r0.w, du, fmaf(r1.x, dv, r0.z));
        const float A = fmaf(r1.y, du, fmaf(r1.z, dv, r1.w));
        const float Bq = fmaf(r2.x, du, fmaf(r2.y, dv, r2.z));
        depth = __frcp_rn(iz);
        // rho = (a'^2 + b'^2)/r^2; alpha = 2^(log2 sigma' + log2(alpha_min/sigma') rho)
        const float rho = fmaf(A, A, Bq * Bq) * (depth * depth);
        a = ex2_approx(fmaf(sd.w, rho, x0.w));
        cr = __float_as_uint(x0.x); cg = __float_as_uint(x0.y); cb = __float_as_uint(x0.z);
        ok = (iz > 0.f && iz < izn && depth - s[3].w < Ds) ? 1.f : 0.f;
    } else {
        const GaussRec g = gauss_rec3(s[0], s[1], s[2]);
        float ex;
        a = gauss_alpha(g, B.u, B.v, ex);
        cr = __float_as_uint(g.r); cg = __float_as_uint(g.g); cb = __float_as_uint(g.b);
        ok = g.key < Ds ? 1.f : 0.f;
        if (kGeo) { sd = s[3]; depth = sd.w; }
    }
    // alpha * 2^32 is exact scaling: the clamp decision equals alpha >= alpha_min
    const float a32 = fminf(a * 4294967296.f, kAlpha32Max);
    if (B.in_img && a32 >= amin32 && ok != 0.f) {
        // alpha on the 2^-30 grid (alpha <= 2: below 2^31), one conversion;
        // the colour terms are exact 32 x 32 -> 64-bit products
        const unsigned A = __float2uint_rn(fminf(a, 2.f) * 1073741824.f);
        acc.w += A;
        acc.r += (long long)((unsigned long long)A * cr);
        acc.g += (long long)((unsigned long long)A * cg);
        acc.b += (long long)((unsigned long long)A * cb);
        if (kGeo) {
            acc.d += __float2ll_rn(a32 * depth);
            acc.nx += f2ll_rn(a32 * sd.x);
            acc.ny += f2ll_rn(a32 * sd.y);
            acc.nz += f2ll_rn(a32 * sd.z);
        }
    }
}

// Copies Gaussian id's planes to d.
template <int kG, bool kGeo>
__device__ __forceinline__ void stage_gauss(const float4 *__restrict__ rec, const float4 *__restrict__ side, int64_t id,
                                            float4 *d)
{
    const float4 *rp = rec + 4 * id;
    const float4 r0 = rp[0], r1 = rp[1], r2 = rp[2];
    d[0] = r0; d[1] = r1; d[2] = r2;
    if (kG == 3 && kGeo) d[3] = side[2 * id];
    if (kG == 2) {
        const float4 r3 = rp[3], x0 = side[2 * id], x1 = side[2 * id + 1];
        d[3] = r3; d[4] = x0; d[5] = x1;
    }
}

// Pass 2 over n queued Gaussians (q[0..n)): the lanes copy a record each into
// the warp's shared slots, then every lane evaluates them at its pixel.
template <int kS, int kG, bool kGeo>
__device__ __forceinline__ void gauss_batch(const uint2 *q, int n, const float4 *__restrict__ rec,
                                            const float4 *__restrict__ side, const WarpBlock<kS> &B, float Ds,
                                            float amin32, float izn, unsigned lane, float4 *st, GaussAcc &acc)
{
    constexpr int kQ = gauss_planes<kG, kGeo>();
    if ((int)lane < n) stage_gauss<kG, kGeo>(rec, side, q[lane].x, st + kQ * lane);
    __syncwarp();
    const float4 *s = st;
    for (int j = 0; j < n; ++j, s += kQ) gauss_test<kS, kG, kGeo>(s, B, Ds, amin32, izn, acc);
    __syncwarp();
}

// Pass 2 over one tile list (opened in ring), queued as in pass 1.  No
// Gaussian with key >= wmaxD (the max over the warp's pixels of D_s) can pass
// the depth test there.
template <int kS, int kG, bool kGeo>
__device__ __forceinline__ void gauss_pass(ListRing<kRing> &ring, const float4 *__restrict__ rec,
                                           const float4 *__restrict__ side, int n_list, const WarpBlock<kS> &B,
                                           float Ds, float wmaxD, float amin32, float izn, unsigned lane, uint2 *q,
                                           float4 *st, GaussAcc &acc)
{
    int n = 0;
    for (int k = 0; k < n_list; k += ring.step) {
        const uint2 c = ring.take();
        const bool keep = (c.y & B.need) == B.need && !(__uint_as_float(c.y) >= wmaxD);
        const unsigned mask = __ballot_sync(0xffffffffu, keep);
        ring.more();
        if (keep) q[n + __popc(mask & ((1u << lane) - 1u))] = c;
        n += __popc(mask);
        __syncwarp();
        if (n < 32) continue;
        gauss_batch<kS, kG, kGeo>(q, 32, rec, side, B, Ds, amin32, izn, lane, st, acc);
        n -= 32;
        const uint2 l = q[32 + lane];
        __syncwarp();
        if ((int)lane < n) q[lane] = l;
    }
    if (n) {
        __syncwarp();
        gauss_batch<kS, kG, kGeo>(q, n, rec, side, B, Ds, amin32, izn, lane, st, acc);
    }
}

// Composite (Eq. 5) of one pixel and its outputs.
template <int kS, bool kGeo>
__device__ __forceinline__ void composite_store(const CamParams &C, const OptParams &O, const ViewScratch &X,
                                                const WarpBlock<kS> &B, const SurfelZ<kS> &z, float bmax, float Ds,
                                                const float *Cs, const GaussAcc &acc, float *__restrict__ out_rgb,
                                                float *__restrict__ out_depth, int32_t *__restrict__ out_id,
                                                float *__restrict__ aux, const GeoMaps &geo)
{
    const float k32 = 2.3283064365386963e-10f;   // 2^-32
    const float k30 = 9.3132257461547852e-10f;   // 2^-30
    const float k46 = 1.4210854715202004e-14f;   // 2^-46
    const float WG = __ll2float_rn(acc.w) * k30;
    const float CG[3] = {__ll2float_rn(acc.r) * k46, __ll2float_rn(acc.g) * k46, __ll2float_rn(acc.b) * k46};
    float out[3];
    if (O.mode == GES_MODE_FULL) {
        const float inv = 1.f / (1.f + WG);
        for (int c = 0; c < 3; ++c) out[c] = (Cs[c] + CG[c]) * inv;
    } else if (O.mode == GES_MODE_SURFELS_ONLY) {
        for (int c = 0; c < 3; ++c) out[c] = Cs[c];
    } else {
        for (int c = 0; c < 3; ++c) out[c] = WG > 0.f ? CG[c] / WG : C.bg[c];
    }
    const int64_t HW = (int64_t)C.W * C.H, pix = (int64_t)B.py * C.W + B.px;
    out_rgb[pix] = out[0];
    out_rgb[HW + pix] = out[1];
    out_rgb[2 * HW + pix] = out[2];
    if (out_depth) out_depth[pix] = Ds;
    if (out_id) {
#pragma unroll
        for (int k = 0; k < kS; ++k) out_id[k * HW + pix] = z.bid[k] != 0x7fffffff ? z.bid[k] : -1;
    }
    if (aux) aux[pix] = WG;
    if (kGeo) {
        // Eq. 10-12 with W_s = 1 where a surfel covers the pixel, 0 elsewhere
        float ns[3] = {0.f, 0.f, 0.f};
        const bool covered = bmax > 0.f;
        if (covered) {
            // the nearest sample's surfel (lowest id on a tie)
            int w = 0x7fffffff;
#pragma unroll
            for (int k = 0; k < kS; ++k)
                if (z.best[k] == bmax && z.bid[k] < w) w = z.bid[k];
            surfel_normal(X.s_rec, w, C, ns);
        }
        const float DG = __ll2float_rn(acc.d) * k32;
        const float NG[3] = {__ll2float_rn(acc.nx) * k32, __ll2float_rn(acc.ny) * k32, __ll2float_rn(acc.nz) * k32};
        const float ws = covered ? 1.f : 0.f, wt = ws + WG;
        if (geo.dg) geo.dg[pix] = DG;
        if (geo.dsm) geo.dsm[pix] = wt > 0.f ? ((covered ? Ds : 0.f) + DG) / wt : INFINITY;
        for (int c = 0; c < 3; ++c) {
            if (geo.ns) geo.ns[c * HW + pix] = ns[c];
            if (geo.ng) geo.ng[c * HW + pix] = NG[c];
            if (geo.nsm) geo.nsm[c * HW + pix] = wt > 0.f ? (ws * ns[c] + NG[c]) / wt : 0.f;
        }
    }
}

// Shared space of one raster warp.
template <int kS, int kG, bool kGeo>
struct __align__(16) WarpSpace {
    union {
        float2 slot[32 * kS];                          // pass 1: the batch's winners; a shared block's z-buffer
        float4 st[32 * gauss_planes<kG, kGeo>()];      // pass 2: staged records
        long long sum[32 * (kGeo ? 8 : 4)];            // a shared block's sums
    };
    uint2 q[64];                                       // entries kept for the next batch
    uint2 ring[32 * kRing];
};
constexpr int kRasterWarps = kRasterThreads / 32;

__device__ __forceinline__ void tile_lists(const ViewScratch &X, const OptParams &O, int tile, int2 &sr, int2 &gr)
{
    sr = O.mode != GES_MODE_GAUSSIANS_ONLY ? X.s_rng[tile] : make_int2(0, 0);
    gr = O.mode != GES_MODE_SURFELS_ONLY ? X.g_rng[tile] : make_int2(0, 0);
}

// 8x4 blocks block, block + 1, ... of a tile whose lists have at most
// 32 entries each, by one warp: an entry per lane of both lists at once, their
// records staged once and tested one after another; no queue and no ring.
// A block of few primitives is bound by its chain of dependent reads and by
// the instructions around its tests.  Through the queues of raster_block the
// raster of a 1890x1002 view of 104k surfels took 57 us, this 46; with four
// samples and 2D Gaussians (3733x1917, 119k primitives) 277 and 215 us.
template <int kS, int kG, bool kGeo>
__device__ __forceinline__ void raster_short(const ViewScratch &X, const CamParams &C, const OptParams &O,
                                             float *__restrict__ out_rgb, float *__restrict__ out_depth,
                                             int32_t *__restrict__ out_id, float *__restrict__ aux,
                                             const GeoMaps &geo, int tile, int block, int blocks, const int2 &sr,
                                             const int2 &gr, WarpSpace<kS, kG, kGeo> &w)
{
    constexpr int kQ = gauss_planes<kG, kGeo>();
    static_assert(32 * 3 * sizeof(float4) <= sizeof(w.ring), "staged surfels");
    const unsigned lane = lane_id();
    uint2 se = make_uint2(0u, 0u), ge = make_uint2(0u, 0u);
    if ((int)lane < sr.y - sr.x) se = X.s_list[sr.x + (int)lane];
    if ((int)lane < gr.y - gr.x) ge = X.g_list[gr.x + (int)lane];
    const auto touches = [](unsigned word, unsigned need) { return (word & need) == need; };
    const unsigned need = blocks == 1 ? WarpBlock<kS>(C, tile, block, lane).need : 0u;
    float4 *ss = reinterpret_cast<float4 *>(w.ring);
    // (an entry's word is not 0: it names the blocks it touches)
    if (se.y && touches(se.y, need)) {
        const float4 *rp = X.s_rec + 4 * (int64_t)se.x;
        float4 *d = ss + 3 * lane;
        const float4 r0 = rp[0], r1 = rp[1], r2 = rp[2];
        d[0] = r0; d[1] = r1; d[2] = r2;
    }
    if (ge.y && touches(ge.y, need)) stage_gauss<kG, kGeo>(X.g_rec, X.g_aux, ge.x, w.st + kQ * lane);
    __syncwarp();
#pragma unroll 1
    for (int b = block; b < block + blocks; ++b) {
        const WarpBlock<kS> B(C, tile, b, lane);
        if (!B.wactive) continue;
        SurfelZ<kS> z;
        z.init(B.in_img);
        for (unsigned m = __ballot_sync(0xffffffffu, touches(se.y, B.need)); m; m &= m - 1u) {
            const float4 *r = ss + 3 * (__ffs(m) - 1);
            surfel_test<kS>(r[0], r[1], r[2], B, C.izn, z);
        }
        float bmax, Ds, Cs[3];
        surfel_resolve<kS>(z, B.in_img, X.s_rgb, C.bg, bmax, Ds, Cs);
        GaussAcc acc;
        for (unsigned m = __ballot_sync(0xffffffffu, touches(ge.y, B.need)); m; m &= m - 1u)
            gauss_test<kS, kG, kGeo>(w.st + kQ * (__ffs(m) - 1), B, Ds, O.alpha_min * 4294967296.f, C.izn, acc);
        if (B.in_img)
            composite_store<kS, kGeo>(C, O, X, B, z, bmax, Ds, Cs, acc, out_rgb, out_depth, out_id, aux, geo);
    }
    __syncwarp();       // the staged records are read: the space is free
}

// One 8x4 block: both passes and the composite, by one warp, or (kShared) by
// all warps of the CTA: each takes every eighth group of the lists, and the
// z-buffers (a lexicographic min) and the sums (exact integers) are merged, so
// the result is the same to the bit.  kG: 3D Gaussians (EWA splats) or 2D
// Gaussians of 2D-GES (ray-splat hit, planar depth).  kGeo: also the geometry
// maps of Eq. 10-12.  space: the CTA's warps' shared space.
template <int kS, int kG, bool kGeo, bool kShared>
__device__ __forceinline__ void raster_block(const ViewScratch &X, const CamParams &C, const OptParams &O,
                                             float *__restrict__ out_rgb, float *__restrict__ out_depth,
                                             int32_t *__restrict__ out_id, float *__restrict__ aux,
                                             const GeoMaps &geo, int tile, int block, const int2 &sr, const int2 &gr,
                                             WarpSpace<kS, kG, kGeo> *space)
{
    const unsigned lane = lane_id(), warp = threadIdx.x >> 5;
    WarpSpace<kS, kG, kGeo> &w = space[warp];
    const WarpBlock<kS> B(C, tile, block, lane);
    if (!B.wactive) return;
    const int first = kShared ? 32 * (int)warp : 0, step = kShared ? 32 * kRasterWarps : 32;
    ListRing<kRing> ring;
    ring.open(X.s_list, sr.x + first, sr.y, step, w.ring, lane);

    // ---------------- pass 1: surfel z-buffer ----------------
    SurfelZ<kS> z;
    z.init(B.in_img);
    surfel_pass<kS>(ring, X.s_rec, sr.y - sr.x - first, B, C.izn, lane, w.q, w.slot, z);
    ring.open(X.g_list, gr.x + first, gr.y, step, w.ring, lane);   // on its way while pass 1 resolves
    if (kShared) {
#pragma unroll
        for (int k = 0; k < kS; ++k) w.slot[32 * k + lane] = make_float2(z.best[k], __int_as_float(z.bid[k]));
        __syncthreads();
        for (int o = 0; o < kRasterWarps; ++o)
#pragma unroll
            for (int k = 0; k < kS; ++k) {
                const float2 v = space[o].slot[32 * k + lane];
                const int id = __float_as_int(v.y);
                if (v.x > z.best[k] || (v.x == z.best[k] && id < z.bid[k])) { z.best[k] = v.x; z.bid[k] = id; }
            }
        __syncthreads();
    }
    float bmax, Ds, Cs[3];
    surfel_resolve<kS>(z, B.in_img, X.s_rgb, C.bg, bmax, Ds, Cs);

    // ---------------- pass 2: Gaussians (Eq. 2-4) ----------------
    GaussAcc acc;
    const float wmaxD = __uint_as_float(__reduce_max_sync(0xffffffffu, B.in_img ? __float_as_uint(Ds) : 0u));
    gauss_pass<kS, kG, kGeo>(ring, X.g_rec, X.g_aux, gr.y - gr.x - first, B, Ds, wmaxD, O.alpha_min * 4294967296.f,
                             C.izn, lane, w.q, w.st, acc);
    if (kShared) {
        long long *v = w.sum + lane;
        v[0] = acc.w; v[32] = acc.r; v[64] = acc.g; v[96] = acc.b;
        if (kGeo) { v[128] = acc.d; v[160] = acc.nx; v[192] = acc.ny; v[224] = acc.nz; }
        __syncthreads();
        if (warp == 0)
            for (int o = 1; o < kRasterWarps; ++o) {
                const long long *u = space[o].sum + lane;
                acc.w += u[0]; acc.r += u[32]; acc.g += u[64]; acc.b += u[96];
                if (kGeo) { acc.d += u[128]; acc.nx += u[160]; acc.ny += u[192]; acc.nz += u[224]; }
            }
        __syncthreads();
        if (warp != 0) return;
    }
    if (!B.in_img) return;
    composite_store<kS, kGeo>(C, O, X, B, z, bmax, Ds, Cs, acc, out_rgb, out_depth, out_id, aux, geo);
}

template <int kS, int kG, bool kGeo>
__global__ void __launch_bounds__(kRasterThreads, kRasterCtas)
    k_raster(ViewScratch X, CamParams C, OptParams O, float *__restrict__ out_rgb, float *__restrict__ out_depth,
             int32_t *__restrict__ out_id, float *__restrict__ aux, GeoMaps geo)
{
    __shared__ WarpSpace<kS, kG, kGeo> space[kRasterWarps];
    // one CTA per item (persistent CTAs that take items from a counter took 10 %
    // longer: two barriers per item); the grid has room for the most there can be,
    // and the order array for the grid, so that its word is read with the status
    unsigned item = blockIdx.x;
    if (X.order) item = X.order[blockIdx.x];
    if (X.status[ST_FLAGS] & (FLAG_SOVF | FLAG_GOVF)) return;
    if (X.order && blockIdx.x >= X.status[ST_ITEMS]) return;
    const int tile = (int)(item & 0xffffffu), warp = (int)threadIdx.x >> 5;
    static_assert(kRasterWarps == kOrderItems, "a warp per block of a tile");
    int2 sr, gr;
    tile_lists(X, O, tile, sr, gr);
    if (item >> 24)
        raster_block<kS, kG, kGeo, true>(X, C, O, out_rgb, out_depth, out_id, aux, geo, tile, (int)(item >> 24) - 1,
                                         sr, gr, space);
    else if (short_lists(sr, gr))
        raster_short<kS, kG, kGeo>(X, C, O, out_rgb, out_depth, out_id, aux, geo, tile, warp, 1, sr, gr, space[warp]);
    else
        raster_block<kS, kG, kGeo, false>(X, C, O, out_rgb, out_depth, out_id, aux, geo, tile, warp, sr, gr, space);
}

// ---------------------------------------------------------------------------
// batch: each phase is one launch over all views of all scenes

// largest v with base(v) <= x (bases ascending, base(0) = 0)
template <typename F>
__device__ __forceinline__ int find_view(int n, int x, F base)
{
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (base(mid) <= x) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// The same by a warp, from view lo on: 32 views are compared at a time (two
// dependent reads among 1024 views instead of ten).
template <class F>
__device__ __forceinline__ int warp_find_view(int lo, int n, int x, F base)
{
    int hi = n - 1;
    while (lo < hi) {
        const int step = (hi - lo + 31) >> 5, k = lo + ((int)lane_id() + 1) * step;
        lo += step * __popc(__ballot_sync(0xffffffffu, k <= hi && base(k) <= x));
        hi = min(hi, lo + step - 1);
    }
    return lo;
}

__device__ __forceinline__ void load_view(const BatchView *V, int v, BatchView &dst)
{
    const int *src = reinterpret_cast<const int *>(V + v);
    int *d = reinterpret_cast<int *>(&dst);
    for (int k = threadIdx.x; k < (int)(sizeof(BatchView) / 4); k += blockDim.x) d[k] = src[k];
}

// Preprocess of all views, one launch per primitive kind (kKind 1: the
// surfel ranges, 2: the Gaussian ranges); CTA x of the launch takes the view
// and the range of map[x].  The two set-ups need different registers, and a
// kernel per kind keeps the one from spilling for the other.  kCol: the
// colours too (a batch whose scenes each have one view; otherwise the colour
// pass evaluates them for all views of a scene at once).
template <int kGd, int kKind, int kCol>
__global__ void __launch_bounds__(kPrepThreads, 2) k_bprep(const BatchView *V, const int2 *__restrict__ map,
                                                          OptParams O, unsigned long long *t0)
{
    extern __shared__ __align__(16) unsigned hist[];
    __shared__ unsigned vcnt;
    __shared__ __align__(16) unsigned char bv_raw[sizeof(BatchView)];
    BatchView &bv = *reinterpret_cast<BatchView *>(bv_raw);
    __shared__ int2 sm;
    if (threadIdx.x == 0) {
        // the first CTA to start stamps the batch's start time (t0 is zeroed per launch)
        atomicCAS(t0, 0ull, global_timer_ns());
        sm = map[blockIdx.x];
    }
    __syncthreads();
    load_view(V, sm.x, bv);
    __syncthreads();
    prep_local_body<kGd, false, kKind, kCol>(bv.S, bv.C, O, bv.X, bv.B, sm.y, hist, vcnt);
}

// Colour pass of the batch (Eq. 1): one thread per primitive of one kind,
// for every view of its view group (the views of one scene).  The SH row and
// the position are read once; the views' camera centres and output arrays
// are staged in shared memory kColourViews at a time.  Per view, the
// direction from the centre to that view's camera, the basis and the colour
// are evaluated with the same operations, in the same order, as the inline
// set-up of the per-view path, so both paths store bit-identical colours.
// Surfels: the view's colour array; Gaussians: the view's Gaussian colour
// array in 2^-16 units (dense 16-byte stores; the set-up, which runs after
// this pass, copies them into the records).  Primitives a view does not draw
// get colours that nothing reads.
template <int K>
__device__ __forceinline__ void colour_views(const BatchView *V, const int *__restrict__ gview, int gofs, int gn,
                                             bool surf, int64_t i, bool act, const SceneView &S, float4 *s_cam,
                                             float4 **s_out)
{
    float px = 0.f, py = 0.f, pz = 0.f, c[3 * K];
    if (act) {
        const float *pos = surf ? S.s_pos : S.g_pos;
        px = __ldg(pos + 3 * i); py = __ldg(pos + 3 * i + 1); pz = __ldg(pos + 3 * i + 2);
        load_sh_row<K>(surf ? S.s_sh : S.g_sh, i, S.sh_dtype, c);
    }
    for (int k0 = 0; k0 < gn; k0 += kColourViews) {
        const int m = min(kColourViews, gn - k0);
        __syncthreads();
        if ((int)threadIdx.x < m) {
            const BatchView *bv = V + __ldg(gview + gofs + k0 + threadIdx.x);
            s_cam[threadIdx.x] = make_float4(bv->C.ocam[0], bv->C.ocam[1], bv->C.ocam[2], 0.f);
            s_out[threadIdx.x] = surf ? bv->X.s_rgb : bv->X.g_col;
        }
        __syncthreads();
        if (!act) continue;
        for (int k = 0; k < m; ++k) {
            const float4 o = s_cam[k];
            float dir[3], L;
            view_dir_o(o.x, o.y, o.z, px, py, pz, dir, L);
            float Y[16];
            sh_basis(K, dir[0], dir[1], dir[2], Y);
            float r = 0.5f, g = 0.5f, b = 0.5f;
#pragma unroll
            for (int q = 0; q < K; ++q) {
                r = fmaf(c[3 * q], Y[q], r);
                g = fmaf(c[3 * q + 1], Y[q], g);
                b = fmaf(c[3 * q + 2], Y[q], b);
            }
            r = fmaxf(r, 0.f); g = fmaxf(g, 0.f); b = fmaxf(b, 0.f);
            s_out[k][i] = surf ? make_float4(r, g, b, 0.f) : make_float4(colour_q(r), colour_q(g), colour_q(b), 0.f);
        }
    }
}

__global__ void __launch_bounds__(kColourThreads) k_bcolour(const BatchView *V, const int4 *__restrict__ items,
                                                            const int *__restrict__ gview, unsigned long long *t0)
{
    __shared__ float4 s_cam[kColourViews];
    __shared__ float4 *s_out[kColourViews];
    // the first CTA to start stamps the batch's start time (t0 is zeroed per launch)
    if (threadIdx.x == 0) atomicCAS(t0, 0ull, global_timer_ns());
    const int4 it = items[blockIdx.x];
    const bool surf = it.x == 0;
    const SceneView &S = V[__ldg(gview + it.y)].S;
    const int64_t i = (int64_t)it.w + threadIdx.x;
    const bool act = i < (surf ? S.N : S.M);
    switch ((S.deg + 1) * (S.deg + 1)) {
    case 16: colour_views<16>(V, gview, it.y, it.z, surf, i, act, S, s_cam, s_out); break;
    case 9: colour_views<9>(V, gview, it.y, it.z, surf, i, act, S, s_cam, s_out); break;
    case 4: colour_views<4>(V, gview, it.y, it.z, surf, i, act, S, s_cam, s_out); break;
    default: colour_views<1>(V, gview, it.y, it.z, surf, i, act, S, s_cam, s_out); break;
    }
}

__global__ void __launch_bounds__(256) k_bcolscan(const BatchView *V, int n)
{
    __shared__ unsigned part[9][kColTiles + 1];
    __shared__ __align__(16) unsigned char bv_raw[sizeof(BatchView)];
    BatchView &bv = *reinterpret_cast<BatchView *>(bv_raw);
    __shared__ int sv;
    if (threadIdx.x == 0) sv = find_view(n, blockIdx.x, [&](int k) { return V[k].colscan_base; });
    __syncthreads();
    load_view(V, sv, bv);
    __syncthreads();
    colscan_body<8>(bv.X, bv.T, bv.B, blockIdx.x - bv.colscan_base, blockIdx.y == 0, part);
}

__global__ void __launch_bounds__(kFillThreads, 2) k_bfill(const BatchView *V, int n, int lb)
{
    extern __shared__ unsigned cur[];
    __shared__ __align__(16) unsigned char bv_raw[sizeof(BatchView)];
    BatchView &bv = *reinterpret_cast<BatchView *>(bv_raw);
    __shared__ int sv;
    // the first n CTAs: the views' tile orders
    const int c = (int)blockIdx.x - n;
    if (threadIdx.x == 0) sv = c < 0 ? c + n : find_view(n, c, [&](int k) { return V[k].prep_base; });
    __syncthreads();
    load_view(V, sv, bv);
    __syncthreads();
    if (c < 0) {
        // list entries of all views (their status words lie together)
        __shared__ unsigned long long total;
        if (threadIdx.x == 0) total = 0ull;
        __syncthreads();
        unsigned *st = bv.X.status - (size_t)sv * ST_WORDS;
        unsigned long long mine = 0ull;
        for (int v = threadIdx.x; v < n; v += kFillThreads)
            mine += (unsigned long long)st[(size_t)v * ST_WORDS + ST_SPAIRS] + st[(size_t)v * ST_WORDS + ST_GPAIRS];
        for (int d = 16; d > 0; d >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, d);
        if (lane_id() == 0 && mine) atomicAdd(&total, mine);
        __syncthreads();
        const uint2 c2 = order_body<ORDER_BATCH>(bv.X, bv.T, total, cur);
        if (threadIdx.x == 0) {
            // lists that overflowed: all tiles are counted, none is drawn
            const bool skip = bv.X.status[ST_FLAGS] & (FLAG_SOVF | FLAG_GOVF);
            const unsigned shared = skip ? 0u : c2.x, few = skip ? (unsigned)bv.T : c2.y;
            bv.X.status[ST_ITEMS] = shared | few << 16;
            bv.X.status[ST_LEFT] = batch_items(bv.T, shared, few, lb);
            if (shared) st[(size_t)n * ST_WORDS + BW_SHARED] = 1u;
        }
    }
    else fill_local_body(bv.X, bv.T, bv.C.tiles_x, bv.C.tsx, bv.C.tsy, bv.B, c - bv.prep_base, cur, false);
}

// Persistent raster over the tiles of the whole batch.  First the shared tiles
// of every view (order_body), their blocks dealt out to the CTAs; then the other
// tiles, by warps that wait for no other and take items until none is left, so
// uneven views balance across the GPU.
// An item is a block of a tile (with whole tiles five uneven scenes of at most
// 1000x600 pixels took 958 us instead of 582), or half or all of a tile of short
// lists (1 << lb blocks), whose records the warp stages once for these blocks.
// Each view has a counter; a warp takes items of one view until none is left,
// then of another.  One counter for the batch, an item per block everywhere
// and every block counted at its view by an atomic that the warp waited for
// bounded batches of sparse views: eight 1080p views of 126k primitives took 650
// us of raster, with a counter per view 370, 256 views of 256x192 460 and 225, the
// 16-view orbit 2460 and 2400 (now 360, 200 and 2190, with pass 1's rows rolled up).
// kOne: a small batch (of `tiles` tiles, a few blocks for each warp) and one
// counter, a block per item, the views in turn: there the last long blocks decide,
// and four uneven views of at most 750x565 pixels (1.4M primitives) take 190 us so,
// 215 with a counter per view.
template <int kS, int kG, bool kIds, bool kOne>
__global__ void __launch_bounds__(kRasterThreads, kRasterCtas) k_braster(const BatchView *V, int n, OptParams O,
                                                                        unsigned *bw, int lb, int tiles)
{
    __shared__ WarpSpace<kS, kG, false> space[kRasterWarps];
    __shared__ __align__(16) unsigned char bv_raw[kRasterWarps][sizeof(BatchView)];
    const unsigned warp = threadIdx.x >> 5;
    BatchView &bv = *reinterpret_cast<BatchView *>(bv_raw[warp]);    // the warp's view
    const auto load = [&](int v) {
        __syncwarp();
        const int *src = reinterpret_cast<const int *>(V + v);
        int *d = reinterpret_cast<int *>(bv_raw[warp]);
        for (int k = lane_id(); k < (int)(sizeof(BatchView) / 4); k += 32) d[k] = src[k];
        __syncwarp();
    };
    // per-view completion time: whoever finishes the view's last blocks stamps it
    const auto retire = [&](unsigned blocks) {
        const unsigned all = (unsigned)bv.T * kOrderItems;
        if (lane_id() == 0 && blocks && atomicAdd(bv.X.status + ST_RETIRED, blocks) + blocks == all)
            *reinterpret_cast<unsigned long long *>(bv.X.status + ST_TDONE) = global_timer_ns();
    };
    // the views with shared tiles, found 32 at a time (a view at a time, two
    // dependent reads each, a batch of 1024 small views took 0.4 ms to look)
    unsigned dealt = blockIdx.x;     // the CTA's next one among the shared blocks of all views
    const unsigned *st = V[0].X.status;      // (the views' status words lie together)
    for (int v0 = bw[BW_SHARED] ? 0 : n; v0 < n; v0 += 32) {
        const int vl = v0 + (int)lane_id();
        unsigned mine = 0u;
        if (vl < n) mine = st[(size_t)vl * ST_WORDS + ST_ITEMS] & 0xffffu;
        for (unsigned m = __ballot_sync(0xffffffffu, mine != 0u); m; m &= m - 1u) {
            const int o = __ffs(m) - 1;
            const unsigned shared = __shfl_sync(0xffffffffu, mine, o) * kOrderItems;
            if (dealt < shared) load(v0 + o);
            for (; dealt < shared; dealt += gridDim.x) {
                const int tile = (int)bv.X.order[dealt / kOrderItems];
                int2 sr, gr;
                tile_lists(bv.X, O, tile, sr, gr);
                raster_block<kS, kG, false, true>(bv.X, bv.C, O, bv.rgb, bv.depth, kIds ? bv.id : nullptr,
                                                  kIds ? bv.aux : nullptr, GeoMaps{}, tile, (int)(dealt % kOrderItems),
                                                  sr, gr, space);
                if (warp == 0) retire(1u);
            }
            dealt -= shared;
        }
    }
    // blocks block, block + 1, ... of tile number k of the view's order
    const auto raster = [&](unsigned k, int block, int blocks, bool brief) {
        const int tile = (int)bv.X.order[k];
        int32_t *const id = kIds ? bv.id : nullptr;
        float *const aux = kIds ? bv.aux : nullptr;
        int2 sr, gr;
        tile_lists(bv.X, O, tile, sr, gr);
        if (brief)
            raster_short<kS, kG, false>(bv.X, bv.C, O, bv.rgb, bv.depth, id, aux, GeoMaps{}, tile, block, blocks, sr,
                                        gr, space[warp]);
        else
            raster_block<kS, kG, false, false>(bv.X, bv.C, O, bv.rgb, bv.depth, id, aux, GeoMaps{}, tile, block, sr,
                                               gr, space);
    };
    // What a warp keeps of its view from item to item, in shared memory: nothing of
    // it holds a register through the raster.
    struct Own {
        int v;
        unsigned done;                  // blocks done, not yet counted at the view (lane 0's)
        unsigned shared, few;           // the view's shared and short tiles
        bool skip;                      // its lists overflowed
    };
    __shared__ Own own[kRasterWarps];
    volatile Own &my = own[warp];
    const auto enter = [&](int v) {
        load(v);
        const unsigned w = bv.X.status[ST_ITEMS];
        my.v = v;
        my.done = 0u;
        my.shared = w & 0xffffu;
        my.few = w >> 16;
        my.skip = bv.X.status[ST_FLAGS] & (FLAG_SOVF | FLAG_GOVF);
        __syncwarp();
    };
    // (the next item is always taken before this one is rastered, and used after
    // it: the atomic's round trip overlaps the raster)
    if constexpr (kOne) {
        unsigned at = 0;
        if (lane_id() == 0) at = atomicAdd(bw + BW_NEXT, 1u);
        at = __shfl_sync(0xffffffffu, at, 0);
        my.v = -1;
        while (at < (unsigned)tiles * kOrderItems) {
            unsigned nxt = 0;
            if (lane_id() == 0) nxt = atomicAdd(bw + BW_NEXT, 1u);
            if (my.v < 0 || (int)(at / kOrderItems) >= bv.tile_base + bv.T) {
                if (my.v >= 0) retire(my.done);
                const int v = warp_find_view(max(my.v, 0), n, (int)(at / kOrderItems), [&](int k) { return V[k].tile_base; });
                enter(v);
            }
            const unsigned k = at / kOrderItems - (unsigned)bv.tile_base;
            if (k >= my.shared) {
                if (lane_id() == 0) my.done = my.done + 1u;
                if (!my.skip) raster(k, (int)(at % kOrderItems), 1, k >= (unsigned)bv.T - my.few);
            }
            at = __shfl_sync(0xffffffffu, nxt, 0);
        }
        if (my.v >= 0) retire(my.done);
    } else {
        // A view with items left, by their numbers: the takers (CTAs, later warps)
        // spread over the views as the work does (evenly, or to the next view with
        // any items, they went from one small view to another), but no farther than
        // 32 items for each warp, so that the first views are also done first (eight
        // uneven scenes: the smallest done after 1.58 ms without this limit; the
        // batch's time is the same, with 16 items it grows by 2 %, with 8 by 6 %).
        const int windows = (n + 31) >> 5;
        const unsigned ahead = 32u * gridDim.x * kRasterWarps;
        int from = (int)((uint64_t)blockIdx.x * windows / gridDim.x) * 32;     // the 32 views looked at
        const auto pick = [&](unsigned taker, unsigned takers) {
            for (int r = 0; r < windows; ++r) {
                const int u = from + (int)lane_id();
                unsigned incl = u < n ? (unsigned)max((int)__ldcg(st + (size_t)u * ST_WORDS + ST_LEFT), 0) : 0u;
                for (int d = 1; d < 32; d <<= 1) {
                    const unsigned y = __shfl_up_sync(0xffffffffu, incl, d);
                    if ((int)lane_id() >= d) incl += y;
                }
                const unsigned all = __shfl_sync(0xffffffffu, incl, 31);
                const unsigned k = (unsigned)((uint64_t)taker * min(all, ahead) / takers);
                if (all) return from + __ffs(__ballot_sync(0xffffffffu, incl > k)) - 1;
                from = from + 32 < n ? from + 32 : 0;
            }
            return -1;
        };
        const auto take = [&](int v, int items) {
            return atomicSub(reinterpret_cast<int *>(V[0].X.status) + (size_t)v * ST_WORDS + ST_LEFT, items);
        };
        // the first items are taken by the CTA, one for each warp (4864 warps that
        // picked and took for themselves waited 10 us for the counters' lines)
        __shared__ int first_v, first_at;
        __syncthreads();
        if (warp == 0) {
            const int v = pick(blockIdx.x, gridDim.x);
            if (lane_id() == 0) {
                first_v = v;
                if (v >= 0) first_at = take(v, kRasterWarps);
            }
        }
        __syncthreads();
        int v = first_v, at = first_at - (int)warp;
        while (v >= 0) {
            enter(v);
            while (at > 0) {
                int nxt = 0;
                if (lane_id() == 0) nxt = atomicSub(reinterpret_cast<int *>(bv.X.status + ST_LEFT), 1);
                // a block of a longer tile, or 1 << lb blocks of a short one
                const unsigned shared = my.shared, few = my.few, cut = (bv.T - shared - few) * kOrderItems;
                const unsigned i = (unsigned)(batch_items(bv.T, shared, few, lb) - at);
                const bool brief = i >= cut;
                if (lane_id() == 0) my.done = my.done + (brief ? 1u << lb : 1u);
                const unsigned blk = brief ? cut + ((i - cut) << lb) : i;
                if (!my.skip) raster(shared + blk / kOrderItems, (int)(blk % kOrderItems), 1 << lb, brief);
                at = __shfl_sync(0xffffffffu, nxt, 0);
            }
            retire(my.done);
            v = pick(blockIdx.x * kRasterWarps + warp, gridDim.x * kRasterWarps);
            if (v >= 0 && lane_id() == 0) at = take(v, 1);
            at = __shfl_sync(0xffffffffu, at, 0);
        }
    }
}

}  // namespace

static size_t stage_smem(int T, int row_bytes);

cudaError_t launch_batch(const BatchView *d_views, const BatchPlan &P, const OptParams &O, unsigned *batch_words,
                         cudaStream_t st, cudaEvent_t *ev, bool ids)
{
    // ev (7 events or null): recorded as graph event nodes when captured
    auto mark = [&](int k) { if (ev) cudaEventRecordWithFlags(ev[k], st, cudaEventRecordExternal); };
    mark(0);
    {
        unsigned long long *t0 = reinterpret_cast<unsigned long long *>(batch_words + BW_START);
        const size_t sm = local_bins_smem(P.max_T, false);
        const bool col = P.total_colour > 0;   // colours in the colour pass, not in the set-up
        if (col) {
            // before the set-up, which copies the Gaussian colours into the records
            if (ev) cudaEventRecordWithFlags(ev[5], st, cudaEventRecordExternal);
            k_bcolour<<<P.total_colour, kColourThreads, 0, st>>>(d_views, P.cmap, P.gview, t0);
            if (ev) cudaEventRecordWithFlags(ev[6], st, cudaEventRecordExternal);
        }
        // the colours: in the pass above, or here, from staged rows where the
        // batch's rows allow it
        const auto prep = [&](auto pass, auto here, auto staged, unsigned g, const int2 *map) {
            if (g == 0) return;
            if (col) pass<<<g, kPrepThreads, sm, st>>>(d_views, map, O, t0);
            else if (P.stage_bytes) staged<<<g, kPrepThreads, stage_smem(P.max_T, P.stage_bytes), st>>>(d_views, map, O, t0);
            else here<<<g, kPrepThreads, sm, st>>>(d_views, map, O, t0);
        };
        if (P.gdim == 2) {
            prep(k_bprep<2, 1, COL_PASS>, k_bprep<2, 1, COL_HERE>, k_bprep<2, 1, COL_STAGED>, P.total_sprep, P.smap);
            prep(k_bprep<2, 2, COL_PASS>, k_bprep<2, 2, COL_HERE>, k_bprep<2, 2, COL_STAGED>, P.total_gprep, P.gmap);
        } else {
            prep(k_bprep<3, 1, COL_PASS>, k_bprep<3, 1, COL_HERE>, k_bprep<3, 1, COL_STAGED>, P.total_sprep, P.smap);
            prep(k_bprep<3, 2, COL_PASS>, k_bprep<3, 2, COL_HERE>, k_bprep<3, 2, COL_STAGED>, P.total_gprep, P.gmap);
        }
    }
    mark(1);
    k_bcolscan<<<dim3(P.total_colscan, 2), 256, 0, st>>>(d_views, P.n);
    mark(2);
    k_bfill<<<P.n + P.total_prep, kFillThreads, local_bins_smem(P.max_T, true), st>>>(d_views, P.n, P.lb);
    mark(3);
    // P.gdim: the Gaussian kind shared by all scenes of the batch
    const unsigned grid = P.raster_ctas;
    const int kind = (O.samples == 4 ? 2 : 0) + (P.gdim == 2 ? 1 : 0);
    auto go = [&](auto one, auto many) {
        if (P.one_counter) one<<<grid, kRasterThreads, 0, st>>>(d_views, P.n, O, batch_words, P.lb, P.total_tiles);
        else many<<<grid, kRasterThreads, 0, st>>>(d_views, P.n, O, batch_words, P.lb, P.total_tiles);
    };
    switch (kind + (ids ? 4 : 0)) {
    case 0: go(k_braster<1, 3, false, true>, k_braster<1, 3, false, false>); break;
    case 1: go(k_braster<1, 2, false, true>, k_braster<1, 2, false, false>); break;
    case 2: go(k_braster<4, 3, false, true>, k_braster<4, 3, false, false>); break;
    case 3: go(k_braster<4, 2, false, true>, k_braster<4, 2, false, false>); break;
    case 4: go(k_braster<1, 3, true, true>, k_braster<1, 3, true, false>); break;
    case 5: go(k_braster<1, 2, true, true>, k_braster<1, 2, true, false>); break;
    case 6: go(k_braster<4, 3, true, true>, k_braster<4, 3, true, false>); break;
    default: go(k_braster<4, 2, true, true>, k_braster<4, 2, true, false>); break;
    }
    mark(4);
    return cudaGetLastError();
}

// (the fill's order CTA needs 67 words)
size_t local_bins_smem(int T, bool fill) { return fill ? (size_t)(T > 67 ? T : 67) * 4 : (size_t)((T + 1) / 2) * 4; }

// Shared memory of the set-up with staged SH rows.
static size_t stage_smem(int T, int row_bytes)
{
    return (local_bins_smem(T, false) + 15) / 16 * 16 + (size_t)kPrepThreads * row_bytes;
}

int staged_row_bytes(const SceneView &S, int T)
{
    const int row = 3 * kShRows * (S.sh_dtype == GES_F32 ? 4 : 2);
    // two CTAs of an SM (1 KB of each is the system's, the batch's keep a view
    // entry): with one the set-up is slower than with direct loads
    return S.deg == 3 && sh_rows_aligned(S) && 2 * (stage_smem(T, row) + 2048) <= (size_t)228 * 1024 ? row : 0;
}

cudaError_t prepare_forward_kernels()
{
    const int hs = (int)local_bins_smem(kLocalMaxTiles, false), ss = 113 * 1024;
    cudaError_t e = cudaSuccess;
    const auto smem = [&](auto k, int bytes) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    };
    smem(k_prep_local<3, false, COL_HERE>, hs);
    smem(k_prep_local<2, false, COL_HERE>, hs);
    smem(k_prep_local<3, true, COL_HERE>, hs);
    smem(k_prep_local<3, false, COL_STAGED>, ss);
    smem(k_prep_local<2, false, COL_STAGED>, ss);
    smem(k_prep_local<3, true, COL_STAGED>, ss);
    smem(k_bprep<3, 1, COL_PASS>, hs);
    smem(k_bprep<3, 2, COL_PASS>, hs);
    smem(k_bprep<2, 1, COL_PASS>, hs);
    smem(k_bprep<2, 2, COL_PASS>, hs);
    smem(k_bprep<3, 1, COL_HERE>, hs);
    smem(k_bprep<3, 2, COL_HERE>, hs);
    smem(k_bprep<2, 1, COL_HERE>, hs);
    smem(k_bprep<2, 2, COL_HERE>, hs);
    smem(k_bprep<3, 1, COL_STAGED>, ss);
    smem(k_bprep<3, 2, COL_STAGED>, ss);
    smem(k_bprep<2, 1, COL_STAGED>, ss);
    smem(k_bprep<2, 2, COL_STAGED>, ss);
    smem(k_fill_local, (int)local_bins_smem(kLocalMaxTiles, true));
    smem(k_bfill, (int)local_bins_smem(kLocalMaxTiles, true));
    return e;
}

// preprocess + binning of one view (everything before the raster)
cudaError_t launch_binning(const SceneView &S, const CamParams &C, const OptParams &O, const ViewScratch &X,
                           cudaStream_t st, cudaEvent_t *ev)
{
    const int T = C.tiles_x * C.tiles_y;
    SceneView Sv = S;
    if (O.mode == GES_MODE_GAUSSIANS_ONLY) Sv.N = 0;
    if (O.mode == GES_MODE_SURFELS_ONLY) Sv.M = 0;
    const bool local = local_binning(X, T);
    if (ev) cudaEventRecord(ev[0], st);
    LocalBins B{};
    if (local) {
        int dev = 0, sms = 152;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        B = plan_local_bins(Sv.N, Sv.M, sms);
        if (B.Ps + B.Pg > 0) {
            const size_t sm = local_bins_smem(T, false);
            const int row = staged_row_bytes(Sv, T);
            const auto prep = [&](auto here, auto staged) {
                if (row) staged<<<B.Ps + B.Pg, kPrepThreads, stage_smem(T, row), st>>>(Sv, C, O, X, B);
                else here<<<B.Ps + B.Pg, kPrepThreads, sm, st>>>(Sv, C, O, X, B);
            };
            if (X.s_tside) prep(k_prep_local<3, true, COL_HERE>, k_prep_local<3, true, COL_STAGED>);
            else if (Sv.gdim == 2) prep(k_prep_local<2, false, COL_HERE>, k_prep_local<2, false, COL_STAGED>);
            else prep(k_prep_local<3, false, COL_HERE>, k_prep_local<3, false, COL_STAGED>);
        }
    } else {
        const int nsb = (int)((Sv.N + 255) / 256), ngb = (int)((Sv.M + 255) / 256);
        if (nsb + ngb > 0) {
            if (X.s_tside) k_prep_atomic<3, true><<<nsb + ngb, 256, 0, st>>>(Sv, C, O, X, nsb);
            else if (Sv.gdim == 2) k_prep_atomic<2><<<nsb + ngb, 256, 0, st>>>(Sv, C, O, X, nsb);
            else k_prep_atomic<3><<<nsb + ngb, 256, 0, st>>>(Sv, C, O, X, nsb);
        }
    }
    if (ev) cudaEventRecord(ev[1], st);
    if (local) k_colscan<<<dim3((T + kColTiles - 1) / kColTiles, 2), 1024, 0, st>>>(X, T, B);
    else k_alloc<<<dim3((T + kAllocTiles - 1) / kAllocTiles, 2), kAllocTiles, 0, st>>>(X, T);
    if (ev) cudaEventRecord(ev[2], st);
    if (local) {
        k_fill_local<<<B.Ps + B.Pg + 1, kFillThreads, local_bins_smem(T, true), st>>>(X, T, C.tiles_x, C.tsx, C.tsy, B);
    } else {
        k_fill_atomic<<<152 * 8, 256, 0, st>>>(X, S.gdim, C.tiles_x, C.tsx, C.tsy);
    }
    if (ev) cudaEventRecord(ev[3], st);
    return cudaGetLastError();
}

namespace {
// Exact work counts of one view: every (sample, surfel) fragment inside the
// opaque disc in front of the near plane, and every (pixel, Gaussian) pair
// with alpha >= alpha_min, over the full tile lists (no culling).
__global__ void __launch_bounds__(256) k_count(SceneView S, ViewScratch X, CamParams C, OptParams O)
{
    __shared__ float4 st[3][256];
    __shared__ unsigned red[2][8];
    if (X.status[ST_FLAGS] & (FLAG_SOVF | FLAG_GOVF)) return;
    const int tile = blockIdx.x, t = threadIdx.x;
    const int tx = tile % C.tiles_x, ty = tile / C.tiles_x;
    const int px = (tx << C.tsx) + (t & ((1 << C.tsx) - 1)), py = (ty << C.tsy) + (t >> C.tsx);
    const bool in_img = px < C.W && py < C.H;
    const float u = px + 0.5f, v = py + 0.5f;
    unsigned ns = 0, ng = 0;
    for (int kind = 0; kind < 2; ++kind) {
        if (kind == 0 && O.mode == GES_MODE_GAUSSIANS_ONLY) continue;
        if (kind == 1 && O.mode == GES_MODE_SURFELS_ONLY) continue;
        const int2 rng = (kind == 0 ? X.s_rng : X.g_rng)[tile];
        const uint2 *list = kind == 0 ? X.s_list : X.g_list;
        const float4 *rec = kind == 0 ? X.s_rec : X.g_rec;
        const int a = rng.x, b = rng.y;
        for (int base = a; base < b; base += 256) {
            __syncthreads();
            if (base + t < b) {
                const float4 *rp = rec + 4 * (int64_t)list[base + t].x;
                st[0][t] = rp[0]; st[1][t] = rp[1]; st[2][t] = rp[2];
            }
            __syncthreads();
            const int n = min(256, b - base);
            if (!in_img) continue;
            for (int j = 0; j < n; ++j) {
                if (kind == 0) {
                    const float4 r0 = st[0][j], r1 = st[1][j], r2 = st[2][j];
                    for (int k = 0; k < O.samples; ++k) {
                        const float uk = O.samples == 4 ? px + 0.25f + 0.5f * (k & 1) : u;
                        const float vk = O.samples == 4 ? py + 0.25f + 0.5f * (k >> 1) : v;
                        const float du = uk - r0.x, dv = vk - r0.y;
                        const float iz = fmaf(r0.w, du, fmaf(r1.x, dv, r0.z));
                        const float A = fmaf(r1.y, du, fmaf(r1.z, dv, r1.w));
                        const float B = fmaf(r2.x, du, fmaf(r2.y, dv, r2.z));
                        ns += (fmaf(A, A, fmaf(B, B, -iz * iz)) <= 0.f && iz > 0.f && iz < C.izn) ? 1u : 0u;
                    }
                } else if (S.gdim == 2) {
                    const float4 r0 = st[0][j], r1 = st[1][j], r2 = st[2][j];
                    const int id = __float_as_int(st[2][j].w);
                    const float4 x0 = X.g_aux[2 * (int64_t)id], x1 = X.g_aux[2 * (int64_t)id + 1];
                    const float du = u - r0.x, dv = v - r0.y;
                    const float iz = fmaf(r0.w, du, fmaf(r1.x, dv, r0.z));
                    const float A = fmaf(r1.y, du, fmaf(r1.z, dv, r1.w));
                    const float B = fmaf(r2.x, du, fmaf(r2.y, dv, r2.z));
                    const float z = __frcp_rn(iz);
                    const float a = ex2_approx(fmaf(x1.w, fmaf(A, A, B * B) * (z * z), x0.w));
                    ng += (iz > 0.f && iz < C.izn && a >= O.alpha_min) ? 1u : 0u;
                } else {
                    const GaussRec g = gauss_rec3(st[0][j], st[1][j], make_float4(0.f, 0.f, 0.f, 0.f));
                    float e;
                    ng += gauss_alpha(g, u, v, e) >= O.alpha_min ? 1u : 0u;
                }
            }
        }
    }
    for (int d = 16; d >= 1; d >>= 1) {
        ns += __shfl_xor_sync(0xffffffffu, ns, d);
        ng += __shfl_xor_sync(0xffffffffu, ng, d);
    }
    if ((t & 31) == 0) { red[0][t >> 5] = ns; red[1][t >> 5] = ng; }
    __syncthreads();
    if (t == 0) {
        unsigned a = 0, b = 0;
        for (int w = 0; w < 8; ++w) { a += red[0][w]; b += red[1][w]; }
        atomicAdd(X.status + ST_SFRAG, a);
        atomicAdd(X.status + ST_GFRAG, b);
    }
}
}  // namespace

namespace {
template <int kS, int kG>
void launch_raster(const ViewScratch &X, const CamParams &C, const OptParams &O, float *out_rgb, float *out_depth,
                   int32_t *out_id, float *aux, const GeoMaps &geo, cudaStream_t st)
{
    // fewer than kShareSlots tiles can be above their share of the entries
    const unsigned T = (unsigned)(C.tiles_x * C.tiles_y);
    const unsigned shared = T < (unsigned)kShareSlots ? T : (unsigned)kShareSlots;
    const unsigned grid = X.order ? T + (kOrderItems - 1) * shared : T;
    if (O.geo) k_raster<kS, kG, true><<<grid, kRasterThreads, 0, st>>>(X, C, O, out_rgb, out_depth, out_id, aux, geo);
    else k_raster<kS, kG, false><<<grid, kRasterThreads, 0, st>>>(X, C, O, out_rgb, out_depth, out_id, aux, geo);
}
}  // namespace

cudaError_t launch_forward(const SceneView &S, const CamParams &C, const OptParams &O, const ViewScratch &Xs,
                           float *out_rgb, float *out_depth, int32_t *out_id, float *aux, cudaStream_t st,
                           cudaEvent_t *ev, const float *const *geo_maps)
{
    cudaError_t e = launch_binning(S, C, O, Xs, st, ev);
    if (e != cudaSuccess) return e;
    ViewScratch X = Xs;
    if (!local_binning(X, C.tiles_x * C.tiles_y)) X.order = nullptr;   // atomic binning makes none
    GeoMaps geo{};
    if (geo_maps) geo = GeoMaps{const_cast<float *>(geo_maps[0]), const_cast<float *>(geo_maps[1]),
                                const_cast<float *>(geo_maps[2]), const_cast<float *>(geo_maps[3]),
                                const_cast<float *>(geo_maps[4])};
    if (O.samples == 4 && S.gdim == 2) launch_raster<4, 2>(X, C, O, out_rgb, out_depth, out_id, aux, geo, st);
    else if (O.samples == 4) launch_raster<4, 3>(X, C, O, out_rgb, out_depth, out_id, aux, geo, st);
    else if (S.gdim == 2) launch_raster<1, 2>(X, C, O, out_rgb, out_depth, out_id, aux, geo, st);
    else launch_raster<1, 3>(X, C, O, out_rgb, out_depth, out_id, aux, geo, st);
    if (ev) cudaEventRecord(ev[4], st);
    return cudaGetLastError();
}

namespace {
// Mip-GES 3D filter variance (Sec. 6.1, Mip-Splatting's world filter): per
// Gaussian, the highest sampling rate max(fx, fy)/z over the cameras whose
// image rectangle holds the projected centre at z > znear; v = s3d / rate^2,
// -1 while unseen.  The largest v seen is kept in *vmax (non-negative floats
// order like their bit patterns, so an integer max is exact and order free).
constexpr int kFiltCams = 32;

__global__ void __launch_bounds__(256) k_filter3d(SceneView S, const CamParams *__restrict__ cams, int n_cams,
                                                  float s3d, float *__restrict__ out, unsigned *vmax)
{
    __shared__ __align__(16) unsigned char cbuf[kFiltCams * sizeof(CamParams)];
    const CamParams *sc = reinterpret_cast<const CamParams *>(cbuf);
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    float px = 0.f, py = 0.f, pz = 0.f;
    if (i < S.M) { px = __ldg(S.g_pos + 3 * i); py = __ldg(S.g_pos + 3 * i + 1); pz = __ldg(S.g_pos + 3 * i + 2); }
    float nu = 0.f;
    for (int c0 = 0; c0 < n_cams; c0 += kFiltCams) {
        const int nc = min(kFiltCams, n_cams - c0);
        __syncthreads();
        const int *src = reinterpret_cast<const int *>(cams + c0);
        int *dst = reinterpret_cast<int *>(cbuf);
        for (int k = threadIdx.x; k < nc * (int)(sizeof(CamParams) / 4); k += blockDim.x) dst[k] = src[k];
        __syncthreads();
        if (i >= S.M) continue;
        for (int c = 0; c < nc; ++c) {
            const CamParams &C = sc[c];
            const df tz = df_dot3_plus(C.R + 6, px, py, pz, C.t[2]);
            if (!(tz.hi > C.znear || (tz.hi == C.znear && tz.lo > 0.f))) continue;
            const df tx = df_dot3_plus(C.R, px, py, pz, C.t[0]);
            const df ty = df_dot3_plus(C.R + 3, px, py, pz, C.t[1]);
            const float u = df_add_f(df_mul_f(df_div(tx, tz), C.fx), C.cx).hi;
            const float v = df_add_f(df_mul_f(df_div(ty, tz), C.fy), C.cy).hi;
            if (!(u >= 0.f && u <= (float)C.W && v >= 0.f && v <= (float)C.H)) continue;
            nu = fmaxf(nu, fmaxf(C.fx, C.fy) / tz.hi);
        }
    }
    if (i >= S.M) return;
    if (nu > 0.f) {
        const float v = s3d / (nu * nu);
        out[i] = v;
        atomicMax(vmax, __float_as_uint(v));
    } else {
        out[i] = -1.f;
    }
}

__global__ void __launch_bounds__(256) k_filter3d_fill(int64_t M, float *__restrict__ out, const unsigned *vmax)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < M && out[i] < 0.f) out[i] = __uint_as_float(*vmax);
}
}  // namespace

cudaError_t launch_filter3d(const SceneView &S, const CamParams *d_cams, int n_cams, float s3d, float *out,
                            unsigned *d_vmax, cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(d_vmax, 0, sizeof(unsigned), st);
    if (e != cudaSuccess || S.M == 0) return e;
    const unsigned blocks = (unsigned)((S.M + 255) / 256);
    k_filter3d<<<blocks, 256, 0, st>>>(S, d_cams, n_cams, s3d, out, d_vmax);
    k_filter3d_fill<<<blocks, 256, 0, st>>>(S.M, out, d_vmax);
    return cudaGetLastError();
}

cudaError_t launch_count(const SceneView &S, const CamParams &C, const OptParams &O, const ViewScratch &X,
                         cudaStream_t st)
{
    cudaError_t e = launch_binning(S, C, O, X, st, nullptr);
    if (e != cudaSuccess) return e;
    k_count<<<C.tiles_x * C.tiles_y, 256, 0, st>>>(S, X, C, O);
    return cudaGetLastError();
}

}  // namespace ges
