// render.cu -- per-tile blending (Algorithm 2, BlendInOrder) and its backward pass (Sec. 6).
//
// A tile is made of 8x8-pixel sub-blocks (four in a 16x16 tile, two in 16x8, one in 8x8).  A group
// of 8, 16 or 32 lanes of one warp owns a sub-block, each lane 8, 4 or 2 pixels of one row; a warp
// (one per block) holds 4, 2 or 1 groups and no two warps wait on one another.  A warp stages the
// next 32 Gaussians of its tile's depth-sorted list in shared memory (its tiles', when a tile has
// fewer sub-blocks than the warp has groups) and each group then walks only the staged splats of
// its own 32-bit word: in the forward those that can reach its sub-block, in the backward those
// it blended.  The groups of a warp run through different splats in the same instructions, so the
// per-splat work (loads, row setup, reduction) is shared by up to four splats.  Arithmetic on
// pixel pairs is packed (f32x2).  What bounds the kernels is the issue slots and the latency of
// few warps, not memory (profiles of the earlier one-warp-per-half-tile kernels: 77 % of the issue
// slots at 59 % blended lanes per visited splat; 8x8 sub-blocks: 70 %).
// A staged splat carries its offset from the tile's first pixel centre, the Cholesky factor of
// its conic pre-scaled to log2 units and log2 of its opacity (Entry), so that for a pixel at
// offset d:
//   p = l11' dx + l21' dy, q = l22' dy, s = p^2 + q^2 = -log2(e) power,  o exp(power) = 2^(lo - s)
// and "alpha < 1/255" is the single comparison s > thr with thr = lo - log2(1/255).  Pixels of
// one row share dy, q and q^2; p is evaluated as that of one of the first four columns plus a
// multiple of the step of four columns.
//
// Forward (eq. front-to-back, App. C): a = min(0.99, o exp(power)); skip a < 1/255; stop before
//   T (1 - a) < 1e-4; C += a T c; T *= 1 - a.  A pixel that stopped has the sign bit of T set; a
//   group stops when all its pixels have.  Writes C + T bg, T and the 1-based list position of the
//   last blended Gaussian, and per sub-block one contribution word per 32 positions: the splats
//   some pixel of the sub-block blended.
// Backward: each group walks the splats its contribution words name back to front (it blends
//   exactly the forward's pairs); each pixel only processes positions below its own last position, recovers
//   T_i = T_{i+1} / (1 - a_i) from the stored final T, and keeps R . dL/dC, the projection of
//   the colour behind the current Gaussian (normalised by the transmittance in front of it; R
//   starts at bg) on the pixel's dL/dC, which is all the recurrence needs:
//     dL/dc_i = a_i T_i dL/dC,  dL/da_i = T_i (c_i - R_{i+1}) . dL/dC,  R_i = a_i c_i + (1 - a_i) R_{i+1}.
//   Through a = o G (zero when clamped), with g = Sigma'^-1 d = L (p, q) (L the Cholesky factor
//   of the conic, (p, q) = L^T d): d(power)/d(mean) = g and d(power)/d(Sigma') = g g^T / 2.  The
//   mean and Sigma' sums are kept in the whitened frame of L: sum dL/dpower (p, q) and
//   (1/2) sum dL/dpower (p, q)(p, q)^T =: K; the per-Gaussian stage maps them back with the same
//   stored L (dL/dmean2D = L (p, q) sums, dL/dSigma' = L K L^T contracted without forming it).
//   In pixel coordinates the three entries of dL/dSigma' of an elongated splat are all dominated
//   by its minor axis and their major-axis part, which the scale along the long axis needs, is
//   lost to cancellation in fp32 sums over many pixels; in the whitened frame every direction of
//   the splat has the same scale.  q being the row's, a lane sums dL/dpower with 1, p and p^2 over
//   its pixels and multiplies by q and q^2 once; the nine sums of a group's lanes (of all the warp's,
//   when its groups walk the same splats) are reduced by a transposed reduce-scatter and every lane
//   adds the one or two totals it holds.
//
// Limited-BW (cfg.grad_limit = N > 0, the ablation of Sec. 7.3): the forward pass also records
// the number of blended splats of every pixel (COUNT); the backward pass (LIMIT) keeps the
// recurrences over all of them but adds gradients only for the N front-most, i.e. it skips the
// gradient terms of the first (count - N) blended splats it meets from the back.
//
// The forward and the backward evaluate a (pixel, splat) pair with the same staging and the same
// operation sequence (stage_splat, splat_row), whatever the pixels per lane, so their skip and
// clamp decisions agree bit for bit.
//
// Block order: warps take the tiles in the order of order[], the frame's tiles by decreasing list
// length (tilesort.cu).  The work of a tile grows with its
// list and varies by a factor of several across a frame; blocks start roughly in index order, so
// in row-major order the longest tiles (the frame's centre) could start late and finish alone.
#include <type_traits>

#include "gs_device.cuh"
#include "gs_kernels.h"

namespace gs {

namespace {

// sqrt(log2(e) / 2): scales the Cholesky factor so that p^2 + q^2 = -log2(e) power.
constexpr float kScaleLog2 = 0.84932180028801907f;
// 1 / kScaleLog2 = sqrt(2 ln 2): scaled p, q back to the whitened frame of the unscaled factor.
constexpr float kUnscale = 1.1774100225154747f;
// (1/2) / kScaleLog2^2 = ln 2: scaled (p, q)(p, q)^T sums to K = (1/2) sum dL/dpower (p, q)(p, q)^T.
constexpr float kLn2 = 0.69314718055994531f;
// Side of a sub-block in pixels: the unit of culling, contribution bits and lane groups.
constexpr int kSub = 8;
// Magnitude of dL/dC, colour or conic from which pixels' products are kept apart (backward_unit):
// three products of two smaller values, their sum, and a conic entry times a pixel offset are finite.
constexpr float kWild = 1.0e18f;

struct Staged {
    float4 a;   // (ox, oy, thr, lo): tile-relative offset, skip threshold, log2(opacity)
    float4 b;   // (l11', l21', l22', 1/o)
};

__device__ __forceinline__ void stage_splat(float4 m, float4 L, int x0, int y0, float log2_amin, Staged& s) {
    const float ox = tile_offset(x0, m.x, m.z);
    const float oy = tile_offset(y0, m.y, m.w);
    const float lo = __log2f(L.w);
    const float thr = __fsub_rn(lo, log2_amin);
    s.a = make_float4(ox, oy, thr, lo);
    s.b = make_float4(__fmul_rn(L.x, kScaleLog2), __fmul_rn(L.y, kScaleLog2), __fmul_rn(L.z, kScaleLog2),
                      __frcp_rn(L.w));
}

// Minimum of s = (l11 x + l21 y)^2 + (l22 y)^2 (the staged splat's scaled quadratic form) over
// the rectangle [xa, xb] x [ya, yb] of pixel-centre offsets: 0 when the splat centre is inside,
// else the smallest of the four edge minima (each a one-dimensional convex quadratic).
__device__ __forceinline__ float rect_min_s(const Staged& st, float xa, float xb, float ya, float yb) {
    const float l11 = st.b.x, l21 = st.b.y, l22 = st.b.z;
    if (xa <= 0.f && 0.f <= xb && ya <= 0.f && 0.f <= yb) return 0.f;
    const float i11 = 1.0f / l11, A = fmaf(l21, l21, l22 * l22), iA = 1.0f / A;
    auto at = [&](float x, float y) { const float p = fmaf(l11, x, l21 * y), q = l22 * y; return fmaf(p, p, q * q); };
    float m = 3.0e38f;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const float y = e ? yb : ya;                          // horizontal edge: x* = -l21 y / l11
        m = fminf(m, at(fminf(fmaxf(-l21 * y * i11, xa), xb), y));
        const float x = e ? xb : xa;                          // vertical edge: y* = -l11 l21 x / A
        m = fminf(m, at(x, fminf(fmaxf(-l11 * l21 * x * iA, ya), yb)));
    }
    return m;
}

// Whether the staged splat can reach alpha_min at a point of an 8x8 sub-block whose first pixel
// centre is at offset (xa, ya) from the splat: the minimum of its quadratic form over the
// sub-block's rectangle (continuous, so it covers every pixel centre) within a small margin of the
// threshold.  False proves no pixel of the sub-block blends the splat.
__device__ __forceinline__ bool sub_reach(const Staged& st, float xa, float ya) {
    const float thr = st.a.z;
    if (!(thr > 0.f)) return false;
    const float lim = fmaf(thr, 1.0009765625f, 0.0009765625f);   // thr (1 + 2^-10) + 2^-10
    return rect_min_s(st, xa, xa + (float)(kSub - 1), ya, ya + (float)(kSub - 1)) <= lim;
}

// The part of the frame a lane works on.  Groups (sub-blocks) are numbered tile by tile in the
// render order; a warp takes GW consecutive groups.  With more groups in a warp than sub-blocks
// in a tile, the warp holds several tiles, each staged by its own lanes.
template <int PX, int SUBS>
struct Lanes {
    static constexpr int LPR = kSub / PX;                    // lanes per pixel row of a sub-block
    static constexpr int GL = kSub * LPR;                    // lanes of a group
    static constexpr int GW = 32 / GL;                       // groups of a warp
    static constexpr int SX = SUBS >= 2 ? 2 : 1;             // sub-blocks per tile row
    static constexpr int NS = SUBS < GW ? SUBS : GW;         // sub-blocks of one tile in a warp
    static constexpr int TPW = GW / NS;                      // tiles in a warp
    static constexpr int SL = 32 / TPW;                      // lanes staging one tile
    static constexpr int ROUNDS = 32 / SL;                   // splats a lane stages per window
    static constexpr int PAIRS = PX / 2;
    // fetch the next window's splats while one is blended (registers allow it with one splat per lane)
    static constexpr bool AHEAD = ROUNDS == 1 && PX < 8;
    // blend every splat with care (Entry): with few pixels per lane that costs less than a second path
    static constexpr bool ONE_PATH = PX == 2;
    int lane, group, slot, tl, sub, sx, sy, row, col;
    uint32_t index;                                          // of the tile in the render order
    __device__ __forceinline__ explicit Lanes(uint32_t unit) {
        lane = threadIdx.x & 31;
        group = lane / GL;
        slot = lane / SL;
        tl = lane % SL;
        const uint32_t gid = unit * GW + (uint32_t)group;
        index = gid / SUBS;
        sub = (int)(gid % SUBS);
        sx = sub % SX;
        sy = sub / SX;
        row = (lane % GL) / LPR;
        col = (lane % LPR) * PX;                             // first owned column in the sub-block
    }
    // Column of the i-th owned pixel in the tile is 8 sx + col + i; its offset is evaluated as
    // that of column c0 = (col + i) & 3 plus j() steps of four columns.
    __device__ __forceinline__ float j(int i) const { return (float)(2 * sx + (PX == 8 ? i / 4 : col / 4)); }
    __device__ __forceinline__ float c0(int i) const { return PX == 2 ? (float)((col & 3) + i) : (float)(i & 3); }
    // Sub-blocks of this warp's tiles: the s-th of NS is sub0() + s.
    __device__ __forceinline__ int sub0() const { return sub - (group % NS); }
};

// A staged splat in shared memory: what the packed arithmetic broadcasts is stored twice, so that a
// 16-byte load yields register pairs (20 move instructions fewer per splat and warp).
struct __align__(16) Entry {
    f32x2 ox, oy;         // offset of the tile's first pixel centre from the mean
    f32x2 l11, l21;       // scaled Cholesky factor of the conic
    f32x2 l22, lo;        // lo = log2(opacity)
    f32x2 r, g;           // colour
    f32x2 b;
    float ko;             // 1 / opacity
    uint32_t id;          // Gaussian
};

__device__ __forceinline__ Entry entry_of(const Staged& st, float4 col, uint32_t gid) {
    Entry e;
    e.ox = pack2(st.a.x, st.a.x);
    e.oy = pack2(st.a.y, st.a.y);
    e.l11 = pack2(st.b.x, st.b.x);
    e.l21 = pack2(st.b.y, st.b.y);
    e.l22 = pack2(st.b.z, st.b.z);
    e.lo = pack2(st.a.w, st.a.w);
    e.r = pack2(col.x, col.x);
    e.g = pack2(col.y, col.y);
    e.b = pack2(col.z, col.z);
    e.ko = st.b.w;
    e.id = gid;
    return e;
}

// Whether a splat's pairs need care: its alpha can reach alpha_max, its conic is not finite (a
// degenerate splat without dilation) or its colour could overflow a product.
__device__ __forceinline__ bool needs_care(const Staged& st, float4 col, float lo_care) {
    return !(st.a.w <= lo_care) || !(fabsf(st.b.x) + fabsf(st.b.y) + fabsf(st.b.z) < kWild) ||
           !(col.x + col.y + col.z < kWild);   // colours are clamped at 0
}

// A ballot of the lanes that stage a window, round r, as bits of the window's 32 positions (of the
// lane's own tile).
template <typename LN>
__device__ __forceinline__ uint32_t window_bits(const LN& ln, bool v, int r) {
    const uint32_t bal = __ballot_sync(0xffffffffu, v);
    if (LN::SL == 32) return bal;
    return ((bal >> (ln.slot * LN::SL & 31)) & ((1u << (LN::SL & 31)) - 1u)) << (r * LN::SL & 31);
}

// What a lane fetches of a splat it stages.
struct Fetched {
    float4 xy, conic, rgb;
    uint32_t id;
};
// The Gaussians a lane stages of a window: positions first, first + SL, ... of its tile's list,
// those below `len`.
template <int ROUNDS, int SL>
__device__ __forceinline__ void fetch_ids(uint32_t (&id)[ROUNDS], const uint32_t* vals, uint32_t first, uint32_t len) {
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) id[r] = first + (uint32_t)(r * SL) < len ? vals[first + (uint32_t)(r * SL)] : 0u;
}
template <typename A>
__device__ __forceinline__ void fetch_splat(Fetched& f, uint32_t g, const A& a) {
    if (g >= (uint32_t)a.n) {   // only reachable after a timed-out sort
        debug_fail(a.status);
        g = 0;
    }
    f.id = g;
    f.xy = a.xy[g];
    f.conic = a.conic_opacity[g];
    f.rgb = a.rgb[g];
}

// log2 of an opacity whose alpha stays below alpha_max whatever the rounding of 2^x.
__device__ __forceinline__ float log2_care(float alpha_max) { return __log2f(alpha_max) - 1.0e-5f; }

// A splat along the lane's pixel row: p at the pairs of columns (0, 1) and (2, 3) of the
// four-column step, its step dp, q and q^2 (in both halves).
struct RowPairs {
    f32x2 p0[2], dp, q, qq;
};
template <int PX, int SUBS>
__device__ __forceinline__ RowPairs splat_row(const Lanes<PX, SUBS>& ln, const Entry& e, f32x2 ly) {
    RowPairs r;
    const f32x2 dy = add2(ly, e.oy);
    r.q = mul2(e.l22, dy);
    r.qq = mul2(r.q, r.q);
#pragma unroll
    for (int h = 0; h < (PX == 2 ? 1 : 2); ++h) {
        const f32x2 dx0 = add2(pack2(ln.c0(2 * h), ln.c0(2 * h + 1)), e.ox);
        r.p0[h] = fma2(e.l21, dy, mul2(e.l11, dx0));
    }
    r.dp = mul2(pack2(4.0f, 4.0f), e.l11);
    return r;
}
__device__ __forceinline__ float low(f32x2 v) {
    float lo, hi;
    unpack2(v, lo, hi);
    return lo;
}

// Sum over the lanes of a group of 9 values by a transposed reduce-scatter: each round halves the
// values a lane keeps (it sends the half its partner keeps and adds the half it receives).  The
// totals of slots [first, first + n) of reduce_slots are left in a[.][0..1].
// U sets at once, so that their shuffles overlap.
template <int GL, int U>
__device__ __forceinline__ void group_reduce9(float (&a)[U][9], int lane) {
    int n = 9;
#pragma unroll
    for (int m = GL / 2; m > 0; m >>= 1) {
        const bool hi = lane & m;
        const int half = (n + 1) / 2;
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            if (i >= half) continue;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (half + i < n) {
                    const float keep = hi ? a[u][half + i] : a[u][i], send = hi ? a[u][i] : a[u][half + i];
                    a[u][i] = keep + __shfl_xor_sync(0xffffffffu, send, m);
                } else {   // the odd value: both sides keep its sum
                    a[u][i] += __shfl_xor_sync(0xffffffffu, a[u][i], m);
                }
            }
        }
        n = half;
    }
}

// Slots [first, first + n) whose totals group_reduce9 leaves in this lane (n <= 2; a slot is
// owned by one lane of the group).
template <int GL>
__device__ __forceinline__ void reduce_slots(int lane, int& first, int& n) {
    first = 0;
    n = 9;
    int len = 9;
#pragma unroll
    for (int m = GL / 2; m > 0; m >>= 1) {
        const int half = (len + 1) / 2;
        const bool odd_tail = len == 1;   // one value left: both sides hold it, the lower lane owns it
        if (lane & m) {
            first += half;
            n = odd_tail ? 0 : (n > half ? n - half : 0);
        } else {
            n = n < half ? n : half;
        }
        len = half;
    }
}

// The decisions of a pixel pair against one splat: alpha >= 1/255 (s <= thr), and stop before T (1 - alpha)
// < T_min.  A pixel that blends takes `te` and its `last`; one that stops gets its sign bit set.
// Returns the blend weights alpha T (0 when not blended); a0, a1: the bits of the blended alphas.
// Written in PTX for the dual-output comparison and in-place selects.  `on`
// false skips the pair.
__device__ __forceinline__ f32x2 blend_pair(f32x2 s, float thr, f32x2 al, f32x2 te, float tmin, uint32_t pos, bool on,
                                            f32x2& T, uint32_t& last0, uint32_t& last1, uint32_t& a0, uint32_t& a1) {
    f32x2 w;
    asm("{\n\t.reg .pred h0, h1, k0, k1, z0, z1;\n\t.reg .f32 s0, s1, t0, t1, e0, e1, x0, x1;\n\t.reg .b64 A;\n\t"
            "mov.b64 {s0, s1}, %6;\n\tmov.b64 {t0, t1}, %1;\n\tmov.b64 {e0, e1}, %9;\n\tmov.b64 {x0, x1}, %8;\n\t"
            "setp.ne.s32 h0, %12, 0;\n\tsetp.leu.and.f32 h1, s1, %7, h0;\n\tsetp.leu.and.f32 h0, s0, %7, h0;\n\t"
            "setp.geu.and.f32 k0|z0, e0, %10, h0;\n\tsetp.geu.and.f32 k1|z1, e1, %10, h1;\n\t"
            "selp.f32 x0, x0, 0f00000000, k0;\n\tselp.f32 x1, x1, 0f00000000, k1;\n\t"
            "mov.b64 A, {x0, x1};\n\tmul.rn.f32x2 %0, A, %1;\n\t"
            "selp.f32 t0, e0, t0, k0;\n\tselp.f32 t1, e1, t1, k1;\n\t"
            "@z0 or.b32 t0, t0, 0x80000000;\n\t@z1 or.b32 t1, t1, 0x80000000;\n\t"
            "mov.b64 %1, {t0, t1};\n\t@k0 mov.u32 %2, %11;\n\t@k1 mov.u32 %3, %11;\n\t"
            "mov.b32 %4, x0;\n\tmov.b32 %5, x1;\n\t}"
            : "=l"(w), "+l"(T), "+r"(last0), "+r"(last1), "=r"(a0), "=r"(a1)
            : "l"(s), "f"(thr), "l"(al), "l"(te), "f"(tmin), "r"(pos), "r"((int)on));
    return w;
}

__device__ __forceinline__ uint32_t bits_of(float v) { return __float_as_uint(v); }
__device__ __forceinline__ uint32_t bits_of(uint32_t v) { return v; }

// Forward pass of the groups of one warp (`unit`) of a frame with ntiles tiles.
template <int PX, int SUBS, bool COUNT>
__device__ __forceinline__ void forward_unit(const RenderFwdArgs& a, uint32_t unit, uint32_t ntiles) {
    using LN = Lanes<PX, SUBS>;
    constexpr int U = PX == 2 ? 4 : 2;
    __shared__ Entry s_e[LN::TPW][32];
    const LN ln(unit);
    const CamK& c = a.cam;
    const uint32_t full = 0xffffffffu;
    uint32_t tile = ln.index < ntiles ? a.order[ln.index] : 0u;
    const bool live = ln.index < ntiles && tile < ntiles;
    if (ln.index < ntiles && !live && ln.tl == 0) debug_fail(a.status);   // an order not written by gs_bin_sort
    if (!live) tile = 0;
    const int tx = (int)tile % c.tiles_x, ty = (int)tile / c.tiles_x;
    const int x0 = tx * (kSub * LN::SX), y0 = ty * c.tile_h;
    const int ly = kSub * ln.sy + ln.row, py = y0 + ly, px0 = x0 + kSub * ln.sx + ln.col;
    const f32x2 lyf = pack2((float)ly, (float)ly);
    uint32_t start = 0, len = 0;
    if (live) {
        const uint2 r = *reinterpret_cast<const uint2*>(a.ranges + 2 * tile);
        start = r.x;
        len = r.y - r.x;
        if (GS_DEBUG && (r.y < r.x || r.y > a.capacity)) {   // a range outside the instance lists
            if (ln.tl == 0) debug_fail(a.status);
            len = 0;
        }
    }
    uint32_t* const bits = a.contrib + (size_t)((start >> 5) + tile) * SUBS + ln.sub;
    const float amax = a.cfg.alpha_max, tmin = a.cfg.T_min;
    const float log2_amin = __log2f(a.cfg.alpha_min), lo_care = log2_care(amax);
    const uint32_t* const vals = a.vals + start;
    const f32x2 one = pack2(1.f, 1.f), neg = pack2(-1.f, -1.f);

    // a pixel is done (stopped, or outside the image) when its T is negative
    f32x2 T[LN::PAIRS], Cr[LN::PAIRS], Cg[LN::PAIRS], Cb[LN::PAIRS];
    uint32_t last[PX], nblended[PX];
#pragma unroll
    for (int i = 0; i < PX; ++i) last[i] = nblended[i] = 0;
#pragma unroll
    for (int i = 0; i < LN::PAIRS; ++i) {
        const bool row_in = live && py < c.H;
        T[i] = pack2(row_in && px0 + 2 * i < c.W ? 1.0f : -1.0f, row_in && px0 + 2 * i + 1 < c.W ? 1.0f : -1.0f);
        Cr[i] = Cg[i] = Cb[i] = pack2(0.f, 0.f);
    }

    Fetched fetched;
    uint32_t ids[LN::ROUNDS];
    if (a.n > 0) {
        fetch_ids<LN::ROUNDS, LN::SL>(ids, vals, (uint32_t)ln.tl, len);
        if (LN::AHEAD) {
            fetch_splat(fetched, ids[0], a);
            fetch_ids<LN::ROUNDS, LN::SL>(ids, vals, 32u + (uint32_t)ln.tl, len);
        }
    }
    const uint32_t gmask = LN::GL == 32 ? full : ((1u << (LN::GL & 31)) - 1u) << (ln.group * LN::GL & 31);
    for (uint32_t base = 0;; base += 32) {
        bool alive = false;
#pragma unroll
        for (int i = 0; i < LN::PAIRS; ++i) {
            float t[2];
            unpack2(T[i], t[0], t[1]);
            alive |= t[0] > 0.f || t[1] > 0.f;
        }
        const uint32_t who = __ballot_sync(full, alive && base < len);
        if (who == 0) break;
        const bool active = (who & gmask) != 0;                // this group
        // stage the next 32 splats of the tile; bit k of a group's word: splat base + k can
        // reach its sub-block
        uint32_t word = 0, careful = 0;
        __syncwarp();
#pragma unroll
        for (int r = 0; r < LN::ROUNDS; ++r) {
            const int k = ln.tl + r * LN::SL;
            uint32_t reach = 0;
            bool care = false;
            if (base + (uint32_t)k < len) {
                if (!LN::AHEAD) fetch_splat(fetched, ids[r], a);
                Staged st;
                stage_splat(fetched.xy, fetched.conic, x0, y0, log2_amin, st);
                s_e[ln.slot][k] = entry_of(st, fetched.rgb, fetched.id);
                care = needs_care(st, fetched.rgb, lo_care);
                const int s0 = ln.sub0();
#pragma unroll
                for (int s = 0; s < LN::NS; ++s) {
                    const int sx = (s0 + s) % LN::SX, sy = (s0 + s) / LN::SX;
                    if (sub_reach(st, st.a.x + (float)(kSub * sx), st.a.y + (float)(kSub * sy))) reach |= 1u << s;
                }
            }
#pragma unroll
            for (int s = 0; s < LN::NS; ++s) {
                const uint32_t bits = window_bits(ln, (reach >> s) & 1u, r);
                if (ln.group % LN::NS == s) word |= bits;
            }
            if (!LN::ONE_PATH) careful |= window_bits(ln, care, r);
        }
        if (!active) word = 0;
        // one path for the warp and the window: groups on different ones would take turns (1M opaque
        // splats at 1080p: 176 us, so 134); a group's own choice per iteration where blended splats are
        // counted, as care costs more there (3M: 459 us the one way, 450 the other)
        const bool care = LN::ONE_PATH || (!COUNT && __any_sync(full, (word & careful) != 0));
        // in flight while this window is blended
        if (LN::AHEAD) fetch_splat(fetched, ids[0], a);
        fetch_ids<LN::ROUNDS, LN::SL>(ids, vals, base + (LN::AHEAD ? 64u : 32u) + (uint32_t)ln.tl, len);
        __syncwarp();
        uint32_t mb = 0;   // bit k: a pixel of this lane blended splat base + k
        while (word) {
            // the next U splats of the group, front to back
            Entry e[U];
            uint32_t bit[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int k = word ? __ffs(word) - 1 : 0;
                bit[u] = word & (0u - word);                   // 0: none left
                word &= word - 1u;
                e[u] = s_e[ln.slot][k];
            }
            auto blend = [&](auto care) {
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const RowPairs row = splat_row(ln, e[u], lyf);
                    const float thr = __fsub_rn(low(e[u].lo), log2_amin);
                    const bool on = bit[u] != 0 && !(low(row.qq) > thr);   // s >= q^2: else the whole row skips
                    const uint32_t pos = base + 32u - (uint32_t)__clz((int)bit[u]);
                    uint32_t any = 0;
#pragma unroll
                    for (int i = 0; i < LN::PAIRS; ++i) {
                        const float jj = ln.j(2 * i);
                        const f32x2 p = fma2(pack2(jj, jj), row.dp, row.p0[i & 1]);
                        const f32x2 s = fma2(p, p, row.qq);
                        const f32x2 x = fma2(s, neg, e[u].lo);     // lo - s
                        float xv[2], al[2];
                        unpack2(x, xv[0], xv[1]);
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            al[h] = hw_exp2(xv[h]);
                            if (decltype(care)::value) al[h] = fminf(amax, al[h]);
                        }
                        const f32x2 al2 = pack2(al[0], al[1]);
                        const f32x2 te = mul2(T[i], fma2(al2, neg, one));   // T (1 - alpha)
                        uint32_t a0, a1;
                        const f32x2 w = blend_pair(s, thr, al2, te, tmin, pos, on, T[i], last[2 * i], last[2 * i + 1], a0, a1);
                        any |= a0 | a1;
                        if (COUNT) {
                            nblended[2 * i] += a0 != 0;
                            nblended[2 * i + 1] += a1 != 0;
                        }
                        Cr[i] = fma2(w, e[u].r, Cr[i]);
                        Cg[i] = fma2(w, e[u].g, Cg[i]);
                        Cb[i] = fma2(w, e[u].b, Cb[i]);
                    }
                    if (any) mb |= bit[u];
                }
            };
            uint32_t mine = 0;
            if (COUNT && !LN::ONE_PATH)
#pragma unroll
                for (int u = 0; u < U; ++u) mine |= bit[u] & careful;
            if (LN::ONE_PATH || care || mine) blend(std::true_type{});
            else blend(std::false_type{});
        }
#pragma unroll
        for (int m = LN::GL / 2; m > 0; m >>= 1) mb |= __shfl_xor_sync(full, mb, m);
        // every word the group walks is written: the backward pass reads no other
        if (active && ln.lane % LN::GL == 0) bits[(size_t)(base >> 5) * SUBS] = mb;
    }
    // Out through shared memory, two planes at a time, so that consecutive lanes store consecutive
    // pixels: stored from the lane that blended it, each pixel of a warp's store lies in a row of its
    // own (1,000 splats at 1080p: 46 us, so 16 at any width; 3M 408 -> 406).
    float t[PX], r[PX], g[PX], b[PX];
#pragma unroll
    for (int i = 0; i < LN::PAIRS; ++i) {
        unpack2(T[i], t[2 * i], t[2 * i + 1]);
        unpack2(Cr[i], r[2 * i], r[2 * i + 1]);
        unpack2(Cg[i], g[2 * i], g[2 * i + 1]);
        unpack2(Cb[i], b[2 * i], b[2 * i + 1]);
    }
#pragma unroll
    for (int i = 0; i < PX; ++i) {
        t[i] = fabsf(t[i]);
        r[i] += t[i] * a.bg[0];
        g[i] += t[i] * a.bg[1];
        b[i] += t[i] * a.bg[2];
    }
    constexpr int ROW = kSub + 1, BLOCK = kSub * ROW;   // words of a row and of a sub-block (no bank conflicts)
    static_assert(sizeof(s_e) >= 2 * LN::GW * BLOCK * sizeof(uint32_t), "two planes of the warp's sub-blocks");
    uint32_t* const s_px = reinterpret_cast<uint32_t*>(s_e) + ln.group * (2 * BLOCK);
    const size_t P = (size_t)c.W * c.H;
    auto store = [&](auto* p0, const auto (&v0)[PX], auto* p1, const auto (&v1)[PX], bool second) {
        __syncwarp();
#pragma unroll
        for (int i = 0; i < PX; ++i) {
            uint32_t* const w = s_px + ln.row * ROW + ln.col + i;
            w[0] = bits_of(v0[i]);
            if (second) w[BLOCK] = bits_of(v1[i]);
        }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < PX; ++j) {
            const int q = j * LN::GL + ln.lane % LN::GL, row = q / kSub, col = q % kSub;
            const int x = x0 + kSub * ln.sx + col, y = y0 + kSub * ln.sy + row;
            if (live && x < c.W && y < c.H) {
                const size_t p = (size_t)y * c.W + x;
                reinterpret_cast<uint32_t*>(p0)[p] = s_px[row * ROW + col];
                if (second) reinterpret_cast<uint32_t*>(p1)[p] = s_px[BLOCK + row * ROW + col];
            }
        }
    };
    store(a.out_rgb, r, a.out_rgb + P, g, true);
    store(a.out_rgb + 2 * P, b, a.out_T, t, true);
    store(a.out_last, last, a.out_count, nblended, COUNT);
}

// One warp per block.  A single frame reads its arguments straight from the parameter bank; a
// batch copies its frame's block of arguments into registers once (measured on four 1M-Gaussian
// views: half the instructions of a shared-memory copy, whose compiled form executed the blend
// loop's skipped pairs at the cost of blended ones).
template <int PX, int SUBS, int MAXF, bool COUNT>
__global__ void __launch_bounds__(32, 16) k_render_forward_t(const __grid_constant__ Multi<RenderFwdArgs, MAXF> m) {
    if constexpr (MAXF == 1) {
        forward_unit<PX, SUBS, COUNT>(m.a[0], blockIdx.x, (uint32_t)(m.a[0].cam.tiles_x * m.a[0].cam.tiles_y));
    } else {
        const int f = find_frame<MAXF>(m.base, m.frames, blockIdx.x);
        const RenderFwdArgs a = m.a[f];
        forward_unit<PX, SUBS, COUNT>(a, blockIdx.x - m.base[f], (uint32_t)(a.cam.tiles_x * a.cam.tiles_y));
    }
}

// A lane's PX consecutive pixels of one plane (src: the first), 0 outside the image (`in` pixels are
// inside), as quads or pairs if `wide`: eight loads of one pixel each read a sector eight times, from L2
// where the rows' stride makes them share a cache set (1,000 splats at 1080p: 33 us, so 24).
template <int PX>
constexpr int kRowVec = PX >= 4 ? 4 : 2;
template <int PX, typename T>
__device__ __forceinline__ void load_row(const T* src, int in, bool wide, T (&v)[PX]) {
    constexpr int VEC = kRowVec<PX>;
    struct __align__(sizeof(T) * VEC) Vec { T e[VEC]; };
    if (wide) {
#pragma unroll
        for (int i = 0; i < PX; i += VEC) {
            const Vec x = *reinterpret_cast<const Vec*>(src + i);
#pragma unroll
            for (int k = 0; k < VEC; ++k) v[i + k] = x.e[k];
        }
    } else {
#pragma unroll
        for (int i = 0; i < PX; ++i) v[i] = i < in ? src[i] : T(0);
    }
}

// Backward pass of the groups of one warp (`unit`) of a frame with ntiles tiles.
template <int PX, int SUBS, bool LIMIT>
__device__ __forceinline__ void backward_unit(const RenderBwdArgs& a, uint32_t unit, uint32_t ntiles) {
    using LN = Lanes<PX, SUBS>;
    constexpr int U = 2;
    __shared__ Entry s_e[LN::TPW][32];
    const LN ln(unit);
    const CamK& c = a.cam;
    const uint32_t full = 0xffffffffu;
    uint32_t tile = ln.index < ntiles ? a.order[ln.index] : 0u;
    const bool live = ln.index < ntiles && tile < ntiles;
    if (ln.index < ntiles && !live && ln.tl == 0) debug_fail(a.status);   // an order not written by gs_bin_sort
    if (!live) tile = 0;
    const int tx = (int)tile % c.tiles_x, ty = (int)tile / c.tiles_x;
    const int x0 = tx * (kSub * LN::SX), y0 = ty * c.tile_h;
    const int ly = kSub * ln.sy + ln.row, py = y0 + ly, px0 = x0 + kSub * ln.sx + ln.col;
    const f32x2 lyf = pack2((float)ly, (float)ly);
    uint32_t start = 0, len = 0;
    if (live) {
        const uint2 r = *reinterpret_cast<const uint2*>(a.ranges + 2 * tile);
        start = r.x;
        len = r.y - r.x;
        if (GS_DEBUG && (r.y < r.x || r.y > a.capacity)) {
            if (ln.tl == 0) debug_fail(a.status);
            len = 0;
        }
    }
    const uint32_t* const bits = a.contrib + (size_t)((start >> 5) + tile) * SUBS + ln.sub;
    const float amax = a.cfg.alpha_max;
    const float log2_amin = __log2f(a.cfg.alpha_min), lo_care = log2_care(amax);
    const size_t P = (size_t)c.W * c.H;
    const uint32_t* const vals = a.vals + start;
    float* const grad2d = a.grad2d;
    const f32x2 one = pack2(1.f, 1.f), neg = pack2(-1.f, -1.f);

    // Per pixel: T, -R . dL/dC (only this projection of the colour behind is ever needed), dL/dC.
    f32x2 T[LN::PAIRS], nRd[LN::PAIRS], dLr[LN::PAIRS], dLg[LN::PAIRS], dLb[LN::PAIRS];
    uint32_t mylast[PX];
    // LIMIT: the first `skip` blended splats met from the back (all but the grad_limit front-most)
    // get no gradient; the recurrences for T and R . dL/dC still run through them
    uint32_t skip[PX], seen[PX];
    uint32_t gmax = 0;
    bool odd = false;
    const int in = live && py < c.H ? min(PX, max(0, c.W - px0)) : 0;   // the lane's pixels inside the image
    const size_t first = in ? (size_t)py * c.W + px0 : 0;
    float tf[PX], dr_[PX], dg_[PX], db_[PX];
    auto wide = [&](const void* p) { return in == PX && reinterpret_cast<uintptr_t>(p) % (4 * kRowVec<PX>) == 0; };
    auto load = [&](auto wide_of) {
        load_row<PX>(a.last + first, in, wide_of(a.last + first), mylast);
        load_row<PX>(a.T_final + first, in, wide_of(a.T_final + first), tf);
        load_row<PX>(a.dL_drgb + first, in, wide_of(a.dL_drgb + first), dr_);
        load_row<PX>(a.dL_drgb + P + first, in, wide_of(a.dL_drgb + P + first), dg_);
        load_row<PX>(a.dL_drgb + 2 * P + first, in, wide_of(a.dL_drgb + 2 * P + first), db_);
    };
    if constexpr (LIMIT) {   // short of registers: one choice for all planes (500k Limited-BW 179 -> 177 us)
        if (wide(a.last + first) && wide(a.T_final + first) && wide(a.dL_drgb + first) && wide(a.dL_drgb + P + first))
            load([](const void*) { return true; });
        else
            load([](const void*) { return false; });
        load_row<PX>(a.count + first, in, false, skip);
    } else {
        load(wide);
    }
#pragma unroll
    for (int i = 0; i < PX; ++i) {
        mylast[i] = min(mylast[i], len);   // last positions never exceed the tile's list
        gmax = max(gmax, mylast[i]);
        if (i >= in) tf[i] = 1.0f;
        const uint32_t lim = (uint32_t)a.cfg.grad_limit;
        skip[i] = LIMIT && skip[i] > lim ? skip[i] - lim : 0u;
        seen[i] = 0;
    }
#pragma unroll
    for (int i = 0; i < LN::PAIRS; ++i) {
        const float dr[2] = {dr_[2 * i], dr_[2 * i + 1]}, dg[2] = {dg_[2 * i], dg_[2 * i + 1]},
                    db[2] = {db_[2 * i], db_[2 * i + 1]};
        T[i] = pack2(tf[2 * i], tf[2 * i + 1]);
        dLr[i] = pack2(dr[0], dr[1]);
        dLg[i] = pack2(dg[0], dg[1]);
        dLb[i] = pack2(db[0], db[1]);
        float rd[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            rd[h] = a.bg[0] * dr[h] + a.bg[1] * dg[h] + a.bg[2] * db[h];
            // not finite, or so large that a product could overflow
            odd |= !(fabsf(dr[h]) <= kWild && fabsf(dg[h]) <= kWild && fabsf(db[h]) <= kWild && fabsf(rd[h]) <= kWild);
        }
        nRd[i] = pack2(-rd[0], -rd[1]);
    }
#pragma unroll
    for (int m = LN::GL / 2; m > 0; m >>= 1) gmax = max(gmax, __shfl_xor_sync(full, gmax, m));
    const uint32_t wmax = __reduce_max_sync(full, gmax);
    uint32_t nblend = 0;
    int slot0, nslots;
    reduce_slots<LN::GL>(ln.lane, slot0, nslots);
    // constant factors of the (up to two) totals this lane adds: the log2-scaled (p, q) back to
    // the whitened frame, and the sign (the sums are of negated terms)
    auto factor = [](int s) { return s < 2 ? -kUnscale : s < 5 ? -kLn2 : -1.0f; };
    const float f0 = factor(slot0), f1 = factor(slot0 + 1);

    // the contribution word of window w: the splats some pixel of the group blended
    auto word_of = [&](int w) {
        uint32_t v = 0;
        const uint32_t base = 32u * (uint32_t)w;
        if (w >= 0 && base < gmax) {
            v = bits[(size_t)w * SUBS];
            if (gmax - base < 32) v &= (1u << (gmax - base)) - 1u;
        }
        return v;
    };
    Fetched fetched;
    uint32_t ids[LN::ROUNDS];
    const int wlast = (int)((wmax + 31) / 32) - 1;
    uint32_t next = word_of(wlast);
    if (wlast >= 0) {
        fetch_ids<LN::ROUNDS, LN::SL>(ids, vals, 32u * (uint32_t)wlast + (uint32_t)ln.tl, len);
        if (LN::AHEAD) {
            fetch_splat(fetched, ids[0], a);
            fetch_ids<LN::ROUNDS, LN::SL>(ids, vals, 32u * (uint32_t)max(0, wlast - 1) + (uint32_t)ln.tl, len);
        }
    }
    for (int w = wlast; w >= 0; --w) {
        const uint32_t base = 32u * (uint32_t)w;
        uint32_t word = next;
        next = word_of(w - 1);
        uint32_t careful = 0;
        __syncwarp();
#pragma unroll
        for (int r = 0; r < LN::ROUNDS; ++r) {
            if (!LN::AHEAD) fetch_splat(fetched, ids[r], a);
            Staged st;
            stage_splat(fetched.xy, fetched.conic, x0, y0, log2_amin, st);
            s_e[ln.slot][ln.tl + r * LN::SL] = entry_of(st, fetched.rgb, fetched.id);
            if (!LN::ONE_PATH) careful |= window_bits(ln, needs_care(st, fetched.rgb, lo_care), r);
        }
        // care: alpha may be clamped (its gradient then stops), or a product of a pixel that does not
        // blend a splat may not be finite (`odd` dL/dC, a wild colour or conic): its terms are then
        // cleared before they meet a sum or the pixel's recurrence, 0 x inf included.  Without care
        // they are finite (kWild), and 0 as alpha is.  One path for the warp and the window: groups
        // on different ones would take turns (1M opaque splats at 1080p: 267 us, so 214).
        const bool care_w = LN::ONE_PATH || __any_sync(full, odd || (word & careful) != 0);
        // in flight while this window is walked
        if (LN::AHEAD) fetch_splat(fetched, ids[0], a);
        fetch_ids<LN::ROUNDS, LN::SL>(ids, vals, 32u * (uint32_t)max(0, w - (LN::AHEAD ? 2 : 1)) + (uint32_t)ln.tl, len);
        __syncwarp();
        // Groups that walk the same positions (splats that cover all the warp's sub-blocks) add their
        // sums as one: the atomics of a few splats that cover the frame meet at few addresses (50 of
        // them at 1080p: 855 us, so 140; 1280x720 217 -> 119).  Decided per window and in a loop of
        // its own: tested per splat in the common loop it cost the ordinary frame 3 % (3M: 596 us,
        // 610; so 589).
        const uint32_t word0 = __shfl_sync(full, word, 0);
        const bool joint = LN::GW > 1 && __all_sync(full, word == word0);
        auto walk = [&](auto joint_c) {
        while (__any_sync(full, word != 0)) {   // every group its own splats, back to front
            Entry es[U];
            uint32_t at[U];
            float qs[U];
            f32x2 sums[U][6];
            bool any_grad = false;
#pragma unroll
            for (int u = 0; u < U; ++u) {   // the next U splats of the group, back to front
                const int k = word ? 31 - __clz((int)word) : 0;
                at[u] = word ? base + (uint32_t)k : 0xffffffffu;
                word &= ~(1u << k);
                es[u] = s_e[ln.slot][k];
            }
            auto blend = [&](auto care_c) {
            constexpr bool care = decltype(care_c)::value;
#pragma unroll
            for (int u = 0; u < U; ++u) {
            const Entry& e = es[u];
            const RowPairs row = splat_row(ln, e, lyf);
            const float thr = __fsub_rn(low(e.lo), log2_amin);
            // past every last position when the group is idle or, as s >= q^2, the whole row skips
            const uint32_t pos = low(row.qq) > thr ? 0xffffffffu : at[u];
            f32x2 S0 = 0, S1 = 0, S2 = 0, Gr = 0, Gg = 0, Gb = 0;
            bool contrib = false;
#pragma unroll
                for (int i = 0; i < LN::PAIRS; ++i) {
                    const float jj = ln.j(2 * i);
                    const f32x2 p = fma2(pack2(jj, jj), row.dp, row.p0[i & 1]);
                    const f32x2 s = fma2(p, p, row.qq);
                    const f32x2 x = fma2(s, neg, e.lo);
                    float sv[2], xv[2], na[2], om[2];
                    unpack2(s, sv[0], sv[1]);
                    unpack2(x, xv[0], xv[1]);
                    bool blends[2], grad[2], grad_a[2];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float oG = hw_exp2(xv[h]);
                        const bool ok = pos < mylast[2 * i + h] && !(sv[h] > thr);
                        if (ok) ++nblend;
                        blends[h] = grad[h] = ok;
                        if (LIMIT) {
                            grad[h] = ok && seen[2 * i + h] >= skip[2 * i + h];
                            seen[2 * i + h] += ok;
                            contrib |= grad[h];
                        }
                        grad_a[h] = grad[h] && (!care || oG <= amax);
                        na[h] = ok ? (care ? fmaxf(-amax, -oG) : -oG) : 0.f;       // -alpha; 0 when skipped
                    }
                    auto only = [](f32x2 v, const bool (&on)[2]) {
                        float y[2];
                        unpack2(v, y[0], y[1]);
                        return pack2(on[0] ? y[0] : 0.f, on[1] ? y[1] : 0.f);
                    };
                    const f32x2 na2 = pack2(na[0], na[1]);
                    unpack2(add2(na2, one), om[0], om[1]);                     // 1 - alpha >= 0.01
                    const f32x2 Ti = mul2(T[i], pack2(hw_rcp(om[0]), hw_rcp(om[1])));   // T_i = T_{i+1} / (1 - alpha_i)
                    f32x2 nw = mul2(na2, Ti);
                    // dL/dalpha = T_i (c_i - R_{i+1}) . dL/dC;  R_i . dL/dC = R_{i+1} . dL/dC + alpha (c_i - R_{i+1}) . dL/dC
                    f32x2 diff = fma2(e.r, dLr[i], fma2(e.g, dLg[i], fma2(e.b, dLb[i], nRd[i])));
                    if (care) diff = only(diff, blends);
                    nRd[i] = fma2(na2, diff, nRd[i]);
                    T[i] = Ti;
                    // -dL/d(power) = -alpha dL/dalpha; its sums with 1, p, p^2 (q is the row's)
                    f32x2 ndp = mul2(nw, diff), pg = p;
                    if (care) {
                        ndp = only(ndp, grad_a);
                        pg = only(p, grad_a);
                        Gr = add2(Gr, only(mul2(nw, dLr[i]), grad));
                        Gg = add2(Gg, only(mul2(nw, dLg[i]), grad));
                        Gb = add2(Gb, only(mul2(nw, dLb[i]), grad));
                    } else {
                        if (LIMIT) {
                            nw = only(nw, grad);
                            ndp = only(ndp, grad);
                        }
                        Gr = fma2(nw, dLr[i], Gr);
                        Gg = fma2(nw, dLg[i], Gg);
                        Gb = fma2(nw, dLb[i], Gb);
                    }
                    const f32x2 ndpp = mul2(ndp, pg);
                    S0 = add2(S0, ndp);
                    S1 = add2(S1, ndpp);
                    S2 = fma2(ndpp, pg, S2);
                }
            sums[u][0] = S0; sums[u][1] = S1; sums[u][2] = S2;
            sums[u][3] = Gr; sums[u][4] = Gg; sums[u][5] = Gb;
            qs[u] = care && (S0 | S1) == 0 ? 0.f : low(row.q);   // no term of this row: q may be infinite
            any_grad |= contrib;
            }
            };
            if (LN::ONE_PATH || care_w) blend(std::true_type{});
            else blend(std::false_type{});
            if (LIMIT && !__any_sync(full, any_grad)) continue;
            float v[U][9];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const float q = qs[u], t0 = sum2(sums[u][0]), t1 = sum2(sums[u][1]), qt0 = q * t0;
                v[u][0] = t1; v[u][1] = qt0; v[u][2] = sum2(sums[u][2]);
                v[u][3] = q * t1; v[u][4] = q * qt0; v[u][5] = es[u].ko * t0;
                v[u][6] = sum2(sums[u][3]); v[u][7] = sum2(sums[u][4]); v[u][8] = sum2(sums[u][5]);
            }
            bool as_one = decltype(joint_c)::value;
            if (LN::TPW > 1 && decltype(joint_c)::value) {   // two tiles may list other splats at a position
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const uint32_t id0 = __shfl_sync(full, es[u].id, 0);
                    const bool same = __all_sync(full, es[u].id == id0);
                    as_one = as_one && same;
                }
            }
            if (LN::GW > 1 && as_one) {   // warp-uniform
                group_reduce9<32, U>(v, ln.lane);
                int lane = ln.lane, slot, n;
                asm volatile("" : "+r"(lane));   // this path's slots are worked out here, not kept in registers
                reduce_slots<32>(lane, slot, n);
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (at[u] != 0xffffffffu && n > 0) atomicAdd(grad2d + 12 * (size_t)es[u].id + slot, factor(slot) * v[u][0]);
            } else {
                group_reduce9<LN::GL, U>(v, ln.lane);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (at[u] != 0xffffffffu) {
                        float* dst = grad2d + 12 * (size_t)es[u].id + slot0;
                        if (nslots > 0) atomicAdd(dst, f0 * v[u][0]);
                        if (nslots > 1) atomicAdd(dst + 1, f1 * v[u][1]);
                    }
                }
            }
        }
        };
        if constexpr (LN::GW > 1) {
            if (joint) walk(std::true_type{});
            else walk(std::false_type{});
        } else {
            walk(std::false_type{});
        }
    }
    const uint32_t wblend = __reduce_add_sync(full, nblend);
    if (ln.lane == 0 && wblend) atomicAdd(a.blended, (unsigned long long)wblend);
}

// One warp per block, arguments as in k_render_forward_t.
template <int PX, int SUBS, int MAXF, bool LIMIT>
__global__ void __launch_bounds__(32, 12) k_render_backward_t(const __grid_constant__ Multi<RenderBwdArgs, MAXF> m) {
    if constexpr (MAXF == 1) {
        backward_unit<PX, SUBS, LIMIT>(m.a[0], blockIdx.x, (uint32_t)(m.a[0].cam.tiles_x * m.a[0].cam.tiles_y));
    } else {
        const int f = find_frame<MAXF>(m.base, m.frames, blockIdx.x);
        const RenderBwdArgs a = m.a[f];
        backward_unit<PX, SUBS, LIMIT>(a, blockIdx.x - m.base[f], (uint32_t)(a.cam.tiles_x * a.cam.tiles_y));
    }
}

// Warps of every frame, in frame order (frames without Gaussians still get their background
// and transmittance written); all frames of a batch share the tile shape.
template <int PX, int SUBS, typename A, int MAXF>
uint32_t unit_split(Multi<A, MAXF>& m) {
    constexpr int GW = Lanes<PX, SUBS>::GW;
    m.base[0] = 0;
    for (int f = 0; f < m.frames; ++f)
        m.base[f + 1] = m.base[f] + (uint32_t)((m.a[f].cam.tiles_x * m.a[f].cam.tiles_y * SUBS + GW - 1) / GW);
    return m.base[m.frames];
}

template <int PX, int SUBS, int MAXF>
cudaError_t forward_px(Multi<RenderFwdArgs, MAXF>& m, cudaStream_t s) {
    const uint32_t units = unit_split<PX, SUBS>(m);
    if (units == 0) return cudaSuccess;
    // gradient-limited frames also record the blended splats per pixel
    if (m.a[0].out_count) k_render_forward_t<PX, SUBS, MAXF, true><<<units, 32, 0, s>>>(m);
    else k_render_forward_t<PX, SUBS, MAXF, false><<<units, 32, 0, s>>>(m);
    return cudaGetLastError();
}

template <int PX, int SUBS, int MAXF>
cudaError_t backward_px(Multi<RenderBwdArgs, MAXF>& m, cudaStream_t s) {
    const uint32_t units = unit_split<PX, SUBS>(m);
    if (units == 0) return cudaSuccess;
    if (m.a[0].count) k_render_backward_t<PX, SUBS, MAXF, true><<<units, 32, 0, s>>>(m);
    else k_render_backward_t<PX, SUBS, MAXF, false><<<units, 32, 0, s>>>(m);
    return cudaGetLastError();
}

// Pixels per lane, by the 8x8 sub-blocks of the launch.  Eight per lane take the fewest
// instructions per splat (four sub-blocks share a warp's iteration) but give one warp per 16x16
// tile: a frame of few tiles leaves the chip idle behind its longest lists.  Measured, 8 / 4 / 2
// pixels per lane, forward and backward in us:
//   16 tiles (64x64, 5k Gaussians, 64 sub-blocks)        176 / 115 /  74    283 / 177 / 133
//   813x611 in 8x8 tiles (60k, 7,854)                     80 /  57 /  45    109 /  90 /  87
//   979x546 (150k, 8,680)                                125 /  90 /  84    154 / 123 / 145
//   1601x901 in 16x8 tiles (500k, 22,826, Limited-BW)    140 / 138 / 160    177 / 173 / 211
//   1920x1080 (200k, 32,640)                             165 / 180 / 217    239 / 285 / 376
//   1920x1080 (3M, 32,640)                               263 / 285 / 333    406 / 470 / 593
int forward_px_for(unsigned long long groups) { return groups < 12000 ? 2 : groups < 26000 ? 4 : 8; }
int backward_px_for(unsigned long long groups) { return groups < 3000 ? 2 : groups < 16000 ? 4 : 8; }

template <typename A, int MAXF>
unsigned long long sub_blocks(const Multi<A, MAXF>& m, int subs) {
    unsigned long long g = 0;
    for (int f = 0; f < m.frames; ++f) g += (unsigned long long)(m.a[f].cam.tiles_x * m.a[f].cam.tiles_y) * subs;
    return g;
}

template <int SUBS, int MAXF>
cudaError_t forward_subs(Multi<RenderFwdArgs, MAXF>& m, cudaStream_t s) {
    switch (forward_px_for(sub_blocks(m, SUBS))) {
        case 2: return forward_px<2, SUBS>(m, s);
        case 4: return forward_px<4, SUBS>(m, s);
        default: return forward_px<8, SUBS>(m, s);
    }
}

template <int SUBS, int MAXF>
cudaError_t backward_subs(Multi<RenderBwdArgs, MAXF>& m, cudaStream_t s) {
    switch (backward_px_for(sub_blocks(m, SUBS))) {
        case 2: return backward_px<2, SUBS>(m, s);
        case 4: return backward_px<4, SUBS>(m, s);
        default: return backward_px<8, SUBS>(m, s);
    }
}

}  // namespace

template <int MAXF>
cudaError_t launch_render_forward(Multi<RenderFwdArgs, MAXF>& m, cudaStream_t s) {
    const CamK& c = m.a[0].cam;   // all frames of a batch share the tile shape
    const int subs = (c.tile_w / kSub) * (c.tile_h / kSub);
    return subs == 4 ? forward_subs<4>(m, s) : subs == 2 ? forward_subs<2>(m, s) : forward_subs<1>(m, s);
}

template <int MAXF>
cudaError_t launch_render_backward(Multi<RenderBwdArgs, MAXF>& m, cudaStream_t s) {
    const CamK& c = m.a[0].cam;
    const int subs = (c.tile_w / kSub) * (c.tile_h / kSub);
    return subs == 4 ? backward_subs<4>(m, s) : subs == 2 ? backward_subs<2>(m, s) : backward_subs<1>(m, s);
}

template cudaError_t launch_render_forward<1>(Multi<RenderFwdArgs, 1>&, cudaStream_t);
template cudaError_t launch_render_forward<kMaxFrames>(Multi<RenderFwdArgs, kMaxFrames>&, cudaStream_t);
template cudaError_t launch_render_backward<1>(Multi<RenderBwdArgs, 1>&, cudaStream_t);
template cudaError_t launch_render_backward<kMaxFrames>(Multi<RenderBwdArgs, kMaxFrames>&, cudaStream_t);

}  // namespace gs
