// Projection and Precise Tile Intersection binning (Sec. 3.2) for sm_103a.
//
// k_project   one thread per (view, surfel) item: homogeneous transform T,
//             its adjugate about the projected centre, opacity-aware cutoff,
//             screen conic, SnugBox pixel range; appends visible items to a
//             compact list (unbounded conics to a per-view list instead).
//             Also counts each item's tiles (AccuTile per-row or per-column
//             intervals) into per-tile counters; a narrow item's pairs (tile,
//             place in the tile, item) go into a buffer in the same pass.
// k_emit      computes the double-float render records; one of its CTAs
//             scans the per-tile counts (tile ranges, total pairs, capacity,
//             the heavy-first tile order) while the others build records;
//             then stores the buffered pairs at their tile's cursor + place and
//             writes each wide item into a slot of each of its tiles (slot
//             order is arbitrary; the per-tile sort restores a total order).
//
// Every tile decision is taken in binary32 with the fixed operation order
// that the FP64 checker's binning mirror also follows, so tile lists compare
// bit for bit.  This translation unit is compiled with -fmad=false and
// spells each rounding with an _rn intrinsic, so no multiply-add is fused.
#include "fss_internal.cuh"
#include "kernels.cuh"

#include <algorithm>
#include <cmath>

namespace fss {

namespace {

__device__ __forceinline__ float fm(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float fa(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float fs(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float fdv(float a, float b) { return __fdiv_rn(a, b); }
__device__ __forceinline__ float fq(float a) { return __fsqrt_rn(a); }

// frexpf and ldexpf for the chain below, from the binary32 layout: for a
// normal x > 0, x = m 2^e with m in [1/2, 1) takes the exponent field and
// the mantissa bits; x 2^k (one rounding, as ldexpf) is a multiply by the
// exact power of two whenever 2^k is a normal number.  Other cases (zero,
// subnormal, non-finite, exponents out of that range) call the library.
__device__ __forceinline__ float frexp32(float x, int* e) {
    const uint32_t b = __float_as_uint(x);
    const uint32_t be = (b >> 23) & 0xffu;
    if (be == 0u || be == 0xffu || (b >> 31)) return frexpf(x, e);
    *e = (int)be - 126;
    return __uint_as_float((b & 0x807fffffu) | 0x3f000000u);
}
__device__ __forceinline__ float ldexp32(float x, int k) {
    if (k < -126 || k > 127) return ldexpf(x, k);
    return __fmul_rn(x, __uint_as_float((uint32_t)(k + 127) << 23));
}

// natural logarithm of x > 0 in binary32, the same operation sequence as the
// checker's binning mirror: x = m 2^e with m in [sqrt(1/2), sqrt(2)),
// ln m = 2 atanh(s), s = (m - 1)/(m + 1), series to s^9 (|s| <= 0.1716).
__device__ __forceinline__ float ln32(float x) {
    int e;
    float m = frexp32(x, &e);
    if (m < 0.70710677f) { m = fm(m, 2.0f); e = e - 1; }
    const float s = fdv(fs(m, 1.0f), fa(m, 1.0f));
    const float s2 = fm(s, s);
    float p = fm(s2, 1.0f / 9.0f);
    p = fm(fa(p, 1.0f / 7.0f), s2);
    p = fm(fa(p, 1.0f / 5.0f), s2);
    p = fm(fa(p, 1.0f / 3.0f), s2);
    p = fa(p, 1.0f);
    return fa(fm((float)e, 0.6931472f), fm(fm(2.0f, s), p));
}

// ---- double-float arithmetic (hi + lo, ~48 significant bits) ----------------
// Error-free sums (Knuth's two-sum, 6 operations) and products (the exact
// low part of a*b from one fused multiply-add), renormalised after every
// operation.  Used only for the per-surfel render record, whose ray-splat
// homography is ill-conditioned for surfels seen close to edge-on.
struct df {
    float hi, lo;
};
__device__ __forceinline__ df two_sum(float a, float b) {
    const float s = fa(a, b), bb = fs(s, a);
    return {s, fa(fs(a, fs(s, bb)), fs(b, bb))};
}
__device__ __forceinline__ df quick_two_sum(float s, float e) {
    const float h = fa(s, e);
    return {h, fs(e, fs(h, s))};
}
__device__ __forceinline__ df two_prod(float a, float b) {
    const float p = fm(a, b);
    return {p, fmaf(a, b, -p)};
}
__device__ __forceinline__ df dadd(df x, df y) {
    const df s = two_sum(x.hi, y.hi);
    return quick_two_sum(s.hi, fa(s.lo, fa(x.lo, y.lo)));
}
__device__ __forceinline__ df dneg(df x) { return {-x.hi, -x.lo}; }
__device__ __forceinline__ df dsub(df x, df y) { return dadd(x, dneg(y)); }
__device__ __forceinline__ df dmul(df x, df y) {
    const df p = two_prod(x.hi, y.hi);
    return quick_two_sum(p.hi, fa(p.lo, fa(fm(x.hi, y.lo), fm(x.lo, y.hi))));
}
__device__ __forceinline__ df dmulf(df x, float f) {
    const df p = two_prod(x.hi, f);
    return quick_two_sum(p.hi, fa(p.lo, fm(x.lo, f)));
}
__device__ __forceinline__ df dfrom(float a) { return {a, 0.0f}; }
// (R v)_r with binary32 R and double-float v
__device__ __forceinline__ void dmvec(const float* R, const df v[3], df o[3]) {
#pragma unroll
    for (int r = 0; r < 3; ++r) o[r] = dadd(dadd(dmulf(v[0], R[3 * r]), dmulf(v[1], R[3 * r + 1])), dmulf(v[2], R[3 * r + 2]));
}
__device__ __forceinline__ void dcross(const df a[3], const df b[3], df o[3]) {
    o[0] = dsub(dmul(a[1], b[2]), dmul(a[2], b[1]));
    o[1] = dsub(dmul(a[2], b[0]), dmul(a[0], b[2]));
    o[2] = dsub(dmul(a[0], b[1]), dmul(a[1], b[0]));
}

// (R v)_r = (R_r0 v0 + R_r1 v1) + R_r2 v2
__device__ __forceinline__ void mvec(const float* R, const float v[3], float o[3]) {
#pragma unroll
    for (int r = 0; r < 3; ++r) o[r] = fa(fa(fm(R[3 * r], v[0]), fm(R[3 * r + 1], v[1])), fm(R[3 * r + 2], v[2]));
}

__device__ __forceinline__ void crossf(const float a[3], const float b[3], float o[3]) {
    o[0] = fs(fm(a[1], b[2]), fm(a[2], b[1]));
    o[1] = fs(fm(a[2], b[0]), fm(a[0], b[2]));
    o[2] = fs(fm(a[0], b[1]), fm(a[1], b[0]));
}

// Q_ab = (m0_a m0_b + m1_a m1_b) - kk (m2_a m2_b), (A,B,C,D,E,F) = (Q00,Q01,Q11,Q02,Q12,Q22)
__device__ __forceinline__ void conic(const float m[9], float kk, float q[6]) {
    const int ia[6] = {0, 0, 1, 0, 1, 2}, ib[6] = {0, 1, 1, 2, 2, 2};
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const int a = ia[k], b = ib[k];
        const float s = fa(fm(m[a], m[b]), fm(m[3 + a], m[3 + b]));
        const float t = fm(kk, fm(m[6 + a], m[6 + b]));
        q[k] = fs(s, t);
    }
}

// centre and half extents of the ellipse q <= 0; false if it is empty
__device__ __forceinline__ bool ellipse(const float q[6], float& X0, float& Y0, float& hx, float& hy) {
    const float A = q[0], B = q[1], C = q[2], D = q[3], E = q[4], F = q[5];
    const float g = fs(fm(A, C), fm(B, B));
    X0 = fdv(fs(fm(B, E), fm(C, D)), g);
    Y0 = fdv(fs(fm(B, D), fm(A, E)), g);
    const float Fp = fa(fa(F, fm(D, X0)), fm(E, Y0));
    if (!(Fp < 0.0f)) return false;
    const float nF = -Fp;
    hx = fq(fdv(fm(nF, C), g));
    hy = fq(fdv(fm(nF, A), g));
    return true;
}

// pixel indices whose centres lie in [lo + 0.5, hi + 0.5], clipped to [0, n-1]
__device__ __forceinline__ bool pix_range(float lo, float hi, int n, int& a, int& b) {
    const float fl = ceilf(lo), fh = floorf(hi);
    if (!(fl <= fh)) return false;
    if (fh < 0.0f || fl > (float)(n - 1)) return false;
    a = fl < 0.0f ? 0 : (int)fl;
    b = fh > (float)(n - 1) ? n - 1 : (int)fh;
    return a <= b;
}

// S20b: pixel interval [a, b] (clipped to [lo_clip, hi_clip]) of the
// low-pass screen disc of radius^2 rd2 about the local origin on the strip
// [Sa, Sb] of the other coordinate; a > b when it misses the strip
__device__ __forceinline__ void disc_strip(float rd2, float Sa, float Sb, float origin, int lo_clip, int hi_clip,
                                           int& a, int& b) {
    a = 1;
    b = 0;
    const float Sn = Sa > 0.0f ? Sa : (Sb < 0.0f ? Sb : 0.0f);
    const float s2 = fm(Sn, Sn);
    if (!(s2 <= rd2)) return;
    const float hw = fq(fs(rd2, s2));
    const float fl = ceilf(fs(fa(-hw, origin), 0.5f)), fh = floorf(fs(fa(hw, origin), 0.5f));
    if (!(fl <= fh) || fh < (float)lo_clip || fl > (float)hi_clip) return;
    a = fl < (float)lo_clip ? lo_clip : (int)fl;
    b = fh > (float)hi_clip ? hi_clip : (int)fh;
}

// union of an ellipse interval [a, b] (empty if a > b) with a disc interval
__device__ __forceinline__ void hull_interval(int& a, int& b, int da, int db) {
    if (da > db) return;
    if (a > b) { a = da; b = db; return; }
    a = min(a, da);
    b = max(b, db);
}

// AccuTile: the inner tile interval of one outer tile line (a row of tiles
// when `rows`, else a column).  On a row strip [Ya, Yb] (local coordinates)
// the ellipse's extreme abscissae are its left/right tangent points when
// these fall inside the strip, else the roots of
//   A x^2 + 2(B y + D) x + (C y^2 + 2 E y + F) = 0
// at the nearer strip edge.  A column is the same with x and y exchanged
// (A <-> C, D <-> E, and the centre, half extents and pixel ranges), so one
// code path serves both, its operands picked by selects; both candidates of
// each side are computed and one is selected.  The lanes of a warp,
// holding different items and line kinds, then never split on these
// branches (a divergent version measured ~1800 cycles per call).
__device__ __forceinline__ bool accu_line(const BinRec& r, bool rows, int ts, int o, int& ta, int& tb) {
    const float A = rows ? r.A : r.C, C = rows ? r.C : r.A, D = rows ? r.D : r.E, E = rows ? r.E : r.D;
    const float X0 = rows ? r.X0 : r.Y0, hx = rows ? r.hx : r.hy;
    const float xc = rows ? r.xc : r.yc, yc = rows ? r.yc : r.xc;
    const int p0 = rows ? r.px0 : r.py0, p1 = rows ? r.px1 : r.py1;  // inner pixel range
    const int q0 = rows ? r.py0 : r.px0, q1 = rows ? r.py1 : r.px1;  // outer pixel range
    const int ra = max(o * ts, q0), rb = min(o * ts + ts - 1, q1);
    if (ra > rb) return false;
    const float Ya = fs(fa((float)ra, 0.5f), yc), Yb = fs(fa((float)rb, 0.5f), yc);
    int da = 1, db = 0;  // S20b
    if (r.flags & BR_LOWPASS) disc_strip(r.rd2, Ya, Yb, xc, p0, p1, da, db);
    if (!(r.flags & BR_ELL)) {
        if (da > db) return false;
        ta = da >> (__ffs(ts) - 1);
        tb = db >> (__ffs(ts) - 1);
        return true;
    }
    float ext[2];
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        const float Xs = side == 0 ? fs(X0, hx) : fa(X0, hx);
        const float t = fa(fm(r.B, Xs), E);
        const float Yt = fdv(-t, C);
        const bool tangent = Yt >= Ya && Yt <= Yb;
        const float Y = Yt < Ya ? Ya : Yb;
        const float bb = fa(fm(r.B, Y), D);
        const float cc = fa(fa(fm(fm(C, Y), Y), fm(fm(2.0f, E), Y)), r.F);
        float disc = fs(fm(bb, bb), fm(A, cc));
        disc = disc < 0.0f ? 0.0f : disc;
        const float sq = fq(disc), nb = -bb;
        const float root = fdv(side == 0 ? fs(nb, sq) : fa(nb, sq), A);
        ext[side] = tangent ? Xs : root;
    }
    const float fl = ceilf(fs(fa(ext[0], xc), 0.5f)), fh = floorf(fs(fa(ext[1], xc), 0.5f));
    const bool hit = fl <= fh && !(fh < (float)p0 || fl > (float)p1);
    int a = hit ? (fl < (float)p0 ? p0 : (int)fl) : 1;
    int b = hit ? (fh > (float)p1 ? p1 : (int)fh) : 0;
    hull_interval(a, b, da, db);
    if (a > b) return false;
    ta = a >> (__ffs(ts) - 1);
    tb = b >> (__ffs(ts) - 1);
    return true;
}

// Outer lines of an item's tile set: rows if the tile span in y does not
// exceed the span in x (or for the box modes), else columns (SnugBox's
// traversal over the smaller span).
struct Lines {
    int n;          // number of outer lines
    int first;      // first outer coordinate
    bool rows;      // outer loop over tile rows
    bool accurate;  // per-line AccuTile interval (else the full rectangle)
};

__device__ __forceinline__ Lines lines_of(const BinRec& r, int bin_mode) {
    Lines L;
    const int xs = r.tx1 - r.tx0 + 1, ys = r.ty1 - r.ty0 + 1;
    L.accurate = bin_mode == FSS_BIN_ACCU;
    L.rows = !L.accurate || ys <= xs;
    L.n = L.rows ? ys : xs;
    L.first = L.rows ? r.ty0 : r.tx0;
    return L;
}

// inner tile interval [a, b] of outer line `o` (an absolute tile row/column)
__device__ __forceinline__ bool line_interval(const BinRec& r, const Lines& L, int ts, int o, int& a, int& b) {
    if (!L.accurate) {
        a = L.rows ? r.tx0 : r.ty0;
        b = L.rows ? r.tx1 : r.ty1;
        return true;
    }
    return accu_line(r, L.rows, ts, o, a, b);
}

// view of item (items are view-major, view * N + surfel, < 2^32)
__device__ __forceinline__ int view_of_item(int64_t item, int64_t N) {
    return N >= ((int64_t)1 << 32) || item < N ? 0 : (int)((uint32_t)item / (uint32_t)N);
}

// Tile work of a warp's items spread over its lanes.  The outer lines of
// the 32 lanes' items are numbered in lane order ((lane, line) units) and
// taken 32 at a time, one per lane, so that an item with many lines no
// longer runs them one after another in its own lane while the others wait.
// The warp's slices of shared memory hold each lane's binning record and
// item, and the inclusive prefix of the line counts.
struct WarpLines {
    BinRec* br;      // [32]
    uint32_t* item;  // [32]
    int* pre;        // [32]
};

// every lane of the warp calls this with its own line count (0 for no
// item) after writing its record and item; returns the warp's total
__device__ __forceinline__ int warp_line_prefix(const WarpLines& w, int nl) {
    const int lane = threadIdx.x & 31;
    int incl = nl;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += y;
    }
    w.pre[lane] = incl;
    __syncwarp();
    return __shfl_sync(0xffffffffu, incl, 31);
}

// owner lane of unit u: the first lane whose inclusive prefix exceeds u
__device__ __forceinline__ int unit_owner(const WarpLines& w, int u) {
    int j = 0;
#pragma unroll
    for (int step = 16; step > 0; step >>= 1) j += w.pre[j + step - 1] <= u ? step : 0;
    return j;
}

}  // namespace

// S3 (centre), S4 (near plane), S5 (opacity) and S5b (conservative frustum
// test): the cheap culls, which remove most surfels of a view before the
// rest of the chain.  Returns false when the item is culled; pc and o as
// computed (o = 0 if the depth test failed first).
// the surfel inputs the culls read, loaded together so that their latencies overlap
struct CullIn {
    float pm[3];
    float o;
    float2 sc;
};
__device__ __forceinline__ CullIn load_cull_in(const float* __restrict__ means, const float* __restrict__ scales,
                                               const float* __restrict__ opac, int64_t s) {
    CullIn c;
    c.pm[0] = __ldg(means + 3 * s);
    c.pm[1] = __ldg(means + 3 * s + 1);
    c.pm[2] = __ldg(means + 3 * s + 2);
    c.o = __ldg(opac + s);
    c.sc = __ldg(reinterpret_cast<const float2*>(scales) + s);
    return c;
}

__device__ __forceinline__ bool early_culls(const CamDev& cam, const RParams& P, const CullIn& in, float pc[3],
                                            float& o) {
    float e[3];
    mvec(cam.R, in.pm, e);
#pragma unroll
    for (int i = 0; i < 3; ++i) pc[i] = fa(e[i], cam.t[i]);
    o = 0.0f;
    if (!(pc[2] > cam.near_plane)) return false;
    // S5
    o = in.o;
    if (!(o >= P.alpha_min)) return false;
    // S5b: the binning disk lies in the sphere of radius
    // rho = sqrt(k^2 (1 + 2^-10)) max(r_u, r_v) about the centre; if that
    // sphere is in front of the camera and its projection's bounding box
    // misses every pixel centre by more than a pixel, no pixel can be reached.
    const float2 scp = in.sc;
    const float kk = fm(fm(2.0f, ln32(fdv(o, P.alpha_min))), 1.0009765625f);
    const float rho = fa(fm(fm(fq(fmaxf(kk, 0.0f)), fmaxf(scp.x, scp.y)), 1.001f), 1e-6f);
    const float zlo = fs(pc[2], rho), zhi = fa(pc[2], rho);
    if (zlo > 0.0f) {
        const float xa = fs(pc[0], rho), xb = fa(pc[0], rho), ya = fs(pc[1], rho), yb = fa(pc[1], rho);
        // extremes of x/z and y/z over the box [xa, xb] x [ya, yb] x [zlo, zhi]
        const float uxmax = fdv(xb, xb >= 0.0f ? zlo : zhi), uxmin = fdv(xa, xa >= 0.0f ? zhi : zlo);
        const float uymax = fdv(yb, yb >= 0.0f ? zlo : zhi), uymin = fdv(ya, ya >= 0.0f ? zhi : zlo);
        const float pxmax = fa(fm(cam.fx, uxmax), cam.cx), pxmin = fa(fm(cam.fx, uxmin), cam.cx);
        const float pymax = fa(fm(cam.fy, uymax), cam.cy), pymin = fa(fm(cam.fy, uymin), cam.cy);
        // S5b': the low-pass filter's screen disc widens the margins
        const float mg = P.lowpass ? fa(0.5f, fq(fm(fmaxf(kk, 0.0f), 0.5f))) : 0.5f;
        if (pxmax < -mg || pxmin > fa((float)cam.W, mg) || pymax < -mg || pymin > fa((float)cam.H, mg))
            return false;
    }
    return true;
}

// A cheap superset of early_culls: true only for items that it culls.  The
// depth and opacity tests are its own; the frustum test takes the largest
// radius that an opacity of at most 1 can give (`rmax` times the larger scale:
// a larger sphere's box contains the smaller one's), multiplies instead of
// dividing, and leaves half a pixel and 1e-5 of the image coordinates for its
// rounding.  Opacities above 1 and non-finite values go on to early_culls.
__device__ __forceinline__ bool surely_culled(const CamDev& cam, const RParams& P, const CullIn& in, float rmax,
                                              float mmax) {
    float e[3], pc[3];
    mvec(cam.R, in.pm, e);
#pragma unroll
    for (int i = 0; i < 3; ++i) pc[i] = fa(e[i], cam.t[i]);
    if (!(pc[2] > cam.near_plane) || !(in.o >= P.alpha_min)) return true;
    const float r = fmaf(rmax, fmaxf(in.sc.x, in.sc.y), 1e-5f);
    const float zlo = pc[2] - r, zhi = pc[2] + r;
    const float sx = mmax + 1e-5f * (fabsf(cam.cx) + (float)cam.W), sy = mmax + 1e-5f * (fabsf(cam.cy) + (float)cam.H);
    const float xa = pc[0] - r, xb = pc[0] + r, ya = pc[1] - r, yb = pc[1] + r;
    const bool out = cam.fx * xb < -(cam.cx + sx) * (xb >= 0.0f ? zlo : zhi) ||
                     cam.fx * xa > ((float)cam.W + sx - cam.cx) * (xa >= 0.0f ? zhi : zlo) ||
                     cam.fy * yb < -(cam.cy + sy) * (yb >= 0.0f ? zlo : zhi) ||
                     cam.fy * ya > ((float)cam.H + sy - cam.cy) * (ya >= 0.0f ? zhi : zlo);
    return out && zlo > 0.0f && in.o <= 1.0f;
}

constexpr int PROJ_THREADS = 256;

// ---------------------------------------------------------------------------
// k_project: (view, surfel) items, ROUNDS * PER * 256 per CTA
//
// Stage A drops the items that the cheap superset of the culls is sure about,
// one thread per item, and queues the rest in shared memory; stage B runs the
// exact culls and the chain one thread per queued item, so the few visible
// surfels of a view fill whole warps instead of one lane in each.  A visible
// item with a bounded conic is appended to the narrow list, or to the wide list
// when its outer rectangle has more than WIDE_TILES tiles; an unbounded item
// goes to its view's list instead (every tile of the view includes it).  A
// narrow item's pairs are made here: each takes the next slot of its tile (the
// value its add to the tile's counter returns) and goes into a pair buffer as
// (tile, slot, item), so that k_emit only has to place them once the tiles'
// first places are known.  A wide item only counts its tiles.  Appends and gradient-slot claims are
// aggregated per warp.
//
// PER = 4 packs stage B well where most items are culled; PER = 1 spreads few
// items over the SMs: below 1024 items per SM (1,000 surfels in a 128 x 128
// frame: 66 -> 41 us for the whole forward, with PER = 4 62; 150k in a room 73
// -> 69, 71; 300k 87 -> 89, 85).  From 4096 and 8192 items per SM a CTA runs stage A
// two and three times before its stage B: the survivors of 1024 items (a twentieth)
// leave most of its warps without a stage B, whose chain the CTA waits for, and the CTAs
// are one wave again (4 an SM).  Whole forwards, one / two / three rounds: 800k items
// 116 / 110 / 113 us, 1M 121 / 115 / 122, 1.5M 253 / 254 / 246 (four: 255), 3M in five
// views 295 / 288 / 286 (four: 296), 12M in twelve 1397 / 1331 / 1316.  Stage A is bound by the latency of its loads;
// with the exact culls in it (a logarithm, a square root and four divisions per
// item) 1.5M items took 50 us where this takes 42, and 12M items 279 / 220.
// ---------------------------------------------------------------------------
// Wide items: outer rectangles of more tiles than this.  They pay a walk over
// their lines in k_emit with a warp per line, so only those whose runs would
// keep one lane busy for long are wide (at 32 the forward of 1.5M surfels at 1280
// x 720 took 443 us, at 64 417, at 128 408, from 256 on 407).
constexpr uint32_t WIDE_TILES = 256;
constexpr int PAIR_BATCH = 8;  // tile counters added to at once by a lane (4: 411 us)
constexpr int64_t PROJ_SPREAD = 1024;  // items per SM below which a CTA takes 256 of them
constexpr int64_t PROJ_TWO = 4096, PROJ_THREE = 8192;  // ... from which it takes twice, three times 1024

template <int PER, int ROUNDS>
__global__ void __launch_bounds__(PROJ_THREADS, 4) k_project(const __grid_constant__ Cams cams, const __grid_constant__ RParams P,
                                                 const float* __restrict__ means, const float* __restrict__ scales,
                                                 const float* __restrict__ quats, const float* __restrict__ opac,
                                                 float4* __restrict__ rec, BinRec* __restrict__ binrec,
                                                 uint32_t* __restrict__ count, uint32_t* __restrict__ tile_cnt,
                                                 uint32_t* __restrict__ vis_list, uint32_t* __restrict__ wide_list,
                                                 uint32_t* __restrict__ unb_list, int32_t* __restrict__ splat_slot,
                                                 int32_t* __restrict__ slot_surf, uint32_t* __restrict__ pairs,
                                                 Status* __restrict__ st, float rmax, float mmax) {
    constexpr int PROJ_ITEMS = ROUNDS * PER * PROJ_THREADS;
    __shared__ uint32_t s_q[PROJ_ITEMS];
    __shared__ int s_nq;
    __shared__ BinRec s_br[PROJ_THREADS];
    __shared__ uint32_t s_item[PROJ_THREADS], s_cnt[PROJ_THREADS];
    __shared__ int s_pre[PROJ_THREADS];
    const int wb = threadIdx.x & ~31;
    const WarpLines wl{s_br + wb, s_item + wb, s_pre + wb};
    const int lane = threadIdx.x & 31;
    const bool one_view = cams.n == 1;  // every item is a surfel of its own: its gradient slot is written here
    if (st->err) {                      // an error not read yet: nothing but the empty slots
        for (int k = threadIdx.x; one_view && k < PROJ_ITEMS; k += PROJ_THREADS)
            if ((int64_t)blockIdx.x * PROJ_ITEMS + k < P.n_items) splat_slot[(int64_t)blockIdx.x * PROJ_ITEMS + k] = -1;
        return;
    }
    if (threadIdx.x == 0) s_nq = 0;
    __syncthreads();
    // stage A: the superset of the culls for PROJ_ITEMS items (each thread's items
    // loaded together first); the rest queued in shared memory
    const int64_t base = (int64_t)blockIdx.x * PROJ_ITEMS;
#pragma unroll 1
    for (int k0 = threadIdx.x; k0 < PROJ_ITEMS; k0 += PER * PROJ_THREADS) {
    CullIn in[PER];
    int vw[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int64_t it = base + k0 + i * PROJ_THREADS;
        vw[i] = 0;
        if (it < P.n_items) {
            vw[i] = view_of_item(it, P.N);
            in[i] = load_cull_in(means, scales, opac, it - (int64_t)vw[i] * P.N);
        }
    }
#pragma unroll
    for (int i = 0; i < PER; ++i) {
        const int k = k0 + i * PROJ_THREADS;
        const int64_t it = base + k;
        const bool keep = it < P.n_items && !surely_culled(cams.c[vw[i]], P, in[i], rmax, mmax);
        if (one_view && !keep && it < P.n_items) splat_slot[it] = -1;
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        int b = 0;
        if (lane == 0 && m) b = atomicAdd(&s_nq, __popc(m));
        b = __shfl_sync(0xffffffffu, b, 0);
        if (keep) s_q[b + __popc(m & ((1u << lane) - 1u))] = (uint32_t)k;
    }
    }
    __syncthreads();
    const int nq = s_nq;
    // stage B: the whole chain for the queued items, packed densely into warps
    // (warp-uniform loop: the appends below use whole-warp ballots)
    for (int q0 = threadIdx.x & ~31; q0 < nq; q0 += blockDim.x) {
    const int64_t item = q0 + lane < nq ? base + s_q[q0 + lane] : P.n_items;
    bool vis = false, wide = false, unb = false, claim = false;
    int64_t claim_s = 0;
    int view = 0;
    BinRec br;
    if (item < P.n_items) {
        view = view_of_item(item, P.N);
        const int64_t s = item - (int64_t)view * P.N;
        const CamDev& cam = cams.c[view];
        br.flags = 0;
        br.px0 = br.py0 = br.tx0 = br.ty0 = 1;
        br.px1 = br.py1 = br.tx1 = br.ty1 = 0;
        br.A = br.B = br.C = br.D = br.E = br.F = 0.0f;
        br.X0 = br.Y0 = br.hx = br.hy = br.xc = br.yc = 0.0f;
        br.rd2 = 0.0f;
        br.z = 0.0f;
        br.pad = 0;
        float4 r0 = make_float4(0.f, 0.f, 0.f, 0.f), r1 = r0, r2 = r0, r3 = r0;
        do {
            // S3 (centre), S4, S5, S5b first: the order of the cull tests does not change the result
            // (the rotation is loaded beside the cull inputs, so that the latencies overlap)
            const CullIn ci = load_cull_in(means, scales, opac, s);
            const float4 q4 = __ldg(reinterpret_cast<const float4*>(quats) + s);
            float pc[3], o;
            const bool pass = early_culls(cam, P, ci, pc, o);
            r3.y = pc[2];
            br.z = pc[2];
            r3.x = o;
            if (!pass) break;
            // S1
            const float qw = q4.x, qx = q4.y, qy = q4.z, qz = q4.w;
            const float n2 = fa(fa(fa(fm(qw, qw), fm(qx, qx)), fm(qy, qy)), fm(qz, qz));
            if (!(n2 > 0.0f)) break;
            const float nn = fq(n2);
            const float w = fdv(qw, nn), x = fdv(qx, nn), y = fdv(qy, nn), z = fdv(qz, nn);
            // S2
            float tu[3], tv[3];
            tu[0] = fs(1.0f, fm(2.0f, fa(fm(y, y), fm(z, z))));
            tu[1] = fm(2.0f, fa(fm(x, y), fm(w, z)));
            tu[2] = fm(2.0f, fs(fm(x, z), fm(w, y)));
            tv[0] = fm(2.0f, fs(fm(x, y), fm(w, z)));
            tv[1] = fs(1.0f, fm(2.0f, fa(fm(x, x), fm(z, z))));
            tv[2] = fm(2.0f, fa(fm(y, z), fm(w, x)));
            // S3 (tangent columns)
            const float su = ci.sc.x, sv = ci.sc.y;
            float au[3], av[3], e[3];
            mvec(cam.R, tu, e);
#pragma unroll
            for (int i = 0; i < 3; ++i) au[i] = fm(su, e[i]);
            mvec(cam.R, tv, e);
#pragma unroll
            for (int i = 0; i < 3; ++i) av[i] = fm(sv, e[i]);
            // S6: k^2 = 2 ln(o / alpha_min)
            const float k2 = fm(2.0f, ln32(fdv(o, P.alpha_min)));
            r3.z = k2;
            // S7
            float c[3][3];
            const float* src[3] = {au, av, pc};
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                c[j][0] = fa(fm(cam.fx, src[j][0]), fm(cam.cx, src[j][2]));
                c[j][1] = fa(fm(cam.fy, src[j][1]), fm(cam.cy, src[j][2]));
                c[j][2] = src[j][2];
            }
            // S8
            const float xc = fdv(c[2][0], c[2][2]);
            const float yc = fdv(c[2][1], c[2][2]);
            // S9
            float d[3][3];
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                d[j][0] = fs(c[j][0], fm(xc, c[j][2]));
                d[j][1] = fs(c[j][1], fm(yc, c[j][2]));
                d[j][2] = c[j][2];
            }
            // S10
            float m[9];
            crossf(d[1], d[2], &m[0]);
            crossf(d[2], d[0], &m[3]);
            crossf(d[0], d[1], &m[6]);
            // S11
            float det = fa(fa(fm(d[0][0], m[0]), fm(d[0][1], m[1])), fm(d[0][2], m[2]));
            // S12: edge-on cull
            const float pn = fq(fa(fa(fm(pc[0], pc[0]), fm(pc[1], pc[1])), fm(pc[2], pc[2])));
            const float lim = fm(1e-3f, fm(fm(fm(fm(cam.fx, cam.fy), su), sv), pn));
            if (!(fabsf(det) > lim)) break;
            // S13: exact power-of-two rescale
            float mx = 0.0f;
#pragma unroll
            for (int i = 0; i < 9; ++i) mx = fabsf(m[i]) > mx ? fabsf(m[i]) : mx;
            if (!(mx > 0.0f)) break;
            int ex;
            frexp32(mx, &ex);
#pragma unroll
            for (int i = 0; i < 9; ++i) m[i] = ldexp32(m[i], -ex);
            det = ldexp32(det, -ex);
            r3.w = ldexp32(1.0f, -ex);
            r0 = make_float4(m[0], m[1], m[2], xc);
            r1 = make_float4(m[3], m[4], m[5], yc);
            r2 = make_float4(m[6], m[7], m[8], det);
            br.xc = xc;
            br.yc = yc;
            // S14
            const float kb = fm(k2, 1.0009765625f);
            float q[6];
            conic(m, kb, q);
            br.A = q[0]; br.B = q[1]; br.C = q[2]; br.D = q[3]; br.E = q[4]; br.F = q[5];
            int px0, px1, py0, py1;
            // S15
            const float g = fs(fm(q[0], q[2]), fm(q[1], q[1]));
            if (!(q[0] > 0.0f && g > 0.0f)) {
                br.flags |= BR_UNBOUNDED;
                px0 = 0; px1 = cam.W - 1; py0 = 0; py1 = cam.H - 1;
            } else {
                // S16, S17: the ellipse's pixel range
                int e0 = 0, e1 = 0, f0 = 0, f1 = 0;
                bool ell = ellipse(q, br.X0, br.Y0, br.hx, br.hy);
                if (ell)
                    ell = pix_range(fs(fa(fs(br.X0, br.hx), xc), 0.5f), fs(fa(fa(br.X0, br.hx), xc), 0.5f), cam.W, e0,
                                    e1) &&
                          pix_range(fs(fa(fs(br.Y0, br.hy), yc), 0.5f), fs(fa(fa(br.Y0, br.hy), yc), 0.5f), cam.H, f0,
                                    f1);
                // S17b: the low-pass screen disc's, then the union
                int g0 = 0, g1 = 0, h0 = 0, h1 = 0;
                bool disc = false;
                if (P.lowpass) {
                    br.flags |= BR_LOWPASS;
                    br.rd2 = fm(kb, 0.5f);
                    const float rd = fq(br.rd2);
                    disc = pix_range(fs(fs(xc, rd), 0.5f), fs(fa(xc, rd), 0.5f), cam.W, g0, g1) &&
                           pix_range(fs(fs(yc, rd), 0.5f), fs(fa(yc, rd), 0.5f), cam.H, h0, h1);
                }
                if (!ell && !disc) break;
                if (ell) br.flags |= BR_ELL;
                px0 = ell ? (disc ? min(e0, g0) : e0) : g0;
                px1 = ell ? (disc ? max(e1, g1) : e1) : g1;
                py0 = ell ? (disc ? min(f0, h0) : f0) : h0;
                py1 = ell ? (disc ? max(f1, h1) : f1) : h1;
            }
            br.flags |= BR_VISIBLE;
            br.px0 = (int16_t)px0; br.px1 = (int16_t)px1; br.py0 = (int16_t)py0; br.py1 = (int16_t)py1;
            // S18
            const int ts = P.ts;
            const int lts = __ffs(ts) - 1;  // tile sizes are powers of two; pixel indices are >= 0
            int tx0 = px0 >> lts, tx1 = px1 >> lts, ty0 = py0 >> lts, ty1 = py1 >> lts;
            // S19
            if (P.bin_mode == FSS_BIN_AABB && !(br.flags & BR_UNBOUNDED)) {
                float k2a = fm(2.0f, ln32(fdv(1.0f, P.alpha_min)));
                if (kb > k2a) k2a = kb;
                float qa[6], X0, Y0, hx, hy;
                conic(m, k2a, qa);
                const float ga = fs(fm(qa[0], qa[2]), fm(qa[1], qa[1]));
                int ax0 = 0, ax1 = cam.W - 1, ay0 = 0, ay1 = cam.H - 1;
                if (qa[0] > 0.0f && ga > 0.0f && ellipse(qa, X0, Y0, hx, hy)) {
                    const float h = hx > hy ? hx : hy;
                    if (!pix_range(fs(fa(fs(X0, h), xc), 0.5f), fs(fa(fa(X0, h), xc), 0.5f), cam.W, ax0, ax1)) {
                        ax0 = px0; ax1 = px1;
                    }
                    if (!pix_range(fs(fa(fs(Y0, h), yc), 0.5f), fs(fa(fa(Y0, h), yc), 0.5f), cam.H, ay0, ay1)) {
                        ay0 = py0; ay1 = py1;
                    }
                }
                ax0 = min(ax0, px0); ax1 = max(ax1, px1);
                ay0 = min(ay0, py0); ay1 = max(ay1, py1);
                tx0 = ax0 >> lts; tx1 = ax1 >> lts; ty0 = ay0 >> lts; ty1 = ay1 >> lts;
            }
            br.tx0 = (int16_t)tx0; br.tx1 = (int16_t)tx1; br.ty0 = (int16_t)ty0; br.ty1 = (int16_t)ty1;
        } while (0);
        vis = (br.flags & BR_VISIBLE) && !(br.flags & BR_UNBOUNDED);
        unb = (br.flags & BR_VISIBLE) && (br.flags & BR_UNBOUNDED);
        if (vis || unb) {  // records of culled items are never read
            float4* rr = rec + 4 * item;
            rr[0] = r0; rr[1] = r1; rr[2] = r2; rr[3] = r3;
            binrec[item] = br;
            // one gradient slot per surfel visible in any view (-1 -> -2 claims it);
            // with one view every item is a distinct surfel, so no round trip
            claim = one_view || atomicCAS(&splat_slot[s], -1, -2) == -1;
            claim_s = s;
        } else if (one_view) {
            splat_slot[s] = -1;
        }
    }
    // the pairs (S20 intervals), the warp's lines spread over its lanes
    wide = vis && (br.tx1 - br.tx0 + 1) * (br.ty1 - br.ty0 + 1) > (int)WIDE_TILES;
    {
        const int lane = threadIdx.x & 31;
        if (vis) wl.br[lane] = br;
        wl.item[lane] = (uint32_t)item;
        s_cnt[threadIdx.x] = 0u;
        const unsigned wides = __ballot_sync(0xffffffffu, wide);
        const int total = warp_line_prefix(wl, vis ? lines_of(br, P.bin_mode).n : 0);
        for (int u0 = 0; u0 < total; u0 += 32) {  // warp-uniform
            const int u = u0 + lane;
            int j = 0, len = 0, t0 = 0, step = 1;  // the run of tiles t0 + i * step of one line
            if (u < total) {
                j = unit_owner(wl, u);
                const BinRec r = wl.br[j];
                const Lines L = lines_of(r, P.bin_mode);
                const int o = L.first + (u - (wl.pre[j] - L.n));
                int a, b;
                if (line_interval(r, L, P.ts, o, a, b)) {
                    const CamDev& cam = cams.c[view_of_item(wl.item[j], P.N)];
                    len = b - a + 1;
                    t0 = cam.tile_off + (L.rows ? o * cam.tiles_x + a : a * cam.tiles_x + o);
                    step = L.rows ? 1 : cam.tiles_x;
                    atomicAdd(&s_cnt[wb + j], (uint32_t)len);
                }
            }
            const bool many = (wides >> j) & 1u;
            // places of the narrow runs in the pair buffer (one atomic per 32 lines)
            const int mine = many ? 0 : len;
            int incl = mine;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, off);
                if (lane >= off) incl += y;
            }
            uint32_t at = 0u;
            if (lane == 31 && incl) at = atomicAdd(&st->npair, (uint32_t)incl);
            if (many) {
                for (int i = 0; i < len; ++i)
                    if (in_bounds(st, SITE_TILE, t0 + i * step, cams.total_tiles))
                        atomicAdd(&tile_cnt[(size_t)(t0 + i * step) * TC_STRIDE + 1], 1u);
            }
            // each pair takes the next slot of its tile; PAIR_BATCH adds in flight
            uint32_t slot[PAIR_BATCH];
#pragma unroll
            for (int i = 0; i < PAIR_BATCH; ++i)
                slot[i] = i < mine && in_bounds(st, SITE_TILE, t0 + i * step, cams.total_tiles)
                              ? atomicAdd(&tile_cnt[(size_t)(t0 + i * step) * TC_STRIDE], 1u) : 0u;
            at = __shfl_sync(0xffffffffu, at, 31) + (uint32_t)(incl - mine);
            const uint32_t cap = (uint32_t)P.pair_cap, it = wl.item[j];
            uint32_t* const p_tile = pairs;
            uint32_t* const p_slot = pairs + cap;
            uint32_t* const p_item = pairs + 2 * (size_t)cap;
            for (int i0 = 0; i0 < mine; i0 += PAIR_BATCH) {
                if (i0 > 0) {
#pragma unroll
                    for (int i = 0; i < PAIR_BATCH; ++i)
                        slot[i] = i0 + i < mine && in_bounds(st, SITE_TILE, t0 + (i0 + i) * step, cams.total_tiles)
                                      ? atomicAdd(&tile_cnt[(size_t)(t0 + (i0 + i) * step) * TC_STRIDE], 1u) : 0u;
                }
#pragma unroll
                for (int i = 0; i < PAIR_BATCH; ++i) {
                    const uint32_t q = at + (uint32_t)(i0 + i);
                    if (i0 + i < mine && q < cap) {  // (over capacity: counted, the frame is reported)
                        p_tile[q] = (uint32_t)(t0 + (i0 + i) * step);
                        p_slot[q] = slot[i];
                        p_item[q] = it;
                    }
                }
            }
        }
        __syncwarp();
        if (vis) count[item] = s_cnt[threadIdx.x];
        __syncwarp();  // the slices are reused by the warp's next survivors
    }
    // warp-aggregated appends (one global atomic per warp and counter, no CTA barrier)
    {
        const int lane = threadIdx.x & 31;
        const unsigned lt = (1u << lane) - 1u;
        const bool narrow = vis && !wide, wid = vis && wide;
        const unsigned mn = __ballot_sync(0xffffffffu, narrow), mw = __ballot_sync(0xffffffffu, wid);
        const unsigned mc = __ballot_sync(0xffffffffu, claim);
        uint32_t bn = 0, bw = 0, bc = 0;
        if (lane == 0) {
            if (mn) bn = atomicAdd(&st->nvis, (uint32_t)__popc(mn));
            if (mw) bw = atomicAdd(&st->nwide, (uint32_t)__popc(mw));
            if (mc) bc = atomicAdd(&st->nslot, (uint32_t)__popc(mc));
        }
        bn = __shfl_sync(0xffffffffu, bn, 0);
        bw = __shfl_sync(0xffffffffu, bw, 0);
        bc = __shfl_sync(0xffffffffu, bc, 0);
        if (narrow && in_bounds(st, SITE_VIS_LIST, bn + __popc(mn & lt), P.n_items))
            vis_list[bn + __popc(mn & lt)] = (uint32_t)item;
        if (wid && in_bounds(st, SITE_VIS_LIST, bw + __popc(mw & lt), P.n_items))
            wide_list[bw + __popc(mw & lt)] = (uint32_t)item;
        if (claim) {
            const int32_t sl = (int32_t)(bc + __popc(mc & lt));
            if (in_bounds(st, SITE_SLOT, sl, P.N) && in_bounds(st, SITE_SLOT, claim_s, P.N)) {
                splat_slot[claim_s] = sl;
                slot_surf[sl] = (int32_t)claim_s;
            }
        }
    }
    if (unb) {
        const uint32_t k = atomicAdd(&st->unb_cnt[view], 1u);
        if (in_bounds(st, SITE_VIS_LIST, k, P.N)) unb_list[(int64_t)view * P.N + k] = (uint32_t)item;
    }
    }  // survivors
}

// Before binning: zeros for the status block's per-frame words and the tile counts
// (16-byte vectors), -1 for the gradient slots (none with one view).  One launch of a
// few microseconds where each of the regions took a memset; not one of the kernels that the
// measurement hook counts.
__global__ void __launch_bounds__(256) k_bin_clear(uint32_t* status, int status_words, uint4* tile_cnt, int64_t tile_vecs,
                                                   int32_t* slot, int64_t slots) {
    const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, n = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = i0; i < status_words; i += n) status[i] = 0u;
    for (int64_t i = i0; i < tile_vecs; i += n) tile_cnt[i] = make_uint4(0u, 0u, 0u, 0u);
    for (int64_t i = i0; i < slots / 4; i += n) reinterpret_cast<int4*>(slot)[i] = make_int4(-1, -1, -1, -1);
    for (int64_t i = slots / 4 * 4 + i0; i < slots; i += n) slot[i] = -1;
}

cudaError_t launch_bin_clear(uint32_t* status, int status_words, uint4* tile_cnt, int64_t tile_vecs, int32_t* slot,
                             int64_t slots, int num_sms, cudaStream_t stream) {
    const int64_t work = std::max<int64_t>(status_words, std::max<int64_t>(tile_vecs, slots / 4));
    const unsigned blocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>((work + 255) / 256, 4 * (int64_t)num_sms));
    k_bin_clear<<<blocks, 256, 0, stream>>>(status, status_words, tile_cnt, tile_vecs, slot, slots);
    return cudaGetLastError();
}

cudaError_t launch_project(const Cams& cams, const RParams& P, const float* means, const float* scales, const float* quats,
                           const float* opac, float4* rec, BinRec* binrec, uint32_t* count, uint32_t* tile_cnt,
                           uint32_t* vis_list, uint32_t* wide_list, uint32_t* unb_list, int32_t* splat_slot,
                           int32_t* slot_surf, uint32_t* pairs, Status* st, int num_sms, cudaStream_t stream) {
    // the largest binning radius per unit scale and screen margin of an opacity <= 1, widened (see surely_culled)
    const double k2 = 2.0 * std::log(1.0 / (double)P.alpha_min) * 1.0009765625;
    const float rmax = (float)(std::sqrt(std::max(k2, 0.0)) * 1.0015);
    const float mmax = (float)(1.0 + (P.lowpass ? std::sqrt(std::max(k2, 0.0) * 0.5) * 1.0015 : 0.0));
    auto go = [&](auto kern, int64_t items) {
        const int64_t blocks = std::max<int64_t>(1, (P.n_items + items - 1) / items);
        kern<<<(unsigned)blocks, PROJ_THREADS, 0, stream>>>(cams, P, means, scales, quats, opac, rec, binrec, count, tile_cnt,
                                                            vis_list, wide_list, unb_list, splat_slot, slot_surf, pairs, st,
                                                            rmax, mmax);
        return cudaGetLastError();
    };
    if (P.n_items < PROJ_SPREAD * num_sms) return go(k_project<1, 1>, PROJ_THREADS);
    if (P.n_items < PROJ_TWO * num_sms) return go(k_project<4, 1>, 4 * PROJ_THREADS);
    if (P.n_items < PROJ_THREE * num_sms) return go(k_project<4, 2>, 8 * PROJ_THREADS);
    return go(k_project<4, 3>, 12 * PROJ_THREADS);
}

// ---------------------------------------------------------------------------
// Tile scan, run by one CTA of k_emit (any block size, a multiple of 32):
// per-tile totals (bounded pairs + the view's unbounded items) -> exclusive
// scan -> ranges; the tile counters become the emit cursors.  Then the
// heavy-first tile order: a counting sort of the tiles by pair count,
// descending, in buckets of 16 pairs (the order within a bucket is
// arbitrary).  The tile kernels take tiles in this order, so that the last
// tiles to start are light ones: the work per tile varies severalfold, and
// in index order a heavy tile starting late sets the kernel's end.
// ---------------------------------------------------------------------------
constexpr int ORDER_BUCKETS = 256;  // 32 lanes x 8
__device__ __forceinline__ int order_bucket(int2 r) { return min(ORDER_BUCKETS - 1, (r.y - r.x) >> 4); }

__device__ void scan_tiles(const Cams& cams, const RParams& P, uint32_t* __restrict__ tile_cnt,
                           int2* __restrict__ ranges, Status* __restrict__ st) {
    __shared__ uint32_t warp_tot[32];
    __shared__ uint64_t carry_s;
    if (threadIdx.x == 0) carry_s = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int nt = cams.total_tiles;
    constexpr int ITEMS = 8;
    for (int base = 0; base < nt; base += blockDim.x * ITEMS) {
        uint32_t v[ITEMS], narrow[ITEMS];
        uint32_t sum = 0;
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const int t = base + threadIdx.x * ITEMS + k;
            // (both words of the sector at once)
            const uint2 c = t < nt ? *reinterpret_cast<const uint2*>(tile_cnt + (size_t)t * TC_STRIDE) : make_uint2(0u, 0u);
            narrow[k] = c.x;
            v[k] = t < nt ? c.x + c.y + st->unb_cnt[view_of_tile(cams, t)] : 0u;
            sum += v[k];
        }
        uint32_t incl = sum;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += y;
        }
        if (lane == 31) warp_tot[wid] = incl;
        __syncthreads();
        if (wid == 0) {
            uint32_t w = lane < nw ? warp_tot[lane] : 0u, wi = w;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, wi, off);
                if (lane >= off) wi += y;
            }
            warp_tot[lane] = wi - w;  // exclusive
        }
        __syncthreads();
        uint64_t run = carry_s + warp_tot[wid] + (incl - sum);
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const int t = base + threadIdx.x * ITEMS + k;
            if (t < nt) {
                const uint64_t s0 = run;
                run += v[k];
                const bool fits = run <= (uint64_t)P.pair_cap;
                ranges[t] = make_int2(fits ? (int)s0 : 0, fits ? (int)run : 0);
                // first place of the narrow pairs, cursor of the wide ones
                *reinterpret_cast<uint2*>(tile_cnt + (size_t)t * TC_STRIDE) =
                    fits ? make_uint2((uint32_t)s0, (uint32_t)s0 + narrow[k]) : make_uint2(0u, 0u);
            }
        }
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) carry_s = run;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        st->pairs_needed = (int64_t)carry_s;
        if (carry_s > (uint64_t)P.pair_cap) atomicOr(&st->err, ERR_CAPACITY);
    }
}

// heavy-first order of the tiles from their ranges (a frame over capacity
// has empty ranges: any order)
__device__ void heavy_first_order(const Cams& cams, const int2* __restrict__ ranges, int32_t* __restrict__ order) {
    __shared__ uint32_t ord[ORDER_BUCKETS];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nt = cams.total_tiles;
    for (int b = threadIdx.x; b < ORDER_BUCKETS; b += blockDim.x) ord[b] = 0u;
    __syncthreads();
    for (int t = threadIdx.x; t < nt; t += blockDim.x) atomicAdd(&ord[order_bucket(ranges[t])], 1u);
    __syncthreads();
    if (wid == 0) {  // first position of each bucket, heaviest bucket first
        uint32_t c[8], sum = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            c[k] = ord[ORDER_BUCKETS - 1 - (8 * lane + k)];
            sum += c[k];
        }
        uint32_t incl = sum;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += y;
        }
        uint32_t run = incl - sum;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            ord[ORDER_BUCKETS - 1 - (8 * lane + k)] = run;
            run += c[k];
        }
    }
    __syncthreads();
    for (int t = threadIdx.x; t < nt; t += blockDim.x) order[atomicAdd(&ord[order_bucket(ranges[t])], 1u)] = t;
}

// failure-detection test hook (fss_test_hold_scan): when set, the scanning
// CTA keeps its result to itself, so the other CTAs' bounded wait runs out
__device__ int g_hold_scan = 0;

cudaError_t set_hold_scan(int hold) { return cudaMemcpyToSymbol(g_hold_scan, &hold, sizeof(int)); }

// Rounds of the bounded wait for the scanning CTA (each about 0.1-0.2 us of
// sleep: about a second in all), after which the waiting CTA raises
// ERR_TIMEOUT and returns.
constexpr int SCAN_WAIT = 1 << 23;

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release(uint32_t* p, uint32_t v) {
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// ---------------------------------------------------------------------------
// precise render record (record_item), written in double-float
//
// The ray-splat solve u ~ adj(T') (x - xc, y - yc, 1) is evaluated per pixel
// in binary32, but the adjugate itself is computed here in double-float from
// the binary32 inputs and rounded once: for a surfel seen nearly edge-on the
// intersection amplifies a relative error e in T by about (depth / size) /
// cos(view angle), so a binary32 chain (the binning mirror above) would put
// ~1e-3 relative error into alpha.  The binning record keeps the binary32
// values; only the render record r0..r2 and the rescale r3.w change.
// With n2 = |q|^2, R(q/|q|) = R'(q) / n2 where R' is the homogeneous
// (unnormalised) rotation polynomial, so n2 * T = K [r_u Rv t_u', r_v Rv t_v',
// n2 (Rv p + t)] needs no square root; its adjugate is n2^2 adj(T).
// ---------------------------------------------------------------------------
// One thread per item.  (A quad of lanes per item, one column each, formed the
// rotation in every lane and exchanged the columns: 2.2 times the instructions, and
// 433 us instead of 430 for the forward of 1.5M surfels at 1280 x 720.)
__device__ __forceinline__ void record_item(const Cams& cams, const RParams& P, const float* __restrict__ means,
                                            const float* __restrict__ scales, const float* __restrict__ quats,
                                            float4* __restrict__ rec, uint32_t item) {
    const int view = view_of_item(item, P.N);
    const int64_t s = (int64_t)item - (int64_t)view * P.N;
    const CamDev& cam = cams.c[view];
    float4* rr = rec + 4 * (size_t)item;
    const float xc = rr[0].w, yc = rr[1].w;
    const float4 q4 = __ldg(reinterpret_cast<const float4*>(quats) + s);
    const float2 sc = __ldg(reinterpret_cast<const float2*>(scales) + s);
    const float pm[3] = {__ldg(means + 3 * s), __ldg(means + 3 * s + 1), __ldg(means + 3 * s + 2)};
    const float qw = q4.x, qx = q4.y, qy = q4.z, qz = q4.w;
    const df ww = two_prod(qw, qw), xx = two_prod(qx, qx), yy = two_prod(qy, qy), zz = two_prod(qz, qz);
    const df n2 = dadd(dadd(ww, xx), dadd(yy, zz));
    df d[3][3];  // the columns of n2 T, shifted about (xc, yc)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        // column j of n2 T (camera frame, before the intrinsics): R t_u' r_u, R t_v' r_v or n2 (R p + t)
        df v[3], col[3];
        if (j == 0) {
            v[0] = dsub(dadd(ww, xx), dadd(yy, zz));
            v[1] = dmulf(dadd(two_prod(qx, qy), two_prod(qw, qz)), 2.0f);
            v[2] = dmulf(dsub(two_prod(qx, qz), two_prod(qw, qy)), 2.0f);
        } else if (j == 1) {
            v[0] = dmulf(dsub(two_prod(qx, qy), two_prod(qw, qz)), 2.0f);
            v[1] = dsub(dadd(ww, yy), dadd(xx, zz));
            v[2] = dmulf(dadd(two_prod(qy, qz), two_prod(qw, qx)), 2.0f);
        } else {
#pragma unroll
            for (int i = 0; i < 3; ++i) v[i] = dfrom(pm[i]);
        }
        dmvec(cam.R, v, col);
#pragma unroll
        for (int i = 0; i < 3; ++i)
            col[i] = j < 2 ? dmulf(col[i], j == 0 ? sc.x : sc.y) : dmul(dadd(col[i], dfrom(cam.t[i])), n2);
        d[j][0] = dsub(dadd(dmulf(col[0], cam.fx), dmulf(col[2], cam.cx)), dmulf(col[2], xc));
        d[j][1] = dsub(dadd(dmulf(col[1], cam.fy), dmulf(col[2], cam.cy)), dmulf(col[2], yc));
        d[j][2] = col[2];
    }
    // adjugate rows m_j = d_{j+1} x d_{j+2}
    df m[3][3];
    dcross(d[1], d[2], m[0]);
    dcross(d[2], d[0], m[1]);
    dcross(d[0], d[1], m[2]);
    float mx = 0.0f;
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
        for (int i = 0; i < 3; ++i) mx = fmaxf(mx, fabsf(m[j][i].hi));
    if (!(mx > 0.0f)) return;
    const df det = dadd(dadd(dmul(d[0][0], m[0][0]), dmul(d[0][1], m[0][1])), dmul(d[0][2], m[0][2]));  // det(n2 T')
    int ex = 0;
    frexp32(mx, &ex);
    // hit depth det(T') / c2: with M = 2^-ex n2^2 adj(T'), store 2^-ex det(n2 T') / n2
    const float detr = ldexp32(fdv(det.hi, n2.hi), -ex);
#pragma unroll
    for (int j = 0; j < 3; ++j)
        rr[j] = make_float4(ldexp32(m[j][0].hi, -ex), ldexp32(m[j][1].hi, -ex), ldexp32(m[j][2].hi, -ex),
                            j == 0 ? xc : (j == 1 ? yc : detr));
    rr[3].w = ldexp32(fm(n2.hi, n2.hi), -ex);  // total scale of M relative to adj(T' of the normalised surfel)
}

// ---------------------------------------------------------------------------
// k_emit: writes every bounded visible item into one slot of each of its
// tiles (slot order is arbitrary; the per-tile sort restores a total order)
// and replaces the render records by their double-float versions.
//   scan:         the first CTA to take the ticket scans the per-tile counts
//                 into ranges and emit cursors and publishes them (release
//                 store of a flag); it never waits, so the others' bounded
//                 wait for the flag ends however the CTAs are scheduled;
//   records:      one thread per narrow, wide or unbounded item (they need no
//                 ranges, so they run while the scan does);
//   narrow pairs: one thread per (tile, slot, item) that k_project made: the
//                 item goes to the slot's place in the tile's range (a second
//                 walk over the lines with one more add per pair took
//                 24 us for 500k surfels at 640 x 480 where this and the pair's
//                 making take 19);
//   wide items:   one warp per (item, outer line), lanes over the line's tiles;
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_emit(const __grid_constant__ Cams cams, const __grid_constant__ RParams P,
                                              const BinRec* __restrict__ binrec, const uint32_t* __restrict__ vis_list,
                                              const uint32_t* __restrict__ wide_list,
                                              const uint32_t* __restrict__ unb_list, uint32_t* __restrict__ cursor,
                                              int2* __restrict__ ranges, int32_t* __restrict__ order,
                                              uint32_t* __restrict__ list, const uint32_t* __restrict__ pairs,
                                              const float* __restrict__ means, const float* __restrict__ scales,
                                              const float* __restrict__ quats, float4* __restrict__ rec,
                                              Status* __restrict__ st, int max_lines) {
    __shared__ int s_scanner, s_go;
    if (st->err) return;
    Status* const stw = st;
    if (threadIdx.x == 0) s_scanner = atomicAdd(&st->scan_ticket, 1u) == 0u;
    __syncthreads();
    if (s_scanner) {
        scan_tiles(cams, P, cursor, ranges, st);
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0 && !g_hold_scan) st_release(&st->scan_done, 1u);
        heavy_first_order(cams, ranges, order);
    }
    const int lane = threadIdx.x & 31;
    const uint32_t nvis = st->nvis, nwide = st->nwide;
    const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t gstride = (int64_t)gridDim.x * blockDim.x;
    uint32_t nunb = 0;
    for (int v = 0; v < cams.n; ++v) nunb += st->unb_cnt[v];
    // render records of all visible items (narrow, wide, unbounded), one thread
    // each, from the lowest threads up
    const uint32_t nrec = nvis + nwide + nunb;
    for (int64_t ri = gtid; ri < nrec; ri += gstride) {
        uint32_t item = 0;
        if (!in_bounds(stw, SITE_VIS_LIST, ri, P.n_items)) break;
        if (ri < nvis) {
            item = vis_list[ri];
        } else if (ri < (int64_t)nvis + nwide) {
            item = wide_list[ri - nvis];
        } else {
            uint32_t k = (uint32_t)(ri - nvis - nwide);
            int v = 0;
            while (FSS_CHECKED(v < cams.n) && k >= st->unb_cnt[v]) k -= st->unb_cnt[v++];
            if (!in_bounds(stw, SITE_VIS_LIST, v, cams.n) || !in_bounds(stw, SITE_VIS_LIST, k, P.N)) continue;
            item = unb_list[(int64_t)v * P.N + k];
        }
        if (in_bounds(stw, SITE_ITEM, item, P.n_items)) record_item(cams, P, means, scales, quats, rec, item);
    }
    // the emit cursors: published by the scanning CTA (bounded wait)
    if (threadIdx.x == 0) {
        bool done = s_scanner != 0;
        for (int i = 0; !done && i < SCAN_WAIT; ++i) {
            done = ld_acquire(&st->scan_done) != 0u;
            if (!done) __nanosleep(128);
        }
        if (!done) atomicOr(&st->err, ERR_TIMEOUT);
        s_go = done && !(ld_acquire(reinterpret_cast<const uint32_t*>(&st->err)) & ERR_CAPACITY);
    }
    __syncthreads();
    if (!s_go) return;
    // the narrow pairs, each to its slot of its tile's range
    const int64_t npair = min((int64_t)st->npair, P.pair_cap);
    for (int64_t i = gstride - 1 - gtid; i < npair; i += gstride) {  // (from the threads without a record up)
        const uint32_t t = pairs[i], slot = pairs[P.pair_cap + i];
        if (!in_bounds(stw, SITE_TILE, t, cams.total_tiles)) continue;
        const uint32_t pos = __ldcg(cursor + (size_t)t * TC_STRIDE) + slot;  // (written during this kernel: from L2)
        if (pos < (uint32_t)P.pair_cap) list[pos] = pairs[2 * P.pair_cap + i];
    }
    const int64_t warps = gstride >> 5;
    // wide items: one warp per (item, outer line), lanes over the line's tiles,
    // so that a surfel spanning many tiles is spread over many warps
    const int64_t units = (int64_t)nwide * max_lines;
    for (int64_t u = gtid >> 5; u < units; u += warps) {
        const int64_t wi = u / max_lines;
        const int li = (int)(u - wi * max_lines);
        if (!in_bounds(stw, SITE_VIS_LIST, wi, P.n_items)) break;
        const uint32_t item = wide_list[wi];
        if (!in_bounds(stw, SITE_ITEM, item, P.n_items)) continue;
        const BinRec r = binrec[item];
        const Lines L = lines_of(r, P.bin_mode);
        if (li >= L.n) continue;  // warp-uniform
        const CamDev& cam = cams.c[view_of_item(item, P.N)];
        const int o = L.first + li;
        int a, b;
        if (!line_interval(r, L, P.ts, o, a, b)) continue;
        for (int k = a + lane; k <= b; k += 32) {
            const int tx = L.rows ? k : o, ty = L.rows ? o : k;
            const int tt = cam.tile_off + ty * cam.tiles_x + tx;
            if (!in_bounds(stw, SITE_TILE, tt, cams.total_tiles)) continue;
            const uint32_t pos = atomicAdd(&cursor[(size_t)tt * TC_STRIDE + 1], 1u);
            if (pos < (uint32_t)P.pair_cap) list[pos] = item;
        }
    }
}

}  // namespace fss
