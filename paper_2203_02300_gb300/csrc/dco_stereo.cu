// GB300 (sm_103a) AD-census stereo matcher: kernels and C ABI.
//
// Method: arXiv 2203.02300, Sect. 4 (census + AD cost with adaptive weight,
// Eq. 1; cross-support region aggregation, Eq. 2; winner-take-all, Eq. 3;
// outlier removal by left-right consistency, Sect. 4.3).
//
// Pipeline per pair (one stream, no host round trip):
//   k_pack   RGB -> packed colour words (with the two edge bits of the arm
//            rule's predecessor test) and the grey level, both images
//   k_prep   census (shared-memory grey tile) + the four arms (walks over the
//            packed colours) -> census and colour planes + arm words
//   per pass of dc disparities:
//     k_hagg  Eq. 1 cost in fixed point for every (column, disparity) of a
//             row, their row prefixes in shared memory, and the horizontal
//             segment sum of every pixel -> sh slices
//     k_vagg  column prefix of the sh slice, the vertical sum over the
//             up/down arms (Eq. 2) and the minimum over the disparities
//             (Eq. 3), merged into one key per pixel; k_vcol, a block per
//             column, in small launches
//   k_end    keys -> disparities; left-right consistency -> disparity map
// Every kernel is launched with programmatic stream serialization and waits
// for its predecessors before its first global access.
// A lane of k_hagg and k_vagg holds four consecutive disparities (of five
// columns, of one), so that a warp's prefix rows hit distinct banks and the
// slices are written and read as whole sectors of 128-byte lines.

#include "kernels.cuh"
#include "dco_stereo.h"

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <string>
#include <type_traits>
#include <vector>

namespace dco {

// Programmatic dependent launch: every kernel of the paths is launched with
// programmatic stream serialization, so the launch of a kernel overlaps the
// end of the previous one in the stream.  Before touching global memory a
// block waits until the previous grids have completed and their writes are
// visible.  No block triggers its dependents early: blocks of the next
// kernel parked on free SMs while a multi-pass run's last waves drain made
// those runs slower (1920x1080 in passes of 32: 5.12 against 4.31 ms);
// with the trigger at grid exit the launch latency alone is hidden
// (640x480 D=64: 165 -> 156 us per pair, 320x240 D=32: 46 -> 36.5 us).
__device__ __forceinline__ void pdl_enter()
{
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
}


// ------------------------------------------------------------------ k_pack
// RGB (3 bytes per pixel) -> packed 32-bit colour and the integer grey level
// of the census, for both images; four pixels (12 bytes) per thread.
__device__ __forceinline__ uint32_t grey_of(uint32_t c)
{
    return (77u * (c & 0xffu) + 150u * ((c >> 8) & 0xffu) + 29u * ((c >> 16) & 0xffu) + 128u) >> 8;
}

// Colour r | g<<8 | b<<16 spread into three 10-bit fields r | g<<10 | b<<20.
// With K holding tau - 1 + 512 in every field, (E(c) + K - E(p)) keeps each
// field in [1, 1023] (no carry or borrow between fields) and has the field's
// bit 9 set exactly when c_i - p_i + tau - 1 >= 0; the same with c and p
// swapped gives the other side, so every channel has |c_i - p_i| < tau
// exactly when all six bit-9s are set.
constexpr uint32_t kM9 = (1u << 9) | (1u << 19) | (1u << 29);
__device__ __forceinline__ uint32_t spread10(uint32_t c)
{
    return (c & 0xffu) | ((c & 0xff00u) << 2) | ((c & 0xff0000u) << 4);
}
// back to bytes r | g<<8 | b<<16 (bits 30, 31 ignored)
__device__ __forceinline__ uint32_t unspread10(uint32_t e)
{
    return (e & 0xffu) | ((e >> 2) & 0xff00u) | ((e >> 4) & 0xff0000u);
}

// The two bits above the fields of a packed colour: every arm step's colour
// difference to its predecessor must be below tau1 (Sect. 4.1), a property
// of the pixel edge alone, so k_pack stores it once per pixel: bit 30 for
// the edge to the left neighbour, bit 31 for the edge to the one above.
constexpr uint32_t kEdgeL = 1u << 30, kEdgeU = 1u << 31, kColour = 0x3fffffffu;

// all channels within tau of p, given Kp = K - E(p) and pK = E(p) + K
__device__ __forceinline__ bool within(uint32_t ec, uint32_t Kp, uint32_t pK)
{
    return ((ec + Kp) & (pK - ec) & kM9) == kM9;
}

__device__ __forceinline__ uint32_t rgb_at(const uint8_t *rgb, size_t i)
{
    const uint8_t *p = rgb + 3 * i;
    return uint32_t(__ldg(p)) | (uint32_t(__ldg(p + 1)) << 8) | (uint32_t(__ldg(p + 2)) << 16);
}

// k_pack stores every colour spread (the arm walks read each candidate many
// times; the record keeps the bytes) with its two edge bits
__device__ __forceinline__ void pack_body(const PackArgs &a, int q, int img)   // pixels 4q .. 4q+3
{
    const int i0 = 4 * q;
    if (i0 >= a.npx) return;
    const uint8_t *rgb = img ? a.rgb[1] : a.rgb[0];
    uint32_t *rgbx = img ? a.rgbx[1] : a.rgbx[0];
    uint8_t *grey = img ? a.grey[1] : a.grey[0];
    uint32_t c[4];
    if (i0 + 4 <= a.npx && ((reinterpret_cast<uintptr_t>(rgb) & 3u) == 0)) {
        const uint32_t *w = reinterpret_cast<const uint32_t *>(rgb + 3 * (size_t)i0);
        const uint32_t w0 = __ldg(w), w1 = __ldg(w + 1), w2 = __ldg(w + 2);
        c[0] = w0 & 0x00ffffffu;
        c[1] = __funnelshift_r(w0, w1, 24) & 0x00ffffffu;
        c[2] = __funnelshift_r(w1, w2, 16) & 0x00ffffffu;
        c[3] = w2 >> 8;
    } else {
        for (int k = 0; k < 4; k++) {
            const int i = min(i0 + k, a.npx - 1);
            const uint8_t *p = rgb + 3 * (size_t)i;
            c[k] = uint32_t(__ldg(p)) | (uint32_t(__ldg(p + 1)) << 8) | (uint32_t(__ldg(p + 2)) << 16);
        }
    }
    // edge bits: the left neighbour (pixel i - 1 in the same row) and the
    // one above (pixel i - W)
    uint32_t e[4], u[4];
#pragma unroll
    for (int k = 0; k < 4; k++) e[k] = spread10(c[k]);
    const int W = a.W;
    const int up0 = i0 - W;
    if (up0 >= 0 && i0 + 4 <= a.npx && ((reinterpret_cast<uintptr_t>(rgb + 3 * (size_t)up0) & 3u) == 0)) {
        const uint32_t *w = reinterpret_cast<const uint32_t *>(rgb + 3 * (size_t)up0);
        const uint32_t w0 = __ldg(w), w1 = __ldg(w + 1), w2 = __ldg(w + 2);
        u[0] = w0 & 0x00ffffffu;
        u[1] = __funnelshift_r(w0, w1, 24) & 0x00ffffffu;
        u[2] = __funnelshift_r(w1, w2, 16) & 0x00ffffffu;
        u[3] = w2 >> 8;
    } else {
#pragma unroll
        for (int k = 0; k < 4; k++) u[k] = up0 + k >= 0 ? rgb_at(rgb, (size_t)min(up0 + k, a.npx - 1)) : 0u;
    }
    // pixel i0 - 1: the top three bytes of the word before this group (the
    // group starts 4-byte aligned on the aligned path)
    uint32_t prev = 0u;
    if (i0 > 0)
        prev = spread10(((reinterpret_cast<uintptr_t>(rgb) & 3u) == 0)
                            ? __ldg(reinterpret_cast<const uint32_t *>(rgb + 3 * (size_t)i0) - 1) >> 8
                            : rgb_at(rgb, (size_t)(i0 - 1)));
    int x = i0 % W;
    uint32_t out[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const uint32_t Kp = a.k1 - e[k], pK = e[k] + a.k1;
        uint32_t v = e[k];
        if (x > 0 && within(prev, Kp, pK)) v |= kEdgeL;
        if (up0 + k >= 0 && within(spread10(u[k]), Kp, pK)) v |= kEdgeU;
        out[k] = v;
        prev = e[k];
        x = x + 1 == W ? 0 : x + 1;
    }
    if (i0 + 4 <= a.npx) {
        *reinterpret_cast<uint4 *>(rgbx + i0) = make_uint4(out[0], out[1], out[2], out[3]);
        *reinterpret_cast<uint32_t *>(grey + i0) =
            grey_of(c[0]) | (grey_of(c[1]) << 8) | (grey_of(c[2]) << 16) | (grey_of(c[3]) << 24);
    } else {
        for (int k = 0; i0 + k < a.npx; k++) {
            rgbx[i0 + k] = out[k];
            grey[i0 + k] = (uint8_t)grey_of(c[k]);
        }
    }
}

// The same for images in host memory (read over NVLink-C2C, where every
// extra read costs): one thread per block of 4 columns x kRows rows, so the
// row above is read once per block instead of once per row.
template <int kRows>
__device__ __forceinline__ void pack_rows_body(const PackArgs &a, int t, int img)
{
    const int W = a.W, H = a.npx / W;
    const int ngx = (W + 3) >> 2, nby = (H + kRows - 1) / kRows;
    const int band = t / ngx, qx = t - band * ngx;
    if (band >= nby) return;
    const int x0 = 4 * qx, y0 = kRows * band, nx = min(4, W - x0);
    const uint8_t *rgb = img ? a.rgb[1] : a.rgb[0];
    uint32_t *rgbx = img ? a.rgbx[1] : a.rgbx[0];
    uint8_t *grey = img ? a.grey[1] : a.grey[0];
    // rows start 4-byte aligned in the input and 16-byte aligned in the
    // outputs when W is a multiple of 4
    const bool vec = nx == 4 && (W & 3) == 0 && (reinterpret_cast<uintptr_t>(rgb) & 3u) == 0;
    // the four colours of row y at x0 .. x0 + 3 (repeating the last one past
    // the row's end) and the left neighbour (x0 - 1)
    auto load_row = [&](int y, uint32_t (&c)[4], uint32_t &left) {
        const size_t i = (size_t)y * W + x0;
        if (vec) {
            const uint32_t *w = reinterpret_cast<const uint32_t *>(rgb + 3 * i);
            const uint32_t w0 = __ldg(w), w1 = __ldg(w + 1), w2 = __ldg(w + 2);
            c[0] = w0 & 0x00ffffffu;
            c[1] = __funnelshift_r(w0, w1, 24) & 0x00ffffffu;
            c[2] = __funnelshift_r(w1, w2, 16) & 0x00ffffffu;
            c[3] = w2 >> 8;
            left = x0 > 0 ? __ldg(w - 1) >> 8 : 0u;   // the top three bytes of the word before
        } else {
#pragma unroll
            for (int k = 0; k < 4; k++) c[k] = rgb_at(rgb, i + min(k, nx - 1));
            left = x0 > 0 ? rgb_at(rgb, i - 1) : 0u;
        }
    };
    uint32_t up[4] = {0u, 0u, 0u, 0u};   // spread colours of the row above
    if (y0 > 0) {
        uint32_t c[4], l;
        load_row(y0 - 1, c, l);
#pragma unroll
        for (int k = 0; k < 4; k++) up[k] = spread10(c[k]);
    }
#pragma unroll
    for (int r = 0; r < kRows; r++) {
        const int y = y0 + r;
        if (y >= H) break;
        uint32_t c[4], l, e[4], out[4];
        load_row(y, c, l);
#pragma unroll
        for (int k = 0; k < 4; k++) e[k] = spread10(c[k]);
        uint32_t prev = spread10(l);
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const uint32_t Kp = a.k1 - e[k], pK = e[k] + a.k1;
            uint32_t v = e[k];
            if (x0 + k > 0 && within(prev, Kp, pK)) v |= kEdgeL;
            if (y > 0 && within(up[k], Kp, pK)) v |= kEdgeU;
            out[k] = v;
            prev = e[k];
            up[k] = e[k];
        }
        const size_t i = (size_t)y * W + x0;
        if (vec) {
            *reinterpret_cast<uint4 *>(rgbx + i) = make_uint4(out[0], out[1], out[2], out[3]);
            *reinterpret_cast<uint32_t *>(grey + i) =
                grey_of(c[0]) | (grey_of(c[1]) << 8) | (grey_of(c[2]) << 16) | (grey_of(c[3]) << 24);
        } else {
            for (int k = 0; k < nx; k++) {
                rgbx[i + k] = out[k];
                grey[i + k] = (uint8_t)grey_of(c[k]);
            }
        }
    }
}

// ------------------------------------------------------------------ k_prep
// One thread per pixel of a 32 x 8 tile.  Census (Sect. 4.2.1) from the grey
// tile with its window halo in shared memory (clamp-to-edge on load); the
// four arms (Sect. 4.1) by walking the packed colours through L1 (arms are
// short on textured input, so no L1-wide halo is staged).  The 9x7 census
// compares four neighbours per SIMD byte comparison.
constexpr int kTX = 32, kTY = 8;
constexpr int kMaxCW = 15, kMaxCH = 15;
constexpr int kArmRun = 8;   // candidates of an arm walk loaded together
constexpr int kGW = 48;   // grey tile row pitch (>= kTX + kMaxCW - 1, multiple of 4)

// 4 flags f_i = [byte_i(w) < byte_i(c4)] -> bits f0 | f1<<1 | f2<<2 | f3<<3.
// Per byte: (w|0x80) - (c&0x7f) never borrows into the next byte, and its top
// bit is clear exactly when the low seven bits compare w < c; the top bits
// of w and c decide the rest.
__device__ __forceinline__ uint32_t lt4(uint32_t w, uint32_t c4, uint32_t c4lo)
{
    const uint32_t x = (w | 0x80808080u) - c4lo;
    const uint32_t lt = ((~w & c4) | (~(w ^ c4) & ~x)) & 0x80808080u;
    return (lt * 0x00204081u) >> 28;
}

template <int CW, int CH>
__device__ __forceinline__ void prep_body(const PrepArgs &a, int bx, int by, int img)
{
    __shared__ __align__(16) uint8_t gs[kTY + kMaxCH - 1][kGW];
    const uint32_t *__restrict__ rgbx = img ? a.rgbx[1] : a.rgbx[0];
    const uint8_t *__restrict__ grey = img ? a.grey[1] : a.grey[0];
    const int W = a.W, H = a.H;
    const int cw = CW ? CW : a.cw, ch = CH ? CH : a.ch;
    const int rx = cw / 2, ry = ch / 2;
    const int x0 = bx * kTX, y0 = by * kTY;
    const int tx = threadIdx.x % kTX, ty = threadIdx.x / kTX;   // 1-D block of kTX x kTY threads
    for (int r = ty; r < kTY + 2 * ry; r += kTY) {
        const int y = min(max(y0 - ry + r, 0), H - 1);
        for (int c = tx; c < kTX + 2 * rx; c += kTX) {
            const int x = min(max(x0 - rx + c, 0), W - 1);
            gs[r][c] = __ldg(grey + (size_t)y * W + x);
        }
    }
    __syncthreads();
    const int x = x0 + tx, y = y0 + ty;
    if (x >= W || y >= H) return;

    // census: bit k = [Y(n) < Y(p)], window row-major, centre skipped
    const uint32_t yc = gs[ty + ry][tx + rx];
    unsigned long long bits = 0ull;
    if (CW == 9 && CH == 7) {
        const uint32_t c4 = yc * 0x01010101u, c4lo = c4 & 0x7f7f7f7fu;
        const int al = tx & ~3, sh = 8 * (tx & 3);
        int k = 0;
#pragma unroll
        for (int dy = 0; dy < 7; dy++) {
            const uint32_t *row = reinterpret_cast<const uint32_t *>(&gs[ty + dy][al]);
            const uint32_t a0 = row[0], a1 = row[1], a2 = row[2];
            const uint32_t w0 = __funnelshift_r(a0, a1, sh);   // bytes dx 0..3
            const uint32_t w1 = __funnelshift_r(a1, a2, sh);   // bytes dx 4..7
            const uint32_t b8 = (__funnelshift_r(a2, 0u, sh) & 0xffu) < yc ? 1u : 0u;   // dx 8
            const uint32_t f0 = lt4(w0, c4, c4lo), f1 = lt4(w1, c4, c4lo);
            uint32_t rowbits;
            int nb;
            if (dy == 3) {   // centre row: dx 4 is the centre itself
                rowbits = f0 | ((f1 >> 1) << 4) | (b8 << 7);
                nb = 8;
            } else {
                rowbits = f0 | (f1 << 4) | (b8 << 8);
                nb = 9;
            }
            bits |= (unsigned long long)rowbits << k;
            k += nb;
        }
    } else {
        int k = 0;
        for (int dy = 0; dy < ch; dy++) {
            for (int dx = 0; dx < cw; dx++) {
                if (dy == ry && dx == rx) continue;
                if (gs[ty + dy][tx + dx] < yc) bits |= 1ull << k;
                k++;
            }
        }
    }

    // arms: largest k <= L1 whose steps all pass the double threshold
    const size_t i = (size_t)y * W + x;
    const uint32_t praw = __ldg(rgbx + i);   // colours are stored spread (k_pack), with edge bits
    const uint32_t p = praw & kColour;
    const int L1 = a.L1, L2 = a.L2;
    // K = t - 1 + 512 in each 10-bit field, t = min(tau, 256): the field of
    // E(c) + K - E(q) has bit 9 set exactly when c - q > -t, and with t = 256
    // every pair passes (a threshold of 256 or more never stops an arm).
    // Up to L2 a step is tested against p with tau1; beyond L2 against p
    // with min(tau1, tau2) (both must hold).  The test against the step's
    // predecessor (tau1) is the edge bit k_pack stored: the candidate's own
    // for walks right and down (its edge towards p), the predecessor's for
    // walks left and up.
    auto kfield = [](int tau) { return 0x00100401u * (uint32_t)(min(tau, 256) + 511); };
    const uint32_t k1 = kfield(a.tau1), k2 = kfield(min(a.tau1, a.tau2));
    const uint32_t K1p = k1 - p, pK1 = p + k1, K2p = k2 - p, pK2 = p + k2;
    auto fails = [](uint32_t c, uint32_t Kp, uint32_t pK, uint32_t ew, uint32_t bit) {
        return ((~((c + Kp) & (pK - c)) & kM9) | (~ew & bit)) != 0u;
    };
    // Steps n + 1 .. end of one direction, with one pair of constants; true if
    // all of them pass.  kArmRun candidates are loaded together, and tested one
    // by one with a way out after each, so a step costs its load, the two sums
    // and the two logic operations of its test and a branch.
    auto walk = [&](auto own_c, const uint32_t *&q, ptrdiff_t st, uint32_t &prev, int &n, int end, uint32_t Kp, uint32_t pK,
                    uint32_t bit) -> bool {
        constexpr bool kOwn = decltype(own_c)::value;   // right, down: the candidate's own edge bit; left, up: its predecessor's
        for (; n + kArmRun <= end; n += kArmRun) {
            uint32_t c[kArmRun];
#pragma unroll
            for (int u = 0; u < kArmRun; u++) c[u] = __ldg(q + (u + 1) * st);
#pragma unroll
            for (int u = 0; u < kArmRun; u++)
                if (fails(c[u], Kp, pK, kOwn ? c[u] : u ? c[u ? u - 1 : 0] : prev, bit)) {
                    n += u;
                    return false;
                }
            prev = c[kArmRun - 1];
            q += kArmRun * st;
        }
        for (; n < end; n++) {
            q += st;
            const uint32_t c = __ldg(q);
            if (fails(c, Kp, pK, kOwn ? c : prev, bit)) return false;
            prev = c;
        }
        return true;
    };
    // the first candidate of all four directions is loaded at once (in-image
    // addresses only)
    constexpr int kArmBatch = 1;
    int arm[4];
    uint32_t cand[4][kArmBatch];
    int lim[4];
    ptrdiff_t step[4];
#pragma unroll
    for (int e = 0; e < 4; e++) {
        const int room = e == 0 ? x : (e == 1 ? W - 1 - x : (e == 2 ? y : H - 1 - y));
        step[e] = e == 0 ? -1 : (e == 1 ? 1 : (e == 2 ? -(ptrdiff_t)W : (ptrdiff_t)W));
        lim[e] = min(L1, room);
#pragma unroll
        for (int u = 0; u < kArmBatch; u++)
            cand[e][u] = u < lim[e] ? __ldg(rgbx + i + (u + 1) * step[e]) : 0u;
    }
#pragma unroll
    for (int e = 0; e < 4; e++) {
        const uint32_t bit = e < 2 ? kEdgeL : kEdgeU;
        const bool own = e & 1;   // right, down: the candidate's own edge bit
        uint32_t prev = praw;     // left, up: the predecessor's (p itself before step 1)
        int n = 0;
        bool open = true;
#pragma unroll
        for (int u = 0; u < kArmBatch; u++) {
            const int j = u + 1;
            const bool far = j > L2;
            const uint32_t c = cand[e][u];
            if (open && j <= lim[e] && !fails(c, far ? K2p : K1p, far ? pK2 : pK1, own ? c : prev, bit)) {
                n = j;
                prev = c;
            } else {
                open = false;
            }
        }
        if (open) {   // longer arms: up to L2, then beyond
            const uint32_t *q = rgbx + i + (ptrdiff_t)n * step[e];
            if (own) {
                if (walk(std::true_type{}, q, step[e], prev, n, min(lim[e], L2), K1p, pK1, bit))
                    walk(std::true_type{}, q, step[e], prev, n, lim[e], K2p, pK2, bit);
            } else {
                if (walk(std::false_type{}, q, step[e], prev, n, min(lim[e], L2), K1p, pK1, bit))
                    walk(std::false_type{}, q, step[e], prev, n, lim[e], K2p, pK2, bit);
            }
        }
        arm[e] = n;
    }
    const int lmin = min(min(arm[0], arm[1]), min(arm[2], arm[3]));
    const uint32_t colour = unspread10(p) | (uint32_t(lmin) << 24);
    const size_t pe = (size_t)y * a.pw + x;
    (img ? a.cen[1] : a.cen[0])[pe] = make_uint2((uint32_t)bits, (uint32_t)(bits >> 32));
    (img ? a.col[1] : a.col[0])[pe] = colour;
    (img ? a.arms[1] : a.arms[0])[i] = make_uchar4((uint8_t)arm[0], (uint8_t)arm[1], (uint8_t)arm[2], (uint8_t)arm[3]);
}

// The same for launches that leave most of the SMs idle, where the time is that
// of one pixel's four walks: block = a 32 x 4 tile, four threads per pixel,
// warp = (direction, row).  Every thread walks one arm of its pixel and takes
// two rows of its census window; one warp per row puts the parts together.
// 96x64 13.0 -> 9.9 us, 320x240 18.8 us either way, 640x480 46.7 against 35.3 us
// (four times the set-up per pixel): the line lies at two blocks of prep_body
// per SM.
constexpr int kTYd = 4, kDirs = 4, kPrepThreads = kTX * kTYd * kDirs;
constexpr int kArmRunDirs = 4;

template <int CW, int CH>
__device__ __forceinline__ void prep_dirs_body(const PrepArgs &a, int bx, int by, int img)
{
    __shared__ __align__(16) uint8_t gs[kTYd + kMaxCH - 1][kGW];
    __shared__ uint2 part_s[kDirs][kTYd][kTX];   // census bits
    __shared__ uint8_t arm_s[kDirs][kTYd][kTX];
    constexpr bool kStd = CW == 9 && CH == 7;
    const uint32_t *__restrict__ rgbx = img ? a.rgbx[1] : a.rgbx[0];
    const uint8_t *__restrict__ grey = img ? a.grey[1] : a.grey[0];
    const int W = a.W, H = a.H;
    const int cw = CW ? CW : a.cw, ch = CH ? CH : a.ch;
    const int rx = cw / 2, ry = ch / 2;
    const int x0 = bx * kTX, y0 = by * kTYd;
    const int warp = threadIdx.x >> 5, tx = threadIdx.x & 31, ty = warp % kTYd, dir = warp / kTYd;   // left, right, up, down
    const int x = x0 + tx, y = y0 + ty;
    const bool in = x < W && y < H;
    const size_t i = (size_t)min(y, H - 1) * W + min(x, W - 1);
    const uint32_t praw = __ldg(rgbx + i);   // colours are stored spread (k_pack), with edge bits
    for (int r = warp; r < kTYd + 2 * ry; r += kTYd * kDirs) {
        const uint8_t *g = grey + (size_t)min(max(y0 - ry + r, 0), H - 1) * W;
        for (int c = tx; c < kTX + 2 * rx; c += kTX) gs[r][c] = __ldg(g + min(max(x0 - rx + c, 0), W - 1));
    }

    // the arm: the rule of prep_body
    {
        const uint32_t p = praw & kColour;
        auto kfield = [](int tau) { return 0x00100401u * (uint32_t)(min(tau, 256) + 511); };
        const uint32_t k1 = kfield(a.tau1), k2 = kfield(min(a.tau1, a.tau2));
        const uint32_t bit = dir < 2 ? kEdgeL : kEdgeU;
        const int st = dir == 0 ? -1 : dir == 1 ? 1 : dir == 2 ? -W : W;
        const int room = dir == 0 ? x : dir == 1 ? W - 1 - x : dir == 2 ? y : H - 1 - y;
        const int lim = in ? min(a.L1, room) : 0;
        const uint32_t *q = rgbx + i;
        uint32_t prev = praw;
        int n = 0;
        auto fails = [&](uint32_t c, uint32_t Kp, uint32_t pK, uint32_t ew) {
            return ((~((c + Kp) & (pK - c)) & kM9) | (~ew & bit)) != 0u;
        };
        // steps n + 1 .. end; true if all of them pass
        auto walk = [&](auto own_c, int end, uint32_t k) -> bool {
            constexpr bool kOwn = decltype(own_c)::value;
            const uint32_t Kp = k - p, pK = p + k;
            for (; n + kArmRunDirs <= end; n += kArmRunDirs) {
                uint32_t c[kArmRunDirs];
#pragma unroll
                for (int u = 0; u < kArmRunDirs; u++) {
                    q += st;
                    c[u] = __ldg(q);
                }
#pragma unroll
                for (int u = 0; u < kArmRunDirs; u++)
                    if (fails(c[u], Kp, pK, kOwn ? c[u] : u ? c[u ? u - 1 : 0] : prev)) {
                        n += u;
                        return false;
                    }
                prev = c[kArmRunDirs - 1];
            }
            for (; n < end; n++) {
                q += st;
                const uint32_t c = __ldg(q);
                if (fails(c, Kp, pK, kOwn ? c : prev)) return false;
                prev = c;
            }
            return true;
        };
        if (dir & 1) {
            if (walk(std::true_type{}, min(lim, a.L2), k1)) walk(std::true_type{}, lim, k2);
        } else {
            if (walk(std::false_type{}, min(lim, a.L2), k1)) walk(std::false_type{}, lim, k2);
        }
        arm_s[dir][ty][tx] = (uint8_t)n;
    }
    __syncthreads();   // (the grey tile)

    // census: bit k = [Y(n) < Y(p)], window row-major, centre skipped
    const uint32_t yc = gs[ty + ry][tx + rx];
    if (kStd) {
        const uint32_t c4 = yc * 0x01010101u, c4lo = c4 & 0x7f7f7f7fu;
        const int al = tx & ~3, sh = 8 * (tx & 3);
        auto row_bits = [&](int dy) -> uint32_t {
            const uint32_t *row = reinterpret_cast<const uint32_t *>(&gs[ty + dy][al]);
            const uint32_t a0 = row[0], a1 = row[1], a2 = row[2];
            const uint32_t w0 = __funnelshift_r(a0, a1, sh);   // bytes dx 0..3
            const uint32_t w1 = __funnelshift_r(a1, a2, sh);   // bytes dx 4..7
            const uint32_t b8 = (__funnelshift_r(a2, 0u, sh) & 0xffu) < yc ? 1u : 0u;   // dx 8
            const uint32_t f0 = lt4(w0, c4, c4lo), f1 = lt4(w1, c4, c4lo);
            return dy == 3 ? f0 | ((f1 >> 1) << 4) | (b8 << 7)   // centre row: dx 4 is the centre itself
                           : f0 | (f1 << 4) | (b8 << 8);
        };
        // window rows 2 dir, 2 dir + 1; rows start at bits 0, 9, 18, 27, 35, 44, 53
        const int first = 18 * dir - (dir > 1), second = dir == 1 ? 27 : first + 9;
        unsigned long long bits = (unsigned long long)row_bits(2 * dir) << first;
        if (dir < 3) bits |= (unsigned long long)row_bits(2 * dir + 1) << second;
        part_s[dir][ty][tx] = make_uint2((uint32_t)bits, (uint32_t)(bits >> 32));
    }
    __syncthreads();
    if (dir != 0 || !in) return;
    uint2 census;
    if (kStd) {
        const uint2 b0 = part_s[0][ty][tx], b1 = part_s[1][ty][tx], b2 = part_s[2][ty][tx], b3 = part_s[3][ty][tx];
        census = make_uint2(b0.x | b1.x | b2.x | b3.x, b0.y | b1.y | b2.y | b3.y);
    } else {
        unsigned long long bits = 0ull;
        int k = 0;
        for (int dy = 0; dy < ch; dy++) {
            for (int dx = 0; dx < cw; dx++) {
                if (dy == ry && dx == rx) continue;
                if (gs[ty + dy][tx + dx] < yc) bits |= 1ull << k;
                k++;
            }
        }
        census = make_uint2((uint32_t)bits, (uint32_t)(bits >> 32));
    }
    const int l = arm_s[0][ty][tx], r = arm_s[1][ty][tx], u = arm_s[2][ty][tx], d = arm_s[3][ty][tx];
    const uint32_t lmin = (uint32_t)min(min(l, r), min(u, d));
    const size_t pe = (size_t)y * a.pw + x;
    (img ? a.cen[1] : a.cen[0])[pe] = census;
    (img ? a.col[1] : a.col[0])[pe] = unspread10(praw) | (lmin << 24);
    (img ? a.arms[1] : a.arms[0])[i] = make_uchar4((uint8_t)l, (uint8_t)r, (uint8_t)u, (uint8_t)d);
}

// --------------------------------------------------------------- k_smooth
// Smooth cross-support window (Sect. 4.1, morphological processing): the
// opening of each arm map is a 3x3 minimum (kMax = false) followed by a 3x3
// maximum (kMax = true), windows cut to the image.  An opening never
// lengthens an arm, so arms stay inside the image and <= L1.  The maximum
// pass also rewrites the colour word's L_min (Eq. 1's weight).
// A thread takes four pixels of a column, six rows of three arm words: the
// four arms of a word are compared at once (byte-wise minimum or maximum), and
// coordinates past the border repeat the border, which changes neither.
// 640x480: 13.3 -> 8.1 us (nine words per pixel, arm by arm, before).
constexpr int kSmRows = 4;
template <bool kMax>
__device__ __forceinline__ void smooth_body(const SmoothArgs &a, int t, int img)
{
    const int W = a.W, H = a.H, x = t % W, y0 = kSmRows * (t / W);
    if (y0 >= H) return;
    const uint32_t *src = reinterpret_cast<const uint32_t *>(img ? a.src[1] : a.src[0]);
    const int xl = max(x - 1, 0), xr = min(x + 1, W - 1);
    auto pick = [](uint32_t u, uint32_t v) { return kMax ? __vmaxu4(u, v) : __vminu4(u, v); };
    uint32_t row[kSmRows + 2];   // of the three words of each row
#pragma unroll
    for (int k = 0; k < kSmRows + 2; k++) {
        const uint32_t *p = src + (size_t)min(max(y0 - 1 + k, 0), H - 1) * W;
        row[k] = pick(pick(p[xl], p[x]), p[xr]);
    }
#pragma unroll
    for (int k = 0; k < kSmRows; k++) {
        const int y = y0 + k;
        if (y >= H) break;
        const uint32_t v = pick(pick(row[k], row[k + 1]), row[k + 2]);
        reinterpret_cast<uint32_t *>(img ? a.dst[1] : a.dst[0])[(size_t)y * W + x] = v;
        if (kMax) {
            const uint32_t lmin = min(min(v & 0xffu, (v >> 8) & 0xffu), min((v >> 16) & 0xffu, v >> 24));
            uint32_t *c = (img ? a.col[1] : a.col[0]) + (size_t)y * a.pw + x;
            *c = (*c & 0x00ffffffu) | (lmin << 24);
        }
    }
}

// ------------------------------------------------------------ copies, waits
__device__ __forceinline__ void cp_async16(void *dst, const void *src)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async4(void *dst, const void *src)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async8(void *dst, const void *src)
{
    const unsigned s = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

constexpr int kWaitLimit = 1 << 22;   // mbarrier polls before a copy is declared lost
constexpr int kTestWaitLimit = 64;    // the same, under the lost-copy failure test
constexpr int kStatusCopyTimeout = 1; // status word: k_hagg's staging copies did not complete

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n" ::"r"(bar),
                 "r"(bytes)
                 : "memory");
}
// bounded wait for the phase of the given parity to complete: false after
// `limit` polls without completion
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int limit)
{
    for (int i = 0; i < limit; i++) {
        uint32_t ok;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                     " selp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(ok)
                     : "r"(bar), "r"(parity)
                     : "memory");
        if (ok) return true;
    }
    return false;
}
// bulk copy of n bytes (a multiple of 16; both addresses 16-byte aligned)
// from global memory to shared memory, completing on mbarrier `bar`
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t n, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(n), "r"(bar)
                 : "memory");
}

// ------------------------------------------------------------------ k_hagg
// Eq. 1 costs and their horizontal segment sums (the first 1-D sum of Eq. 2).
// Block = (row, view, 32 disparities, a range of columns): a warp per four
// disparities and up to 320 columns, so eight warps for ranges of at most 320 reference
// columns (four blocks per SM), sixteen up to 640 (two).  The records of both
// images, the arms and the tables arrive in shared memory by bulk copies on one mbarrier
// (bounded wait).  Then:
//   A. a warp walks its part in segments of 160 columns (ends in one of 96 or
//      32), lane = five (three, one)
//      consecutive columns x four disparities: the reference records stay in
//      registers and each candidate loaded serves up to four costs; costs
//      rounded to fixed point, prefixes within the lane, a scan of the lanes'
//      totals, and the prefixes stored as one 16-byte word per column
//      (G[quad][x], lanes an odd number of words apart: no bank conflicts);
//   B. every output column: S_H = G(end) - G(start), eight lanes (quads) per
//      column, a 128-byte line of the slice per column; the planes' stride
//      puts the eight quads of a column on distinct banks whatever the arms.
// Bound by the shared-memory data path (15 M wavefronts at 640x480, D = 64, 88 %
// of the L1 throughput, a third of them the table gathers of Eq. 1).  Against
// one block per task with a disparity pair per lane and sixteen-column
// segments: 46 M instead of 52 M instructions; 640x480, D = 64, one pass 70 -> 66
// us (in two passes 82), 1280x720, D = 128 481 -> 416 us, 1920x1080, D = 256 in
// eight passes 1960 -> 1817 us.  Blocks of sixteen warps alone left half of them
// idle on rows of up to 160 columns and an SM with two blocks in the same phase on
// rows of up to 320: 64 pairs of 160x120, D = 32 206 us against 140 with eight warps (one
// block per row and group before: 121), of 320x240 574 against 465 (502), 256x192,
// D = 64 22.1 against 17.7 us (17.1).  Both views in one block from one
// evaluation of every pixel pair (16 disparities, 96 registers, one set of
// table gathers for two costs) took 72-75 us: 13.5 M wavefronts, but sixteen
// warps per SM, and right-view windows that move with the disparity.
constexpr int kHD = 32;        // disparities per block
constexpr int kHQuads = kHD / 4;
constexpr int kHCols = 5;      // columns per lane (odd: conflict-free stores)
constexpr int kHSegCols = 32 * kHCols;
constexpr int kHScan = 40;     // words per value of the scan of the lanes' totals (eight lanes' 16-byte reads hit distinct banks)
constexpr int kTabBytes = kTabFloats * 4;

// Byte offsets of the shared memory of a block of kParts warps per quad: each
// copied range has room for its 16-byte alignment; the arms of two tasks.
template <int kParts>
struct HSmem {
    static constexpr int warps = kParts * kHQuads, cols = kParts * 2 * kHSegCols;   // cols: reference columns
    static constexpr int plane = cols + 1;   // 16-byte words per plane: odd
    static constexpr int e = cols + 4, f = cols + kHD + 4;   // reference and candidate columns
    // (a second copy of the AD table for every other lane: 67.7 against 65.8 us at
    // 640x480, D = 64: neighbouring columns often read the same entry)
    static constexpr int rcen = kTabBytes, ccen = rcen + 8 * e, rcol = ccen + 8 * f, ccol = rcol + 4 * e;
    static constexpr int arm = ccol + 4 * f, arms = 4 * e, g = arm + 2 * arms;
    static constexpr int total = g + kHQuads * plane * 16;
};

// one unit of a block's work: a range of output columns of a row, view and group
struct HTask {
    int live;
    int W, p0, n, q0, nq;      // reference columns p0 .. p0 + n - 1, candidates q0 .. q0 + nq - 1
    int m, lead;               // output columns, the first at relative column `lead`
    int view, dlo, dend, arm;  // arm: entries before the first output's arm word in the copy
    float S;
    uint32_t Sint;
    size_t ds4;                // slice words of a pixel / 4
    uint4 *out;                // slice of the first output column, this group
    unsigned long long *init;  // keys to set (null: none)
};

// Blocks are resident and take tasks in turn: the next task's copies are in
// flight during phase B, which does not read the records.  Warp 0 prepares them (a
// thread's chain of about a microsecond) and takes no part in B.
// find(t, bx, by, bz): the arguments of task t and its place in their grid.
template <int kParts, class Find>
__device__ __forceinline__ void hagg_tasks(int ntasks, Find find)
{
    using hsm = HSmem<kParts>;
    extern __shared__ __align__(16) uint8_t smem_raw[];
    __shared__ __align__(8) unsigned long long hbar_s;
    __shared__ HTask task_s[2];
    __shared__ uint4 half_s[kHQuads];   // totals of the first half
    __shared__ int lost_s;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t bar = (uint32_t)__cvta_generic_to_shared(&hbar_s);
    const float *sTC = reinterpret_cast<const float *>(smem_raw) + kTabAD, *sAl = sTC + kTabCen;

    // thread 0: task t's description, and its copies.  Each starts on the
    // 16-byte boundary at or below its first entry and ends on the one at or
    // above its last.
    auto prepare = [&](int t, int slot) {
        HTask k;
        k.live = t < ntasks;
        if (!k.live) {
            task_s[slot].live = 0;
            return;
        }
        int y, part, bz;   // rows first, then ranges: the short last ranges come last
        const HArgs &a = find(t, y, part, bz);
        const int W = a.W, L1 = a.L1, xs = part ? a.first + (part - 1) * a.chunk : 0;
        const int xe = min(W, part ? xs + a.chunk : a.first);
        const int view = bz / a.ngroups, g32 = bz - view * a.ngroups, dlo = a.d0 + kHD * g32;
        const int p0 = max(0, xs - L1), pe = min(W, xe + L1);
        const int q0 = max(0, min(W, view ? p0 + dlo : p0 - dlo - (kHD - 1)));
        const int q1 = max(q0, min(W, view ? pe + dlo + kHD - 1 : pe - dlo));
        const size_t row = (size_t)y * a.pw, arow = (size_t)y * W, ga = (arow + xs) & ~(size_t)3;
        k.W = W;
        k.p0 = p0;
        k.n = pe - p0;
        k.q0 = q0;
        k.nq = q1 - q0;
        k.m = xe - xs;
        k.lead = xs - p0;
        k.view = view;
        k.dlo = dlo;
        k.dend = min(a.d0 + a.dc, a.D);
        k.arm = (int)(arow + xs - ga);
        k.S = a.S;
        k.Sint = a.Sint;
        k.ds4 = (size_t)a.dstride / 4;
        k.out = reinterpret_cast<uint4 *>((view ? a.sh[1] : a.sh[0]) + (arow + xs) * a.dstride + kHD * g32);
        unsigned long long *init = view ? a.init[1] : a.init[0];
        k.init = init && g32 == 0 ? init + arow + xs : nullptr;
        task_s[slot] = k;
        auto bytes = [](int x0, int x1, int size) -> uint32_t {   // of entries [x0, x1) from the boundary below x0
            const int per = 16 / size;
            return x1 > x0 ? (uint32_t)((x1 - (x0 & ~(per - 1)) + per - 1) & ~(per - 1)) * size : 0u;
        };
        const uint32_t nrc = bytes(p0, pe, 8), ncc = bytes(q0, q1, 8), nrk = bytes(p0, pe, 4), nck = bytes(q0, q1, 4);
        const uint32_t na = 4u * ((uint32_t)(arow + xe - ga + 3) & ~3u);
        mbar_expect_tx(bar, nrc + ncc + nrk + nck + na);
        if (a.skip_copy) return;   // (the failure test arms the barrier and issues nothing)
        const uint2 *cr = view ? a.cen[1] : a.cen[0], *cc = view ? a.cen[0] : a.cen[1];
        const uint32_t *kr = view ? a.col[1] : a.col[0], *kc = view ? a.col[0] : a.col[1];
        bulk_g2s(smem_raw + hsm::rcen, cr + row + (p0 & ~1), nrc, bar);
        bulk_g2s(smem_raw + hsm::rcol, kr + row + (p0 & ~3), nrk, bar);
        if (ncc) bulk_g2s(smem_raw + hsm::ccen, cc + row + (q0 & ~1), ncc, bar);
        if (nck) bulk_g2s(smem_raw + hsm::ccol, kc + row + (q0 & ~3), nck, bar);
        bulk_g2s(smem_raw + hsm::arm + slot * hsm::arms, (view ? a.arms[1] : a.arms[0]) + ga, na, bar);
    };
    int next = blockIdx.x;
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        lost_s = 0;
        prepare(next, 0);
    }
    if (next < ntasks) {
        int bx, by, bz;
        const float *tables = find(next, bx, by, bz).tables;   // (one set per handle: the same for every task)
        for (int i = threadIdx.x; i < kTabFloats; i += blockDim.x) reinterpret_cast<float *>(smem_raw)[i] = __ldg(tables + i);
    }
    for (int it = 0;; it++) {
        const int slot = it & 1;
        if (threadIdx.x == 0 && task_s[slot].live) {
            int bx, by, bz;
            const HArgs &a = find(next, bx, by, bz);
            if (!mbar_wait(bar, (uint32_t)slot, a.wait_limit)) {
                // report, and wait (bounded) once more before the block's shared memory is released
                if (a.status) atomicOr(a.status, kStatusCopyTimeout);
                mbar_wait(bar, (uint32_t)slot, a.wait_limit);
                lost_s = 1;
            }
        }
        __syncthreads();   // (also: the last task's outputs have been read from G)
        const HTask &k = task_s[slot];
        if (!k.live || lost_s) return;
        if (unsigned long long *init = k.init)   // the keys the V pass minimises into
            for (int i = threadIdx.x; i < k.m; i += blockDim.x) init[i] = ~0ull;

        // ---- A: prefixes of the warp's quad over its half of the columns
        const int n = k.n, view = k.view;
        // first column of the second half: whole segments (of 160 and 96) before it
        const int split = kParts == 1 ? n : n <= 352 ? min(n, 160) : n <= 448 ? 256 : 320;
        {
            const int quad = warp & (kHQuads - 1), half = warp / kHQuads, d0 = k.dlo + 4 * quad;
            const int W = k.W, p0 = k.p0, q0 = k.q0, nq = k.nq;
            const uint2 *rcen = reinterpret_cast<const uint2 *>(smem_raw + hsm::rcen) + (p0 & 1);
            const uint32_t *rcol = reinterpret_cast<const uint32_t *>(smem_raw + hsm::rcol) + (p0 & 3);
            // indexed by candidate column - q0
            const uint2 *ccen = reinterpret_cast<const uint2 *>(smem_raw + hsm::ccen) + (q0 & 1);
            const uint32_t *ccol = reinterpret_cast<const uint32_t *>(smem_raw + hsm::ccol) + (q0 & 3);
            uint4 *g = reinterpret_cast<uint4 *>(smem_raw + hsm::g) + quad * hsm::plane;
            const float S = k.S;
            const uint32_t one = k.Sint;
            // Cost j of column c meets candidate c + 3 - j of the lane's eight:
            // disparity d0 + j in the left view, d0 + 3 - j in the right one.
            const int cand = view ? p0 + d0 - q0 : p0 - d0 - 3 - q0;   // of relative column 0, relative to q0
            uint32_t carry = 0;   // of cost lane & 3: the prefix before the segment
            // columns s .. s + 32 kCols - 1 (relative); kEdge: some lie past the range, or
            // meet candidates outside the image
            auto segment = [&](int s, auto cols_c, auto edge_c) {
                constexpr int kCols = decltype(cols_c)::value;
                constexpr bool kEdge = decltype(edge_c)::value;
                const int x = s + kCols * lane;   // the lane's first column
                uint32_t lo[kCols], hi[kCols], rgb[kCols];
                float av[kCols];
#pragma unroll
                for (int c = 0; c < kCols; c++) {
                    const int i = kEdge ? min(x + c, n - 1) : x + c;
                    const uint2 ce = rcen[i];
                    lo[c] = ce.x;
                    hi[c] = ce.y;
                    rgb[c] = rcol[i];
                    av[c] = sAl[rgb[c] >> 24];
                }
                // c - j of the costs inside the image: [first, last)
                const int first = view ? -4 : d0 - p0 - x, last = view ? W - p0 - x - d0 - 3 : kCols;
                uint32_t pl[kCols][4];   // prefixes within the lane
#pragma unroll
                for (int i = 0; i < kCols + 3; i++) {
                    const int r = kEdge ? max(0, min(cand + x + i, nq - 1)) : cand + x + i;
                    const uint2 ce = ccen[r];
                    const uint32_t rc = ccol[r];
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        const int c = i - 3 + j;
                        if (c < 0 || c >= kCols) continue;   // (resolved at compile time)
                        const int h = __popc(lo[c] ^ ce.x) + __popc(hi[c] ^ ce.y);
                        const uint32_t k4 = __dp4a(__vabsdiffu4(rgb[c], rc), 0x00040404u, 0u);   // byte offset
                        const float ta = *reinterpret_cast<const float *>(smem_raw + k4), tc = sTC[h];
                        uint32_t q = __float2uint_rn(fmaf(av[c], ta, (S - av[c]) * tc));
                        if (kEdge && (c - j < first || c - j >= last)) q = one;   // match outside the image: cost 1
                        pl[c][j] = c ? pl[c ? c - 1 : 0][j] + q : q;
                    }
                }
                // offsets of the lanes: exclusive scan of their four totals, by way
                // of shared memory (the segment's own columns of G, not yet
                // written): lane = (value, four lanes' worth of it)
                uint32_t *scan = reinterpret_cast<uint32_t *>(g + s + 1);
#pragma unroll
                for (int j = 0; j < 4; j++) scan[j * kHScan + lane] = pl[kCols - 1][j];
                __syncwarp();
                uint4 *mine = reinterpret_cast<uint4 *>(scan + (lane & 3) * kHScan + (lane >> 2) * 4);
                const uint4 t = *mine;
                const uint32_t a2 = t.x + t.y, a3 = a2 + t.z, a4 = a3 + t.w;
                uint32_t incl = a4;
#pragma unroll
                for (int o = 4; o < 32; o <<= 1) {
                    const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += u;
                }
                const uint32_t before = carry + incl - a4;
                *mine = make_uint4(before, before + t.x, before + a2, before + a3);
                carry += __shfl_sync(0xffffffffu, incl, 28 + (lane & 3));
                __syncwarp();
                uint32_t off[4];
#pragma unroll
                for (int j = 0; j < 4; j++) off[j] = scan[j * kHScan + lane];
                __syncwarp();
#pragma unroll
                for (int c = 0; c < kCols; c++) {
                    if (kEdge && x + c >= n) break;
                    const uint4 v = make_uint4(pl[c][0] + off[0], pl[c][1] + off[1], pl[c][2] + off[2], pl[c][3] + off[3]);
                    g[x + c + 1] = view ? make_uint4(v.w, v.z, v.y, v.x) : v;
                }
            };
            if (d0 < k.dend) {
                const int s1 = half ? n : split;
                for (int s = half ? split : 0; s < s1; s += kHSegCols) {
                    const bool inside = view ? p0 + s + kHSegCols + d0 + 3 <= W : p0 + s >= d0 + 3;
                    if (s1 - s <= 32) segment(s, std::integral_constant<int, 1>{}, std::true_type{});
                    else if (s1 - s <= 96) segment(s, std::integral_constant<int, 3>{}, std::true_type{});
                    else if (inside && s + kHSegCols <= n) segment(s, std::integral_constant<int, kHCols>{}, std::false_type{});
                    else segment(s, std::integral_constant<int, kHCols>{}, std::true_type{});
                }
                if (half == 0) {
                    if (lane == 0) g[0] = make_uint4(0u, 0u, 0u, 0u);
                    if (kParts > 1 && lane < 4) reinterpret_cast<uint32_t *>(&half_s[quad])[view ? 3 - lane : lane] = carry;
                }
            }
        }
        __syncthreads();
        next += gridDim.x;
        if (threadIdx.x == 0) prepare(next, slot ^ 1);

        // ---- B: segment sums; lane = (column, quad).  Whole 32-byte sectors are
        // written, a dead quad beside a live one too (half a sector is read back from
        // memory when the line leaves the L2: 1920x1080, D = 10 243 us against 146)
        const int quad = lane & (kHQuads - 1), c0 = 32 / kHQuads * (warp - 1);
        if (warp > 0 && k.dlo + 4 * (quad & ~1) < k.dend) {
            constexpr int kStep = (hsm::warps - 1) * 32 / kHQuads;
            const int lead = k.lead, cross = split - lead, m = k.m, col = lane / kHQuads;
            const uint4 *g = reinterpret_cast<const uint4 *>(smem_raw + hsm::g) + quad * hsm::plane + lead + col;
            const uchar4 *arm = reinterpret_cast<const uchar4 *>(smem_raw + hsm::arm + slot * hsm::arms) + k.arm + col;
            const size_t ds4 = k.ds4, ostep = kStep * ds4;
            uint4 *o = k.out + (c0 + col) * ds4 + quad;
            const uint4 tot = kParts > 1 ? half_s[quad] : make_uint4(0u, 0u, 0u, 0u);
            // columns i + col
            auto sum = [&](int i) {
                const uchar4 am = arm[i];
                const int hi = i + am.y + 1, lo = i - am.x;
                const uint4 h = g[hi], w = g[lo];
                uint4 v = make_uint4(h.x - w.x, h.y - w.y, h.z - w.z, h.w - w.w);
                if (kParts > 1 && i + kMaxL1 + 4 > cross && i - kMaxL1 <= cross) {   // near the halves' border (the same in the warp)
                    if (hi + col > cross && lo + col <= cross) v = make_uint4(v.x + tot.x, v.y + tot.y, v.z + tot.z, v.w + tot.w);
                }
                return v;
            };
            int i = c0;
            for (; i + kStep + 3 < m; i += 2 * kStep, o += 2 * ostep) {
                const uint4 v0 = sum(i), v1 = sum(i + kStep);
                o[0] = v0;
                o[ostep] = v1;
            }
            for (; i + col < m; i += kStep, o += ostep) o[0] = sum(i);
        }
    }
}

// The output phase of a pass whose lanes hold one disparity each (k_vcost):
// every output position c (n_out of them,
// prefix index base + c): S_H = F(c + r) - F(c - l - 1), F the prefix of the
// costs along the scan.  P holds prefixes local to segments of 1 << kSegLog
// positions and OFF the exclusive prefix of the segment totals, so
// F(x) = OFF[x >> kSegLog] + P(x) and F(-1) = 0 (the zero row in front of P,
// segment 0 whose offset is 0); no pass over P adds offsets.  Each
// quarter-warp takes one column, lane j of the quarter the disparities
// 4j .. 4j + 3 of the group (16-byte loads and stores, one 128-byte prefix
// row per quarter).  Unsigned wrap-around makes the differences exact.
template <int kSegLog>
__device__ __forceinline__ void hagg_out_quads(const uint32_t *P, const uint32_t *OFF, const uchar4 *sarm, int n_out,
                                               int base, uint32_t *o, size_t ds)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int l8 = lane & 7;
    const uint4 *P4 = reinterpret_cast<const uint4 *>(P) + l8;
    const uint4 *F4 = reinterpret_cast<const uint4 *>(OFF) + l8;
    uint4 *o4 = reinterpret_cast<uint4 *>(o) + l8;
    const size_t ds4 = ds / 4;
    auto column = [&](int i) -> uint4 {
        const uchar4 am = sarm[i];
        const int hi = base + i + am.y, lo = base + i - am.x - 1;   // lo >= -1
        const uint4 a = P4[hi * 8], b = P4[lo * 8];
        uint4 v = make_uint4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
        const int sh = hi >> kSegLog, sl = max(lo, 0) >> kSegLog;
        if (sh != sl) {   // the arm interval crosses segment boundaries
            const uint4 fh = F4[sh * 8], fl = F4[sl * 8];
            v.x += fh.x - fl.x;
            v.y += fh.y - fl.y;
            v.z += fh.z - fl.z;
            v.w += fh.w - fl.w;
        }
        return v;
    };
    int i = 4 * warp + (lane >> 3);
    const int step = 4 * nw;
    for (; i + step < n_out; i += 2 * step) {
        const uint4 v0 = column(i), v1 = column(i + step);
        o4[(size_t)i * ds4] = v0;
        o4[(size_t)(i + step) * ds4] = v1;
    }
    if (i < n_out) o4[(size_t)i * ds4] = column(i);
}

// Segment offsets and outputs of a pass (k_vcost) whose warps each
// scanned one segment of 1 << kSegLog positions: P holds every warp's local
// inclusive prefix of its segment, T the segment totals (visible after a
// barrier).
//   B. T is replaced by the exclusive prefix of the totals (segment offsets);
//   C. hagg_out_quads with those offsets.
template <int kSegLog>
__device__ __forceinline__ void hagg_tail(const uint32_t *P, uint32_t *T, const uchar4 *sarm, int n_out, int base,
                                          uint32_t *o, size_t ds)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t offs = 0;
#pragma unroll 4
    for (int w = 0; w < warp; w++) offs += T[w * 32 + lane];
    __syncthreads();
    T[warp * 32 + lane] = offs;
    __syncthreads();
    hagg_out_quads<kSegLog>(P, T, sarm, n_out, base, o, ds);
}

// ---------------------------------------------------------------- k_vcost
// The other aggregation order, first pass: Eq. 1 costs and their vertical
// segment sums S_V(q, d) over q's vertical arm.  Block = one column x (a
// chunk of rows) of one reference view for one group of 32 disparities;
// lane = disparity.  The reference records of the column are staged in
// shared memory; the candidates of each row (32 neighbouring pixels of the
// other view's row) are read straight from the planes.  Then the
// phases of a horizontal pass along the column: local prefixes over warp
// segments of 32 rows, segment offsets, segment sums (hagg_tail, with the
// up / down arms), written to the same slice layout.
// Bound by the L1 data path and its latency (76 % of its throughput; fewer
// instructions per row changed nothing), so by the warps that fit: with the
// plane entry as one 32-bit index the loop takes 38 registers (44 with two
// pointers), and two blocks of 720 rows share an SM: 1280x720, D = 128 974 -> 752
// us, 320x240, D = 32 22.7 -> 20.7, 333x211, D = 50 27.5 -> 29.3.
struct CSmem {
    int ref, arm, p, t, total;
    __host__ __device__ CSmem(int len, int chunk, int nw)
    {
        ref = kTabBytes;
        arm = ref + len * 16;
        p = arm + (chunk + 3) / 4 * 16 + 128;   // one zero row in front: P[-1]
        t = p + len * 128;
        total = t + nw * 128;
    }
};

__device__ __forceinline__ void vcost_body(const HArgs &a, int bx, int by, int bz)
{
    extern __shared__ __align__(16) uint8_t smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int W = a.W, H = a.H, L1 = a.L1;
    const int x = bx;
    const int view = bz / a.ngroups, g = bz % a.ngroups;
    const int ys = by * a.chunk, ye = min(H, ys + a.chunk);
    const int ya = max(0, ys - L1), yb = min(H, ye + L1), len = yb - ya;
    const CSmem L(len, a.chunk, nw);
    const float *sTC = reinterpret_cast<const float *>(smem_raw) + kTabAD;   // (the AD table comes first)
    uint4 *sref = reinterpret_cast<uint4 *>(smem_raw + L.ref);
    uchar4 *sarm = reinterpret_cast<uchar4 *>(smem_raw + L.arm);   // (up, down) of the output rows
    uint32_t *P = reinterpret_cast<uint32_t *>(smem_raw + L.p);    // [len][32], P[-1] = 0
    uint32_t *T = reinterpret_cast<uint32_t *>(smem_raw + L.t);
    const uint2 *cref = (view ? a.cen[1] : a.cen[0]) + x, *coth = view ? a.cen[0] : a.cen[1];
    const uint32_t *kref = (view ? a.col[1] : a.col[0]) + x, *koth = view ? a.col[0] : a.col[1];
    const uchar4 *aref = view ? a.arms[1] : a.arms[0];
    unsigned long long *init = view ? a.init[1] : a.init[0];
    if (init && g == 0)   // the keys the second pass minimises into
        for (int i = threadIdx.x; i < ye - ys; i += blockDim.x) init[(size_t)(ys + i) * W + x] = ~0ull;

    for (int i = threadIdx.x; i < kTabBytes / 16; i += blockDim.x)
        cp_async16(smem_raw + 16 * i, reinterpret_cast<const uint8_t *>(a.tables) + 16 * i);
    // a warp stages the rows of its own segment
    const int sa = warp * kHSegCost, sb = min(len, sa + kHSegCost), own = sa + lane;   // rows relative to ya
    if (own < len) {
        cp_async8(sref + own, cref + (size_t)(ya + own) * a.pw);
        cp_async4(&sref[own].z, kref + (size_t)(ya + own) * a.pw);
    }
    for (int i = threadIdx.x; i < ye - ys; i += blockDim.x) {
        const uchar4 am = aref[(size_t)(ys + i) * W + x];
        sarm[i] = make_uchar4(am.z, am.w, 0, 0);   // backward = up, forward = down
    }
    if (threadIdx.x < 32) P[(int)threadIdx.x - 32] = 0u;
    cp_async_wait_all();
    __syncthreads();
    if (own < len) reinterpret_cast<float *>(&sref[own])[3] = sTC[kTabCen + (sref[own].z >> 24)];   // alpha
    __syncwarp();

    const int dlo = a.d0 + 32 * g;
    const int dhi = min(min(a.d0 + a.dc, a.D), dlo + 32) - 1;
    const int d = dlo + lane;
    const int dd = d <= dhi ? d : dlo;                // dead lanes read a real candidate, results unused
    const int xo = view ? x + dd : x - dd;            // candidate column
    const bool outside = xo < 0 || xo >= W;           // match outside the image: cost 1
    const uint32_t pw = (uint32_t)a.pw;
    uint32_t at = (uint32_t)(ya + warp * kHSegCost) * pw + (uint32_t)max(0, min(xo, W - 1));   // the candidate's plane entry
    const float Sf = a.S;
    const uint32_t Sint = a.Sint;

    // ---- A: costs down this warp's segment of rows, local prefix
    uint32_t run = 0;
    auto rows = [&](auto edge_c) {
        constexpr bool kEdge = decltype(edge_c)::value;   // some lane's match lies outside the image
        int u = sa;
        auto cost = [&](int row, uint2 pc, uint32_t po) {
            const uint4 pr = sref[row];
            const int hm = __popc(pr.x ^ pc.x) + __popc(pr.y ^ pc.y);
            const uint32_t k4 = __dp4a(__vabsdiffu4(pr.z, po), 0x00040404u, 0u);   // byte offset
            const float av = __uint_as_float(pr.w), ta = *reinterpret_cast<const float *>(smem_raw + k4);
            const uint32_t q = __float2uint_rn(fmaf(av, ta, (Sf - av) * sTC[hm]));
            run += kEdge && outside ? Sint : q;
            P[row * 32 + lane] = run;
        };
        constexpr int kRows = 16;
        for (; u + kRows <= sb; u += kRows) {
            uint2 pc[kRows];
            uint32_t po[kRows];
#pragma unroll
            for (int k = 0; k < kRows; k++) {
                pc[k] = __ldg(coth + at);
                po[k] = __ldg(koth + at);
                at += pw;
            }
#pragma unroll
            for (int k = 0; k < kRows; k++) cost(u + k, pc[k], po[k]);
        }
        for (; u < sb; u++, at += pw) cost(u, __ldg(coth + at), __ldg(koth + at));
    };
    if (__any_sync(0xffffffffu, outside)) rows(std::true_type{});
    else rows(std::false_type{});
    T[warp * 32 + lane] = run;
    __syncthreads();
    // consecutive output rows are one slice row (W * dstride words) apart
    static_assert(kHSegCost == 1 << 5, "k_vcost segments: 32 rows per warp");
    hagg_tail<5>(P, T, sarm, ye - ys, ys - ya, (view ? a.sh[1] : a.sh[0]) + ((size_t)ys * W + x) * a.dstride + g * 32,
                 (size_t)W * a.dstride);
}

// ---------------------------------------------------------------- k_hvote
// Horizontal pass of the parallax optimisation (Sect. 4.3, Eq. 4): block =
// (row, group of 32 disparities), lane = disparity, local prefixes over warp
// segments of 64 columns of the indicator [disp(x, y) == d] of the map being
// voted on (-1 matches no d), then the output phase of the horizontal passes,
// so S_H holds the number of pixels of each horizontal segment that vote for
// d.  A local prefix counts at most 64 columns, so P keeps it in one byte
// per disparity (32 bytes per column): a quarter of the 4-byte prefix rows
// of the cost pass, so that more blocks fit an SM.
struct HVSmem {
    int disp, arm, p, t, total;
    __host__ __device__ HVSmem(int len, int chunk, int nw)
    {
        disp = 0;
        arm = (len * 2 + 15) / 16 * 16;
        p = arm + (chunk + 3) / 4 * 16 + 32;    // one zero row in front: P[-1]
        t = p + (len * 32 + 15) / 16 * 16;
        total = t + nw * 128;
    }
};

// The output phase of k_hvote: as hagg_out_quads, with byte prefixes (each
// lane of a quarter-warp reads the four counts of its disparities 4j .. 4j + 3
// as one word and widens them; unsigned wrap-around keeps the differences
// exact once the segment offsets are added).
template <int kSegLog>
__device__ __forceinline__ void hvote_out_quads(const uint8_t *P, const uint32_t *OFF, const uchar4 *sarm,
                                                int n_out, int base, uint32_t *o, size_t ds)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int l8 = lane & 7;
    const uint32_t *P4 = reinterpret_cast<const uint32_t *>(P) + l8;   // rows of 8 words
    const uint4 *F4 = reinterpret_cast<const uint4 *>(OFF) + l8;
    uint4 *o4 = reinterpret_cast<uint4 *>(o) + l8;
    const size_t ds4 = ds / 4;
    auto column = [&](int i) -> uint4 {
        const uchar4 am = sarm[i];
        const int hi = base + i + am.y, lo = base + i - am.x - 1;   // lo >= -1
        const uint32_t a = P4[hi * 8], b = P4[lo * 8];
        uint4 v = make_uint4((a & 0xffu) - (b & 0xffu), ((a >> 8) & 0xffu) - ((b >> 8) & 0xffu),
                             ((a >> 16) & 0xffu) - ((b >> 16) & 0xffu), (a >> 24) - (b >> 24));
        const int sh = hi >> kSegLog, sl = max(lo, 0) >> kSegLog;
        if (sh != sl) {   // the arm interval crosses segment boundaries
            const uint4 fh = F4[sh * 8], fl = F4[sl * 8];
            v.x += fh.x - fl.x;
            v.y += fh.y - fl.y;
            v.z += fh.z - fl.z;
            v.w += fh.w - fl.w;
        }
        return v;
    };
    int i = 4 * warp + (lane >> 3);
    const int step = 4 * nw;
    for (; i + step < n_out; i += 2 * step) {
        const uint4 v0 = column(i), v1 = column(i + step);
        o4[(size_t)i * ds4] = v0;
        o4[(size_t)(i + step) * ds4] = v1;
    }
    if (i < n_out) o4[(size_t)i * ds4] = column(i);
}

__device__ __forceinline__ void hvote_body(const HVArgs &a, int bx, int by, int bz)
{
    extern __shared__ __align__(16) uint8_t smem_raw[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int W = a.W, L1 = a.L1;
    const int y = by, g = bz;
    const int xs = bx * a.chunk, xe = min(W, xs + a.chunk);
    const int xa = max(0, xs - L1), xb = min(W, xe + L1), len = xb - xa;
    const HVSmem L(len, a.chunk, nw);
    int16_t *sd = reinterpret_cast<int16_t *>(smem_raw + L.disp);
    uchar4 *sarm = reinterpret_cast<uchar4 *>(smem_raw + L.arm);
    uint8_t *P = smem_raw + L.p;                                   // [len][32] bytes, P[-1] = 0
    uint32_t *T = reinterpret_cast<uint32_t *>(smem_raw + L.t);   // [nw][32]
    if (threadIdx.x < 32) P[(int)threadIdx.x - 32] = 0;
    const int16_t *drow = a.disp + (size_t)y * W;
    const uchar4 *aref = a.arms + (size_t)y * W;
    if (a.keys) {   // a later round: the previous round's winners where the first map was valid
        const unsigned long long *krow = a.keys + (size_t)y * W;
#pragma unroll 4
        for (int i = threadIdx.x; i < len; i += blockDim.x) {
            const int v = drow[xa + i];
            sd[i] = v >= a.dmin && v < a.D ? (int16_t)(krow[xa + i] & 0xffffu) : (int16_t)-1;
        }
    } else {
        for (int i = threadIdx.x; i < len; i += blockDim.x) sd[i] = drow[xa + i];
    }
    if (a.init && g == 0)   // the keys the V pass minimises into
        for (int i = threadIdx.x; i < xe - xs; i += blockDim.x) a.init[(size_t)y * W + xs + i] = ~0ull;
    for (int i = threadIdx.x; i < xe - xs; i += blockDim.x) sarm[i] = aref[xs + i];
    __syncthreads();

    // ---- A: votes and local prefix of this warp's segment (lane = d)
    const int d = a.d0 + 32 * g + lane;
    const int sa = warp * kHSeg, sb = min(len, sa + kHSeg);   // relative to xa
    static_assert(kHSeg <= 255, "k_hvote: local prefixes in one byte");
    uint32_t run = 0;
#pragma unroll 8
    for (int x = sa; x < sb; x++) {
        run += sd[x] == d ? 1u : 0u;
        P[x * 32 + lane] = (uint8_t)run;
    }
    T[warp * 32 + lane] = run;
    __syncthreads();
    // B: exclusive prefix of the segment totals (segment offsets), then C
    uint32_t offs = 0;
    for (int w = 0; w < warp; w++) offs += T[w * 32 + lane];
    __syncthreads();
    T[warp * 32 + lane] = offs;
    __syncthreads();
    hvote_out_quads<kHSegLog>(P, T, sarm, xe - xs, xs - xa, a.sh + ((size_t)y * W + xs) * a.dstride + g * 32,
                              a.dstride);
}

// ------------------------------------------------------------------ k_vagg
// Second 1-D sum (Eq. 2) and winner-take-all (Eq. 3).  A block of four warps
// walks down strips of four neighbouring columns for one group of 32
// disparities of one view, 32 slice rows per step, eight per warp; lane =
// (column, four consecutive disparities), so a row of the strip is one
// 16-byte load per lane (four 128-byte slice lines), issued a step ahead.
// A step:
//   - the totals of the warps' rows and the prefix before the step give each
//     warp its start; it writes the column prefix Q of its rows to a ring in
//     shared memory that holds the last 2 L1 + 1 rows besides the step's;
//   - V(d) = Q(y + down, d) - Q(y - up - 1, d) of the output rows that the
//     entered rows complete: two 16-byte reads per lane, on the same eight
//     bank quads whatever the arms are;
//   - the minimum over a lane's four disparities goes through a small tile to
//     the lane that owns the row, which finds the minimum over the group
//     (smallest d on ties) and minimises (V << 32 | d) into the pixel's key.
// A run of rows starts up to 2 L1 + 1 rows before its first output, so strips
// are split only where whole ones do not fill the SMs evenly (vagg_geom).
// Bound by the shared-memory and L1 data path (70 % of its cycles, DRAM at
// 45 %): per 32 evaluations one wavefront each for the load and the prefix's
// store and two for the window.  Three blocks (61 KB, L1 = 34) per SM; four,
// with the tile inside the totals, were slower (eight passes 1060 us).
// Against one block per column that held its whole column's prefix, lane =
// disparity: 1920x1080, D = 256, eight passes 2117 -> 998 us, one pass 1073
// -> 882 us; 640x480, D = 64, two passes 66.3 -> 50.5 us; small launches, which
// the longer chain of a strip would bind, take k_vcol.  Walks of one
// warp per strip with no block barrier (six or four warps per SM, by loads or
// TMA boxes) were latency bound: 55-65 us and 1090-1390 us.
//
// kMax: the WTA takes the largest V (the vote counts of Eq. 4, at most
// (2 L1 + 1)^2): it minimises 0x7fffffff - V.
// kRow: the other aggregation order: the walk runs along x over the vertical
// segment sums of four neighbouring rows, with p's horizontal arms.  Below,
// "rows" are the positions of the walk and "columns" the lines across it.
constexpr int kVCols = 4;        // columns per strip
constexpr int kVWarps = 4;
constexpr int kVThreads = 32 * kVWarps;
constexpr int kVSub = 8;         // rows per warp and step
constexpr int kVStep = kVWarps * kVSub;
constexpr int kVRow = 512;       // ring bytes per row: 32 lanes x 16
constexpr int kVTile = 128;      // reduction tile: bytes per output row (4 columns x 8 words)
constexpr int kVResident = 4;   // blocks per SM that the registers allow (128 each)
constexpr int kVHalf = 2;        // output rows whose window ends are loaded together (4 and 8: 1-2 % slower)
// the output rows of a step read back to 2 L1 + 1 rows above it
__host__ __device__ inline uint32_t vagg_ring_bytes(int L1)
{
    return (uint32_t)((2 * L1 + 1 + kVSub - 1) / kVSub * kVSub + kVStep) * kVRow;
}
__host__ __device__ inline size_t vagg_smem_bytes(int L1)
{
    return vagg_ring_bytes(L1) + (kVWarps + 2) * 512 + kVWarps * (kVSub * kVTile + 128);
}
static_assert(((2 * kMaxL1 + kVSub) / kVSub * kVSub + kVStep) * kVRow <= 1 << 16, "k_vagg: ring offsets in 16 bits");

template <bool kMax, bool kRow>
__device__ __forceinline__ void vagg_body(const VArgs &a, int blk)
{
    extern __shared__ __align__(128) uint8_t vring[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, col = lane >> 3, dq = lane & 7;
    const int E = kRow ? a.W : a.H, F = kRow ? a.H : a.W;     // extents along and across the walk
    const int pstep = kRow ? 1 : a.W, pcol = kRow ? a.W : 1;   // the same as pixel steps
    const int L1 = a.L1;
    const uint32_t rb = vagg_ring_bytes(L1);
    uint4 *sums = reinterpret_cast<uint4 *>(vring + rb);                 // [kVWarps][32]: totals of the warps' rows
    uint4 *carry = sums + kVWarps * 32;                                  // [2][32]: prefix before the step
    uint8_t *tile = reinterpret_cast<uint8_t *>(carry + 2 * 32) + warp * (kVSub * kVTile + 128);   // [8 rows][32 lanes]
    uint8_t *offs = tile + kVSub * kVTile;                               // ring offsets: [4 columns][8 rows]
    uint8_t *own = vring + 16 * lane;                                    // the lane's words of ring row 0
    const uint32_t step = (uint32_t)pstep * (uint32_t)a.dstride * 4u;    // slice bytes per row

    // the block's runs of output rows: whole strips first, then its share of
    // the strips that are left over
    for (int k = 0;; k++) {
        int strip, ys, ye;
        if (k < a.rounds) {
            strip = k * a.nblk + blk;
            ys = 0;
            ye = E;
        } else {
            int first, f, f1;   // strip and rows among those that are left
            if (a.bands) {
                first = blk / a.bands;
                if (k > a.rounds || first >= a.rest) return;
                f = (blk - first * a.bands) * a.share;
                f1 = min(E, f + a.share);
            } else {
                const int f0 = blk * a.share;
                f1 = min(f0 + a.share, a.rest * E);
                first = f0 / E + k - a.rounds;
                f = k == a.rounds ? f0 : first * E;
                if (f >= f1) return;
                f -= first * E;
                f1 = min(E, f1 - first * E);
            }
            strip = a.rounds * a.nblk + first;
            ys = f;
            ye = f1;
        }
        const int layer = strip / a.strips, view = layer / a.ng, g = layer - view * a.ng;
        const int line = kVCols * (strip - layer * a.strips) + col;
        const size_t pix0 = (size_t)min(line, F - 1) * pcol;   // lanes past the last column repeat it
        const int dbase = a.d0 + 32 * g, nlive = min(32, min(a.dc - 32 * g, a.D - dbase));
        const uint32_t *arms = reinterpret_cast<const uint32_t *>(view ? a.arms[1] : a.arms[0]) + pix0;
        unsigned long long *best = (view ? a.best[1] : a.best[0]) + pix0;
        // Rows enter the ring kVStep at a time, eight per warp; row ys + L1 is
        // the first, at ring row 0.  The nfill rows before it end at the last
        // ring row, and the row before them counts as zeros.
        const int ya = max(0, ys - L1), yb = min(E, ye + L1);
        int y = ys + kVSub * warp;   // the output row that the warp's first entering row completes
        const uint8_t *src = reinterpret_cast<const uint8_t *>((view ? a.sh[1] : a.sh[0]) + pix0 * a.dstride + 32 * g) + 16 * dq;
        uint4 v[kVSub];
        auto load = [&](int row) {   // the warp's eight rows from `row` on
            const uint8_t *p = src + (ptrdiff_t)row * (ptrdiff_t)step;
            if (row + kVSub <= yb) {
#pragma unroll
                for (int r = 0; r < kVSub; r++) v[r] = __ldg(reinterpret_cast<const uint4 *>(p + (size_t)r * step));
            } else {   // (rows past the image are never read)
#pragma unroll
                for (int r = 0; r < kVSub; r++)
                    v[r] = row + r < yb ? __ldg(reinterpret_cast<const uint4 *>(p + (size_t)r * step))
                                        : make_uint4(0u, 0u, 0u, 0u);
            }
        };
        auto arm_word = [&](int row) { return row < ye ? __ldg(arms + (size_t)row * pstep) : 0u; };
        // the fill: a quarter of its rows per warp, all in flight at once
        const int nfill = ys + L1 - ya, quarter = (nfill + kVWarps - 1) / kVWarps;
        const int i0 = min(quarter * warp, nfill), i1 = min(i0 + quarter, nfill);
        uint8_t *fill = own + rb - (uint32_t)nfill * kVRow;   // ring row of row ya
        {
            const uint8_t *p = src + (size_t)(ya + i0) * step;
#pragma unroll 4
            for (int i = i0; i < i1; i++, p += step)
                if (ya + i < yb) cp_async16(fill + i * kVRow, p);
        }
        load(y + L1);
        uint32_t aw = arm_word(y + dq);   // the lane's own row of the warp's eight
        cp_async_wait_all();   // (a lane reads only what it copied itself)
        uint4 t = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 4
        for (int i = i0; i < i1; i++) {
            const uint4 w = *reinterpret_cast<const uint4 *>(fill + i * kVRow);
            t = make_uint4(t.x + w.x, t.y + w.y, t.z + w.z, t.w + w.w);
        }
        sums[32 * warp + lane] = t;
        __syncthreads();
        uint4 run = make_uint4(0u, 0u, 0u, 0u);
        if (warp == 0) *reinterpret_cast<uint4 *>(fill - kVRow) = run;
        for (int w = 0; w < warp; w++) {
            const uint4 s = sums[32 * w + lane];
            run = make_uint4(run.x + s.x, run.y + s.y, run.z + s.z, run.w + s.w);
        }
#pragma unroll 4
        for (int i = i0; i < i1; i++) {
            uint4 *p = reinterpret_cast<uint4 *>(fill + i * kVRow);
            const uint4 w = *p;
            run = make_uint4(run.x + w.x, run.y + w.y, run.z + w.z, run.w + w.w);
            *p = run;
        }
        if (warp == kVWarps - 1) carry[lane] = run;
        __syncthreads();   // (the totals have been read)
        uint32_t in = kVSub * kVRow * warp;   // ring offset of the warp's first entering row
        int buf = 0;
        for (int yb0 = ys; yb0 < ye; yb0 += kVStep) {
            // ---- the column prefix over the block's kVStep rows
            t = v[0];
#pragma unroll
            for (int r = 1; r < kVSub; r++) t = make_uint4(t.x + v[r].x, t.y + v[r].y, t.z + v[r].z, t.w + v[r].w);
            sums[32 * warp + lane] = t;
            __syncthreads();   // (also: the window reads of the last step are done)
            run = carry[32 * buf + lane];
            for (int w = 0; w < warp; w++) {
                const uint4 s = sums[32 * w + lane];
                run = make_uint4(run.x + s.x, run.y + s.y, run.z + s.z, run.w + s.w);
            }
            {
                uint8_t *p = own + in;
#pragma unroll
                for (int r = 0; r < kVSub; r++) {
                    run = make_uint4(run.x + v[r].x, run.y + v[r].y, run.z + v[r].z, run.w + v[r].w);
                    *reinterpret_cast<uint4 *>(p + r * kVRow) = run;
                }
            }
            buf ^= 1;
            if (warp == kVWarps - 1) carry[32 * buf + lane] = run;
            load(y + kVStep + L1);   // the next step's rows are in flight during this one's output
            // and the lines of the step after it, one per lane, on their way to
            // L2 (a second step in registers made every wait on the first one
            // wait for both: 860 against 1190 us at 1920x1080, D = 256)
            if (const int row = y + 2 * kVStep + L1 + dq; row < yb)
                asm volatile("prefetch.global.L2 [%0];\n" ::"l"(src - 16 * dq + (ptrdiff_t)row * (ptrdiff_t)step));
            const uint32_t aw_next = arm_word(y + kVStep + dq);
            // ring offsets of the windows, each lane its own row's, passed to
            // the lanes of its column packed in one word
            const uint32_t back = kRow ? aw & 0xffu : (aw >> 16) & 0xffu, fwd = kRow ? (aw >> 8) & 0xffu : aw >> 24;
            uint32_t h = in + (dq + fwd) * kVRow + rb - L1 * kVRow, l = in + dq * kVRow + rb - (L1 + 1 + back) * kVRow;
            h = min(h, h - rb);   // modulo the ring (h below 3 rb, l below 2 rb)
            h = min(h, h - rb);
            l = min(l, l - rb);
            *reinterpret_cast<uint32_t *>(offs + 4 * lane) = h | l << 16;
            __syncthreads();
            // ---- the warp's output rows y .. y + 7
            if (y < ye) {
                const uint4 o0 = *reinterpret_cast<const uint4 *>(offs + 32 * col);
                const uint4 o1 = *reinterpret_cast<const uint4 *>(offs + 32 * col + 16);
                const uint32_t ov[kVSub] = {o0.x, o0.y, o0.z, o0.w, o1.x, o1.y, o1.z, o1.w};
                uint32_t who = 0;   // per row, which of the lane's four disparities wins
#pragma unroll
                for (int r0 = 0; r0 < kVSub; r0 += kVHalf) {
                    uint4 hi[kVHalf], lo[kVHalf];
#pragma unroll
                    for (int r = 0; r < kVHalf; r++) {
                        hi[r] = *reinterpret_cast<const uint4 *>(vring + ((ov[r0 + r] & 0xffffu) | 16 * lane));
                        lo[r] = *reinterpret_cast<const uint4 *>(vring + (ov[r0 + r] >> 16) + 16 * lane);
                    }
#pragma unroll
                    for (int u = 0; u < kVHalf; u++) {
                        const int r = r0 + u;
                        uint32_t c[4] = {hi[u].x - lo[u].x, hi[u].y - lo[u].y, hi[u].z - lo[u].z, hi[u].w - lo[u].w};
#pragma unroll
                        for (int j = 0; j < 4; j++)
                            if (kMax) c[j] = 0x7fffffffu - c[j];
                        if (nlive < 32) {
#pragma unroll
                            for (int j = 0; j < 4; j++) c[j] = 4 * dq + j < nlive ? c[j] : 0xffffffffu;
                        }
                        bool p01, p23, p;
                        const uint32_t m01 = __vibmin_u32(c[0], c[1], &p01), m23 = __vibmin_u32(c[2], c[3], &p23);
                        const uint32_t m = __vibmin_u32(m01, m23, &p);   // p: m01 <= m23
                        who = 4u * who + (p ? (p01 ? 0u : 1u) : (p23 ? 2u : 3u));
                        // 16-byte chunks of row r permuted by r: the reads below hit distinct banks
                        *reinterpret_cast<uint32_t *>(tile + r * kVTile + ((4 * lane) ^ (16 * r))) = m;
                    }
                }
                __syncwarp();
                // the lane's row y + dq: the minimum over the eight lanes of its
                // column, and which of that lane's four disparities has it
                const uint8_t *row = tile + dq * kVTile;
                const uint4 t0 = *reinterpret_cast<const uint4 *>(row + ((32 * col) ^ (16 * dq)));
                const uint4 t1 = *reinterpret_cast<const uint4 *>(row + ((32 * col + 16) ^ (16 * dq)));
                const uint32_t tv[8] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w};
                uint32_t m = tv[0];
                int q = 0;
#pragma unroll
                for (int i = 1; i < 8; i++) {
                    q = tv[i] < m ? i : q;   // strict: the smallest d on ties
                    m = min(m, tv[i]);
                }
                const uint32_t w = __shfl_sync(0xffffffffu, who, (lane & 24) | q);
                const uint32_t j = (w >> (2 * (kVSub - 1 - dq))) & 3u;
                if (line < F && y + dq < ye) {
                    const unsigned long long key = ((unsigned long long)m << 32) | (uint32_t)(dbase + 4 * q + j);
                    unsigned long long *b = best + (size_t)(y + dq) * pstep;
                    if (a.single) *b = key;
                    else atomicMin(b, key);
                }
            }
            aw = aw_next;
            y += kVStep;
            in += kVStep * kVRow;
            in = min(in, in - rb);
        }
        __syncthreads();   // the ring is the next run's
    }
}

// ------------------------------------------------------------------ k_vcol
// The same second sum and winner, a block per line: for short lines, for
// launches whose strips of k_vagg do not fill the SMs (whole_lines), and for
// cost volumes.  Block = one column x of one view (kRow: one
// row y), a chunk of output rows and their reach; a warp per 32 rows.  Per
// group of 32 disparities:
//   0. the warp's 32 slice rows (128 bytes each) into its rows of Q by 16-byte
//      asynchronous copies, all in flight;
//   A. lane = disparity: the rows into registers, their sum exchanged with the
//      other warps, and the column prefix in their place;
//   C. lane = output row: V(d) = Q(y + down, d) - Q(y - up - 1, d), four
//      disparities per 16-byte load, the running minimum with the smallest d
//      on ties in registers across the groups.
// One store per pixel and pass (a line belongs to one block), and N(p) of
// Eq. 2 from a prefix of the segment lengths, so costs and volumes are written
// here.  Q rows are 36 words: 32 rows of 16-byte loads spread over the banks.
// Bound by latency: a copy, two block barriers and a row's window per group, all
// blocks resident at once.  Against the strips (event times, us): 96x64, D = 16 8.3
// -> 6.9; 320x240, D = 32 14.3 -> 11.9, D = 64 18.6 -> 16.3; 333x211, D = 50 18.4 -> 14.6.
// A cost volume of 640x480, D = 64 takes 162 us here; summing N(p) from the arms
// for every group, as the strips would have to, 369.
constexpr int kQS = 36;        // Q row stride in words
constexpr int kColSeg = 32;    // rows per warp
constexpr int kColMax = 512;   // rows of a block's prefix range (16 warps)
// words: Q[-1] (zeros), Q [nw * 32], T [nw][32], NQ [nw * 32], NT [nw]
__host__ __device__ inline size_t vcol_smem_bytes(int nw) { return 4 * (size_t)(kQS + nw * (kColSeg * (kQS + 2) + 1)); }

template <bool kMax, bool kRow>
__device__ __forceinline__ void vcol_body(const VArgs &a, int fix, int view, int part)
{
    extern __shared__ __align__(16) uint32_t vsmem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const int W = a.W, H = a.H, L1 = a.L1;
    const int E = kRow ? W : H;
    const int ys = part * a.chunk, ye = min(E, ys + a.chunk);
    const int ya = max(0, ys - L1), len = min(E, ye + L1) - ya;
    const size_t pix0 = kRow ? (size_t)fix * W : (size_t)fix, pstep = kRow ? 1 : (size_t)W;   // pixels along the line
    uint32_t *Q = vsmem + kQS, *T = Q + nw * kColSeg * kQS, *NQ = T + nw * 32, *NT = NQ + nw * kColSeg;
    const uint32_t *arms = reinterpret_cast<const uint32_t *>(view ? a.arms[1] : a.arms[0]) + pix0;
    const size_t step = pstep * (size_t)a.dstride;
    const int r = warp * kColSeg + lane;   // the lane's row, relative to ya
    // group g's rows of the warp into its rows of Q: eight lanes per row, four
    // rows per instruction.  Rows past the range keep what they held: they are
    // summed after its last row, and the last warp's total is read by no other.
    const uint32_t *src = (view ? a.sh[1] : a.sh[0]) +
                          (pix0 + (size_t)(ya + warp * kColSeg + (lane >> 3)) * pstep) * a.dstride + 4 * (lane & 7);
    uint32_t *dst = Q + (warp * kColSeg + (lane >> 3)) * kQS + 4 * (lane & 7);
    const int nrow = len - warp * kColSeg - (lane >> 3);   // copied: the lane's rows 4 i < nrow
    auto load = [&](int g) {
#pragma unroll
        for (int i = 0; i < kColSeg / 4; i++)
            if (4 * i < nrow) cp_async16(dst + 4 * i * kQS, src + (size_t)(4 * i) * step + 32 * g);
    };
    load(0);
    const uint32_t aw = r < len ? __ldg(arms + (size_t)(ya + r) * pstep) : 0u;
    const int back = kRow ? aw & 0xffu : (aw >> 16) & 0xffu, fwd = kRow ? (aw >> 8) & 0xffu : aw >> 24;
    float *cost = view ? a.cost[1] : a.cost[0];
    const bool vol = a.vol != nullptr && view == a.vol_view;
    if (cost || vol) {   // the prefix of the segment lengths (the other arms)
        uint32_t n = r >= len ? 0u : kRow ? ((aw >> 16) & 0xffu) + (aw >> 24) + 1u : (aw & 0xffu) + ((aw >> 8) & 0xffu) + 1u;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, n, o);
            if (lane >= o) n += t;
        }
        if (lane == 31) NT[warp] = n;
        __syncthreads();
        for (int w = 0; w < warp; w++) n += NT[w];
        NQ[r] = n;   // (read after the barriers below)
    }
    if (warp == 0) vsmem[lane] = 0u;   // Q[-1]: read by rows whose arm reaches the line's start
    const bool out = r < len && ya + r >= ys && ya + r < ye;
    const uint4 *qh = reinterpret_cast<const uint4 *>(Q + (r + fwd) * kQS);
    const uint4 *ql = reinterpret_cast<const uint4 *>(Q + (r - back - 1) * kQS);
    uint32_t bv = 0xffffffffu, bd = 0;
    for (int g = 0; g < a.ng; g++) {
        // ---- A
        cp_async_wait_all();
        __syncwarp();
        uint32_t *q = Q + warp * kColSeg * kQS + lane;
        uint32_t v[kColSeg], tot = 0;
#pragma unroll
        for (int u = 0; u < kColSeg; u++) {
            v[u] = q[u * kQS];
            tot += v[u];
        }
        T[warp * 32 + lane] = tot;
        __syncthreads();
        uint32_t run = 0;
        for (int w = 0; w < warp; w++) run += T[w * 32 + lane];
#pragma unroll
        for (int u = 0; u < kColSeg; u++) {
            run += v[u];
            q[u * kQS] = run;
        }
        __syncthreads();
        // ---- C
        const int dbase = a.d0 + 32 * g, nlive = min(32, min(a.dc - 32 * g, a.D - dbase));
        if (out) {
            uint32_t bj = 0xffffffffu, bmin = bv;   // strict <: the smallest d on ties
            auto quad = [&](int j4, int live) {
                const uint4 h = qh[j4], l = ql[j4];
                const uint32_t c[4] = {h.x - l.x, h.y - l.y, h.z - l.z, h.w - l.w};
#pragma unroll
                for (int k = 0; k < 4; k++) {
                    const uint32_t s = k < live ? (kMax ? 0x7fffffffu - c[k] : c[k]) : 0xffffffffu;
                    bj = s < bmin ? (uint32_t)(4 * j4 + k) : bj;
                    bmin = min(bmin, s);
                }
                return make_uint4(c[0], c[1], c[2], c[3]);
            };
            if (vol) {
                const float n = float(NQ[r + fwd] - (r > back ? NQ[r - back - 1] : 0u));
                float *o = a.vol + (size_t)(dbase - a.dmin) * H * W + pix0 + (size_t)(ya + r) * pstep;
                for (int j4 = 0; 4 * j4 < nlive; j4++) {
                    const uint4 w = quad(j4, nlive - 4 * j4);
                    const uint32_t c[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                    for (int k = 0; k < 4; k++)
                        if (4 * j4 + k < nlive) o[(size_t)(4 * j4 + k) * H * W] = float(c[k]) / (n * a.S);
                }
            } else if (nlive == 32) {
#pragma unroll 2
                for (int j4 = 0; j4 < 8; j4++) quad(j4, 4);
            } else {
                for (int j4 = 0; 4 * j4 < nlive; j4++) quad(j4, nlive - 4 * j4);
            }
            if (bj != 0xffffffffu) {
                bv = bmin;
                bd = (uint32_t)dbase + bj;
            }
        }
        if (g + 1 < a.ng) {
            __syncthreads();   // Q and T are the next group's
            load(g + 1);
        }
    }
    if (!out) return;
    const size_t i = pix0 + (size_t)(ya + r) * pstep;
    unsigned long long *best = (view ? a.best[1] : a.best[0]) + i;
    unsigned long long key = ((unsigned long long)bv << 32) | bd;
    if (!a.first) key = min(key, *best);   // (of the earlier passes)
    *best = key;
    if (cost) {
        const uint32_t n = NQ[r + fwd] - (r > back ? NQ[r - back - 1] : 0u);
        cost[i] = float(uint32_t(key >> 32)) / (float(n) * a.S);
    }
}

// ------------------------------------------------------------------ k_lr
__device__ __forceinline__ void lr_body(const LrArgs &a, size_t i)
{
    if (i >= (size_t)a.W * a.H) return;
    const int x = int(i % a.W);
    const int d = a.dl[i];
    int16_t r = -1;
    if (a.tol < 0) r = (int16_t)d;
    else if (d >= 0 && x - d >= 0) {
        const int d2 = a.dr[i - d];
        if (d2 >= 0 && abs(d - d2) <= a.tol) r = (int16_t)d;
    }
    a.out[i] = r;
}

// -------------------------------------------------------------------- k_end
// The per-pixel end of a match: the winners' keys become the two views'
// disparities and minimum costs (where asked for) and the consistency map.
__device__ __forceinline__ int16_t checked(const EndArgs &a, size_t i, int x, int d)
{
    if (a.tol < 0) return (int16_t)d;
    if (x - d >= 0 && abs(d - (int)(a.best[1][i - d] & 0xffffu)) <= a.tol) return (int16_t)d;
    return -1;
}

__device__ __forceinline__ void end_body(const EndArgs &a, size_t i)
{
    if (i >= (size_t)a.W * a.H) return;
    const int d = (int)(a.best[0][i] & 0xffffu);
    if (a.disp[0]) a.disp[0][i] = (int16_t)d;
    if (a.disp[1]) a.disp[1][i] = (int16_t)(a.best[1][i] & 0xffffu);
    if (a.out) a.out[i] = checked(a, i, int(i % a.W), d);   // last: a caller may pass one buffer as disp_left and disp_out
}

// The same with costs, for one view: a cost is the key's sum over the region
// size N(p) of Eq. 2, the segment lengths along p's second arm.  Block = a 32 x
// 8 tile; the lengths of the tile and its reach along the walk are staged in
// shared memory, every load of a thread in flight at once (bound by latency:
// 333x211 8.1 us; with a walk along the arm in global memory per pixel 11.4,
// with the staging loads one after the other 10.7).
constexpr int kEX = 32, kEY = 8;
template <bool kRow>
__device__ __forceinline__ void end_costs_body(const EndArgs &a, int bx, int by, int view)
{
    constexpr int kPitch = kRow ? kEX + 2 * kMaxL1 : kEX;
    constexpr int kLoads = kRow ? (kEX + 2 * kMaxL1 + 31) / 32 : (kEY + 2 * kMaxL1 + kEY - 1) / kEY;
    __shared__ uint16_t len_s[kRow ? kEY * kPitch : (kEY + 2 * kMaxL1) * kPitch];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int W = a.W, H = a.H, L1 = a.L1, x = kEX * bx + lane, y = kEY * by + warp;
    const uchar4 *arms = view ? a.arms[1] : a.arms[0];
    uchar4 q[kLoads];
#pragma unroll
    for (int j = 0; j < kLoads; j++) {
        const int k = (kRow ? lane : warp) + (kRow ? 32 : kEY) * j;   // position in the walk's reach
        const int qx = kRow ? kEX * bx - L1 + k : x, qy = kRow ? y : kEY * by - L1 + k;
        q[j] = make_uchar4(0, 0, 0, 0);
        if (k < (kRow ? kEX : kEY) + 2 * L1 && qx >= 0 && qx < W && qy >= 0 && qy < H)
            q[j] = arms[(size_t)qy * W + qx];
    }
    const bool in = x < W && y < H;
    const size_t i = (size_t)min(y, H - 1) * W + min(x, W - 1);
    const unsigned long long key = view ? a.best[1][i] : a.best[0][i];
    const uchar4 p = arms[i];
#pragma unroll
    for (int j = 0; j < kLoads; j++) {
        const int k = (kRow ? lane : warp) + (kRow ? 32 : kEY) * j;
        if (k < (kRow ? kEX : kEY) + 2 * L1)
            len_s[kRow ? warp * kPitch + k : k * kPitch + lane] = kRow ? q[j].z + q[j].w + 1 : q[j].x + q[j].y + 1;
    }
    __syncthreads();
    if (!in) return;
    const int d = (int)(key & 0xffffu);
    if (int16_t *disp = view ? a.disp[1] : a.disp[0]) disp[i] = (int16_t)d;
    if (view == 0 && a.out) a.out[i] = checked(a, i, x, d);
    if (float *cost = view ? a.cost[1] : a.cost[0]) {
        const int first = kRow ? -(int)p.x : -(int)p.z, last = kRow ? p.y : p.w;
        const uint16_t *n = kRow ? len_s + warp * kPitch + L1 + lane : len_s + (L1 + warp) * kPitch + lane;
        uint32_t size = 0;
#pragma unroll 8
        for (int k = first; k <= last; k++) size += n[k * (kRow ? 1 : kPitch)];
        cost[i] = float(uint32_t(key >> 32)) / (float(size) * a.S);
    }
}

// ------------------------------------------------------ quarter size, depth
// Sect. 4: the pair is matched at half of each axis; channel c of output
// pixel (x, y) is the rounded mean (sum + 2) >> 2 of its 2x2 input block.
__global__ void __launch_bounds__(256) k_down(const DownArgs a)
{
    pdl_enter();
    const int Wh = a.W / 2, Hh = a.H / 2;
    const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
    if (x >= Wh || y >= Hh) return;
    const uint8_t *s0 = a.src[blockIdx.z] + ((size_t)(2 * y) * a.W + 2 * x) * 3;
    const uint8_t *s1 = s0 + (size_t)a.W * 3;
    uint8_t *d = a.dst[blockIdx.z] + ((size_t)y * Wh + x) * 3;
#pragma unroll
    for (int c = 0; c < 3; c++) d[c] = (uint8_t)((s0[c] + s0[3 + c] + s1[c] + s1[3 + c] + 2) >> 2);
}

// Sect. 4.4: the half-size disparity doubled back to full size, Z = f B / (2 d)
// on the 2x2 block of each half-size pixel; 0 (missing, Eq. 14) where d <= 0
// and on an odd last row or column.  Thread = one 2x2 block (hx, hy) of the
// ceil(W/2) x ceil(H/2) blocks.
__global__ void __launch_bounds__(256) k_depth(const DepthArgs a)
{
    pdl_enter();
    const int hx = blockIdx.x * blockDim.x + threadIdx.x, hy = blockIdx.y;
    if (2 * hx >= a.W) return;
    const int Wh = a.W / 2;
    float z = 0.0f;
    if (hx < Wh && hy < a.H / 2) {
        const int d = a.disp[(size_t)hy * Wh + hx];
        if (d > 0) z = a.fb / (2.0f * (float)d);
    }
    const int x = 2 * hx;
    for (int y = 2 * hy; y < min(a.H, 2 * hy + 2); y++) {
        float *o = a.out + (size_t)y * a.W + x;
        o[0] = z;
        if (x + 1 < a.W) o[1] = z;
    }
}

// ------------------------------------------------------------------ batches
// Every stage is one launch over all pairs of a batch (a single pair is a
// batch of one).  The pairs' arguments travel in the kernel parameters; the
// flat block index is mapped to (pair, block of that pair's own grid).
template <class A, int N>
struct Batch {
    int n;
    int off[N + 1];   // first flat block of each pair; off[n] = total
    int gx[N], gy[N]; // the pair's own grid is gx x gy x gz
    A p[N];
};

// launch with programmatic stream serialization (the kernel calls pdl_enter
// before any global memory access)
template <class... KArgs, class... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

template <class A, int N>
__device__ __forceinline__ int batch_pair(const Batch<A, N> &b, int flat, int &bx, int &by, int &bz)
{
    int lo = 0, hi = b.n - 1;
    while (lo < hi) {   // last pair with off <= flat
        const int mid = (lo + hi + 1) >> 1;
        if (b.off[mid] <= flat) lo = mid;
        else hi = mid - 1;
    }
    const int local = flat - b.off[lo];
    bx = local % b.gx[lo];
    const int t = local / b.gx[lo];
    by = t % b.gy[lo];
    bz = t / b.gy[lo];
    return lo;
}

template <int N, bool kMax>
__global__ void __launch_bounds__(256) k_smooth(const __grid_constant__ Batch<SmoothArgs, N> b)
{
    pdl_enter();
    int bx, by, bz;
    const int i = batch_pair(b, blockIdx.x, bx, by, bz);
    smooth_body<kMax>(b.p[i], bx * 256 + threadIdx.x, by);
}

// kRows 0: the flat mapping (images in device memory); else blocks of
// kRows rows per thread (images in host memory)
template <int N, int kRows = 0>
__global__ void __launch_bounds__(256) k_pack(const __grid_constant__ Batch<PackArgs, N> b)
{
    pdl_enter();
    int bx, by, bz;
    const int i = batch_pair(b, blockIdx.x, bx, by, bz);
    if (kRows == 0) pack_body(b.p[i], bx * 256 + threadIdx.x, by);
    else pack_rows_body<kRows ? kRows : 1>(b.p[i], bx * 256 + threadIdx.x, by);
}

template <int CW, int CH, int N>
__global__ void __launch_bounds__(kTX * kTY) k_prep(const __grid_constant__ Batch<PrepArgs, N> b)
{
    pdl_enter();
    int bx, by, bz;
    const int i = batch_pair(b, blockIdx.x, bx, by, bz);
    prep_body<CW, CH>(b.p[i], bx, by, bz);
}

template <int CW, int CH, int N>
__global__ void __launch_bounds__(kPrepThreads) k_prep_dirs(const __grid_constant__ Batch<PrepArgs, N> b)
{
    pdl_enter();
    int bx, by, bz;
    const int i = batch_pair(b, blockIdx.x, bx, by, bz);
    prep_dirs_body<CW, CH>(b.p[i], bx, by, bz);
}

template <int N, int kParts>
__global__ void __launch_bounds__(HSmem<kParts>::warps * 32, 4 / kParts) k_hagg(const __grid_constant__ Batch<HArgs, N> b)
{
    pdl_enter();
    hagg_tasks<kParts>(b.off[b.n], [&](int t, int &bx, int &by, int &bz) -> const HArgs & {
        return b.p[batch_pair(b, t, bx, by, bz)];
    });
}

template <int N, bool kMax, bool kRow>
__global__ void __launch_bounds__(kVThreads, kVResident) k_vagg(const __grid_constant__ Batch<VArgs, N> b)
{
    pdl_enter();
    int bx, by, bz;
    const int i = batch_pair(b, blockIdx.x, bx, by, bz);
    vagg_body<kMax, kRow>(b.p[i], bx);
}

template <int N, bool kMax, bool kRow>
__global__ void __launch_bounds__(kColMax, 2) k_vcol(const __grid_constant__ Batch<VArgs, N> b)
{
    pdl_enter();
    int bx, by, bz;
    const int i = batch_pair(b, blockIdx.x, bx, by, bz);
    vcol_body<kMax, kRow>(b.p[i], bx, by, bz);
}

template <int N>
__global__ void __launch_bounds__(1024) k_vcost(const __grid_constant__ Batch<HArgs, N> b)
{
    pdl_enter();
    int bx, by, bz;
    const int i = batch_pair(b, blockIdx.x, bx, by, bz);
    vcost_body(b.p[i], bx, by, bz);
}

// (32 registers: with 40 fewer blocks fit an SM, 1280x720, D = 128 266 against 238 us)
template <int N>
__global__ void __launch_bounds__(16 * 32, 4) k_hvote(const __grid_constant__ Batch<HVArgs, N> b)
{
    pdl_enter();
    int bx, by, bz;
    const int i = batch_pair(b, blockIdx.x, bx, by, bz);
    hvote_body(b.p[i], bx, by, bz);
}

template <int N>
__global__ void __launch_bounds__(256) k_lr(const __grid_constant__ Batch<LrArgs, N> b)
{
    pdl_enter();
    int bx, by, bz;
    const int i = batch_pair(b, blockIdx.x, bx, by, bz);
    lr_body(b.p[i], (size_t)bx * 256 + threadIdx.x);
}

template <int N>
__global__ void __launch_bounds__(256) k_end(const __grid_constant__ Batch<EndArgs, N> b)
{
    pdl_enter();
    int bx, by, bz;
    const int i = batch_pair(b, blockIdx.x, bx, by, bz);
    end_body(b.p[i], (size_t)bx * 256 + threadIdx.x);
}

template <int N, bool kRow>
__global__ void __launch_bounds__(kEX * kEY) k_end_costs(const __grid_constant__ Batch<EndArgs, N> b)
{
    pdl_enter();
    int bx, by, bz;
    const int i = batch_pair(b, blockIdx.x, bx, by, bz);
    end_costs_body<kRow>(b.p[i], bx, by, bz);
}

template <int N>
__global__ void __launch_bounds__(256) k_vote_end(const __grid_constant__ Batch<VoteEndArgs, N> b)
{
    pdl_enter();
    int bx, by, bz;
    const int i = batch_pair(b, blockIdx.x, bx, by, bz);
    const VoteEndArgs &a = b.p[i];
    const int k = bx * 256 + threadIdx.x;
    if (k >= a.npx) return;
    const int v = a.mask[k];
    a.out[k] = v >= a.dmin && v < a.D ? (int16_t)(a.best[k] & 0xffffu) : (int16_t)-1;
}

__global__ void k_extract_census(const uint2 *__restrict__ cen, int W, int H, int pw, unsigned long long *out)
{
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (size_t)W * H) return;
    const uint2 r = cen[(i / W) * pw + i % W];
    out[i] = ((unsigned long long)r.y << 32) | r.x;
}

} // namespace dco

// ====================================================================== host
using namespace dco;

namespace {

struct ProfEvent {
    const char *name;
    cudaEvent_t a, b;
};

struct ProfAgg {
    std::string name;
    int launches = 0;
    double ms = 0.0;
};

struct Derived {
    int L1;
    uint32_t Sint;
    float S;
    int order;   // aggregation order: 0 horizontal then vertical, 1 vertical then horizontal
    int dmin;    // smallest disparity of the search
    int hchunk, vchunk;   // tile shapes of the two 1-D passes (0: automatic)
};

struct Layout {
    size_t rgbx[2], grey[2], cen[2], col[2], arms[2], atmp[2], best[2], sh[2], total;
    int dc, dstride, npass, pw;
};

constexpr size_t kAlign = 256;
constexpr size_t kSmShared = 228 << 10, kBlockShared = 1 << 10;   // shared memory of an SM; kept back per block
size_t align_up(size_t v) { return (v + kAlign - 1) / kAlign * kAlign; }

bool derive(const dco_params &p, Derived &d)
{
    d.L1 = p.arm_l1;
    // fixed-point scale: the largest region, (2*L1+1)^2 costs of at most 1
    // (+1 unit of rounding each), must stay below 2^32
    const double n = double(2 * p.arm_l1 + 1) * double(2 * p.arm_l1 + 1);
    double s = std::floor(4294967295.0 / n) - 1.0;
    s = std::min(s, 1048576.0);
    d.Sint = (uint32_t)s;
    d.S = (float)s;
    d.order = p.agg_order;
    d.dmin = p.d_min;
    d.hchunk = p.h_chunk;
    d.vchunk = p.v_chunk;
    return true;
}

// a tile shape: 0 (automatic) or 32 .. 16384 positions
bool tile_valid(int c) { return c == 0 || (c >= 32 && c <= 16384); }

bool params_valid(const dco_params &p)
{
    if (!(p.lambda_ad > 0.f) || !(p.lambda_census > 0.f) || !(p.eps > 0.f) || !(p.gamma_l >= 0.f))
        return false;
    if (p.census_w < 1 || p.census_h < 1 || !(p.census_w & 1) || !(p.census_h & 1)) return false;
    if (p.census_w > kMaxCW || p.census_h > kMaxCH || p.census_w * p.census_h - 1 > 64) return false;
    if (p.arm_l1 < 1 || p.arm_l1 > kMaxL1 || p.arm_l2 < 0 || p.tau1 < 0 || p.tau2 < 0) return false;
    if (p.d_chunk < 0) return false;
    if (p.vote_iters < 0 || p.vote_iters > 64) return false;
    if (p.smooth_arms != 0 && p.smooth_arms != 1) return false;
    if (p.agg_order != 0 && p.agg_order != 1) return false;
    if (p.d_min < 0 || p.d_min > 255) return false;
    if (!tile_valid(p.h_chunk) || !tile_valid(p.v_chunk)) return false;
    return true;
}

bool dims_valid(int W, int H, int D, int dmin = 0)
{
    return W >= 1 && H >= 1 && W <= 16384 && H <= 16384 && D >= 1 && dmin >= 0 && dmin + D <= 256 && dmin + D <= W;
}

// Automatic pass width: both views' slices of a pass within `cap` bytes, at
// least one group of 32 disparities.  Wide passes are fewer, larger launches of
// the two aggregation kernels and whole 128-byte lines per pixel and group:
// first and second pass together at 640x480, D = 64 in one pass 117 us, in two
// 128; 1280x720, D = 128 in two passes 663 us, in four 722.  The narrow cap
// (about the L2) is what the serving lanes admit frames by, and the fallback
// where the device cannot allocate the wide one.
constexpr size_t kSlicesWide = 512u << 20, kSlicesNarrow = 96u << 20;
// all pairs of a call together: from 65 pairs on (more than one launch), the wide cap
// of each is its part of this (at least the narrow one), so that a batch's
// workspace stays bounded by what narrow passes or 32 GiB of slices take
constexpr size_t kSlicesCall = size_t(32) << 30;
size_t wide_cap(size_t pairs) { return std::max(kSlicesNarrow, std::min(kSlicesWide, kSlicesCall / std::max<size_t>(1, pairs))); }
int auto_width(int W, int H, int D, size_t cap)
{
    const size_t per = 8 * (size_t)W * H;   // slice bytes per disparity
    if (per * ((size_t)(D + 31) / 32 * 32) <= cap) return D;
    return (int)std::min<size_t>(D, std::max<size_t>(32, cap / per / 32 * 32));
}

Layout make_layout(int W, int H, int D, const dco_params &p, int dc_override = 0, size_t cap = kSlicesWide)
{
    Layout L{};
    const size_t npx = (size_t)W * H;
    int dc = dc_override > 0 ? dc_override : p.d_chunk;
    if (dc <= 0) dc = auto_width(W, H, D, cap);
    dc = std::min(dc, D);
    L.dc = dc;
    L.dstride = (dc + 31) / 32 * 32;
    L.npass = (D + dc - 1) / dc;
    size_t off = 0;
    L.pw = (W + 3) / 4 * 4;
    for (int v = 0; v < 2; v++) { L.rgbx[v] = off; off = align_up(off + 4 * npx); }
    for (int v = 0; v < 2; v++) { L.grey[v] = off; off = align_up(off + npx); }
    for (int v = 0; v < 2; v++) { L.cen[v] = off; off = align_up(off + 8 * (size_t)H * L.pw); }
    for (int v = 0; v < 2; v++) { L.col[v] = off; off = align_up(off + 4 * (size_t)H * L.pw); }
    // arms: 16 bytes of slack, read by the cost pass's bulk copies past the last pixel
    for (int v = 0; v < 2; v++) { L.arms[v] = off; off = align_up(off + 4 * npx + 16); }
    for (int v = 0; v < 2; v++) { L.atmp[v] = off; off = align_up(off + (p.smooth_arms ? 4 * npx : 0)); }
    for (int v = 0; v < 2; v++) { L.best[v] = off; off = align_up(off + 8 * npx); }
    for (int v = 0; v < 2; v++) { L.sh[v] = off; off = align_up(off + 4 * npx * (size_t)L.dstride); }
    L.total = off;
    return L;
}

// geometry of a pass over lines: output positions per block, warps, grid
struct HGeom {
    int chunk, nw;
    size_t smem;
    dim3 grid;
};

// Output positions per block of a first-pass line of n positions: the whole
// line up to kHMaxLen, else 512 (want = 0); otherwise `want`, capped so that
// a block's prefix range (chunk + 2 L1 halo) stays within kHMaxLen.
int first_pass_chunk(int n, int L1, int want)
{
    if (want <= 0) return n <= kHMaxLen ? n : 512;
    int c = std::min(want, n);
    if (c < n || n > kHMaxLen) c = std::min(c, kHMaxLen - 2 * L1);
    return c;
}

// the other aggregation order: k_vcost takes columns, one chunk of rows per
// block while it fits 32 warps of 32 rows (k_vagg<.., kRow> then walks rows)
HGeom vcost_geom(int W, int H, int dc, int L1, int want)
{
    HGeom g{};
    g.chunk = first_pass_chunk(H, L1, want);
    const int len = std::min(H, g.chunk + 2 * L1);
    g.nw = (len + kHSegCost - 1) / kHSegCost;
    g.smem = CSmem(len, g.chunk, g.nw).total;
    g.grid = dim3(W, (H + g.chunk - 1) / g.chunk, 2 * ((dc + 31) / 32));
    return g;
}

// the vote's horizontal pass: one block per (row, chunk of output columns, group)
HGeom hvote_geom(int W, int H, int dc, int L1, int want)
{
    HGeom g{};
    g.chunk = first_pass_chunk(W, L1, want);
    const int len = std::min(W, g.chunk + 2 * L1);
    g.nw = (len + kHSeg - 1) / kHSeg;
    g.smem = HVSmem(len, g.chunk, g.nw).total;
    g.grid = dim3((W + g.chunk - 1) / g.chunk, H, (dc + 31) / 32);
    return g;
}

// k_hagg: one task per (row, view, 32 disparities, range of output columns): whole
// rows up to what a block of sixteen warps holds, else ranges that fill it with
// their L1 reach on both sides (the first has a reach on one side only)
struct HaggGeom {
    int first, chunk;
    int parts;   // warps per quad: two where a task has more than 320 reference columns
    dim3 grid;   // of tasks: rows, ranges, views and groups
};

HaggGeom hagg_geom(int W, int H, int dc, int L1, int want)
{
    constexpr int most = HSmem<2>::cols;
    HaggGeom g{};
    if (W <= most && (want <= 0 || want >= W)) {
        g.first = g.chunk = W;
    } else {
        g.chunk = most - 2 * L1;
        g.first = most - L1;
        if (want > 0) {   // (ranges of equal length)
            const int ranges = (W + std::min(want, g.chunk) - 1) / std::min(want, g.chunk);
            g.first = g.chunk = (W + ranges - 1) / ranges;
        }
    }
    const int ranges = g.first >= W ? 1 : 1 + (W - g.first + g.chunk - 1) / g.chunk;
    g.parts = (ranges == 1 ? W : std::min(W, std::max(g.first + L1, g.chunk + 2 * L1))) <= HSmem<1>::cols ? 1 : 2;
    g.grid = dim3(H, ranges, 2 * ((dc + kHD - 1) / kHD));
    return g;
}

// V geometry: the walk is dealt out to as many blocks as the SMs hold at once:
// whole strips (kVCols columns of one group and view) round by round,
// neighbouring blocks on neighbouring strips; the strips that are left are
// cut into bands, or, where there are too many for two bands each, into equal
// shares that run on from strip to strip.  A run costs its fill of up to 2 L1
// rows again, so strips of at most kVRunOn rows are not shared (160x120,
// D = 16: 8.4 us in bands, 11.5 us in shares that run on).
struct VGeom {
    int strips;   // per layer (group and view)
    int rounds, rest, share, bands, nblk;   // bands: per strip that is left (0: shares run on)
};
constexpr int kVRunOn = 256;

size_t vagg_units(int F, int layers) { return (size_t)((F + kVCols - 1) / kVCols) * layers; }

// `blocks`: this pair's part of the resident blocks; want > 0: rows per band
VGeom vagg_geom(int E, int F, int layers, int want, int blocks)
{
    VGeom g{};
    g.strips = (F + kVCols - 1) / kVCols;
    const int units = g.strips * layers;
    if (want > 0) {
        g.bands = (E + want - 1) / want;
        g.rest = units;
    } else {
        g.rounds = units / blocks;
        g.rest = units - g.rounds * blocks;
        const int nb = g.rest > 0 ? blocks / g.rest : 1;
        if (nb > 1) g.bands = std::min(nb, (E + kVStep - 1) / kVStep);
        else if (E <= kVRunOn) g.bands = 1;
    }
    const long long rows = g.bands ? E : (long long)g.rest * E;
    const int parts = g.bands ? g.bands : blocks;
    g.share = (int)((rows + parts - 1) / parts);
    if (want <= 0) g.share = std::max(1, (g.share + kVStep - 1) / kVStep) * kVStep;   // whole steps
    if (g.bands) g.bands = (E + g.share - 1) / g.share;
    const int tail = g.bands ? g.rest * g.bands : (int)((rows + g.share - 1) / g.share);
    g.nblk = g.rounds > 0 ? blocks : tail;
    return g;
}

} // namespace

struct dco_stereo {
    int device = 0;
    int nsm = 152;                           // multiprocessors of the device
    bool yield = false;                      // launches of blocks that end after one unit of work (serving, see srv_launch)
    size_t budget = 0;
    char *ws = nullptr;
    size_t ws_cap = 0;
    size_t ws_refused = SIZE_MAX;            // smallest workspace of wide passes that the device could not allocate
    int *d_status = nullptr;
    float *d_tables = nullptr;
    float *h_tables = nullptr;   // pinned staging of the tables
    bool tab_valid = false;
    float tab_key[4] = {0, 0, 0, 0};
    int tab_l1 = -1;
    uint8_t *stage = nullptr;
    size_t stage_cap = 0;
    bool profiling = false;
    int test_flags = 0;                      // DCO_TEST_* failure tests (0 in normal use)
    int groups_last = 1;                     // admission groups of the last batch call
    unsigned long long launches = 0;
    std::vector<ProfEvent> pending;
    std::vector<cudaEvent_t> pool;
    std::vector<ProfAgg> agg;
    std::string last_error;
    int *dn_pin = nullptr;                   // pinned convergence flag of the densify solve
    cudaEvent_t dn_ev[2] = {nullptr, nullptr};
    cudaStream_t dn_stream = nullptr;        // private stream the iteration batch is captured on
    cudaGraphExec_t dn_exec = nullptr;       // one captured batch of iterations
    std::vector<unsigned char> dn_key;       // the arguments it was captured with
    int dn_iters = 0;
    double dn_relres = 0.0;
};

namespace {

// A failed runtime call also leaves its error as the thread's last error;
// it is reported here and then dropped, so that the launch checks of the
// next call (cudaGetLastError after a launch) see only their own launches.
dco_status cuda_fail(dco_stereo *h, cudaError_t e, const char *what)
{
    if (h) h->last_error = std::string(what) + ": " + cudaGetErrorString(e);
    (void)cudaGetLastError();
    return e == cudaErrorMemoryAllocation ? DCO_ENOMEM : DCO_ECUDA;
}

// Entry of a call that launches work: h's device made current, and a
// non-sticky error that an earlier runtime call left in this thread dropped
// (it belongs to that call, not to this one's launches).
cudaError_t enter_device(const dco_stereo *h)
{
    const cudaError_t e = cudaSetDevice(h->device);
    (void)cudaGetLastError();
    return e;
}

// status word -> call status: a lost tile copy is a timed-out wait, any
// other bit a failed internal check
dco_status status_of_word(int v)
{
    if (v == 0) return DCO_OK;
    return (v & kStatusCopyTimeout) ? DCO_ETIMEOUT : DCO_EDEVICE;
}

#define DCO_CUDA(h, call)                                              \
    do {                                                               \
        cudaError_t e_ = (call);                                       \
        if (e_ != cudaSuccess) return cuda_fail((h), e_, #call);       \
    } while (0)

cudaEvent_t take_event(dco_stereo *h)
{
    if (!h->pool.empty()) {
        cudaEvent_t e = h->pool.back();
        h->pool.pop_back();
        return e;
    }
    cudaEvent_t e = nullptr;
    cudaEventCreate(&e);
    return e;
}

void collect_profile(dco_stereo *h)
{
    for (auto &pe : h->pending) {
        float ms = 0.f;
        if (cudaEventElapsedTime(&ms, pe.a, pe.b) == cudaSuccess) {
            ProfAgg *slot = nullptr;
            for (auto &g : h->agg)
                if (g.name == pe.name) slot = &g;
            if (!slot) {
                h->agg.push_back(ProfAgg{pe.name, 0, 0.0});
                slot = &h->agg.back();
            }
            slot->launches += 1;
            slot->ms += ms;
        }
        h->pool.push_back(pe.a);
        h->pool.push_back(pe.b);
    }
    h->pending.clear();
}

struct ProfScope {
    dco_stereo *h;
    cudaStream_t s;
    ProfEvent ev{};
    // name == nullptr: a launch being captured into a graph (counted when the
    // graph runs, never timed)
    ProfScope(dco_stereo *h_, cudaStream_t s_, const char *name) : h(name ? h_ : nullptr), s(s_)
    {
        if (!h) return;
        h->launches++;
        if (h->profiling) {
            ev.name = name;
            ev.a = take_event(h);
            ev.b = take_event(h);
            cudaEventRecord(ev.a, s);
        }
    }
    ~ProfScope()
    {
        if (h && h->profiling) {
            cudaEventRecord(ev.b, s);
            h->pending.push_back(ev);
        }
    }
};

// keep: a workspace that the device cannot enlarge stays as it is
dco_status ensure_ws(dco_stereo *h, size_t need, bool keep = false)
{
    if (need <= h->ws_cap) return DCO_OK;
    if (h->budget && need > h->budget) {
        h->last_error = "workspace of " + std::to_string(need) + " bytes exceeds the budget of " +
                        std::to_string(h->budget);
        return DCO_EBUDGET;
    }
    char *old = h->ws;
    if (old && !keep) {
        DCO_CUDA(h, cudaDeviceSynchronize());
        cudaFree(old);
        h->ws = old = nullptr;
        h->ws_cap = 0;
    }
    char *ws = nullptr;
    DCO_CUDA(h, cudaMalloc((void **)&ws, need));
    if (old) {
        const cudaError_t e = cudaDeviceSynchronize();
        if (e != cudaSuccess) {
            cudaFree(ws);
            return cuda_fail(h, e, "cudaDeviceSynchronize()");
        }
        cudaFree(old);
    }
    h->ws = ws;
    h->ws_cap = need;
    return DCO_OK;
}

// Eq. 1 tables, evaluated in double on the host and rounded once to float:
//   [0, kTabAD)   1 - exp(-(k/3) / lambda_AD), k = 0..765 (the channel sum);
//   [kTabAD, +kTabCen)   1 - exp(-h / lambda_census), h = 0..64;
//   [kTabAD + kTabCen, +kTabAlpha)   alpha(Lmin) * S.
void fill_tables(float *t, const dco_params &p, const Derived &dv)
{
    for (int k = 0; k < kTabAD; k++)
        t[k] = k <= 765 ? (float)(1.0 - std::exp(-(k / 3.0) / (double)p.lambda_ad)) : 1.0f;
    for (int k = 0; k < kTabCen; k++)
        t[kTabAD + k] = k <= 64 ? (float)(1.0 - std::exp(-(double)k / (double)p.lambda_census)) : 1.0f;
    for (int l = 0; l < kTabAlpha; l++) {
        const double alpha = 1.0 - std::exp(-(double)p.gamma_l / ((double)l + (double)p.eps));
        t[kTabAD + kTabCen + l] = (float)(alpha * (double)dv.Sint);
    }
}

dco_status ensure_tables(dco_stereo *h, const dco_params &p, const Derived &dv, cudaStream_t s)
{
    const float key[4] = {p.lambda_ad, p.lambda_census, p.gamma_l, p.eps};
    if (h->tab_valid && !std::memcmp(key, h->tab_key, sizeof key) && h->tab_l1 == p.arm_l1) return DCO_OK;
    float *t = h->h_tables;
    fill_tables(t, p, dv);
    DCO_CUDA(h, cudaMemcpyAsync(h->d_tables, t, sizeof(float) * kTabFloats, cudaMemcpyHostToDevice, s));
    // the pinned staging buffer is reused by the next upload: wait for this one
    DCO_CUDA(h, cudaStreamSynchronize(s));
    std::memcpy(h->tab_key, key, sizeof key);
    h->tab_l1 = p.arm_l1;
    h->tab_valid = true;
    return DCO_OK;
}

template <class T>
T *ws_ptr(dco_stereo *h, size_t off) { return reinterpret_cast<T *>(h->ws + off); }

// ----------------------------------------------------------- batched launches
constexpr int kBatchMax = 64;   // pairs per launch (kernel parameter space)
static_assert(sizeof(Batch<VArgs, kBatchMax>) <= 32764, "kernel parameters of a full V batch");
static_assert(sizeof(Batch<HArgs, kBatchMax>) <= 32764, "kernel parameters of a full H batch");

// The dynamic shared-memory limit is an attribute of the kernel on a device,
// shared by every handle and thread of the process: it is raised under a lock
// and never lowered, so a warmed-up process makes no attribute calls (safe
// inside stream capture) and no handle can shrink another's limit.
std::mutex g_smem_mu;
std::map<std::pair<int, const void *>, size_t> g_smem_set;

dco_status opt_in_smem(dco_stereo *h, const void *kernel, size_t smem)
{
    std::lock_guard<std::mutex> lock(g_smem_mu);
    size_t &done = g_smem_set[{h->device, kernel}];
    if (smem <= done) return DCO_OK;
    DCO_CUDA(h, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    done = smem;
    return DCO_OK;
}

template <class A>
struct Item {
    A a;
    int gx, gy, gz;   // the pair's own grid
};

template <class A, int N, class K>
dco_status launch_group(dco_stereo *h, cudaStream_t s, const char *name, K kernel, const Item<A> *it, int n,
                        int block, size_t smem, int most = INT_MAX)
{
    Batch<A, N> b;
    std::memset(&b, 0, sizeof b);
    b.n = n;
    b.off[0] = 0;
    for (int i = 0; i < n; i++) {
        b.gx[i] = it[i].gx;
        b.gy[i] = it[i].gy;
        b.p[i] = it[i].a;
        b.off[i + 1] = b.off[i] + it[i].gx * it[i].gy * it[i].gz;
    }
    if (b.off[n] == 0) return DCO_OK;
    if (smem > (48u << 10)) {
        dco_status st = opt_in_smem(h, reinterpret_cast<const void *>(kernel), smem);
        if (st != DCO_OK) return st;
    }
    ProfScope ps(h, s, name);
    cudaError_t e = launch_pdl(kernel, dim3((unsigned)std::min(b.off[n], most)), dim3((unsigned)block), smem, s, b);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) {
        h->last_error = std::string(name) + " launch (" + std::to_string(n) + " pairs, " + std::to_string(b.off[n]) +
                        " blocks of " + std::to_string(block) + " threads, " + std::to_string(smem) +
                        " B shared): " + cudaGetErrorString(e);
        return e == cudaErrorMemoryAllocation ? DCO_ENOMEM : DCO_ECUDA;
    }
    return DCO_OK;
}

// most: blocks of a launch whose kernel takes its blocks' tasks in turn
// one launch for a single pair (small parameter block), else groups of
// kBatchMax (kn is the kernel instance for that many)
template <class A, class K1, class KN>
dco_status launch_items(dco_stereo *h, cudaStream_t s, const char *name, K1 k1, KN kn,
                        const std::vector<Item<A>> &items, int block, size_t smem, int most = INT_MAX)
{
    constexpr int nmax = kBatchMax;
    if (items.empty()) return DCO_OK;
    if (items.size() == 1) return launch_group<A, 1>(h, s, name, k1, items.data(), 1, block, smem, most);
    for (size_t i = 0; i < items.size(); i += nmax) {
        const int n = (int)std::min<size_t>(nmax, items.size() - i);
        dco_status st = launch_group<A, nmax>(h, s, name, kn, items.data() + i, n, block, smem, most);
        if (st != DCO_OK) return st;
    }
    return DCO_OK;
}

// one pair of a run
struct Job {
    const uint8_t *left = nullptr, *right = nullptr;
    int W = 0, H = 0, D = 0;
    int16_t *out = nullptr, *disp_l = nullptr, *disp_r = nullptr;
    float *cost_l = nullptr, *cost_r = nullptr, *vol = nullptr;
    int vol_view = 0;
    uchar4 *arms0 = nullptr;   // stage entry point: arms of image 0 go here
    int dchunk = 0;                  // this pair's pass width (0: the call's parameters)
    int hchunk = 0, vchunk = 0;      // this pair's tile shapes (0: the call's parameters)
    int host_in = -1;                // images in host memory: 1, in device memory: 0, -1: ask the driver
    const unsigned long long *vkeys = nullptr;   // Eq. 4 round: the previous round's keys (null: first round)
    unsigned long long *vbest = nullptr;         //   and the keys it minimises into
    bool costs_done = false;   // the second pass wrote the costs
    Layout L{};
    size_t base = 0;           // workspace offset of this pair
};

// workspace plan for all jobs; the pass width shrinks (same for all pairs)
// until the plan fits the handle's budget
size_t plan_jobs(const dco_stereo *h, const dco_params &p, std::vector<Job> &jobs, size_t cap)
{
    // a pair's own pass width (j.dchunk > 0) replaces the call's; a budget
    // override caps both
    auto plan = [&](int dc_override) {
        size_t t = 0;
        for (auto &j : jobs) {
            int dc = j.dchunk > 0 ? j.dchunk : 0;
            if (dc_override > 0) dc = dc > 0 ? std::min(dc, dc_override) : dc_override;
            j.L = make_layout(j.W, j.H, j.D, p, dc, cap);
            j.base = t;
            t = align_up(t + j.L.total);
        }
        return t;
    };
    size_t total = plan(0);
    if (h->budget && total > h->budget) {
        int widest = 32;
        for (auto &j : jobs) widest = std::max(widest, (j.L.dc + 31) / 32 * 32);
        for (int dc = widest; dc >= 32 && total > h->budget; dc -= 32) total = plan(dc);
    }
    return total;
}

// Jobs that run together, and the workspace that the largest group needs.  On
// a handle with a budget, jobs whose workspaces do not fit it together (even
// at the narrowest pass width) are admitted in consecutive groups that do.
struct Plan {
    std::vector<std::vector<Job>> groups;
    size_t need = 0;
};

dco_status make_plan(dco_stereo *h, const dco_params &p, const std::vector<Job> &jobs, size_t cap, size_t front, Plan &plan)
{
    plan.groups.assign(1, jobs);
    plan.need = plan_jobs(h, p, plan.groups[0], cap);
    if (h->budget && plan.need > h->budget && jobs.size() > 1) {
        plan.groups.clear();
        plan.need = 0;
        for (size_t i = 0; i < jobs.size();) {
            std::vector<Job> g{jobs[i]};
            size_t t = plan_jobs(h, p, g, cap);
            if (t > h->budget) {
                h->last_error = "pair " + std::to_string(i) + " needs " + std::to_string(t) +
                                " bytes of workspace, more than the budget of " + std::to_string(h->budget);
                return DCO_EBUDGET;
            }
            size_t j = i + 1;
            for (; j < jobs.size(); j++) {
                std::vector<Job> g2 = g;
                g2.push_back(jobs[j]);
                const size_t t2 = plan_jobs(h, p, g2, cap);
                if (t2 > h->budget) break;
                g.swap(g2);
                t = t2;
            }
            plan.need = std::max(plan.need, t);
            plan.groups.push_back(std::move(g));
            i = j;
        }
    }
    plan.need += front;
    for (auto &g : plan.groups)
        for (auto &j : g) j.base += front;
    return DCO_OK;
}

// Plan of a call and its workspace, behind `front` bytes of the call's own.
// Wide passes are a choice: where the device or the budget cannot hold them,
// the call runs with narrow ones.  A size that the device refused is not asked
// for again while the workspace holds the narrow plan, so a call that has run
// once allocates nothing the next time; a call that needs more than there is in any
// case, and dco_stereo_reserve, try the wide plan afresh.
dco_status plan_ws(dco_stereo *h, const dco_params &p, const std::vector<Job> &jobs, Plan &plan, size_t front = 0)
{
    dco_status st = make_plan(h, p, jobs, wide_cap(jobs.size()), front, plan);
    if (st == DCO_OK && plan.need <= h->ws_cap) return DCO_OK;
    Plan narrow;
    const dco_status nst = make_plan(h, p, jobs, kSlicesNarrow, front, narrow);
    const bool choice = nst == DCO_OK && narrow.need < plan.need, fits = choice && narrow.need <= h->ws_cap;
    if (st == DCO_OK) {
        if (choice && (h->test_flags & DCO_TEST_REFUSE_WIDE)) st = DCO_ENOMEM;
        else if (fits && plan.need >= h->ws_refused) st = DCO_ENOMEM;
        else st = ensure_ws(h, plan.need, fits);
        if (st == DCO_ENOMEM && choice) h->ws_refused = std::min(h->ws_refused, plan.need);
    }
    if (!choice || (st != DCO_ENOMEM && st != DCO_EBUDGET)) return st;
    plan = std::move(narrow);
    return ensure_ws(h, plan.need);
}

template <class T>
T *jptr(dco_stereo *h, const Job &j, size_t off) { return ws_ptr<T>(h, j.base + off); }

// images the kernels read from host memory (pinned or registered; over
// NVLink-C2C on Grace systems)
constexpr int kPackHostRows = 4;   // rows per k_pack thread for those
bool in_host_memory(const void *p)
{
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    return at.type == cudaMemoryTypeHost;
}

// grey/colour packing and census + arms for nimg images (1 or 2) of every job;
// arms of image 0 go to arms0 where it is set (the arms entry point)
dco_status launch_prep(dco_stereo *h, const dco_params &p, const Derived &dv, const std::vector<Job> &jobs,
                       int nimg, cudaStream_t s)
{
    std::vector<Item<PackArgs>> pk, pk_host;
    std::vector<Item<PrepArgs>> pr;
    for (const Job &j : jobs) {
        const int npx = j.W * j.H;
        Item<PackArgs> a{};
        a.a.rgb[0] = j.left; a.a.rgb[1] = j.right;
        for (int v = 0; v < 2; v++) {
            a.a.rgbx[v] = jptr<uint32_t>(h, j, j.L.rgbx[v]);
            a.a.grey[v] = jptr<uint8_t>(h, j, j.L.grey[v]);
        }
        a.a.npx = npx;
        a.a.W = j.W;
        a.a.k1 = 0x00100401u * (uint32_t)(std::min(p.tau1, 256) + 511);   // tau1 in every 10-bit field
        a.gy = nimg;
        a.gz = 1;
        if (j.host_in > 0 || (j.host_in < 0 && (in_host_memory(j.left) || in_host_memory(j.right)))) {
            a.gx = (((j.W + 3) / 4) * ((j.H + kPackHostRows - 1) / kPackHostRows) + 255) / 256;
            pk_host.push_back(a);
        } else {
            a.gx = (npx + 1023) / 1024;   // 256 threads x 4 pixels
            pk.push_back(a);
        }
        Item<PrepArgs> b{};
        for (int v = 0; v < 2; v++) {
            b.a.rgbx[v] = jptr<uint32_t>(h, j, j.L.rgbx[v]);
            b.a.grey[v] = jptr<uint8_t>(h, j, j.L.grey[v]);
            b.a.cen[v] = jptr<uint2>(h, j, j.L.cen[v]);
            b.a.col[v] = jptr<uint32_t>(h, j, j.L.col[v]);
            b.a.arms[v] = jptr<uchar4>(h, j, j.L.arms[v]);
        }
        b.a.pw = j.L.pw;
        if (j.arms0) b.a.arms[0] = j.arms0;
        b.a.W = j.W; b.a.H = j.H;
        b.a.cw = p.census_w; b.a.ch = p.census_h;
        b.a.L1 = dv.L1; b.a.L2 = p.arm_l2; b.a.tau1 = p.tau1; b.a.tau2 = p.tau2;
        b.gx = (j.W + kTX - 1) / kTX;
        b.gy = (j.H + kTY - 1) / kTY;
        b.gz = nimg;
        pr.push_back(b);
    }
    dco_status st = launch_items(h, s, "k_pack", k_pack<1>, k_pack<kBatchMax>, pk, 256, 0);
    if (st != DCO_OK) return st;
    st = launch_items(h, s, "k_pack", k_pack<1, kPackHostRows>, k_pack<kBatchMax, kPackHostRows>, pk_host, 256, 0);
    if (st != DCO_OK) return st;
    int blocks = 0;
    for (const auto &b : pr) blocks += b.gx * b.gy * b.gz;
    const bool dirs = blocks <= 2 * h->nsm;   // a thread per arm instead of one per pixel
    if (dirs)
        for (auto &b : pr) b.gy = (b.a.H + kTYd - 1) / kTYd;
    const bool std_census = p.census_w == 9 && p.census_h == 7;
    if (dirs && std_census)
        st = launch_items(h, s, "k_prep", k_prep_dirs<9, 7, 1>, k_prep_dirs<9, 7, kBatchMax>, pr, kPrepThreads, 0);
    else if (dirs)
        st = launch_items(h, s, "k_prep", k_prep_dirs<0, 0, 1>, k_prep_dirs<0, 0, kBatchMax>, pr, kPrepThreads, 0);
    else if (std_census)
        st = launch_items(h, s, "k_prep", k_prep<9, 7, 1>, k_prep<9, 7, kBatchMax>, pr, kTX * kTY, 0);
    else
        st = launch_items(h, s, "k_prep", k_prep<0, 0, 1>, k_prep<0, 0, kBatchMax>, pr, kTX * kTY, 0);
    if (st != DCO_OK || !p.smooth_arms) return st;
    // Sect. 4.1 smoothing: arms -> 3x3 minimum (atmp) -> 3x3 maximum (arms, records)
    std::vector<Item<SmoothArgs>> er, di;
    for (size_t k = 0; k < jobs.size(); k++) {
        const Job &j = jobs[k];
        Item<SmoothArgs> e{};
        for (int v = 0; v < 2; v++) {
            e.a.src[v] = pr[k].a.arms[v];
            e.a.dst[v] = jptr<uchar4>(h, j, j.L.atmp[v]);
        }
        e.a.W = j.W; e.a.H = j.H; e.a.pw = j.L.pw;
        e.gx = (j.W * ((j.H + kSmRows - 1) / kSmRows) + 255) / 256; e.gy = nimg; e.gz = 1;
        er.push_back(e);
        Item<SmoothArgs> d = e;
        for (int v = 0; v < 2; v++) {
            d.a.src[v] = e.a.dst[v];
            d.a.dst[v] = pr[k].a.arms[v];
            d.a.col[v] = pr[k].a.col[v];
        }
        di.push_back(d);
    }
    if ((st = launch_items(h, s, "k_smooth", k_smooth<1, false>, k_smooth<kBatchMax, false>, er, 256, 0)) != DCO_OK)
        return st;
    return launch_items(h, s, "k_smooth", k_smooth<1, true>, k_smooth<kBatchMax, true>, di, 256, 0);
}

// blocks of k_vagg that are resident at once: by the ring in shared memory, and
// by the registers (the deal for arm_l1 <= 19 counted five to eight blocks per SM by the
// ring alone: 640x480, D = 64, arm_l1 = 17 51.4 us, with four 43.2)
int vagg_slots(const dco_stereo *h, int L1)
{
    return h->nsm * std::max(1, std::min(kVResident, (int)(kSmShared / (vagg_smem_bytes(L1) + kBlockShared))));
}

// The pairs of a call whose second pass runs by whole lines (k_vcol), the others by
// strips (k_vagg).  Lines have to fit a block, and a v_chunk asks for strips.  A
// strip's fill of arm_l1 rows and its last part step weigh on short lines, and its long
// walk leaves the chip idle in small launches; with many lines per SM, k_vcol's one
// line per block and barrier is the slower form.  Strips against lines, us, arm_l1 = 34,
// by warps per SM (a warp per 32 positions of a line and group; k_vcol holds 32 at once):
//   320x240, D = 64    69   18.6, 16.3      1920x100, D = 64    202   40.4, 29.1
//   400x300, D = 64   105   23.3, 20.7      960x256, D = 64     202   43.2, 36.8
//   640x480, D = 32   126   25.4, 28.7      960x256, D = 256    808   127.8, 118.2
//   480x360, D = 64   152   27.4, 31.0      960x320, D = 256   1010   168, 183
//   640x400, D = 64   219   44.7, 45.3      64 x 320x240, D = 32  2156  300, 306
// The length from which strips win falls with arm_l1: 640x256, D = 64, arm_l1 = 40 29.5, 24.8;
// 17 24.5, 24.8; 3 23.5, 24.6.
std::vector<char> whole_lines(const dco_stereo *h, const std::vector<Item<VArgs>> &it, int L1, bool row_scan)
{
    std::vector<char> lines(it.size());
    size_t all = 0, few = 0;   // warps of the pairs whose lines fit, of those with short lines
    for (size_t i = 0; i < it.size(); i++) {
        const auto &b = it[i];
        const int E = row_scan ? b.a.W : b.a.H, F = row_scan ? b.a.H : b.a.W;
        if (b.gy > 0 || E > kColMax) {
            all = SIZE_MAX / 2;   // (strips are launched in any case)
            continue;
        }
        const size_t warps = (size_t)F * b.gz * ((E + kColSeg - 1) / kColSeg);
        lines[i] = E <= 200 + 3 * L1 ? 2 : 1;
        all += warps;
        if (lines[i] == 2) few += warps;
    }
    const int least = all <= 110 * (size_t)h->nsm ? 1 : few <= 1000 * (size_t)h->nsm ? 2 : 3;
    for (char &l : lines) l = l >= least;
    return lines;
}

// Deals the resident V blocks of a launch (of at most kBatchMax pairs) out to its
// pairs by their work (strips x rows; a pair's own v_chunk in it[].gy, the layers
// in it[].gz).
void deal_v_blocks(const dco_stereo *h, std::vector<Item<VArgs>> &it, int L1, bool row_scan)
{
    const int slots = vagg_slots(h, L1);
    for (size_t i0 = 0; i0 < it.size(); i0 += kBatchMax) {
        const size_t i1 = std::min(it.size(), i0 + kBatchMax);
        double all = 0.0;
        for (size_t i = i0; i < i1; i++) {
            const Item<VArgs> &b = it[i];
            all += double(vagg_units(row_scan ? b.a.H : b.a.W, b.gz)) * (row_scan ? b.a.W : b.a.H);
        }
        for (size_t i = i0; i < i1; i++) {
            Item<VArgs> &b = it[i];
            const int E = row_scan ? b.a.W : b.a.H, F = row_scan ? b.a.H : b.a.W;
            int mine = std::max(1, (int)(slots * (double(vagg_units(F, b.gz)) * E / all)));
            if (h->yield) mine = std::max(mine, (int)vagg_units(F, b.gz));   // a strip each
            const VGeom g = vagg_geom(E, F, b.gz, b.gy, mine);
            b.a.strips = g.strips;
            b.a.nblk = g.nblk; b.a.rounds = g.rounds; b.a.rest = g.rest; b.a.share = g.share; b.a.bands = g.bands;
            b.gx = g.nblk;
            b.gy = b.gz = 1;
        }
    }
}

// k_vcol's grids (b.gy: a pair's own v_chunk, b.gz: layers), by warps per block
std::map<int, std::vector<Item<VArgs>>> deal_lines(const std::vector<Item<VArgs>> &it, int L1, bool row_scan)
{
    std::map<int, std::vector<Item<VArgs>>> out;
    for (Item<VArgs> b : it) {
        const int E = row_scan ? b.a.W : b.a.H, want = b.gy > 0 ? b.gy : E;
        const int most = want >= E && E <= kColMax ? E : std::min(want, kColMax - 2 * L1);
        const int parts = (E + most - 1) / most;   // balanced
        b.a.chunk = (E + parts - 1) / parts;
        b.gx = row_scan ? b.a.H : b.a.W;
        b.gy = b.gz / b.a.ng;
        b.gz = (E + b.a.chunk - 1) / b.a.chunk;
        const int len = std::min(E, b.a.chunk + 2 * L1);
        out[(len + kColSeg - 1) / kColSeg].push_back(b);
    }
    return out;
}

template <bool kMax, bool kRow>
dco_status launch_second(dco_stereo *h, const char *name, const std::vector<Item<VArgs>> &it, const std::vector<char> &lines,
                         int L1, cudaStream_t s)
{
    std::vector<Item<VArgs>> part[2];
    for (size_t i = 0; i < it.size(); i++) part[lines[i]].push_back(it[i]);
    deal_v_blocks(h, part[0], L1, kRow);
    const dco_status st = launch_items(h, s, name, k_vagg<1, kMax, kRow>, k_vagg<kBatchMax, kMax, kRow>, part[0], kVThreads,
                                       vagg_smem_bytes(L1));
    if (st != DCO_OK) return st;
    for (const auto &kv : deal_lines(part[1], L1, kRow)) {
        const dco_status ls = launch_items(h, s, name, k_vcol<1, kMax, kRow>, k_vcol<kBatchMax, kMax, kRow>, kv.second,
                                           32 * kv.first, vcol_smem_bytes(kv.first));
        if (ls != DCO_OK) return ls;
    }
    return DCO_OK;
}

// pass `pass` (disparities [pass*dc, pass*dc + dc)) of every job that has it.
// k_vcost and k_vcol: pairs are bucketed by warps per block, one launch per bucket.
dco_status launch_pass(dco_stereo *h, const Derived &dv, std::vector<Job> &jobs, int pass, cudaStream_t s)
{
    std::map<int, std::vector<Item<HArgs>>> cb;   // k_vcost, by warps per block
    std::map<int, size_t> csm;
    std::vector<Item<HArgs>> hb[2];   // k_hagg, by warps per quad
    std::vector<Item<VArgs>> vb;
    const bool vh = dv.order == 1;   // vertical segment sums first (k_vcost), then rows (kRow)
    for (const Job &j : jobs) {
        if (pass >= j.L.npass) continue;
        const int d0 = dv.dmin + pass * j.L.dc, dc = std::min(j.L.dc, dv.dmin + j.D - d0);
        const int ng = (dc + 31) / 32;
        Item<VArgs> b{};
        for (int v = 0; v < 2; v++) {
            b.a.sh[v] = jptr<uint32_t>(h, j, j.L.sh[v]);
            b.a.arms[v] = jptr<uchar4>(h, j, j.L.arms[v]);
            b.a.best[v] = jptr<unsigned long long>(h, j, j.L.best[v]);
        }
        b.a.vol = j.vol; b.a.vol_view = j.vol_view;
        b.a.W = j.W; b.a.H = j.H; b.a.D = dv.dmin + j.D; b.a.dmin = dv.dmin;
        b.a.d0 = d0; b.a.dc = dc; b.a.dstride = j.L.dstride;
        b.a.ng = ng; b.a.single = j.L.npass == 1 && ng == 1; b.a.first = pass == 0;
        b.a.L1 = dv.L1; b.a.S = dv.S;
        b.gy = j.vchunk > 0 ? j.vchunk : dv.vchunk;
        b.gz = 2 * ng;
        vb.push_back(b);
    }
    std::vector<char> lines = whole_lines(h, vb, dv.L1, vh);
    size_t nv = 0;
    for (Job &j : jobs) {
        if (pass >= j.L.npass) continue;
        const int d0 = dv.dmin + pass * j.L.dc, dc = std::min(j.L.dc, dv.dmin + j.D - d0);
        const int ng = (dc + 31) / 32;
        const int hw = j.hchunk > 0 ? j.hchunk : dv.hchunk;
        if (j.vol) lines[nv] = 1;   // (k_vcol writes the volumes)
        const bool init = pass == 0 && !lines[nv] && !(j.L.npass == 1 && ng == 1);
        j.costs_done = lines[nv] && pass == j.L.npass - 1;
        if (j.costs_done) {   // k_vcol knows the costs with the last pass's keys
            vb[nv].a.cost[0] = j.cost_l;
            vb[nv].a.cost[1] = j.cost_r;
        }
        nv++;
        Item<HArgs> a{};
        for (int v = 0; v < 2; v++) {
            a.a.cen[v] = jptr<uint2>(h, j, j.L.cen[v]);
            a.a.col[v] = jptr<uint32_t>(h, j, j.L.col[v]);
            a.a.arms[v] = jptr<uchar4>(h, j, j.L.arms[v]);
            a.a.sh[v] = jptr<uint32_t>(h, j, j.L.sh[v]);
            a.a.init[v] = init ? jptr<unsigned long long>(h, j, j.L.best[v]) : nullptr;
        }
        a.a.pw = j.L.pw;
        a.a.status = h->d_status;
        {   // bounded staging waits; the lost-copy failure test arms the barrier without copies
            const bool lose = (h->test_flags & DCO_TEST_LOSE_TILE_COPIES) != 0;
            a.a.wait_limit = lose ? kTestWaitLimit : kWaitLimit;
            a.a.skip_copy = lose ? 1 : 0;
        }
        a.a.tables = h->d_tables;
        a.a.W = j.W; a.a.H = j.H; a.a.D = dv.dmin + j.D;
        a.a.d0 = d0; a.a.dc = dc; a.a.dstride = j.L.dstride;
        a.a.ngroups = ng;
        a.a.L1 = dv.L1; a.a.S = dv.S; a.a.Sint = dv.Sint;
        if (vh) {
            const HGeom hg = vcost_geom(j.W, j.H, dc, dv.L1, hw);
            a.a.chunk = hg.chunk;
            a.gx = hg.grid.x; a.gy = hg.grid.y; a.gz = hg.grid.z;
            csm[hg.nw] = std::max(csm[hg.nw], hg.smem);
            cb[hg.nw].push_back(a);
        } else {
            const HaggGeom hg = hagg_geom(j.W, j.H, dc, dv.L1, hw);
            a.a.chunk = hg.chunk; a.a.first = hg.first;
            a.gx = hg.grid.x; a.gy = hg.grid.y; a.gz = hg.grid.z;
            hb[hg.parts - 1].push_back(a);
        }
    }
    dco_status st;
    for (auto &kv : cb)
        if ((st = launch_items(h, s, "k_vcost", k_vcost<1>, k_vcost<kBatchMax>, kv.second, kv.first * 32,
                               csm[kv.first])) != DCO_OK)
            return st;
    if ((st = launch_items(h, s, "k_hagg", k_hagg<1, 1>, k_hagg<kBatchMax, 1>, hb[0], HSmem<1>::warps * 32,
                           HSmem<1>::total, h->yield ? INT_MAX : 4 * h->nsm)) != DCO_OK)
        return st;
    if ((st = launch_items(h, s, "k_hagg", k_hagg<1, 2>, k_hagg<kBatchMax, 2>, hb[1], HSmem<2>::warps * 32,
                           HSmem<2>::total, h->yield ? INT_MAX : 2 * h->nsm)) != DCO_OK)
        return st;
    return vh ? launch_second<false, true>(h, "k_hwta", vb, lines, dv.L1, s)
              : launch_second<false, false>(h, "k_vagg", vb, lines, dv.L1, s);
}

dco_status launch_lr(dco_stereo *h, const std::vector<Item<LrArgs>> &items, cudaStream_t s)
{
    return launch_items(h, s, "k_lr", k_lr<1>, k_lr<kBatchMax>, items, 256, 0);
}

// disparities [d0, d0 + dc) of pass `pass` of one Eq. 4 round, every job
// with a map to vote on: vote counts per horizontal segment (k_hvote), then
// vertical sums and the count maximum (k_vagg in vote mode, "k_vvote")
dco_status launch_vote_pass(dco_stereo *h, const Derived &dv, const std::vector<Job> &jobs, int pass,
                            cudaStream_t s)
{
    std::map<int, std::vector<Item<HVArgs>>> hb;
    std::vector<Item<VArgs>> vb;
    std::map<int, size_t> hsm;
    for (const Job &j : jobs) {
        if (!j.vbest || pass >= j.L.npass) continue;
        const int d0 = dv.dmin + pass * j.L.dc, dc = std::min(j.L.dc, dv.dmin + j.D - d0);
        const int ng = (dc + 31) / 32;
        Item<VArgs> b{};
        b.a.sh[0] = jptr<uint32_t>(h, j, j.L.sh[0]);
        b.a.arms[0] = jptr<uchar4>(h, j, j.L.arms[0]);
        b.a.best[0] = j.vbest;
        b.a.W = j.W; b.a.H = j.H; b.a.D = dv.dmin + j.D; b.a.dmin = dv.dmin;
        b.a.d0 = d0; b.a.dc = dc; b.a.dstride = j.L.dstride;
        b.a.ng = ng; b.a.single = j.L.npass == 1 && ng == 1; b.a.first = pass == 0;
        b.a.L1 = dv.L1; b.a.S = dv.S;
        b.gy = j.vchunk > 0 ? j.vchunk : dv.vchunk;
        b.gz = ng;   // the left view only
        vb.push_back(b);
    }
    const std::vector<char> lines = whole_lines(h, vb, dv.L1, false);
    size_t nv = 0;
    for (const Job &j : jobs) {
        if (!j.vbest || pass >= j.L.npass) continue;
        const int d0 = dv.dmin + pass * j.L.dc, dc = std::min(j.L.dc, dv.dmin + j.D - d0);
        const int ng = (dc + 31) / 32;
        const int hw = j.hchunk > 0 ? j.hchunk : dv.hchunk;
        const HGeom hg = hvote_geom(j.W, j.H, dc, dv.L1, hw);
        const bool init = pass == 0 && !lines[nv++] && !(j.L.npass == 1 && ng == 1);
        hsm[hg.nw] = std::max(hsm[hg.nw], hg.smem);
        Item<HVArgs> a{};
        a.a.disp = j.out;
        a.a.keys = j.vkeys;
        a.a.init = init ? j.vbest : nullptr;
        a.a.dmin = dv.dmin; a.a.D = dv.dmin + j.D;
        a.a.arms = jptr<uchar4>(h, j, j.L.arms[0]);
        a.a.sh = jptr<uint32_t>(h, j, j.L.sh[0]);
        a.a.W = j.W; a.a.H = j.H; a.a.d0 = d0; a.a.dstride = j.L.dstride;
        a.a.L1 = dv.L1; a.a.chunk = hg.chunk;
        a.gx = hg.grid.x; a.gy = hg.grid.y; a.gz = hg.grid.z;
        hb[hg.nw].push_back(a);
    }
    for (auto &kv : hb) {
        dco_status st = launch_items(h, s, "k_hvote", k_hvote<1>, k_hvote<kBatchMax>, kv.second, kv.first * 32,
                                     hsm[kv.first]);
        if (st != DCO_OK) return st;
    }
    return launch_second<true, false>(h, "k_vvote", vb, lines, dv.L1, s);
}

// p.vote_iters rounds of Eq. 4 on every job's final map (j.out, in place).
// A round's winners stay keys, which the next round reads (alternating
// between the two views' key arrays, free by then); the last round's become
// the map.  Arms of the left view in the workspace.
dco_status run_vote(dco_stereo *h, const dco_params &p, const Derived &dv, std::vector<Job> &jobs, cudaStream_t s)
{
    if (p.vote_iters == 0) return DCO_OK;
    int maxpass = 0;
    for (const Job &j : jobs) maxpass = std::max(maxpass, j.L.npass);
    for (int it = 0; it < p.vote_iters; it++) {
        for (Job &j : jobs) {
            j.vkeys = it > 0 ? j.vbest : nullptr;
            j.vbest = j.out ? jptr<unsigned long long>(h, j, j.L.best[it & 1]) : nullptr;
        }
        for (int pass = 0; pass < maxpass; pass++) {
            dco_status st = launch_vote_pass(h, dv, jobs, pass, s);
            if (st != DCO_OK) return st;
        }
    }
    std::vector<Item<VoteEndArgs>> end;
    for (const Job &j : jobs) {
        if (!j.out) continue;
        Item<VoteEndArgs> it{};
        it.a.best = j.vbest;
        it.a.mask = j.out; it.a.out = j.out;
        it.a.npx = j.W * j.H; it.a.dmin = dv.dmin; it.a.D = dv.dmin + j.D;
        it.gx = (j.W * j.H + 255) / 256; it.gy = 1; it.gz = 1;
        end.push_back(it);
    }
    return launch_items(h, s, "k_vote_end", k_vote_end<1>, k_vote_end<kBatchMax>, end, 256, 0);
}

// every stage of the path for planned jobs (workspace and tables ready)
dco_status launch_jobs(dco_stereo *h, const dco_params &p, const Derived &dv, std::vector<Job> &jobs,
                       cudaStream_t s)
{
    int maxpass = 0;
    for (const Job &j : jobs) maxpass = std::max(maxpass, j.L.npass);
    dco_status st;
    if ((st = launch_prep(h, p, dv, jobs, 2, s)) != DCO_OK) return st;
    for (int pass = 0; pass < maxpass; pass++)
        if ((st = launch_pass(h, dv, jobs, pass, s)) != DCO_OK) return st;
    std::vector<Item<EndArgs>> end, end_costs;
    for (const Job &j : jobs) {
        if (!j.out && !j.disp_l && !j.disp_r && (j.costs_done || (!j.cost_l && !j.cost_r))) continue;
        Item<EndArgs> it{};
        for (int v = 0; v < 2; v++) {
            it.a.best[v] = jptr<unsigned long long>(h, j, j.L.best[v]);
            it.a.arms[v] = jptr<uchar4>(h, j, j.L.arms[v]);
        }
        it.a.disp[0] = j.disp_l; it.a.disp[1] = j.disp_r; it.a.out = j.out;
        if (!j.costs_done) {
            it.a.cost[0] = j.cost_l;
            it.a.cost[1] = j.cost_r;
        }
        it.a.W = j.W; it.a.H = j.H; it.a.tol = p.lr_tol; it.a.L1 = dv.L1; it.a.S = dv.S;
        if (it.a.cost[0] || it.a.cost[1]) {
            it.gx = (j.W + kEX - 1) / kEX; it.gy = (j.H + kEY - 1) / kEY; it.gz = 2;
            end_costs.push_back(it);
        } else {
            it.gx = (j.W * j.H + 255) / 256; it.gy = 1; it.gz = 1;
            end.push_back(it);
        }
    }
    st = dv.order == 1 ? launch_items(h, s, "k_end", k_end_costs<1, true>, k_end_costs<kBatchMax, true>, end_costs,
                                      kEX * kEY, 0)
                       : launch_items(h, s, "k_end", k_end_costs<1, false>, k_end_costs<kBatchMax, false>, end_costs,
                                      kEX * kEY, 0);
    if (st != DCO_OK) return st;
    if ((st = launch_items(h, s, "k_end", k_end<1>, k_end<kBatchMax>, end, 256, 0)) != DCO_OK) return st;
    return p.vote_iters > 0 ? run_vote(h, p, dv, jobs, s) : DCO_OK;
}

// the whole path for a set of independent pairs: one launch per stage.  The
// groups that a budget makes run one after the other on the stream, each
// reusing the same workspace.  Every group is planned before anything is
// enqueued.
dco_status run_jobs(dco_stereo *h, const dco_params &p, const std::vector<Job> &jobs, cudaStream_t s)
{
    Derived dv;
    derive(p, dv);
    Plan plan;
    dco_status st = plan_ws(h, p, jobs, plan);
    if (st != DCO_OK) return st;
    if ((st = ensure_tables(h, p, dv, s)) != DCO_OK) return st;
    if (plan.groups.size() > 1) h->groups_last = (int)plan.groups.size();
    for (auto &g : plan.groups)
        if ((st = launch_jobs(h, p, dv, g, s)) != DCO_OK) return st;
    return DCO_OK;
}

dco_status check_common(dco_stereo *h, const dco_params *pin, dco_params &p)
{
    if (!h) return DCO_EINVAL;
    if (pin) p = *pin;
    else dco_params_default(&p);
    if (!params_valid(p)) {
        h->last_error = "invalid parameters";
        return DCO_EINVAL;
    }
    DCO_CUDA(h, enter_device(h));
    return DCO_OK;
}

dco_status run_match(dco_stereo *h, const uint8_t *left, const uint8_t *right, int W, int H, int D,
                     const dco_params &p, int16_t *disp_out, int16_t *disp_l, int16_t *disp_r,
                     float *cost_l, float *cost_r, float *vol, int vol_view, cudaStream_t s, int host_in = -1)
{
    std::vector<Job> jobs(1);
    Job &j = jobs[0];
    j.left = left; j.right = right; j.W = W; j.H = H; j.D = D;
    j.host_in = host_in;
    j.out = disp_out; j.disp_l = disp_l; j.disp_r = disp_r;
    j.cost_l = cost_l; j.cost_r = cost_r; j.vol = vol; j.vol_view = vol_view;
    return run_jobs(h, p, jobs, s);
}

} // namespace

// ===================================================================== C ABI
#include "densify.cuh"

extern "C" {

dco_status dco_params_default(dco_params *p)
{
    if (!p) return DCO_EINVAL;
    p->lambda_ad = 10.0f;
    p->lambda_census = 40.0f;
    p->gamma_l = 1.0f;
    p->eps = 0.8f;
    p->census_w = 9;
    p->census_h = 7;
    p->arm_l1 = 34;
    p->arm_l2 = 17;
    p->tau1 = 20;
    p->tau2 = 6;
    p->lr_tol = 1;
    p->d_chunk = 0;
    p->vote_iters = 0;
    p->smooth_arms = 0;
    p->agg_order = 0;
    p->d_min = 0;
    p->h_chunk = 0;
    p->v_chunk = 0;
    return DCO_OK;
}

const char *dco_status_string(dco_status s)
{
    switch (s) {
    case DCO_OK: return "ok";
    case DCO_EINVAL: return "invalid argument";
    case DCO_ENOMEM: return "device allocation failed";
    case DCO_EBUDGET: return "workspace budget exceeded";
    case DCO_ECUDA: return "CUDA runtime error";
    case DCO_ETIMEOUT: return "device-side wait timed out";
    case DCO_EDEVICE: return "kernel reported a failed internal check";
    }
    return "unknown status";
}

dco_status dco_stereo_create(dco_stereo **out, int device, size_t workspace_budget_bytes)
{
    if (!out) return DCO_EINVAL;
    *out = nullptr;
    int n = 0;
    if (cudaGetDeviceCount(&n) != cudaSuccess || device < 0 || device >= n) return DCO_EINVAL;
    dco_stereo *h = new (std::nothrow) dco_stereo();
    if (!h) return DCO_ENOMEM;
    h->device = device;
    h->budget = workspace_budget_bytes;
    cudaError_t e = cudaSetDevice(device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&h->nsm, cudaDevAttrMultiProcessorCount, device);
    if (e == cudaSuccess) e = cudaMalloc((void **)&h->d_status, sizeof(int));
    if (e == cudaSuccess) e = cudaMemset(h->d_status, 0, sizeof(int));
    if (e == cudaSuccess) e = cudaMalloc((void **)&h->d_tables, sizeof(float) * kTabFloats);
    if (e == cudaSuccess) e = cudaMallocHost((void **)&h->h_tables, sizeof(float) * kTabFloats);
    if (e != cudaSuccess) {
        dco_stereo_destroy(h);
        return e == cudaErrorMemoryAllocation ? DCO_ENOMEM : DCO_ECUDA;
    }
    *out = h;
    return DCO_OK;
}

void dco_stereo_destroy(dco_stereo *h)
{
    if (!h) return;
    cudaSetDevice(h->device);
    cudaDeviceSynchronize();
    for (auto &pe : h->pending) { cudaEventDestroy(pe.a); cudaEventDestroy(pe.b); }
    for (auto e : h->pool) cudaEventDestroy(e);
    cudaFree(h->ws);
    cudaFree(h->d_status);
    cudaFree(h->d_tables);
    cudaFree(h->stage);
    if (h->h_tables) cudaFreeHost(h->h_tables);
    if (h->dn_pin) cudaFreeHost(h->dn_pin);
    if (h->dn_exec) cudaGraphExecDestroy(h->dn_exec);
    if (h->dn_stream) cudaStreamDestroy(h->dn_stream);
    for (auto e : h->dn_ev)
        if (e) cudaEventDestroy(e);
    delete h;
}

size_t dco_stereo_workspace_bytes(int W, int H, int D, const dco_params *pin)
{
    dco_params p;
    if (pin) p = *pin;
    else dco_params_default(&p);
    if (!params_valid(p) || !dims_valid(W, H, D, p.d_min)) return 0;
    return make_layout(W, H, D, p).total;
}

dco_status dco_stereo_reserve(dco_stereo *h, int W, int H, int D, const dco_params *pin)
{
    dco_params p;
    dco_status st = check_common(h, pin, p);
    if (st != DCO_OK) return st;
    if (!dims_valid(W, H, D, p.d_min)) return DCO_EINVAL;
    if (p.d_chunk > 0) return ensure_ws(h, make_layout(W, H, D, p).total);
    // the widest automatic passes that the budget and the device allow
    std::vector<Job> jobs(1);
    jobs[0].W = W; jobs[0].H = H; jobs[0].D = D;
    h->ws_refused = SIZE_MAX;
    Plan plan;
    return plan_ws(h, p, jobs, plan);
}

dco_status dco_stereo_match_views(dco_stereo *h, const uint8_t *left, const uint8_t *right, int W, int H,
                                  int D, const dco_params *pin, int16_t *disp_out, int16_t *disp_left,
                                  int16_t *disp_right, float *cost_left, float *cost_right,
                                  dco_stream stream)
{
    dco_params p;
    dco_status st = check_common(h, pin, p);
    if (st != DCO_OK) return st;
    if (!left || !right || !dims_valid(W, H, D, p.d_min)) return DCO_EINVAL;
    return run_match(h, left, right, W, H, D, p, disp_out, disp_left, disp_right, cost_left, cost_right,
                     nullptr, 0, (cudaStream_t)stream);
}

dco_status dco_stereo_match(dco_stereo *h, const uint8_t *left, const uint8_t *right, int W, int H, int D,
                            const dco_params *p, int16_t *disp_out, dco_stream stream)
{
    if (!disp_out) return DCO_EINVAL;
    return dco_stereo_match_views(h, left, right, W, H, D, p, disp_out, nullptr, nullptr, nullptr, nullptr,
                                  stream);
}

// the device can dereference p at the same address (pinned, registered or
// managed host memory)
static bool device_accessible(const void *p)
{
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();   // plain pageable memory: not an error for the caller
        return false;
    }
    return (at.type == cudaMemoryTypeHost || at.type == cudaMemoryTypeManaged) && at.devicePointer == p;
}

dco_status dco_stereo_match_host(dco_stereo *h, const uint8_t *left_host, const uint8_t *right_host, int W,
                                 int H, int D, const dco_params *pin, int16_t *disp_host, dco_stream stream)
{
    dco_params p;
    dco_status st = check_common(h, pin, p);
    if (st != DCO_OK) return st;
    if (!left_host || !right_host || !disp_host || !dims_valid(W, H, D, p.d_min)) return DCO_EINVAL;
    const size_t img = (size_t)W * H * 3, out = (size_t)W * H * 2;
    const size_t need = align_up(img) * 2 + align_up(out);
    cudaStream_t s = (cudaStream_t)stream;
    // Buffers the device can dereference (pinned, registered or managed host
    // memory; over NVLink-C2C on Grace systems) are read by k_pack and
    // written by the consistency check in place, without staging copies.
    // With Eq. 4 rounds the map is rewritten several times: it stays on the
    // device and is copied once.
    if (device_accessible(left_host) && device_accessible(right_host) && device_accessible(disp_host) &&
        p.vote_iters == 0) {
        st = run_match(h, left_host, right_host, W, H, D, p, disp_host, nullptr, nullptr, nullptr, nullptr, nullptr,
                       0, s, 1);
        if (st != DCO_OK) return st;
        DCO_CUDA(h, cudaStreamSynchronize(s));
        return DCO_OK;
    }
    if (h->stage_cap < need) {
        if (h->stage) {
            DCO_CUDA(h, cudaDeviceSynchronize());
            cudaFree(h->stage);
            h->stage = nullptr;
            h->stage_cap = 0;
        }
        DCO_CUDA(h, cudaMalloc((void **)&h->stage, need));
        h->stage_cap = need;
    }
    uint8_t *dl = h->stage, *dr = h->stage + align_up(img);
    int16_t *dd = reinterpret_cast<int16_t *>(h->stage + 2 * align_up(img));
    DCO_CUDA(h, cudaMemcpyAsync(dl, left_host, img, cudaMemcpyHostToDevice, s));
    DCO_CUDA(h, cudaMemcpyAsync(dr, right_host, img, cudaMemcpyHostToDevice, s));
    st = run_match(h, dl, dr, W, H, D, p, dd, nullptr, nullptr, nullptr, nullptr, nullptr, 0, s);
    if (st != DCO_OK) return st;
    DCO_CUDA(h, cudaMemcpyAsync(disp_host, dd, out, cudaMemcpyDeviceToHost, s));
    DCO_CUDA(h, cudaStreamSynchronize(s));
    return DCO_OK;
}

// census + arms of one image (stage entry points): the pack/prep launches
// of a one-job run with a single image
static dco_status prep_one(dco_stereo *h, const dco_params &p, const uint8_t *rgb, int W, int H,
                           uchar4 *arms_out, std::vector<Job> &jobs, cudaStream_t s)
{
    Derived dv;
    derive(p, dv);
    jobs.assign(1, Job{});
    Job &j = jobs[0];
    j.left = rgb; j.right = rgb; j.W = W; j.H = H; j.D = 1; j.arms0 = arms_out;
    dco_status st = ensure_ws(h, plan_jobs(h, p, jobs, kSlicesNarrow));
    if (st != DCO_OK) return st;
    if ((st = ensure_tables(h, p, dv, s)) != DCO_OK) return st;
    return launch_prep(h, p, dv, jobs, 1, s);
}

dco_status dco_stereo_census(dco_stereo *h, const uint8_t *rgb, int W, int H, const dco_params *pin,
                             uint64_t *census_out, dco_stream stream)
{
    dco_params p;
    dco_status st = check_common(h, pin, p);
    if (st != DCO_OK) return st;
    if (!rgb || !census_out || !dims_valid(W, H, 1)) return DCO_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    std::vector<Job> jobs;
    if ((st = prep_one(h, p, rgb, W, H, nullptr, jobs, s)) != DCO_OK) return st;
    const Job &j = jobs[0];
    const size_t n = (size_t)W * H;
    ProfScope ps(h, s, "k_extract_census");
    k_extract_census<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(jptr<uint2>(h, j, j.L.cen[0]), W, H, j.L.pw,
                                                                  reinterpret_cast<unsigned long long *>(census_out));
    DCO_CUDA(h, cudaGetLastError());
    return DCO_OK;
}

dco_status dco_stereo_arms(dco_stereo *h, const uint8_t *rgb, int W, int H, const dco_params *pin,
                           uint8_t *arms_out, dco_stream stream)
{
    dco_params p;
    dco_status st = check_common(h, pin, p);
    if (st != DCO_OK) return st;
    if (!rgb || !arms_out || !dims_valid(W, H, 1)) return DCO_EINVAL;
    std::vector<Job> jobs;
    return prep_one(h, p, rgb, W, H, reinterpret_cast<uchar4 *>(arms_out), jobs, (cudaStream_t)stream);
}

dco_status dco_stereo_vote(dco_stereo *h, const uint8_t *rgb, const int16_t *disp_in, int W, int H, int D,
                           const dco_params *pin, int16_t *disp_out, dco_stream stream)
{
    dco_params p;
    dco_status st = check_common(h, pin, p);
    if (st != DCO_OK) return st;
    if (!rgb || !disp_in || !disp_out || !dims_valid(W, H, D, p.d_min)) return DCO_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    Derived dv;
    derive(p, dv);
    std::vector<Job> jobs(1);
    Job &j = jobs[0];
    j.left = rgb; j.right = rgb; j.W = W; j.H = H; j.D = D; j.out = disp_out;
    Plan plan;
    if ((st = plan_ws(h, p, jobs, plan)) != DCO_OK) return st;
    if ((st = ensure_tables(h, p, dv, s)) != DCO_OK) return st;
    if ((st = launch_prep(h, p, dv, plan.groups[0], 1, s)) != DCO_OK) return st;   // arms of rgb
    if (disp_in != disp_out)
        DCO_CUDA(h, cudaMemcpyAsync(disp_out, disp_in, sizeof(int16_t) * W * H, cudaMemcpyDeviceToDevice, s));
    return run_vote(h, p, dv, plan.groups[0], s);
}

dco_status dco_stereo_downscale(dco_stereo *h, const uint8_t *rgb, int W, int H, uint8_t *out, dco_stream stream)
{
    if (!h || !rgb || !out || W < 2 || H < 2 || W > 2 * 16384 || H > 2 * 16384) return DCO_EINVAL;
    DCO_CUDA(h, enter_device(h));
    cudaStream_t s = (cudaStream_t)stream;
    DownArgs da{};
    da.src[0] = rgb; da.dst[0] = out; da.W = W; da.H = H;
    ProfScope ps(h, s, "k_down");
    launch_pdl(k_down, dim3((unsigned)((W / 2 + 255) / 256), (unsigned)(H / 2), 1), dim3(256), 0, s, da);
    DCO_CUDA(h, cudaGetLastError());
    return DCO_OK;
}

dco_status dco_stereo_depth(dco_stereo *h, const uint8_t *left, const uint8_t *right, int W, int H, int D,
                            const dco_params *pin, double f_px, double baseline, float *depth_out,
                            int16_t *disp_half_out, dco_stream stream)
{
    dco_params p;
    dco_status st = check_common(h, pin, p);
    if (st != DCO_OK) return st;
    if (!left || !right || !depth_out || W < 2 || H < 2 || !dims_valid(W / 2, H / 2, D, p.d_min)) return DCO_EINVAL;
    if (!(f_px > 0.0) || !(baseline > 0.0) || !std::isfinite(f_px * baseline)) return DCO_EINVAL;
    cudaStream_t s = (cudaStream_t)stream;
    const int Wh = W / 2, Hh = H / 2;
    Derived dv;
    derive(p, dv);
    std::vector<Job> jobs(1);
    jobs[0].W = Wh; jobs[0].H = Hh; jobs[0].D = D;
    Plan plan;
    // in front of the pair's workspace: the two half-size images and the map
    const size_t img = align_up(3 * (size_t)Wh * Hh), front = 2 * img + align_up(2 * (size_t)Wh * Hh);
    if ((st = plan_ws(h, p, jobs, plan, front)) != DCO_OK) return st;
    Job &j = plan.groups[0][0];
    if ((st = ensure_tables(h, p, dv, s)) != DCO_OK) return st;
    DownArgs da{};
    da.src[0] = left; da.src[1] = right;
    da.dst[0] = ws_ptr<uint8_t>(h, 0); da.dst[1] = ws_ptr<uint8_t>(h, img);
    da.W = W; da.H = H;
    j.left = da.dst[0]; j.right = da.dst[1];
    j.out = disp_half_out ? disp_half_out : ws_ptr<int16_t>(h, 2 * img);
    {
        ProfScope ps(h, s, "k_down");
        launch_pdl(k_down, dim3((unsigned)((Wh + 255) / 256), (unsigned)Hh, 2), dim3(256), 0, s, da);
        DCO_CUDA(h, cudaGetLastError());
    }
    if ((st = launch_jobs(h, p, dv, plan.groups[0], s)) != DCO_OK) return st;
    DepthArgs za{};
    za.disp = j.out; za.out = depth_out; za.W = W; za.H = H; za.fb = (float)(f_px * baseline);
    ProfScope ps(h, s, "k_depth");
    launch_pdl(k_depth, dim3((unsigned)(((W + 1) / 2 + 255) / 256), (unsigned)((H + 1) / 2)), dim3(256), 0, s, za);
    DCO_CUDA(h, cudaGetLastError());
    return DCO_OK;
}

dco_status dco_stereo_cost_volume(dco_stereo *h, const uint8_t *left, const uint8_t *right, int W, int H,
                                  int D, const dco_params *pin, int view, float *vol_out, dco_stream stream)
{
    dco_params p;
    dco_status st = check_common(h, pin, p);
    if (st != DCO_OK) return st;
    if (!left || !right || !vol_out || (view != 0 && view != 1) || !dims_valid(W, H, D, p.d_min)) return DCO_EINVAL;
    return run_match(h, left, right, W, H, D, p, nullptr, nullptr, nullptr, nullptr, nullptr, vol_out, view,
                     (cudaStream_t)stream);
}

dco_status dco_stereo_lr_check(dco_stereo *h, const int16_t *dl, const int16_t *dr, int W, int H, int tol,
                               int16_t *out, dco_stream stream)
{
    if (!h || !dl || !dr || !out || W < 1 || H < 1) return DCO_EINVAL;
    DCO_CUDA(h, enter_device(h));
    std::vector<Item<LrArgs>> it(1);
    it[0].a.dl = dl; it[0].a.dr = dr; it[0].a.out = out;
    it[0].a.W = W; it[0].a.H = H; it[0].a.tol = tol;
    it[0].gx = (int)(((size_t)W * H + 255) / 256); it[0].gy = 1; it[0].gz = 1;
    return launch_lr(h, it, (cudaStream_t)stream);
}

dco_status dco_stereo_match_batch(dco_stereo *h, const dco_pair_desc *descs, int n, const dco_params *pin,
                                  dco_stream stream)
{
    dco_params p;
    dco_status st = check_common(h, pin, p);
    if (st != DCO_OK) return st;
    h->groups_last = 1;
    if (n < 0 || (n > 0 && !descs)) return DCO_EINVAL;
    for (int i = 0; i < n; i++)
        if (!descs[i].left || !descs[i].right || !descs[i].disp_out ||
            !dims_valid(descs[i].W, descs[i].H, descs[i].D, p.d_min) || descs[i].d_chunk < 0 ||
            !tile_valid(descs[i].h_chunk) || !tile_valid(descs[i].v_chunk))
            return DCO_EINVAL;
    if (n == 0) return DCO_OK;
    std::vector<Job> jobs(n);
    for (int i = 0; i < n; i++) {
        jobs[i].left = descs[i].left; jobs[i].right = descs[i].right;
        jobs[i].W = descs[i].W; jobs[i].H = descs[i].H; jobs[i].D = descs[i].D;
        jobs[i].out = descs[i].disp_out;
        jobs[i].dchunk = descs[i].d_chunk;
        jobs[i].hchunk = descs[i].h_chunk;
        jobs[i].vchunk = descs[i].v_chunk;
    }
    return run_jobs(h, p, jobs, (cudaStream_t)stream);
}

dco_status dco_stereo_sync_status(dco_stereo *h)
{
    if (!h) return DCO_EINVAL;
    DCO_CUDA(h, enter_device(h));
    DCO_CUDA(h, cudaDeviceSynchronize());
    int v = 0;
    DCO_CUDA(h, cudaMemcpy(&v, h->d_status, sizeof v, cudaMemcpyDeviceToHost));
    DCO_CUDA(h, cudaMemset(h->d_status, 0, sizeof v));
    return status_of_word(v);
}

dco_status dco_stereo_stream_status(dco_stereo *h, dco_stream stream)
{
    if (!h) return DCO_EINVAL;
    DCO_CUDA(h, enter_device(h));
    const cudaStream_t s = (cudaStream_t)stream;
    // a device-to-pageable copy returns once it has completed: the word is
    // read after everything enqueued on `stream` before this call
    int v = 0;
    DCO_CUDA(h, cudaMemcpyAsync(&v, h->d_status, sizeof v, cudaMemcpyDeviceToHost, s));
    DCO_CUDA(h, cudaStreamSynchronize(s));
    DCO_CUDA(h, cudaMemsetAsync(h->d_status, 0, sizeof v, s));
    return status_of_word(v);
}

dco_status dco_stereo_set_test_flags(dco_stereo *h, int flags)
{
    if (!h || (flags & ~(DCO_TEST_LOSE_TILE_COPIES | DCO_TEST_LOSE_GRID_ARRIVAL | DCO_TEST_REFUSE_WIDE))) return DCO_EINVAL;
    h->test_flags = flags;
    return DCO_OK;
}

size_t dco_stereo_workspace_allocated(dco_stereo *h)
{
    return h ? h->ws_cap : 0;
}

int dco_stereo_batch_groups(dco_stereo *h)
{
    return h ? h->groups_last : 0;
}

dco_status dco_stereo_set_profiling(dco_stereo *h, int enable)
{
    if (!h) return DCO_EINVAL;
    h->profiling = enable != 0;
    return DCO_OK;
}

dco_status dco_stereo_profile_reset(dco_stereo *h)
{
    if (!h) return DCO_EINVAL;
    cudaSetDevice(h->device);
    cudaDeviceSynchronize();
    collect_profile(h);
    h->agg.clear();
    return DCO_OK;
}

int dco_stereo_profile_count(dco_stereo *h)
{
    if (!h) return 0;
    cudaSetDevice(h->device);
    cudaDeviceSynchronize();
    collect_profile(h);
    return (int)h->agg.size();
}

dco_status dco_stereo_profile_get(dco_stereo *h, int i, const char **name, int *launches, double *total_ms)
{
    if (!h || i < 0 || i >= (int)h->agg.size()) return DCO_EINVAL;
    if (name) *name = h->agg[i].name.c_str();
    if (launches) *launches = h->agg[i].launches;
    if (total_ms) *total_ms = h->agg[i].ms;
    return DCO_OK;
}

unsigned long long dco_stereo_launch_count(dco_stereo *h)
{
    return h ? h->launches : 0ull;
}

const char *dco_stereo_last_error(dco_stereo *h)
{
    return h ? h->last_error.c_str() : "null handle";
}

} // extern "C"

// ======================================================= no-allocation entry
// For callers that may not allocate device memory: the scratch lives in one
// file-scope device array that every GPU loading this library holds until
// exit.  Host code never uses the array's name as a device address: each
// device's address comes from cudaGetSymbolAddress, taken once per device
// on the first call with that device current.
namespace {
constexpr size_t kNoAllocScratchBytes = size_t(32) << 20;
constexpr int kNoAllocMaxDevices = 64;
// scratch layout: the Eq. 1 tables, the status word, the workspace
constexpr size_t kNoAllocTabBytes = (sizeof(float) * kTabFloats + kAlign - 1) / kAlign * kAlign;
constexpr size_t kNoAllocStatusBytes = kAlign;
std::mutex g_noalloc_mu;
void *g_noalloc_base[kNoAllocMaxDevices] = {};

// the tables travel by value in the kernel parameters, so no host buffer
// has to outlive the call
struct TabBlock {
    float t[kTabFloats];
};
__global__ void k_put_tables(const __grid_constant__ TabBlock b, float *dst)
{
    for (int i = threadIdx.x; i < kTabFloats; i += blockDim.x) dst[i] = b.t[i];
}
} // namespace

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

namespace {
dco_status noalloc_base(int dev, void **out)
{
    if (dev < 0 || dev >= kNoAllocMaxDevices) return DCO_EINVAL;
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_base[dev]) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return DCO_ECUDA;
        g_noalloc_base[dev] = p;
    }
    *out = g_noalloc_base[dev];
    return DCO_OK;
}
} // namespace

extern "C" dco_status dco_stereo_match_noalloc(const uint8_t *left, const uint8_t *right, int W, int H, int D,
                                               const dco_params *pin, int16_t *disp_out, dco_stream stream)
{
    dco_params p;
    if (pin) p = *pin;
    else dco_params_default(&p);
    if (!params_valid(p) || !left || !right || !disp_out || !dims_valid(W, H, D, p.d_min)) return DCO_EINVAL;
    p.d_chunk = 32;   // passes of 32 disparities keep the slices small
    Derived dv;
    derive(p, dv);
    const Layout L = make_layout(W, H, D, p);
    if (kNoAllocTabBytes + kNoAllocStatusBytes + L.total > kNoAllocScratchBytes) return DCO_EBUDGET;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return DCO_ECUDA;
    (void)cudaGetLastError();   // an earlier call's error is not this call's launch failure
    void *base = nullptr;
    dco_status st = noalloc_base(dev, &base);
    if (st != DCO_OK) return st;
    cudaStream_t s = (cudaStream_t)stream;

    // Eq. 1 tables (host double, rounded once to float) into the scratch
    TabBlock tb;
    fill_tables(tb.t, p, dv);
    k_put_tables<<<1, 256, 0, s>>>(tb, static_cast<float *>(base));
    if (cudaGetLastError() != cudaSuccess) return DCO_ECUDA;

    // a handle that owns nothing: its workspace and tables are the scratch
    dco_stereo view;
    view.device = dev;
    view.d_status = reinterpret_cast<int *>(static_cast<char *>(base) + kNoAllocTabBytes);
    view.ws = static_cast<char *>(base) + kNoAllocTabBytes + kNoAllocStatusBytes;
    view.ws_cap = kNoAllocScratchBytes - kNoAllocTabBytes - kNoAllocStatusBytes;
    view.d_tables = static_cast<float *>(base);
    view.tab_valid = true;
    view.tab_key[0] = p.lambda_ad;
    view.tab_key[1] = p.lambda_census;
    view.tab_key[2] = p.gamma_l;
    view.tab_key[3] = p.eps;
    view.tab_l1 = p.arm_l1;
    st = run_match(&view, left, right, W, H, D, p, disp_out, nullptr, nullptr, nullptr, nullptr, nullptr, 0, s);
    view.ws = nullptr;
    view.d_tables = nullptr;
    view.d_status = nullptr;
    return st;
}

extern "C" dco_status dco_stereo_noalloc_status(dco_stream stream)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return DCO_ECUDA;
    void *base = nullptr;
    dco_status st = noalloc_base(dev, &base);
    if (st != DCO_OK) return st;
    int *word = reinterpret_cast<int *>(static_cast<char *>(base) + kNoAllocTabBytes);
    const cudaStream_t s = (cudaStream_t)stream;
    // a device-to-pageable copy returns once it has completed, after the
    // work enqueued on `stream` before it
    int v = 0;
    if (cudaMemcpyAsync(&v, word, sizeof v, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess || cudaMemsetAsync(word, 0, sizeof v, s) != cudaSuccess) {
        (void)cudaGetLastError();
        return DCO_ECUDA;
    }
    return status_of_word(v);
}

// ====================================================== serving runtime
#include "serve.cuh"
