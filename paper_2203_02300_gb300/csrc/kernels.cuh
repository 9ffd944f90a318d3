// Device-side types and constants of the AD-census matcher (arXiv 2203.02300, Sect. 4).
//
// Data layout in HBM (row-major, pixel index i = y*W + x):
//   rgbx[i]  uint32 r | g<<10 | b<<20          colour in three 10-bit fields (arm tests)
//   grey[i]  uint8  (77R + 150G + 29B + 128) >> 8
//   cen[y*pw + x]  uint2 {census bits 0-31, census bits 32-63}
//   col[y*pw + x]  uint32 r | g<<8 | b<<16 | Lmin<<24   (pw: W rounded up to a
//                    multiple of 4, so that every row starts on a 16-byte boundary)
//   arms[i]  uchar4 {left, right, up, down}
//   sh[i*dstride + j]  uint32 horizontal segment sum (fixed point) of
//                    disparity d0 + j (one pass of the d range)
//   best[i]  uint64 (aggregate << 32 | d), the WTA's running minimum over the
//            disparity groups and passes
//
// Costs are carried in unsigned fixed point with scale S (an integer below
// 2^20, chosen so a full (2*L1+1)^2 region of costs <= 1 stays below 2^32).
// Prefix sums wrap modulo 2^32, and differences of prefix sums are exact
// region sums, so the Eq. 2 aggregation is exact integer arithmetic on the
// rounded per-pixel costs; only the Eq. 1 evaluation (FP32) and the rounding
// to fixed point differ from the real-valued definition.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace dco {

constexpr int kMaxL1 = 40;
constexpr int kTabAD = 768;   // entries of the AD table (sum of 3 abs diffs, 0..765)
constexpr int kTabCen = 96;   // entries of the census table (Hamming 0..64)
constexpr int kTabAlpha = 64; // alpha*S by Lmin, 0..kMaxL1
constexpr int kTabFloats = kTabAD + kTabCen + kTabAlpha;

// k_vcost gives each warp kHSegCost rows of the prefix range, the vote H pass
// segments of kHSeg columns.
constexpr int kHSegLog = 6, kHSeg = 1 << kHSegLog;
constexpr int kHSegCost = 32;
constexpr int kHMaxLen = 1024;   // prefix positions one k_vcost or k_hvote block holds

struct PackArgs {
    const uint8_t *rgb[2];
    uint32_t *rgbx[2];
    uint8_t *grey[2];
    int npx, W;
    uint32_t k1;           // colour threshold tau1 in every 10-bit field (see kM9)
};

struct PrepArgs {
    const uint32_t *rgbx[2];
    const uint8_t *grey[2];
    uint2 *cen[2];         // planes, row pitch pw
    uint32_t *col[2];
    int pw;
    uchar4 *arms[2];
    int W, H;
    int cw, ch;            // census window (odd)
    int L1, L2, tau1, tau2;
};

struct HArgs {
    const uint2 *cen[2];   // planes, row pitch pw
    const uint32_t *col[2];
    int pw;
    int *status;           // device status word (a lost staging copy sets bit 0)
    int wait_limit;        // mbarrier polls before the staging copies are declared lost
    int skip_copy;         // failure test: arm the staging barrier but issue no copy
    const uchar4 *arms[2];
    uint32_t *sh[2];
    unsigned long long *init[2];   // first pass: keys to set to the maximum (null: none)
    const float *tables;
    int W, H, D;
    int d0, dc;            // this pass covers d in [d0, d0 + dc)
    int dstride;           // uint32 per pixel in sh (dc rounded up to 32)
    int ngroups;           // 32-disparity groups in the pass
    int L1;
    int chunk;             // output positions per block (k_hagg: per task, `first` in a row's first)
    int first;
    float S;               // fixed-point scale (integer valued)
    uint32_t Sint;
};

// horizontal pass of the parallax optimisation (Eq. 4): per-d vote counts
struct HVArgs {
    const int16_t *disp;   // map of the first round, W x H; outside [dmin, D) = invalid
    const unsigned long long *keys;   // later rounds: the previous round's keys (d in the low word)
    unsigned long long *init;         // first pass: keys to set to the maximum (null: none)
    int dmin, D;
    const uchar4 *arms;    // reference-view arms {l, r, u, d}
    uint32_t *sh;          // count slices [y][x][dstride]
    int W, H, d0, dstride, L1, chunk;
};

// quarter-size input (Sect. 4): the two images of a pair, W x H -> W/2 x H/2
struct DownArgs {
    const uint8_t *src[2];
    uint8_t *dst[2];
    int W, H;
};

// sparse depth (Sect. 4.4) of a half-size map on the W x H grid
struct DepthArgs {
    const int16_t *disp;   // (H/2) x (W/2)
    float *out;            // W x H
    int W, H;
    float fb;              // f * B
};

// smoothing of the cross-support window (Sect. 4.1): one pass of a 3x3
// grey-level opening (minimum, then maximum) of the four arm maps
struct SmoothArgs {
    const uchar4 *src[2];
    uchar4 *dst[2];
    uint32_t *col[2];      // dilation pass: colour words whose L_min follows the new arms
    int W, H, pw;
};

struct VArgs {
    const uint32_t *sh[2];        // slices, dstride words per pixel
    const uchar4 *arms[2];
    unsigned long long *best[2];  // (aggregate << 32 | d) per pixel, minimised over every pass and group
    float *vol;            // optional (D, H, W) normalised costs of view `vol_view`
    int vol_view;
    int W, H, D;           // D: one past the largest disparity of the search (d_min + count)
    int dmin;              // smallest disparity of the search
    int d0, dc, dstride;   // this pass covers d in [d0, d0 + dc)
    int ng;                // 32-disparity groups in the pass
    int single;            // k_vagg: the only pass and group: keys are stored, not minimised
    int first;             // k_vcol: the first pass: keys are stored, else minimised
    int chunk;             // k_vcol: output rows per block
    float *cost[2];        // k_vcol: minimum costs (null: none), from this pass's keys
    int L1;
    int strips;            // strips of four columns per layer (group and view)
    int nblk, rounds;      // blocks; whole strips per block
    int rest, share, bands;   // strips left over, rows of them per block, blocks per strip (0: shares run on)
    float S;
};

// the per-pixel end of a match: keys -> disparities and costs of both views,
// left-right consistency -> disparity map (every output optional)
struct EndArgs {
    const unsigned long long *best[2];
    const uchar4 *arms[2];
    int16_t *disp[2], *out;
    float *cost[2];
    int W, H, tol, L1;
    float S;
};

// the end of the Eq. 4 rounds: keys -> map; pixels of `mask` outside the
// range cast no vote and stay invalid
struct VoteEndArgs {
    const unsigned long long *best;
    const int16_t *mask;
    int16_t *out;
    int npx, dmin, D;
};

struct LrArgs {
    const int16_t *dl, *dr;
    int16_t *out;
    int W, H, tol;
};

} // namespace dco
