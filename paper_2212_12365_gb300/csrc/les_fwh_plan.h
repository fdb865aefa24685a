// Host side of les_fwh: block and batch sizes of an evaluation (plain C++, no
// device code).
#pragma once

#include <algorithm>
#include <cmath>
#include <cstddef>

namespace les {

constexpr int FWH_T = 256;   // observer times per CTA of the direct pass
constexpr int FWH_MG = 16;   // microphones per group of the staged pass, at most
constexpr int FWH_PB = 8;    // panels whose geometry is staged together
constexpr size_t FWH_GEO_BYTES = 784;        // staged geometry of a panel (FwhGeo)
constexpr size_t FWH_WIN_SMEM = 110 * 1024;  // shared memory of a staged CTA, at most: two per SM
constexpr int FWH_WIN_MAX = 1024;            // frames of a window, at most (32 mask words)

// Rows of a group's window buffer: its microphones, in pairs.
inline constexpr int fwh_rows(int MG) { return (MG + 1) / 2 * 2; }
// Shared memory of the staged pass for windows of W frames (a multiple of 32)
// and `rows` rows: the rows twice, the records, the geometry.
inline constexpr size_t fwh_win_smem(int W, int rows)
{
    return 8 * (size_t)rows * W + 32 * (size_t)W + FWH_PB * FWH_GEO_BYTES;
}

struct FwhPlan {
    int MG, ngroups;   // microphones per group, groups
    bool staged;       // staged or direct observer pass
    int T, tblocks;    // observer times per block, blocks
    int W, span, nth;  // staged: frames of a window, frames of a block's times, threads
    int NB, nchunk;    // panels per batch; panel chunks of a batch
    size_t b_src, b_rec, b_part; // bytes of source records, panel records and partial sums
    size_t scratch() const { return b_src + b_rec + b_part; }
};

// Microphone groups of equal size, at most FWH_MG.
inline int fwh_group(int nobs)
{
    const int n = (nobs + FWH_MG - 1) / FWH_MG;
    return (nobs + n - 1) / n;
}

// spread: the largest spread of a panel's distances over a microphone group.
inline FwhPlan fwh_plan(int npts, int N, int nobs, int nt, double dt_obs, double dtau, double c0, double spread, int nsm)
{
    FwhPlan P{};
    P.MG = fwh_group(nobs);
    P.ngroups = (nobs + P.MG - 1) / P.MG;
    // The staged pass takes blocks of observer times, in equal parts; per panel a
    // window of W frames: the block's times plus the spread of the group's
    // emission times.  Two CTAs of 256 threads fit an SM by their registers, so a
    // CTA may use 110 KB of shared memory; with a buffer row per microphone of the
    // group a window holds 640 frames for a group of 16 and 1024 for one of 8.  A
    // block of 512 times shares the spread among more evaluations than one of 256,
    // so it comes first (with blocks of 256 only, 8, 24 and 64 microphones x 512
    // times take 3.61, 5.14 and 7.37 ms a call against 3.32, 4.55 and 7.11; no call
    // measured gains); the direct pass is left for windows that fit neither.
    // (With sixteen rows always and no second block size, 98,304 panels of 1024
    // frames took the direct pass at 8, 16, 24 and 32 microphones x 512 times:
    // 3.94, 5.71, 8.58, 10.50 ms a call; so 3.31, 4.23, 4.52, 5.65.)
    const int caps[2] = {512, 256};
    const int rows = fwh_rows(P.MG);
    for (int cap : caps) {
        P.tblocks = (nt + cap - 1) / cap;
        P.T = (nt + P.tblocks - 1) / P.tblocks;
        const double span = std::floor((P.T - 1) * dt_obs / dtau + 2.0) + 1.0;
        const double W = span + std::ceil(spread / (c0 * dtau)) + 6.0;
        if (!(W <= FWH_WIN_MAX)) continue;
        P.W = ((int)W + 31) / 32 * 32;
        P.span = (int)span;
        P.staged = fwh_win_smem(P.W, rows) <= FWH_WIN_SMEM;
        if (P.staged) break;
    }
    if (!P.staged) {
        P.W = P.span = 0;
        P.T = FWH_T;
        P.tblocks = (nt + FWH_T - 1) / FWH_T;
    }
    // threads: half the block's times, so that few are idle in a short block
    P.nth = P.T <= 128 ? 64 : (P.T <= 256 ? 128 : 256);
    // panels per batch: source records of at most 256 MB (and at least 1024
    // panels, so that a batch fills the chip), and in the staged pass panel records
    // of at most 256 MB too (from 8192 microphones on a batch has fewer than 1024
    // panels, but the microphone groups alone fill the chip)
    const long long batch = 256LL << 20;
    P.NB = (int)std::min<long long>(npts, std::max<long long>(1024, batch / (32LL * N) / 256 * 256));
    if (P.staged) P.NB = (int)std::min<long long>(P.NB, std::max<long long>(1, batch / (32LL * nobs)));
    // panel chunks of a batch: the CTAs of one wave (staged: 512 threads or the
    // shared memory of an SM; direct: four CTAs per SM)
    const int cps = P.staged ? std::min(512 / P.nth, (int)(2 * FWH_WIN_SMEM / fwh_win_smem(P.W, rows))) : 4;
    P.nchunk = P.staged ? cps * nsm / (P.tblocks * P.ngroups)
                        : (cps * nsm + P.tblocks * nobs - 1) / (P.tblocks * nobs);
    P.nchunk = std::max(1, std::min(P.nchunk, (P.NB + FWH_PB - 1) / FWH_PB));
    P.b_src = (size_t)P.NB * N * 32;
    P.b_rec = P.staged ? (size_t)P.NB * nobs * 32 : 0;
    P.b_part = (size_t)nobs * nt * (P.nchunk + 1) * sizeof(double);
    return P;
}

} // namespace les
