// Which tiles a frame's plan gets, by rule (where neither BF_TILE_ROWS nor bf_autotune
// decides), from the frames that share it.  Header-only and free of CUDA calls, so that
// the rules can be checked on a machine without a GPU.
#pragma once

#include <algorithm>

#include "bf_internal.h"

namespace bfi {

// 16-row tiles of an image.
inline int image_tiles(int nx, int nz) { return (nx + kTileCols - 1) / kTileCols * ((nz + 15) / 16); }

// Configuration (of kTileConfigs, or a solo one).  tiles: the image's 16-row tiles; alone:
// the frame shares its plan with no other; shares: its combiners can share a job; peers:
// the frames of its plan that are submitted together.
//
// Beamforming time per 512 x 512 frame, 32 frames in a batch, DAS + DMAS of one
// angle / DMAS of three: alone (solo; one angle since at 0.75 of this) 13.7 / 22.3 us,
// in pairs on 32-row tiles 7.4 / 21.0 us, in fours on 16-row tiles 5.9 / 16.2 us.
//
// Alone: split the channels of a row pair over four warps below 3/4 of a tile per SM,
// over two below 3/2 (152 SMs; splits 1 / 2 / 4, DMAS of three angles: 32 tiles 26.2 /
// 16.0 / 11.9 us, 112 tiles 20.4 / 16.0 / 13.9, 128 tiles 20.1 / 16.0 / 20.1, 220 tiles
// 28.3 / 24.2 / 32.4, 325 tiles 26.2 / 26.6 / 36.5, 512 tiles 32.4 / 34.4 / 54.9).  The
// frame's own tiles decide, also in a batch: a lone frame's sums do not depend on what it
// is launched with.
//
// Fours where they give the SMs work: below 3/4 of a CTA per SM pairs, whose CTAs are as
// many and larger, are faster (whole passes of 64 x 64 and 128 x 128 frames, DAS of one
// angle in fours / in pairs: 4 frames 36.9 / 32.9 and 28.8 / 26.9 us, 7 frames 39.4 / 33.5
// and 31.4 / 28.8).  Six or seven frames leave two or three behind the four, which weighs
// where a frame is short (384 x 384, DAS + DMAS of one angle: 6 frames 55.8 / 54.9, 7
// frames 67.7 / 63.2; of three angles 110.6 / 125.0 and 138.2 / 145.1); a fifth frame alone
// on the tiles of the four takes less than three pairs (49.5 / 63.0), and beside them on
// solo tiles more.  IQ records above 4096 samples share no job; four and more of them take
// the 16-row tiles all the same (4 frames of 128 x 128 and 512 x 512: 41.4 and 113.9 us, on
// 32-row tiles 58.4 and 121.2).
inline int rule_config(int prec, int ns, int na, int tiles, int sms, bool alone, bool shares, int peers)
{
    const bool iq = prec == kPrecIQ;
    if (alone && !iq)
        return kSoloConfig + (4 * tiles <= 3 * sms ? 2 : 2 * tiles <= 3 * sms ? 1 : 0);
    if (!shares || peers < kMaxFramesPerJob)
        return 0;
    if (iq && ns > 4096)
        return 4;
    if (4ll * (peers / kMaxFramesPerJob) * tiles < 3ll * sms)
        return 0;
    if (!iq && na == 1 && (peers == 6 || peers == 7))
        return 0;
    return iq ? 4 : 6;
}

// Frames the pairs buffer of frame `index` of `peers` (0 <= index < peers; < 0: not known)
// has room for, in jobs of up to cap: the frame that leads a job holds the pairs of all of
// it, so that cap frames need 2 cap - 1 rooms together instead of cap^2.  fixed: the launch
// is made of just these frames in this order (a batch); otherwise (the serving engine) the
// frames behind the last whole four, too few for one, and pairs may meet others.
inline int pairs_room(int cap, int index, int peers, bool fixed)
{
    if (index < 0 || cap == 1 || (!fixed && (cap == 2 || peers < cap)))
        return cap;
    const int first = index / cap * cap, n = std::min(cap, peers - first);
    if (n == cap)
        return index == first ? cap : 1;
    return !fixed || (n >= 2 && index == first) ? 2 : 1;
}

}  // namespace bfi
