// Which hopping kernel a call takes when the handle names none (one right-hand side
// per thread, no lanes, no tiles): rules on sizes and formats, both sides of each
// line measured. Host code without CUDA, shared by the launcher and the tuner.
// Times are us per M_eo on one GB300; V/2 = 65536 is 16^3 x 32, 331776 24^3 x 48.
#pragma once

namespace weo {

enum class Route {
    OneSite,  // hop_kernel: a site per thread
    Split,    // weo_split.cuh: a site's directions on the warps of a CTA
    Tiles,    // hop_kernel_tile_links: links in shared memory for four right-hand sides at a time
};

// Largest V/2 of the split kernels: their 32-bit offsets address 16-byte elements.
constexpr int kSplitMaxSites = 1 << 28;

// Tiles against the better of the other two. A pass over four right-hand sides costs
// little more than one over three, so what counts is how well the passes are filled;
// with fewer than 2^16 sites there are less than two waves of tiles.
//   FP32 18-real, split : tiles: 65536 sites 4 RHS 50.4 : 51.7, 8 RHS 94.6 : 84.6,
//     9 RHS 104.5 : 105.1, 13 RHS 147 : 137; 331776 sites 3 RHS 188 : 192, 4 RHS
//     243 : 215, 5 RHS 297 : 295, 6 RHS 352 : 314, 12 RHS 680 : 518; 16^4 with 16 RHS
//     92.4 : 93.1
//   FP32 12-real: 65536 sites 8 RHS 86.6 : 82.6, 9 RHS 96.6 : 103, 10 RHS 106.5 : 106.4;
//     331776 sites 4 RHS 221 : 208, 5 RHS 272 : 290, 9 RHS 477 : 436, 12 RHS 630 : 512
//   16 bits, 18-real: 65536 sites 8 RHS 79.5 : 78.6, 9 RHS 88.5 : 97.7, 12 RHS 115 : 110,
//     13 RHS 124 : 129; 331776 sites (one site : tiles) 4 RHS 197 : 198, 5 RHS 240 : 278,
//     6 RHS 283 : 294, 7 RHS 326 : 324, 10 RHS 454 : 434, 12 RHS 539 : 481
//   16 bits, 12-real: 65536 sites 8 RHS 83.2 : 78.0, 9 RHS 92.8 : 96.9; 331776 sites
//     (one site : tiles) 4 RHS 196 : 196, 6 RHS 286 : 292, 9 RHS 419 : 412, 12 RHS 553 : 479
inline bool tiles_pay(bool bits16, bool link12, long long vh, int nrhs)
{
    const long long work = vh * nrhs, slots = (nrhs + 3ll) / 4 * 4;
    if (nrhs < 4 || vh < (1 << 16) || work < (1 << 19)) return false;
    if (bits16) return nrhs > 4 && (nrhs == slots || (4 * nrhs > 3 * slots && work >= (1 << 21)));
    return nrhs == slots || (4 * nrhs >= 3 * slots && (!link12 || work >= (1 << 20)));
}

// Split against one site per thread: with 16-bit storage the split kernel issues more
// instructions per byte, and once the work fills the GPU many times over, the one-site
// kernel's fewer ones win, for several right-hand sides (which share the links it
// reads) earlier than for one. FP16, one site : split:
//   18-real: 331776 sites 2 RHS 112 : 105, 4 RHS 197 : 197, 5 RHS 240 : 243, 6 RHS
//     283 : 289, 9 RHS 411 : 428; 65536 sites 13 RHS 127 : 124; 5308416 sites 1 RHS 867 : 851
//   12-real: 1 RHS 786432 sites 129 : 126, 1048576 168 : 166, 5308416 788 : 817; 2 RHS
//     262144 sites 86.7 : 85.3, 331776 107.0 : 106.5, 589824 179 : 185; 3 RHS 262144 sites
//     121.9 : 123.4; 65536 sites 9 RHS 93.1 : 92.8, 10 RHS 101.3 : 102.2
// FP32 is split at any size (the largest, 5308416 sites: 1358 : 1206 and 1109 : 991).
inline bool split_pays(bool bits16, bool link12, long long vh, int nrhs)
{
    if (vh > kSplitMaxSites) return false;
    if (!bits16) return true;
    if (nrhs == 1) return !link12 || vh <= (1 << 20);
    return vh * nrhs <= (link12 ? 5 << 17 : 5 << 18);
}

inline Route default_route(bool f64, bool bits16, bool link12, long long vh, int nrhs)
{
    if (f64) return vh <= kSplitMaxSites ? Route::Split : Route::OneSite;
    if (tiles_pay(bits16, link12, vh, nrhs)) return Route::Tiles;
    return split_pays(bits16, link12, vh, nrhs) ? Route::Split : Route::OneSite;
}

}  // namespace weo
