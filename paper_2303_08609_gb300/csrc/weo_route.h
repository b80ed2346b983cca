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

// FP64: hop_kernel_rows (16-site CTAs) in the place of hop_kernel_pairs (32 sites). Both
// are bound by the FP64 pipe of each of the 152 SMs, so what counts is how many CTAs the
// fullest SM gets: an odd number of 16-site ones is less work for it than the next 32-site
// one, until the rows' 3 to 6 % of overhead outweigh the half CTA saved; with 12-real
// links both half-warps rebuild the third row, which costs more. Rows : pairs, us per
// M_eo, by 16-site CTAs per SM:
//   18-real: 1 8^4 15.2 : 18.3; 2 8^3 x 16 22.6 : 18.7, 8^4 2 RHS 22.2 : 18.6; 3 8^4 3 RHS
//     28.0 : 32.8; 4 10x6x14x18 35.2 : 33.2; 6 8^3 x 12 4 RHS 49.5 : 47.5; 7 8^3 x 16 4 RHS
//     57.5 : 62.1; 11 8^4 12 RHS 87.6 : 90.0; 13 10x6x14x18 4 RHS 103 : 105; 38 293 : 279
//   12-real: 1 8^4 19.9 : 21.5; 2 8^3 x 12 24.8 : 21.7; 3 8^4 3 RHS 37.4 : 39.6; 4 46.6 : 39.7;
//     7 8^3 x 16 4 RHS 78.8 : 75.2; 11 8^4 12 RHS 121 : 109
inline bool rows_pay(bool link12, long long vh, int nrhs)
{
    const long long per_sm = ((vh + 15) / 16 * nrhs + 151) / 152;
    return per_sm % 2 == 1 && per_sm <= (link12 ? 3 : 7);
}

// The handle's 2x2x2 blocks of rows have CTAs of 8 Lx/2 threads, 64 to 256 of them; on
// another lattice the setting changes nothing.
inline bool site_blocks_apply(bool asked, int lxh) { return asked && 8 * lxh >= 64 && 8 * lxh <= 256; }

inline Route default_route(bool f64, bool bits16, bool link12, long long vh, int nrhs)
{
    if (f64) return vh <= kSplitMaxSites ? Route::Split : Route::OneSite;
    if (tiles_pay(bits16, link12, vh, nrhs)) return Route::Tiles;
    return split_pays(bits16, link12, vh, nrhs) ? Route::Split : Route::OneSite;
}

// whether the handle's threads per CTA reach the default kernel: the others have CTAs
// of one size
inline bool threads_matter(bool f64, bool bits16, bool link12, long long vh, int nrhs)
{
    return default_route(f64, bits16, link12, vh, nrhs) == Route::OneSite;
}

}  // namespace weo
