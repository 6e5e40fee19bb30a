// Launch shapes by sizes: which of a call's kernels runs, and how its work is
// dealt out.  Plain C++ without CUDA, so that the rules can be tested on any
// host.  The constants are fits to times measured on a GB300; each rule says
// over which sizes.
#pragma once

#include <algorithm>

namespace genesis {

constexpr int kSMs = 152;                   // of a whole GB300

// Blocks of so many bytes of shared memory that an SM's 228 KB hold: each takes
// 1 KB beside its own, which come in steps of 256 bytes.
inline int blocks_by_shared(int bytes) { return 228 * 1024 / ((bytes + 255) / 256 * 256 + 1024); }

// FP32 synthesis and Jacobian: how many chunks of 32 wavelengths of one model
// a warp takes (k_models), or 0 for a thread per (model, wavelength)
// (k_points).  k_models forms a model's geometry once per warp and not once
// per lane, but a chunk's lanes beyond the grid idle and equal shares of the
// models' unequal work are dealt to the warps beforehand; k_points leaves no
// lane idle and its blocks are dealt out as they finish.
//  * Fewer than one and a half rounds of resident warps: k_models, which is
//    the faster or within 15 % there, but for heavy models.
//  * Heavy models (more than 40 Zeeman components): k_points below 448
//    wavelengths (69 components, 30 000 models: 64 wavelengths 473 -> 386 us,
//    129 869 -> 638, 384 level, 512 2314 against 2618).
//  * Otherwise the smaller of the costs of a model: a fit to 1100 times of 600
//    to 30 000 models of 3 to 512 wavelengths and 3 to 15 components, which
//    picks the slower kernel by more than 6 % in 6 of them.  30 000 models,
//    k_models against k_points: two lines, 8 wavelengths 35 -> 13 us, 33
//    wavelengths 46 -> 37, 64 45.7 against 54; full pattern and a line, 33
//    wavelengths 93 -> 62, 97 168 -> 139, 192 233 against 259; Jacobians of
//    two lines, 8 wavelengths 62 -> 43, 33 99 against 117.
// ncomp: Zeeman components of all lines; triplets: one or two effective triplets
// without the fill fraction; blocks_per_sm: k_models's.
inline int chunks_per_warp(bool jac, int n, int nl, int n_lines, int ncomp, bool triplets, int blocks_per_sm)
{
    const int resident = kSMs * blocks_per_sm * 4;  // warps of k_models on the chip
    const int chunks = (nl + 31) / 32;
    if (ncomp > 40) {
        if (nl < 448) return 0;
    } else if ((long long)n * chunks * 2 >= 3ll * resident) {
        // per warp: k_points' and k_models' geometry, the closed form, a component
        const double point_geo = jac ? (triplets ? 0.30 : 0.186 * n_lines) : triplets ? 0.052 : 0.0276 * n_lines;
        const double model_geo = jac ? (triplets ? 0.02 : 0.063 * n_lines) : triplets ? 0.032 : 0.021 * n_lines;
        const double closed = jac ? (triplets ? 0.125 : 0.055) : triplets ? 0.012 : 0.0;
        const double comp = jac ? (triplets ? 0.0145 : 0.0212) : triplets ? 0.0092 : 0.0133;
        const double chunk = closed + comp * ncomp;
        if (nl / 32.0 * (point_geo + chunk) < model_geo + chunks * chunk) return 0;
    }
    // the split whose busiest warp has the least to do, the geometry counted in chunks
    const double geometry = jac ? 0.2 : 0.8;
    int per = 1;
    double least = 1e300;
    for (int c = 1; c <= chunks; ++c) {
        const long long items = (long long)n * ((chunks + c - 1) / c);
        const double t = (double)((items + resident - 1) / resident) * (geometry + c);
        if (t < least) {
            least = t;
            per = c;
        }
    }
    return per;
}

// Warps of a kernel of so many registers per thread that fit an SM, in steps of
// four (one to each partition) and no more than a block can have.
inline int resident_warps(int regs) { return std::min(32, 65536 / ((regs + 7) / 8 * 8 * 32)) / 4 * 4; }

// GA: threads per individual (segments) for npix pixels; 1 = no split.
//  * As many as keep an SM's share of the pixels within the warps its
//    registers hold: with few pixels an SM holds only a few warps and the
//    fitness loop is a chain of dependent operations.  FP64 takes a power of
//    two, so that the eight shares of an individual's wavelengths divide
//    evenly.
//  * A split block does more work for the same pixels (each segment forms the
//    geometry, one breeds), which only costs where `others`, the warps that
//    other launches bring meanwhile, fill the GPU twice over: a burst of 24
//    serving requests took 325 ms with each split as if it ran alone and takes
//    300 ms with this rule, while four requests that just fill the GPU take 24
//    ms split, 28 ms unsplit and 48 ms with the first alone split.
//  * An FP32 split block also holds a float per pair of wavelengths and
//    individual, so on wide grids fewer blocks fit an SM and the pixels take
//    turns.  A round of w resident warps, rounded up to the four partitions of
//    an SM, takes max(10, w + 4) units for a warp's work (two lines, population
//    128, 256 wavelengths, 1 to 7 blocks to an SM: 952, 1161, 1524, 1886, 2682
//    and 3063 us at 4, 8, 12, 16, 24 and 28 warps); its work is its pairs and
//    four more for what every segment does.  Where the split blocks do not all
//    fit, the split runs if its rounds take less than those without: of 301
//    measured sizes (111 to 512 wavelengths, populations 32 to 160, 1 to 14
//    pixels to an SM) the slower side is picked by more than 5 % for 4, at most
//    10 %.  Population 128, 456 pixels: 384 wavelengths 2606 us split, 2061
//    not, 512 wavelengths 3414 and 2689; population 64: 1064 pixels, 192
//    wavelengths 1296 and 1448, 608 pixels, 128 wavelengths 536 and 599.
// shared_split, shared_plain: bytes of a block with and without the split.
inline int ga_segments(int npix, int npop, int nl, int regs, bool fp64, int shared_split, int shared_plain,
                       long long others)
{
    const int room = resident_warps(regs), per_sm = (npix + kSMs - 1) / kSMs, each = npop / 32;
    if (others >= 2ll * 28 * kSMs) return 1;
    int s = room / (per_sm * each);
    if (fp64) return s >= 8 ? 8 : s >= 4 ? 4 : s >= 2 ? 2 : 1;
    const int npair = (nl + 1) / 2;
    s = std::min(s, npair);
    if (s < 2) return 1;
    auto fit = [&](int warps, int shared) { return std::max(1, std::min(room / warps, blocks_by_shared(shared))); };
    if (per_sm <= fit(s * each, shared_split)) return s;  // no turns
    auto rounds = [&](int warps, int shared) -> long long {
        const int f = fit(warps, shared), rest = per_sm % f;
        auto round = [](int w) { return w ? std::max(10, (w + 3) / 4 * 4 + 4) : 0; };
        return per_sm / f * round(f * warps) + round(rest * warps);
    };
    const long long split = rounds(s * each, shared_split) * ((npair + s - 1) / s + 4);
    return split < rounds(each, shared_plain) * (npair + 4) ? s : 1;
}

// Line centres: lanes per pixel (32, 8, 2 or 1; 32 / lanes pixels to a one-warp
// block), for n pixels, candidates search positions of 2 W differences and
// elem bytes of shared memory per staged sample.  More lanes shorten a warp's
// chain of dependent sums and the rows it stages, fewer leave no lane idle in
// a ragged last round and start fewer blocks.  The time of a choice is modelled
// as the longer of the chains, one after another where shared memory admits R
// blocks to an SM, and of the SM's issue, plus 0.3 of the other; fitted to 800
// measured calls (1 to 70 000 pixels, 7 to 510 candidates, W = 1, 10, 40,
// float and double), of which it picks a shape more than 1.1 times slower than
// the best for 3.  Lanes by the number of pixels alone took up to ten times the
// best: 70 000 pixels over a whole grid of 512 wavelengths, W = 10, float 1969
// -> 234 us (8.4 x), double 6610 -> 1474 us.
inline int centre_lanes(bool integers, int n, int candidates, int W, int elem)
{
    // in units of one term of a chain: a term's issue, a staged row of 32 samples and its issue, a block's start
    const double term = integers ? 0.018 : 0.265, row = integers ? 3.66 : 1.11;
    const double row_issue = integers ? 0.012 : 0.126, start = integers ? 4.04 : 0.735;
    int best = 1;
    double least = 1e300;
    for (int lanes : {32, 8, 2, 1}) {
        const int pixels = 32 / lanes, span = candidates + 2 * W;
        const double per_sm = (double)(((long long)n * lanes + 31) / 32) / kSMs;
        const int resident = std::max(1, std::min(32, blocks_by_shared(pixels * (span | 1) * elem)));
        const double terms = (double)((candidates + lanes - 1) / lanes + (lanes == 1 ? 2 : 1)) * W;
        const double rows = (double)pixels * ((span + 31) / 32);
        const double chains = std::max(1.0, per_sm / resident) * (terms + row * rows);
        const double issue = per_sm * (term * terms + row_issue * rows + start);
        const double t = std::max(chains, issue) + 0.3 * std::min(chains, issue);
        if (t < least) {
            least = t;
            best = lanes;
        }
    }
    return best;
}

// FP64 synthesis: blocks per model (k_synth64, whose passes of 128 wavelengths
// they share), or 0 for a thread per (model, wavelength) (k_points).
//  * A block works for one model, so on a few wavelengths most of its time goes
//    into the model's tables; from 2000 models of up to 12 wavelengths on (6
//    with more than 40 components) threads of their own are faster: 20 000
//    models, one line, 3 wavelengths 326 -> 66 us, 8 339 -> 143, 16 362 -> 269;
//    two lines, 12 wavelengths 434 -> 352, 16 462 against 460; four full
//    patterns, 6 wavelengths 2802 -> 1797, 12 3257 against 3309.  Below 2000
//    models a block each is faster (600 models of 8 wavelengths 16.5 against
//    20.9 us).
//  * Up to 152 models each get a block per pass, so that the passes run side by
//    side: a call for one model, one line, 257 wavelengths 31.2 -> 17.7 us, 512
//    43.6 -> 17.3, two lines 64 -> 23; 150 models of 512 wavelengths 46 -> 37,
//    but 600 107 against 128 (every block builds the model's tables).
inline int blocks_per_model64(int n, int nl, int ncomp, int pass)
{
    if (n >= 2000 && nl <= (ncomp > 40 ? 6 : 12)) return 0;
    return n <= kSMs ? (nl + pass - 1) / pass : 1;
}

}  // namespace genesis
