// Tile shapes of the RPY pair kernels (shared by the launcher and the kernels).
#pragma once

namespace fil {

// ----------------------------------------------------------------------------
// RPY pair-kernel geometry (tuned on GB300 at 32 000 segments).
// ----------------------------------------------------------------------------
constexpr int kRpyThreads = 128;               // threads per CTA
constexpr int kRpyUnroll = 16;                 // unroll of the per-source loop
constexpr int kRpyTargetsPerThread = 2;        // register-blocked targets
constexpr int kRpyTile = kRpyThreads * kRpyTargetsPerThread;   // targets per tile
constexpr int kRpyMinTile = 64;                // targets per tile of the warp kernel
constexpr int kRpyChunk = 128;                 // sources per shared-memory chunk
constexpr int kRpyComp = 32;                   // sources per compensated partial (FP32)
// Resident CTAs per SM the FP32 pair kernels are compiled for, by targets per
// thread and source split: caps the registers so that this many CTAs fit
// (2 targets: 168 registers, 3 CTAs; 1 target: 96 registers, 5 CTAs; split in
// two: 2 CTAs of 256 threads, 128 registers).
constexpr int kRpyMinBlocksTpt2 = 3;
constexpr int kRpyMinBlocksTpt1 = 5;
constexpr int kRpyMinBlocksSplit2 = 2;
// Most CTAs per SM a schedule of the FP32 kernels may ask for (grids larger
// than the residency run in more than one wave).
constexpr int kRpyMaxCtasTpt2 = 4;
constexpr int kRpyMaxCtasTpt1 = 6;
constexpr int kRpyMaxCtasSplit2 = 2;
// float4 per two FP32 source records (the packed FP32x2 layout), and per group
// of kRpyComp sources (its centre, then the records)
constexpr int kRpyPairF4 = 9;
constexpr int kRpyGroupF4 = 1 + kRpyPairF4 * kRpyComp / 2;

}  // namespace fil
