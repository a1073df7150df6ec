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
// (2 targets: 128 registers; 1 target: 80; split in two, 256 threads: 128).
constexpr int kRpyMinBlocksTpt2 = 4;
constexpr int kRpyMinBlocksTpt1 = 6;
constexpr int kRpyMinBlocksSplit2 = 2;
// float4 per two FP32 source records (the packed FP32x2 layout), and per group
// of kRpyComp sources (its centre, then the records)
constexpr int kRpyPairF4 = 9;
constexpr int kRpyGroupF4 = 1 + kRpyPairF4 * kRpyComp / 2;

}  // namespace fil
