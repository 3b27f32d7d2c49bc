// CTA shapes of the large-vocabulary kernels (the per-method and the three-method kernels of a step take the
// same ones: their results are the same bit for bit).
#pragma once

namespace spechub {

// Draft step and leaf rows: 8 CTAs of 128 threads per SM (64 / 128 / 256 / 512 threads: 0.41 / 0.36 / 0.38 /
// 0.52 ms on V = 128256; 0.078 / 0.081 / 0.102 / 0.165 ms on V = 32000).
constexpr int kLeanDraftThreads = 128;
constexpr int kLeanThreads = 256;  // 4 CTAs per SM measured best (256/512/1024: 1.54/1.65/1.87 ms)
// Verification from draft statistics on shorter rows: 8 CTAs of 128 threads per SM overlap the fixed work of
// a row (reductions, tests, draws) better (V = 32000, 3840 rows: SpecHub 0.180 -> 0.158 ms, RRS 0.230 ->
// 0.205 ms; 64 threads: 0.171 ms; on V = 128256 the 256-thread CTA stays ahead, 1.02 against 1.06 ms).
constexpr int kLeanSmallThreads = 128;
constexpr int kLeanSmallVocab = 65536;

}  // namespace spechub
