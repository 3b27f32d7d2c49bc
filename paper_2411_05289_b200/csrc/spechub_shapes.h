// CTA shapes of the streaming kernels (the per-method and the three-method kernels of a step take the same ones:
// their results are the same bit for bit).
#pragma once

namespace spechub {

constexpr int kSms = 148;

// Threads per row where the rows do not fill the GPU with CTAs of the shape that is best for many rows: one wave of
// 512 (two per SM) or 256 threads (four per SM).
constexpr int threads_for_few(unsigned rows, int many) {
    if (rows <= 2 * kSms) return 512;
    if (rows <= 4 * kSms) return 256;
    return many;
}
// Draft step and leaf rows: 8 CTAs of 128 threads per SM (64 / 128 / 256 / 512 threads: 0.41 / 0.36 / 0.38 /
// 0.52 ms on V = 128256).  Rows too short to feed those take 64, and so do rows below 40960 ids in more than one wave of
// 64 threads: one warp draws while the others' registers idle, which weighs more the shorter the row and the more draws
// it makes (3584 rows: RRSw V = 16384 44.0 -> 37.9 us, V = 32000 67.7 -> 61.8, SpecHub 58.6 -> 59.1; three drafts, 10240
// rows of 32000 216 -> 199; but V = 65472 106 -> 109, SpecHub 95 -> 105, and 1400 rows of 32000 27.8 -> 31.8).
// words: bf16 rows in whole words, of a draft step.  Short ones in more than a quarter of a wave of one-warp CTAs take
// those: no warp idles while one draws, nothing waits at a barrier (64 / 32 threads, 2500 rows: V = 4096 22.5 / 19.2 us,
// 8192 26.6 / 23.5; 20000 rows: V = 2500 88 / 64, 4096 100 / 76, 8192 121 / 102; but 800 rows of 8192 16.4 / 18.4, 5000 of
// 12000 49 / 51, of 24000 74 / 84: more rows in flight than L2 holds until their draws.  Not fp32 or shifted rows, whose
// passes are longer, and not leaf rows, which are half of a call's: a step on 1300 fp32 rows of 9999 ids 82 / 116).
constexpr int draft_threads(int vocab, unsigned rows, bool words) {
    if (words && vocab < 10240 && rows > 8 * kSms) return 32;
    return vocab < 8192 || (vocab < 40960 && rows > 16 * kSms) ? 64 : threads_for_few(rows, 128);
}
// Verification: 4 CTAs of 256 threads per SM (256/512/1024: 1.54/1.65/1.87 ms on V = 128256); 128 threads on rows too
// short to feed those (V = 8192, 1792 rows: SpecHub 28.6 -> 23.3 us, RRSw 30.7 -> 26.2 us).
// (`per_sm`: threads of these kernels that fit an SM)
constexpr int verify_threads(int vocab, unsigned rows, int per_sm) {
    return rows <= unsigned(per_sm / 512 * kSms) ? 512 : rows <= unsigned(per_sm / 256 * kSms) || vocab >= 16384 ? 256 : 128;
}
// More rows than one wave of the draft step's CTAs of these many threads?  (What that decides: RowPass.)
constexpr bool many_rows(int threads, unsigned rows) { return rows > unsigned(1024 / threads * kSms); }
constexpr int kLeanThreads = 256;   // split rows, and the rings of bulk copies

}  // namespace spechub
