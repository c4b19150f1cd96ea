// Estimated time of a Lanczos step, for the balance of a batch's lanes (plain C++).
//
// The systems of a batch go longest first to the least loaded lane, so the estimate
// has to rank them and to weigh K_c, near field and vectors against one another.
// Rates measured on GB300 with kernels one after another; beside other lanes all of
// them share the chip, so the terms add up.
#pragma once

struct StepWork {
    long long Nc, N;                 // coarse and dense dimension
    int chains;
    int kc_bytes;                    // of one K_c entry: 16 (FP64 vectors), 8, 4
    int m3;                          // Method 3's near field
    int common;                      // common-basis path: the near field is the scalar stencil
    long long near_offsets;          // of the stencil
    long long near_pieces;           // general path: (dense point, corner) pieces times transitions
};

// Microseconds.  Coarse 8^3, n_div 4, 4x4 bands, 3 chains, BF16 K_c: 64 (K_c) + 84 (stencil) +
// 83 (restrict, prolong, update) + launches; the general path's tensor-core near field 604.
inline double bse_step_us(const StepWork& w) {
    const double entries = (double)w.Nc * w.Nc, values = (double)w.N * w.chains;
    const bool f64 = w.kc_bytes == 16;
    // one pass over K_c at 4.2 MB/us; in FP64 its 8 operations per entry and chain at 1.1 TFLOP/s
    const double kc = f64 ? 8.0 * entries * w.chains / 1.1e6 : entries * w.kc_bytes / 4.2e6;
    // 4 operations per offset and complex value: 19 TFLOP/s in FP32, 1.1 in FP64
    const double stencil = 4.0 * values * w.near_offsets / (f64 ? 1.1e6 : 19e6);
    const double general = 1.1e-6 * w.near_pieces * w.chains * (f64 ? 16.0 : 1.0);
    return kc + (w.m3 ? (w.common ? stencil : general) : 0.0) + values * (f64 ? 160e-6 : 53e-6) + 25.0;
}
