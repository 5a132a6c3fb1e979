// When a launch of the solver's kernel chain may overlap the drain of the one
// before it (launch_chained, internal.h).  Plain host C++ (no CUDA), so that
// the rule is tested without a GPU.
#pragma once

enum ChainKind {
    CHAIN_F64,    // FP64 kernels
    CHAIN_ONE,    // one-slice FP32 / FP16 kernels
    CHAIN_PAIR,   // two-slice kernels
    CHAIN_STREAM  // elementwise FP32 / FP16 kernels
};

// A chained launch's blocks are placed while the blocks before it are still
// resident, so they fill the SMs that those left emptier, and where the two
// launches together need more than one block an SM, some SMs end up with one
// block more than the even share.  Chaining saves the gap between launches (1.5
// to 2.5 us each); the uneven share costs in proportion to how far a kernel is
// bound by its SM's throughput, most where the even share is a full two blocks.
// us per CG iteration on 152 SMs, plain / chained, at the stated lattice (blocks
// per SM):
//   FP64 (bound by the FP64 pipe): 6^2 x 8^2 x 8 (0.47) 220 / 211, 8^4 x 8 (0.84) 220 / 322, 8^4 x 12
//     (1.7) and 10^2 x 12^2 x 5 (3.0) 0.64 and 0.51 of the plain speed: chained only while two
//     launches fit on separate SMs.
//   one slice a thread: FP32 8^4 x 9 (0.84) 67 / 60, 8^2 x 10^2 x 9 (1.3) 0.96 of the plain speed,
//     8^3 x 16 x 9 (1.7) 73 / 81, 12^4 x 7 (2.1) 127 / 120.
//   two slices: FP32 8^4 x 8 (0.57) 50 / 43, 8^3 x 16 x 8 (1.1) 57 / 49, 10^4 x 10 (1.7) and 8 x 10^2 x
//     12 x 12 (2.0) 0.93 of the plain speed, 8^3 x 16 x 24 (3.4) 79 / 74; FP16 8^4 x 8 54 / 49, 8 x
//     10^2 x 12 x 12 0.90 of the plain speed, 8^3 x 16 x 24 84 / 79; between 1.1 and 1.7 blocks 0.92
//     to 1.18 of it from lattice to lattice.
// Grids of more than one wave are plain: the gap does not show there (16^4 x 16:
// FP32 iteration 0.282 ms either way, FP16 0.252 plain and 0.279 chained).
inline bool chain_pays(ChainKind kind, long long blocks, bool one_wave, int sms) {
    if (!one_wave) return false;
    if (kind == CHAIN_F64) return 2 * blocks <= sms;
    if (kind == CHAIN_STREAM) return true;
    return blocks > 2LL * sms || 10 * blocks <= (kind == CHAIN_PAIR ? 17LL : 11LL) * sms;
}
