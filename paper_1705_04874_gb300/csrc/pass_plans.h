// The FFT plans of the derivative passes, one X(n, R1, R2, R3, T) per candidate:
// radices of the stages in order, R3 = 1 for a two-stage plan, and T threads
// per pencil pair, which divides n and deals the butterflies of the stages (n /
// R1, n / R2, ...) as evenly as it can: 96 = 16 x 6 takes 8 threads (6 of them
// for the radix-16 stages, two radix-6 butterflies each), not 6 with three
// butterflies each.  The first candidate of a length is the default, the
// faster one on batches of 17 M cells: the smaller radix first leaves fewer idle
// threads in the stages that run through shared memory (ps per cell, x passes + y and
// z passes of both halves, first and second candidate: 80 25.1 + 60.7 and 27.0 +
// 63.7, 96 24.9 + 45.5 and 25.1 + 48.6, 128 22.6 + 42.0 and 23.5 + 42.1, 192 26.1 +
// 48.0 and 26.8 + 50.9; 160 the other way, 26.3 + 46.6 and 26.1 + 50.9).
// es_model_autotune may pick another.  Through the C ABI a plan is named (R1, n /
// R1).  Every radix has a register DFT in fft_pass.cuh (2, 3, 4, 5, 6, 8, 10, 12,
// 15, 16, 25).
#pragma once

#define ES_PLANS(X)                                                                                  \
    X(16, 4, 4, 1, 4)                                                                                \
    X(32, 8, 4, 1, 4) X(32, 4, 8, 1, 4)                                                              \
    X(48, 12, 4, 1, 4) X(48, 4, 12, 1, 4)                                                            \
    X(64, 16, 4, 1, 4) X(64, 8, 8, 1, 8) X(64, 4, 16, 1, 4)                                          \
    X(75, 5, 15, 1, 5)  X(75, 3, 5, 5, 25) X(75, 15, 5, 1, 5)                                        \
    X(80, 5, 16, 1, 8) X(80, 16, 5, 1, 8)                                                            \
    X(96, 6, 16, 1, 8) X(96, 16, 6, 1, 8)                                                            \
    X(125, 5, 5, 5, 25) X(125, 25, 5, 1, 5)                                                          \
    X(128, 8, 16, 1, 8) X(128, 16, 8, 1, 8)                                                          \
    X(160, 16, 10, 1, 10) X(160, 10, 16, 1, 16)                                                      \
    X(192, 12, 16, 1, 16) X(192, 16, 12, 1, 16)                                                      \
    X(256, 16, 16, 1, 16)
