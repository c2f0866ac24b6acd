// FFT lengths of the derivative passes for axis lengths without a plan of their
// own (conv_pass.cuh): X(len, R1, R2, R3, T, pairs) runs axes of up to len / 2
// cells as a convolution through an FFT of len points, the smallest that fits
// being taken; T threads per pencil pair, `pairs` pairs per tile row (narrower
// tiles for the long ones, so that several CTAs fit on an SM).
#pragma once

#define ES_CONV_PLANS(X)                                                                            \
    X(160, 16, 10, 1, 10, 16)                                                                       \
    X(256, 16, 16, 1, 16, 16)                                                                       \
    X(320, 20, 16, 1, 20, 8)                                                                        \
    X(400, 20, 20, 1, 20, 8)                                                                        \
    X(500, 25, 20, 1, 25, 8)                                                                        \
    X(625, 25, 25, 1, 25, 8)                                                                        \
    X(1024, 16, 8, 8, 64, 8)
