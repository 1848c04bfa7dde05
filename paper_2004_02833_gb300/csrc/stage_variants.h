// (order, tile x, tile y, tile z, stage buffers, sub-stages per column) variants of the TMA-staged
// kernel, one translation unit each, instantiated for FP32 and BF16 storage where the stage ring fits
// shared memory (the deeper rings fit BF16 only).  The default for a grid is the variant that covers
// it at the least cost (best_variant in kernels_stage.cu), the first listed of equals.  At most one entry per (order, tile, depth).  The
// build reads this list: keep it a single line of X(...) entries.
#pragma once
#define RTPN_STAGE_VARIANTS(X) X(39, 80, 2, 2, 4, 4) X(39, 72, 2, 2, 4, 4) X(39, 64, 2, 2, 5, 4) X(39, 48, 2, 2, 7, 4) X(39, 32, 3, 3, 5, 4) X(39, 40, 2, 2, 2, 1) X(39, 40, 2, 2, 4, 1) X(39, 32, 2, 2, 5, 2) X(39, 32, 2, 2, 3, 1) X(29, 80, 2, 2, 4, 3) X(29, 64, 2, 2, 5, 3) X(29, 32, 3, 3, 5, 3) X(29, 32, 2, 2, 5, 2) X(29, 32, 2, 2, 3, 1) X(29, 40, 2, 2, 2, 1) X(19, 80, 2, 2, 4, 2) X(19, 64, 2, 2, 5, 2) X(19, 48, 2, 2, 4, 2) X(19, 32, 3, 3, 5, 2) X(19, 32, 2, 2, 3, 1) X(19, 40, 2, 2, 2, 1) X(15, 64, 2, 2, 3, 2) X(15, 48, 2, 2, 4, 2) X(15, 96, 2, 2, 4, 2) X(15, 32, 4, 4, 3, 2) X(15, 32, 3, 3, 3, 1) X(15, 32, 2, 2, 3, 1) X(15, 32, 2, 2, 4, 1) X(15, 16, 4, 4, 4, 1) X(7, 64, 2, 2, 3, 1) X(7, 48, 2, 2, 4, 1) X(7, 32, 3, 3, 3, 1) X(7, 32, 2, 2, 4, 1)
