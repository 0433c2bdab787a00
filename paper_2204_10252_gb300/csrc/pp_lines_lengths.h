// (n, N1, N2) of the lengths with compiled two-factor FFT kernels, n = N1 N2.  The
// build compiles pp_lines_unit.cu and pp_cart_unit.cu once for each entry, so that
// every length is a module of its own: the driver loads a module, with all that is in
// it, when the first of its kernels is launched.  In four modules of 6 to 20 lengths
// that first launch took 11 to 15 ms.
#pragma once

// row and column stages (pp_lines.cuh)
#define PP_LINE_LENGTHS(X) \
    X(16, 4, 4) X(18, 3, 6) X(20, 4, 5) X(24, 4, 6) X(30, 5, 6) X(32, 4, 8) X(36, 6, 6) \
    X(40, 5, 8) X(48, 6, 8) X(50, 5, 10) X(54, 6, 9) X(60, 6, 10) X(64, 8, 8) X(72, 8, 9) \
    X(80, 8, 10) X(90, 9, 10) X(96, 8, 12) X(100, 10, 10) X(108, 9, 12) X(120, 10, 12) \
    X(128, 8, 16) X(144, 12, 12) X(150, 10, 15) X(160, 10, 16) X(162, 9, 18) X(180, 12, 15) \
    X(192, 12, 16) X(200, 10, 20) X(216, 12, 18) X(240, 15, 16) X(250, 10, 25) X(256, 16, 16) \
    X(270, 15, 18) X(288, 16, 18) X(300, 15, 20) X(320, 16, 20) X(324, 18, 18) X(360, 18, 20) \
    X(384, 16, 24) X(400, 20, 20) X(432, 18, 24) X(450, 18, 25) X(480, 20, 24) X(486, 18, 27) \
    X(500, 20, 25) X(512, 16, 32) X(540, 20, 27) X(576, 24, 24) X(600, 24, 25) X(640, 20, 32) \
    X(648, 24, 27) X(720, 24, 30) X(750, 25, 30) X(768, 24, 32) X(800, 25, 32) X(810, 27, 30) \
    X(864, 27, 32) X(900, 30, 30) X(960, 30, 32) X(1024, 32, 32)

// column-resident Cartesian chains (pp_cart_cols.cuh)
#define PP_CART_LENGTHS(X) \
    X(32, 4, 8) X(36, 6, 6) X(40, 5, 8) X(48, 6, 8) X(60, 6, 10) X(64, 8, 8) X(72, 8, 9) \
    X(80, 8, 10) X(96, 8, 12) X(100, 10, 10) X(108, 9, 12) X(120, 10, 12) X(128, 8, 16) \
    X(144, 12, 12) X(160, 10, 16) X(180, 12, 15) X(192, 12, 16) X(200, 10, 20) X(216, 12, 18) \
    X(240, 15, 16) X(256, 16, 16) X(288, 16, 18) X(300, 15, 20) X(320, 16, 20) X(324, 18, 18) \
    X(360, 18, 20) X(384, 16, 24) X(400, 20, 20) X(432, 18, 24) X(480, 20, 24) X(500, 20, 25) \
    X(512, 16, 32)
