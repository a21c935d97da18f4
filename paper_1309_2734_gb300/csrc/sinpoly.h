// Generated by gen_sinpoly.py; do not edit.
// sin(2 pi d) = d (S0 + S1 u + ... + S4 u^4), u = d^2, |d| <= 1/4.
// Fit error 3.3e-09; RMS error of a turn's entries in single precision 2.77e-08 (3.68e-08 as rounded).
#pragma once
#define CGH_SIN_0 6.283185005187988f
#define CGH_SIN_1 -41.341651916503906f
#define CGH_SIN_2 81.60100555419922f
#define CGH_SIN_3 -76.54976654052734f
#define CGH_SIN_4 39.53668975830078f
