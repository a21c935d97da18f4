// Generated by gen_sincospoly.py; do not edit.
// sqrt(2) sin(pi r) = r (S0 + S1 u + ... + S4 u^4) and sqrt(2) cos(pi r) = C0 + C1 u + ... + C4 u^4, u = r^2, |r| <= 1/2.
#pragma once
#define CGH_HSIN_0 4.442883014678955f
#define CGH_HSIN_1 -7.308241844177246f
#define CGH_HSIN_2 3.6062874794006348f
#define CGH_HSIN_3 -0.8457623720169067f
#define CGH_HSIN_4 0.10920922458171844f
#define CGH_HCOS_0 1.4142134189605713f
#define CGH_HCOS_1 -6.978850364685059f
#define CGH_HCOS_2 5.739460468292236f
#define CGH_HCOS_3 -1.8835639953613281f
#define CGH_HCOS_4 0.3106975257396698f
