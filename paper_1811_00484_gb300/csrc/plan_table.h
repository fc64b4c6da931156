// Factor plans of the padded edges N = 2n with 16 <= N <= 512 (every 7-smooth
// even N there but 490 = 2 5 7 7, whose factor pairs need a 35-point radix):
//   X(N, Q1, Q2, R1, R2, R3)
// Q1 Q2 = N for the line stages (Q1 even: the radix the zero padding and the
// crop are pruned from), R1 R2 R3 = N for the fused stage.  The line radices are
// as equal as N allows: unequal ones leave threads of the other pass idle (N =
// 128, 3 x 128 x 64 lines: 16 x 8 6.4 us, 32 x 4 15.9 us; N = 192, 96^3 with 16
// right-hand sides: 16 x 12 206 us, 24 x 8 379 us).  The fused stage takes two
// passes up to 256 and three beyond, where two would not fit the registers (N =
// 120, 100 x 144 lines: 10 x 12 20.2 us, 6 x 5 x 4 28.7 us; N = 256, two right-hand
// sides: 16 x 16 353 us, 8 x 8 x 4 446 us; N = 320: 20 x 16 541 us, 8 x 8 x 5 469 us);
// each pair's order is the faster one measured (N = 192, 96^3 with 16 right-hand
// sides: 12 x 16 1018 us, 16 x 12 1120 us, 24 x 8 1224 us).
// The sets only spread the compilation over translation units.
#define VIE_PLAN_SET_0(X) \
  X(16, 4, 4, 4, 4, 1) \
  X(84, 12, 7, 7, 12, 1) \
  X(90, 10, 9, 10, 9, 1) \
  X(210, 14, 15, 14, 15, 1) \
  X(216, 18, 12, 18, 12, 1) \
  X(400, 20, 20, 8, 10, 5) \
  X(420, 20, 21, 10, 7, 6)
#define VIE_PLAN_SET_1(X) \
  X(18, 6, 3, 6, 3, 1) \
  X(80, 10, 8, 10, 8, 1) \
  X(96, 12, 8, 8, 12, 1) \
  X(200, 20, 10, 20, 10, 1) \
  X(224, 16, 14, 14, 16, 1) \
  X(392, 14, 28, 8, 7, 7) \
  X(432, 24, 18, 8, 9, 6)
#define VIE_PLAN_SET_2(X) \
  X(20, 4, 5, 4, 5, 1) \
  X(72, 8, 9, 8, 9, 1) \
  X(98, 14, 7, 14, 7, 1) \
  X(196, 14, 14, 14, 14, 1) \
  X(240, 16, 15, 15, 16, 1) \
  X(384, 24, 16, 8, 8, 6) \
  X(448, 16, 28, 8, 8, 7)
#define VIE_PLAN_SET_3(X) \
  X(24, 6, 4, 6, 4, 1) \
  X(70, 10, 7, 7, 10, 1) \
  X(100, 10, 10, 10, 10, 1) \
  X(192, 16, 12, 12, 16, 1) \
  X(250, 10, 25, 10, 5, 5) \
  X(378, 18, 21, 6, 9, 7) \
  X(450, 18, 25, 10, 9, 5)
#define VIE_PLAN_SET_4(X) \
  X(28, 4, 7, 4, 7, 1) \
  X(64, 8, 8, 8, 8, 1) \
  X(108, 12, 9, 9, 12, 1) \
  X(180, 12, 15, 15, 12, 1) \
  X(252, 18, 14, 18, 14, 1) \
  X(360, 20, 18, 10, 6, 6) \
  X(480, 24, 20, 8, 10, 6)
#define VIE_PLAN_SET_5(X) \
  X(30, 6, 5, 6, 5, 1) \
  X(60, 10, 6, 6, 10, 1) \
  X(112, 14, 8, 14, 8, 1) \
  X(168, 14, 12, 14, 12, 1) \
  X(256, 16, 16, 16, 16, 1) \
  X(350, 14, 25, 10, 7, 5) \
  X(486, 18, 27, 6, 9, 9)
#define VIE_PLAN_SET_6(X) \
  X(32, 8, 4, 8, 4, 1) \
  X(56, 8, 7, 8, 7, 1) \
  X(120, 12, 10, 10, 12, 1) \
  X(162, 18, 9, 18, 9, 1) \
  X(270, 18, 15, 6, 9, 5) \
  X(336, 16, 21, 8, 7, 6) \
  X(500, 20, 25, 10, 10, 5)
#define VIE_PLAN_SET_7(X) \
  X(36, 6, 6, 6, 6, 1) \
  X(54, 6, 9, 6, 9, 1) \
  X(126, 14, 9, 14, 9, 1) \
  X(160, 16, 10, 16, 10, 1) \
  X(280, 20, 14, 8, 7, 5) \
  X(324, 18, 18, 6, 9, 6) \
  X(504, 24, 21, 8, 9, 7)
#define VIE_PLAN_SET_8(X) \
  X(40, 8, 5, 8, 5, 1) \
  X(50, 10, 5, 10, 5, 1) \
  X(128, 16, 8, 16, 8, 1) \
  X(150, 10, 15, 15, 10, 1) \
  X(288, 18, 16, 8, 6, 6) \
  X(320, 20, 16, 8, 8, 5) \
  X(512, 32, 16, 8, 8, 8)
#define VIE_PLAN_SET_9(X) \
  X(42, 6, 7, 6, 7, 1) \
  X(48, 8, 6, 8, 6, 1) \
  X(140, 14, 10, 14, 10, 1) \
  X(144, 12, 12, 12, 12, 1) \
  X(294, 14, 21, 6, 7, 7) \
  X(300, 20, 15, 10, 6, 5)
