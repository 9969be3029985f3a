// The lengths that have register line kernels: X(n, R1, R2) with n = R1 R2, R1 <= R2, radices as close
// as the factors allow.  Sixteen neighbouring points per load (R2 = 16) where there is a choice; one
// line per build unit, of about equal compile time.
#pragma once

#define SWF_LINES_0(X) X(32, 4, 8) X(64, 8, 8) X(96, 8, 12) X(128, 8, 16) X(144, 12, 12) X(160, 10, 16) X(192, 12, 16) X(512, 16, 32) X(450, 18, 25) X(40, 5, 8) X(54, 6, 9)
#define SWF_LINES_1(X) X(256, 16, 16) X(240, 15, 16) X(200, 10, 20) X(100, 10, 10) X(120, 10, 12) X(180, 12, 15) X(48, 6, 8) X(80, 8, 10) X(500, 20, 25) X(45, 5, 9) X(72, 8, 9)
#define SWF_LINES_2(X) X(320, 16, 20) X(288, 16, 18) X(360, 18, 20) X(225, 15, 15) X(150, 10, 15) X(108, 9, 12) X(36, 6, 6) X(60, 6, 10) X(375, 15, 25) X(81, 9, 9) X(250, 10, 25)
#define SWF_LINES_3(X) X(384, 16, 24) X(400, 20, 20) X(300, 15, 20) X(216, 12, 18) X(135, 9, 15) X(90, 9, 10) X(50, 5, 10) X(324, 18, 18) X(432, 18, 24) X(75, 5, 15)
#define SWF_LINES_4(X) X(480, 20, 24) X(270, 15, 18) X(162, 9, 18) X(125, 5, 25) X(30, 5, 6)
