// mr_lengths.h -- every length the composite-radix line passes are compiled
// for: the 2^a 3^b 5^c from 3 to 4096 that are not a power of two, in two
// halves (one translation unit each per layout and direction), and the powers of
// two whose contiguous or strided lines they take too (pow2_on_mr).
#pragma once

#define FB_MR_LENGTHS_A(K) \
    K(3) K(5) K(6) K(9) K(10) K(12) K(15) K(18) K(20) K(24) K(25) K(27) K(30) K(36) K(40) K(45) K(48) K(50) \
    K(54) K(60) K(72) K(75) K(80) K(81) K(90) K(96) K(100) K(108) K(120) K(125) K(135) K(144) K(150) K(160) \
    K(162) K(180) K(192) K(200) K(216) K(225) K(240) K(243) K(250) K(270) K(288) K(300) K(320) K(324) K(360) \
    K(375) K(384) K(400) K(405) K(432) K(450) K(480) K(486) K(500) K(540) K(576) K(600) K(625)

#define FB_MR_LENGTHS_B(K) \
    K(640) K(648) K(675) K(720) K(729) K(750) K(768) K(800) K(810) K(864) K(900) K(960) K(972) K(1000) \
    K(1080) K(1125) K(1152) K(1200) K(1215) K(1250) K(1280) K(1296) K(1350) K(1440) K(1458) K(1500) K(1536) \
    K(1600) K(1620) K(1728) K(1800) K(1875) K(1920) K(1944) K(2000) K(2025) K(2160) K(2187) K(2250) K(2304) \
    K(2400) K(2430) K(2500) K(2560) K(2592) K(2700) K(2880) K(2916) K(3000) K(3072) K(3125) K(3200) K(3240) \
    K(3375) K(3456) K(3600) K(3645) K(3750) K(3840) K(3888) K(4000) K(4050)

#define FB_MR_POW2_NN(K) K(64) K(128) K(256) K(512) K(1024) K(2048) K(4096)
#define FB_MR_POW2_CC(K) K(64) K(128)
