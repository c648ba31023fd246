// Rules by which a launch takes one form of a kernel or another: plain functions of sizes and counts, without CUDA, so
// that the lines they draw can be checked on any machine.
#pragma once

#ifdef __CUDACC__
#define SSVP_HD __host__ __device__
#else
#define SSVP_HD
#endif

namespace ssvp {

// Whether a frustum gather takes the instance that can drop whole blocks of a long hull.  Hulls grow with the image
// and with the distance of the window's frames, and only long ones gain; the instance without it spills next to
// nothing (with it 230 to 280 bytes a thread).  side: the image's longer side; band: the hull's width in input pixels; a
// band of one or two pixels has few candidates to drop, in a wide one few blocks can be dropped.  Both sides, in ms with
// and without:
//   band 3     960 x 540 +-15 1.73, 1.73; 720p +-15 3.21, 3.44; 640 x 360 +-30 1.80, 1.94; 720p +-30 8.15, 11.2;
//              1080p +-30 20.5, 33.6
//   band 9     640 x 360 +-30 6.71, 6.13; 1080p +-15 28.4, 29.9; 6: 720p +-15 6.77, 6.82
//   band 1     720p +-15 1.85, 1.65; 1080p +-15 4.84, 4.58; 720p +-30 4.97, 5.35
//   super-resolution: x 3 of 640 x 360, +-30 (band 0.3, 1) 6.18, 4.39 and 7.58, 6.89; x 2 of 720p, +-15 (0.5, 1.5) 5.93,
//              4.51 and 7.82, 7.62, +-30 16.7, 14.8 and 20.2, 25.3; x 2 of 640 x 360, +-60 (1.5) 10.6, 13.2
// A rule on the whole image and the window, not on the crop: the two sum in different orders.
inline bool frustum_long_hulls(int n_slots, int side, float band) {
    return (long long)n_slots * side >= (band < 1.0f ? 100000 : band < 2.0f ? 70000 : band < 5.0f ? 35000 : 50000);
}

// Whether each pixel's window frames are shared out to four threads, where one thread a pixel fills the chip badly.
// ctas: CTAs of 32 x 8 pixels with one thread a pixel; wave: how many are resident at once.  Four threads cost four
// times the CTAs, each with its own set-up, and with few frames some threads have none, so the fuller the chip the
// longer the window has to be.

// Frustum gather, us with one thread and with four (l = 3): 96 x 54 (0.05 waves) +-1 16.3, 13.4 (super-resolution x 2);
// 320 x 180 (0.5) 0 20.6, 28, +-1 31, 30, +-2 40, 37 (l = 9 118, 108); 480 x 270 (1.1) +-1 48, 53, +-2 70, 75, +-3 92, 85, +-15 450, 378;
// 640 x 360 (2.0) +-3 118, 134, +-8 306, 343, +-15 694, 700
SSVP_HD inline bool frustum_shares(long long ctas, long long wave, int n_slots) {
    return (n_slots >= 3 && 4 * ctas <= wave) || (n_slots >= 5 && 5 * ctas <= 3 * wave) || (n_slots >= 7 && 2 * ctas < 3 * wave);
}

// Window gather, us with one thread and with four (k = 7, and k = 3 where named): 96 x 54 (0.03 waves) 0 13.5, 13.4, +-1
// 17.3, 13.4; 320 x 180 (0.4) 0 16.9, 19.6, +-1 23.6, 21.2, +-15 120, 71; 480 x 270 (0.8) 0 21.8, 31.2, +-2 42.9, 45.7,
// +-3 51.9, 51.3, k = 3 +-2 28.7, 34.0; 560 x 316 (1.2) +-2 59.4, 57.7, +-3 75.8, 64.3, +-5 108, 85, k = 3 +-5 53.7,
// 51.8; 640 x 360 (1.5) +-2 60.3, 65.4, +-3 79.1, 75.1, +-15 321, 262, k = 3 +-5 54.6, 58.4, +-15 147, 133; 853 x 479
// (2.7) +-8 284, 284, k = 3 135, 151; 720p (5.9) +-15 949, 986
SSVP_HD inline bool window_shares(long long ctas, long long wave, int n_slots, int k) {
    return (n_slots >= 3 && 2 * ctas <= wave) || (n_slots >= 7 && ctas < wave) || (n_slots >= 7 && n_slots * k >= 49 && 2 * ctas < 3 * wave) ||
           (n_slots >= 16 && 2 * ctas < 5 * wave);
}

// Virtual aperture, us with one thread and with four (FP32 colour): 320 x 180 (0.4 waves) 0 29.9, 41.3, +-1 62.9, 48.7,
// +-2 95, 79; 640 x 360 (1.5) 0 64.4, 119, +-1 157, 147, +-2 249, 251, +-3 344, 285, +-15 1543, 1153; 853 x 479 (2.7) 0 110,
// 223, +-1 268, 274, +-2 426, 463, +-3 602, 551, +-15 2616, 2190; FP16: 853 x 479 (3.6) +-2 390, 441, +-15 2441, 2096.
// Where the chip is full already the frames have to divide well: five leave three of four threads idle half the time.
SSVP_HD inline bool aperture_shares(long long ctas, long long wave, int n_slots) {
    const int full = 4 * ((n_slots + 3) / 4);
    return n_slots >= 3 && (ctas <= wave || (ctas < 3 * wave && 3 * n_slots >= 2 * full));
}

// Extraction of the learned filter's sets: four CTAs an SM where that is one wave and three an SM are not (figures at
// kLearnCtas)
SSVP_HD inline bool extract_four_ctas(long long ctas, int sms) { return ctas > 3ll * sms && ctas <= 4ll * sms; }

}  // namespace ssvp
