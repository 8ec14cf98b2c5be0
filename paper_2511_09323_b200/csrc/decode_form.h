// Which plan and form a decode call takes, where more than one serves it: rules on sizes.  Host code only, free of CUDA.
#pragma once

#include <cmath>
#include <cstdint>

namespace moc {

constexpr int kGateRows = 64;  // rows of W_gate that a CTA of the gathering plan takes at most, two CTAs to an SM

// Which form of the small-batch plan a decode call takes (Top-K mask, no block form).  us per call over three sets of weights, three
// kernels | four, overlapped | one: 6 and 32 tokens of 768 x 2048 18.3 20.0 | 20.3 22.4 | 26.7 28.7, of 2048 x 5504 30.4 33.3 | 31.4
// 34.8 | 34.9 38.8, of 2560 x 6912 36.0 38.0 | 35.9 39.6 | 39.2 43.3; of 3072 x 8192 43.4 46.2 | 41.9 45.9 | 44.3 48.4, of 4096 x 11008
// 62.9 66.3 | 58.5 61.5 | 59.9 66.0, of 4096 x 16384 83.9 88.0 | 74.7 83.3 | 83.9 89.1; 12 and 24 tokens of 5120 x 20480 142 144 | 111 114
// | 110 122.  More than 32 tokens, three | four: 36 of 3072 x 8192 46.7 | 46.6 and 44 46.9 | 48.4, 44 of 4096 x 11008 68.1 | 66.1 and 52
// 69.0 | 69.5, 48 of 4608 x 12288 79.7 | 78.5.  The overlapped form's last CTA takes channels one by one where they do not come in
// fours: 24 tokens of 5120 x 13653 87.5 | 92.1 | 84.3, of 3584 x 9557 55.4 | 60.2 | 54.9.
// Up to 16 tokens, four | one.  Layers wider than 4224: within 2 % of one another where the rows are whole lines (12 of 4608 x 12288 67.8 |
// 68.7, 16 of 5120 x 13824 80.1 | 80.7, 6 of 8192 x 21888 174.8 | 169.3), the one kernel ahead where they are not (6 and 14 of 4328 x
// 11520 68.0 67.1 | 63.1 65.4, 12 of 4776 x 12736 78.0 | 75.7).  Narrower ones whose rows are not whole 32-byte sectors, 8/3 of the width
// in channels: 6 of 3592 x 9580 55.0 | 52.4, 10 of 4008 x 10688 62.3 | 58.0, 6, 14 and 16 of 4104 x 10944 65.2 65.6 62.2 | 61.5 63.7
// 62.4, 4, 6 and 16 of 3080 x 8216 45.8 46.7 46.6 | 46.8 45.5 46.0; four times the width: 10 of 3592 x 14368 69.3 | 74.1.
enum class SmallBatchForm { kOne, kThree, kOverlapped };
inline SmallBatchForm small_batch_form(int tokens, int d_model, int d_ff, int sms) {
    const int64_t weights = (int64_t)d_model * d_ff;  // of one matrix
    const bool fours = d_ff % 4 == 0;
    if (weights < 300'000) return SmallBatchForm::kOne;  // (fewer than any that was measured)
    if (weights < (fours ? 18'000'000 : 25'000'000)) return SmallBatchForm::kThree;
    if (!fours || sms < 96 || tokens > (weights < 30'000'000 ? 32 : 44)) return SmallBatchForm::kOne;  // (three kernels beyond its 32 tokens)
    if (tokens <= 16 && d_model > 4224) return SmallBatchForm::kOne;
    if (tokens <= (weights < 45'000'000 ? 16 : 14) && d_model % 16 != 0 && d_ff < 3 * d_model && weights >= 28'000'000) return SmallBatchForm::kOne;
    return SmallBatchForm::kOverlapped;
}

// Three to five tokens (Top-K, no block form) for which the gathering plan reads fewer bytes, (1 + 2 u) d F elements against 3 d F with
// a share u of the channels in use: the forms that stream all three matrices have fewer hand-overs and are faster all the same on
//  - layers below 30 million weights of a matrix (25 where the channels do not come in fours: no overlapped form), but from 25 on only
//    with a tenth of the channels in use; below 40 with 0.3; from 90 on with 0.4;
//  - layers with more channels than the gate kernel takes in one go (18944 on 148 SMs): the CTAs left over run behind the others, at the
//    pace of one CTA to an SM or less.  The plan then takes some 33 + 11.9 d / 1000 + (0.19 + 0.82 u) W us, W being millions of weights,
//    against 18.7 + 0.853 W: within 8 and 5 % of 79 calls measured.
// Gathering plan | streaming forms, us, three tokens: 2048 x 5504, K = F / 8 34.0 | 28.7, F / 64 32.1 | 28.2; 2560 x 9728, F / 8 44.4 |
// 39.1, F / 64 40.1 | 38.6; 3072 x 8192, F / 8 44.4 | 41.2, F / 16 41.0 | 40.8, F / 32 39.7 | 40.8; 2560 x 11520, F / 16 43.4 | 42.8, F / 64
// 41.1 | 42.6; 4096 x 9728, F / 8 55.0 | 53.3; 4096 x 11008, F / 8 57.2 | 57.9, F / 16 52.3 | 57.9; 4096 x 18944, F / 8 80.3 | 83.7; 8192 x
// 18000, F / 8 132 | 144, F / 64 106 | 145; 7168 x 18432, F / 8 123 | 129 (four tokens 133 | 128), F / 64 97 | 128.  More channels: 2048 x 19200, F / 64 63.8 |
// 53.4; 4096 x 20480, F / 8 130 | 90.5, F / 64 98.8 | 90.1; 5120 x 20480, F / 8 151 | 107; 6144 x 24576, F / 16 157 | 148, F / 32 145 | 149;
// 8192 x 28672, F / 8 237 | 221, F / 16 208 | 221, F / 64 187 | 221; 4096 x 28672, F / 16 123 | 119, F / 32 113 | 119.
// (Four tokens, F / 8, on layers in between stay with the gathering plan, although it takes 3 to 7 % longer there: 4096 x 11008 59.2 | 57.7, 4096 x
// 12288 66.7 | 62.1, 4096 x 16384 76.9 | 75.1.)
inline bool streaming_beats_gathering(int tokens, int d_model, int d_ff, int k, int sms) {
    const int64_t weights = (int64_t)d_model * d_ff;
    const double used = 1.0 - std::pow(1.0 - (double)k / (double)d_ff, (double)tokens);
    const bool fours = d_ff % 4 == 0;
    if (weights < 300'000) return false;  // (fewer than any that was measured)
    if (d_ff > 2 * sms * kGateRows) return weights * 1e-6 * (0.659 - 0.815 * used) < 12.0 + 11.9e-3 * d_model;
    if (weights < (fours ? 30'000'000 : 25'000'000)) return weights < 25'000'000 || used >= 0.1;
    return (fours && weights < 40'000'000 && used >= 0.3) || (weights >= 90'000'000 && used >= 0.4);
}

}  // namespace moc
