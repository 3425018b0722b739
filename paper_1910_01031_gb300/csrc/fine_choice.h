// How many particles a CTA of the fine stage (qhalf_dev.cuh) takes (host).
#pragma once

namespace iewpf {
namespace qhalf {

// 16 (four warps per strip with 4 particles each), 4 (the four warps share the
// rows of 4 particles) or 1 (they share the rows of one): the form whose waves
// of CTAs take the least time.  A CTA's time hardly depends on how many of its
// places hold a particle: 31, 14 and 11 us (tiles of 64 x 32 cells, c_Omega = 3;
// with c_Omega = 1, or the pull, all three are about 1.5 times that), with 2, 2
// and per_sm1 CTAs per SM.
//   Model error, 16 / 4 / 1 particles per CTA, us:
//     1024^2 x 1: 46 / 24 / 14.5    512^2 x 4: 30 / 13.5 / 15
//     1024^2 x 4: 58 / 27 / 43      512^2 x 16: 31.5 / 27.5 / 44
//     1024^2 x 16: 79 / 96 / 154    256^2 x 9: 30 / 13.6 / 11.7
// ctas(parts) counts the CTAs of `parts` particles each.
template <class F>
inline int fine_choice(F ctas, int sms, int per_sm1)
{
    const struct {
        int parts, per_sm, us;
    } form[3] = {{16, 2, 31}, {4, 2, 14}, {1, per_sm1, 11}};
    int best = 0;
    long long least = 0;
    for (const auto& f : form) {
        const long long at_once = (long long)sms * f.per_sm, us = (ctas(f.parts) + at_once - 1) / at_once * f.us;
        if (best == 0 || us < least) {
            best = f.parts;
            least = us;
        }
    }
    return best;
}

}  // namespace qhalf
}  // namespace iewpf
