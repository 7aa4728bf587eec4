// unbind_teams.cuh -- how the self-boundness check shares its larger groups
// among the CTAs of one launch (host and device; plain C++).
#pragma once

#ifdef __CUDACC__
#define CWTHF_HD __host__ __device__
#else
#define CWTHF_HD
#endif

namespace cwthf {

// Groups up to this size take one CTA (and sort in shared memory); larger ones
// are medium up to kUbBigMin members and big up to kUbBigMax.
constexpr int kUbCtaMax = 2048, kUbBigMin = 1 << 16, kUbBigMax = 1 << 20;
CWTHF_HD constexpr bool ub_big(long long n) { return n > kUbBigMin && n <= kUbBigMax; }

// Most CTAs of the launch (its per-CTA scratch is sized for them).
constexpr int kUbCtaCap = 1024;

// The ways of sharing a group, taken in this order: the whole launch (0: groups
// above kUbBigMax), teams of 128 and 64 CTAs (1, 2: big groups), teams of 8, 4,
// 2 and 1 (3 .. 6: medium ones).  The sizes divide each other, so the CTAs of a
// team have all been in one team of any earlier way, or in none.
constexpr int kUbWays = 7, kUbWhole = 0, kUbMediumWays = 3;
CWTHF_HD constexpr int ub_team_size(int way) {
    return way == kUbWhole ? kUbCtaCap : (way < kUbMediumWays ? 256 >> way : 64 >> way);
}

// CTAs of a team of `want` in a launch of `ctas`: a launch too small for such a
// team is one team itself, so that every group has a team that takes it.
CWTHF_HD constexpr int ub_team_ctas(int want, int ctas) { return want < ctas ? want : ctas; }

// Number of a way's first team among all teams (way kUbWays: their number).
CWTHF_HD constexpr int ub_first_team(int way) {
    int n = 0;
    for (int w = kUbWhole; w < way; w++) n += kUbCtaCap / ub_team_size(w);
    return n;
}

// The way of a group of n members in a launch of `ctas`, where all groups of its
// kind have `total`.
//
// Big groups: 128 CTAs for one that has them nearly to itself, else 64, so that
// four go side by side.  One group (us, whole launch of 304 CTAs / 128 / 64):
// 131,072 members 2720 / 2360 / 2540, 300,000 4270 / 3200 / 4170, 2^20 7760 /
// 7640 / 12,700 or more; two of 300,000 - / 5560 / 6280.
//
// Medium groups: the CTAs that the group's share of all members asks for, or one
// per 4096 members if that is more, at most eight.  A group alone wants eight (a
// CTA by itself works 21 ms on 40,000 members, eight 3.2 ms), but many small
// ones spend most of their time in the teams' barriers: 5000 groups of 2100
// 111 ms with eight CTAs each, 29 with one; 2000 of 4000 56 and 22; 1000 of
// 10,000 47 and 31 (two each); 300 of 40,000 45 with eight, 49 with one.
CWTHF_HD constexpr int ub_big_way(long long n, long long total, int ctas) {
    const long long share = ctas * n / total, w = share < n / 1024 ? share : n / 1024;
    return w >= 128 ? 1 : 2;
}
CWTHF_HD constexpr int ub_medium_way(long long n, long long total, int ctas) {
    const long long share = ctas * n / total, w = share > n / 4096 ? share : n / 4096;
    return w >= 8 ? 3 : (w >= 4 ? 4 : (w >= 2 ? 5 : 6));
}

}  // namespace cwthf
