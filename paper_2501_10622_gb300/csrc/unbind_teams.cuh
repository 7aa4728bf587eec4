// unbind_teams.cuh -- how the self-boundness check shares its larger groups
// among the CTAs of one launch (host and device; plain C++).
#pragma once

#ifdef __CUDACC__
#define CWTHF_HD __host__ __device__
#else
#define CWTHF_HD
#endif

namespace cwthf {

// CTAs of a team of `want` in a launch of `ctas`: a launch too small for such a
// team is one team itself, so that every group has a team that takes it.
CWTHF_HD constexpr int ub_team_ctas(int want, int ctas) { return want < ctas ? want : ctas; }

}  // namespace cwthf
