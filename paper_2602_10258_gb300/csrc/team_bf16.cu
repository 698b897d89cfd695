// Team graph search over BF16 rows (see query_team.cuh).
#include "query_team.cuh"

namespace jag {
template cudaError_t launch_team_fmt<JAG_VEC_BF16>(const SearchLaunch &L, int P, int CPL, TeamTook *took);
}  // namespace jag
