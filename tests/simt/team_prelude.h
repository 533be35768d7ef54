// TEST INFRASTRUCTURE: what simt_prelude.h lacks for teams.  The CTAs of a
// team run side by side, each on a host thread of its own, so that their
// __shared__ variables (thread-local statics) are apart; team_runtime.cpp lets
// one of them run at a time.
#pragma once
#undef __shared__
#define __shared__ static thread_local
#define HM_TEAM_EMULATION 1

namespace simt {
void team_sync();
// grid CTAs in teams of `team` consecutive ones; team after team.
void launch_team(int team, unsigned grid, unsigned block, size_t smem, const std::function<void()>& body);
}  // namespace simt
