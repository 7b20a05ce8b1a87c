// batch_teams.h -- how a chip-resident batched launch splits the SMs into teams, and the
// message memory of a launch.  Host code without CUDA types.
#pragma once

#include <stddef.h>

namespace lap5 {

// Teams of one launch: each has a message word, a slot apart, in the launch's memory.  19
// on a whole chip (teams of eight SMs); a slice of 33 to 37 SMs would have one SM a
// team and more teams than words without the bound.
constexpr int kMaxTeams = 32;
constexpr int kTeamWordStride = 32;      // in 64-bit words
constexpr size_t kTeamWordOffset = 256;  // after the queue head
constexpr size_t kTeamLaunchBytes = kTeamWordOffset + (size_t)kMaxTeams * kTeamWordStride * 8;

// Team sizes that are tried: the chip split into 19 to 1 teams.
constexpr int kTeamSplits[] = {19, 16, 12, 8, 6, 4, 3, 2, 1};
constexpr int team_size(int sms, int split) { return sms / split > 1 ? sms / split : 1; }
constexpr int team_count(int sms, int size) { return sms / size < kMaxTeams ? sms / size : kMaxTeams; }

}  // namespace lap5
