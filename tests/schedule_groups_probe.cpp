// Prints, as one JSON object, the accumulation lists and the batch groups that libhfx makes for
//   n_orb  block  transform_budget_couples  ragged_ok  group_couples
// (the library's own build_schedule and build_groups, host code only), for tests/test_schedule_groups.py.
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "../paper_2309_00651_gb300/csrc/hfx_schedule.h"

static void ints(const char* name, const std::vector<int>& v) {
  std::printf("\"%s\": [", name);
  for (size_t i = 0; i < v.size(); ++i) std::printf("%s%d", i ? ", " : "", v[i]);
  std::printf("], ");
}

int main(int argc, char** argv) {
  if (argc != 6) return 2;
  hfx::Schedule S;
  hfx::build_schedule(S, std::atoi(argv[1]), std::atoi(argv[2]), (size_t)std::atoll(argv[3]), 1, true, true,
                      std::atoi(argv[4]) != 0);
  hfx::build_groups(S, std::atoll(argv[5]));
  std::vector<int> blocks;
  for (const int2& b : S.slot_blocks) { blocks.push_back(b.x); blocks.push_back(b.y); }
  std::printf("{");
  ints("slot_blocks", blocks);
  ints("slot_couple_base", S.slot_couple_base);
  ints("batch_slot_begin", S.batch_slot_begin);
  ints("dense_slots", S.dense_slots);
  ints("diag_slots", S.diag_slots);
  ints("generic_slots", S.generic_slots);
  ints("group_begin", S.group_begin);
  std::printf("\"ngroups\": %d, \"max_group_couples\": %lld}\n", S.ngroups, S.max_group_couples);
  return 0;
}
