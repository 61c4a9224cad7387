// The whole library on top of fake_cuda.cpp: host code only, no kernel ever runs.
#include "../../paper_2607_20125_b200/csrc/headcast_api.cu"
#include "../../paper_2607_20125_b200/csrc/noalloc_scratch.cu"

// What the last attention launch was given.
static hc::AttnParams last_attn;
static void* last_noalloc_list;

// Returns the partial results that the launch uses (a merge launch: those of the attention launch before it).
extern "C" const void* fake_saw_launch(const char* name, void** args) {
  if (std::strstr(name, "attn_kernel")) std::memcpy(&last_attn, args[0], sizeof(last_attn));
  if (std::strstr(name, "noalloc_list_kernel")) std::memcpy(&last_noalloc_list, args[0], sizeof(void*));
  return last_attn.part_o;
}
extern "C" int fake_noalloc_list_is_the_devices() {
  void* now = nullptr;
  cudaGetSymbolAddress(&now, g_noalloc_scratch);
  return last_noalloc_list == now && last_attn.items == static_cast<NoAllocScratch*>(now)->items;
}
extern "C" void* fake_attn_part_o() { return last_attn.part_o; }
extern "C" int fake_attn_radius() { return last_attn.radius; }
// Key tiles of its work list, over all CTAs (without a shared queue).
extern "C" int fake_attn_tile_steps() {
  int sum = 0;
  for (int i = 0; i < last_attn.cta_first[148]; ++i) sum += last_attn.items[i].tile_end - last_attn.items[i].tile_begin;
  return sum;
}
// How the allocation-free call spreads so many query-tile pairs: 0 whole, > 0 in so many equal pieces, < 0 as a line.
extern "C" int fake_noalloc_cuts(int pairs, int n_keys, int n_sm, int head_dim) { return noalloc_plan(pairs, n_keys, n_sm, head_dim).cuts; }
// The first key tile of every CTA's share and, behind the last, their end; returns how many CTAs (0: whole pairs).
extern "C" int fake_noalloc_shares(int pairs, int n_keys, int n_sm, int head_dim, long long* begins, int* slots, int* entries) {
  const NoAllocPlan plan = noalloc_plan(pairs, n_keys, n_sm, head_dim);
  *slots = NOALLOC_SLOTS;
  *entries = NOALLOC_MERGES;
  for (int b = 0; plan.cuts != 0 && b <= plan.n_cta; ++b) begins[b] = plan.share_begin(b);
  return plan.cuts != 0 ? plan.n_cta : 0;
}
