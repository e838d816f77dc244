// Test helper: the interleaved scan form the engine generates for a primer set.
// usage: il_dump source|compile|ops|suits [windows=N] k clamp primer [primer ...]
// (each primer gives its + and - strand patterns and may carry its own budget as "PRIMER:k"; "compile" compiles for
// sm_103a with NVRTC, no device needed; "suits" prints whether plans choose the form for these patterns)
//        il_dump generic threads groups_per_thread tiles
// (the groups that the generic kernel's blocks cover for so many of the form's tiles, and those of a full launch)
#define main jit_dump_main
#include "jit_dump.cpp"
#undef main

#include <string>

int main(int argc, char** argv) {
  const std::string what = argv[1];
  int a = 2;
  ah::ScanConfig cfg;
  cfg.interleaved = 1;
  if (what == "generic") {
    cfg.threads = atoi(argv[2]), cfg.groups_per_thread = atoi(argv[3]);
    const unsigned long long per = 1ull * cfg.threads * cfg.groups_per_thread, tile = ah::scan_tile_groups(cfg);
    const unsigned long long most = ah::generic_tiles_per_launch(cfg);
    printf("%llu %llu %llu\n", (unsigned long long)ah::generic_blocks(cfg, atoll(argv[4]) * tile) * per, most,
           (unsigned long long)ah::generic_blocks(cfg, most * tile));
    return 0;
  }
  if (!strncmp(argv[a], "windows=", 8)) cfg.vote_windows = atoi(argv[a++] + 8);
  const int k = atoi(argv[a]), clamp = atoi(argv[a + 1]);
  std::vector<ah::Pattern> pats;
  for (a += 2; a < argc; ++a)
    for (int strand = 0; strand < 2; ++strand) {
      ah::Pattern P;
      memset(&P, 0, sizeof P);
      const std::string arg = argv[a], primer = arg.substr(0, arg.find(':'));
      const int L = (int)primer.size();
      P.len = (uint8_t)L;
      P.k = (uint8_t)(primer.size() < arg.size() ? atoi(arg.c_str() + primer.size() + 1) : k);
      P.id = (uint16_t)pats.size();
      for (int j = 0; j < L; ++j) P.set[j] = strand == 0 ? set_of(primer[j]) : comp(set_of(primer[L - 1 - j]));
      P.clamp_lo = (uint8_t)(strand == 0 ? L - clamp : 0);
      P.clamp_hi = (uint8_t)(strand == 0 ? L : clamp);
      pats.push_back(P);
    }
  if (what == "suits") {
    printf("%d\n", ah::interleaved_suits(pats) ? 1 : 0);
    return 0;
  }
  int ops = 0;
  const std::string src = ah::scan_source(pats, cfg, &ops);
  if (what == "ops") {
    printf("%d\n", ops);
  } else if (what == "compile") {
    std::vector<char> cubin;
    std::string err;
    if (ah::nvrtc_compile_sm(103, src, "ah_scan_jit.cu", &cubin, &err) != AH_OK) {
      printf("error: %s\n", err.c_str());
      return 1;
    }
    printf("compiled %zu\n", cubin.size());
  } else {
    puts(src.c_str());
  }
  return 0;
}
