// Test helper, included after the generated source: runs the kernel's blocks on the CPU.
// usage: il_run input output order
// input (little-endian words): n_groups, first group, groups, slot_cap (u32 each), then (n_groups + 64) x (lo, hi) and
// n_groups + 64 invalid words; output: the status word, tile counts, slots (u64)
int main(int argc, char** argv) {
  if (argc < 4) return 2;
  FILE* f = fopen(argv[1], "rb");
  unsigned head[4];
  if (!f || fread(head, 4, 4, f) != 4) return 2;
  const u64 n = head[0];
  std::vector<uint2> planes(n + 64);
  std::vector<u32> invalid(n + 64);
  if (fread(planes.data(), 8, n + 64, f) != n + 64 || fread(invalid.data(), 4, n + 64, f) != n + 64) return 2;
  fclose(f);
  const u64 n_tiles = (n + 1023) / 1024;
  std::vector<u64> slots(n_tiles * head[3]);
  std::vector<u32> tile_count(n_tiles);
  u32 status = 0;
  ScanParams P{};
  P.planes = planes.data(), P.invalid = invalid.data();
  P.group_begin = head[1], P.n_groups = head[2], P.slot_cap = head[3];
  P.slots = slots.data(), P.tile_count = tile_count.data(), P.status = &status, P.tile_groups = 1024;
  const unsigned blocks = (head[2] + 1024 * (NT / 32) - 1) / (1024 * (NT / 32));
  for (unsigned b = 0; b < blocks; ++b)
    for (unsigned w = 0; w < NT / 32; ++w) warp::run(b, w, atoi(argv[3]), [&] { ah_scan_jit(P); });
  f = fopen(argv[2], "wb");
  fwrite(&status, 4, 1, f);
  fwrite(tile_count.data(), 4, n_tiles, f);
  fwrite(slots.data(), 8, slots.size(), f);
  fclose(f);
  return 0;
}
