// rundump.cpp -- test helper: the warp programs of a reaction table (compiled by
// csrc/mechanism.cpp on the CPU) with their runs, their device form's groups and
// run tables, as text.
//
// usage: rundump <in.bin> <out.txt>; in.bin = int32 n_species, int32
// n_reactions, then n_reactions chem_reaction records.
#include <cstdio>
#include <utility>
#include <vector>

#include "internal.h"

using namespace chemgpu;

// the constant-memory upload lives with the kernels; the compiler only calls it
namespace chemgpu {
cudaError_t set_constants() { return cudaSuccess; }
}

static void dump(FILE *f, const char *name, const HostProgram &p) {
  std::vector<std::pair<int, int>> groups;
  std::vector<uint32_t> table;
  p.groups(groups, table);
  std::fprintf(f, "program %s\nops", name);
  for (const Op &o : p.ops) std::fprintf(f, " %u %u %u %u", o.t, o.a, o.b, o.c);
  std::fprintf(f, "\nunit");
  for (uint8_t u : p.unit) std::fprintf(f, " %d", (int)u);
  std::fprintf(f, "\nrun");
  for (uint8_t r : p.run) std::fprintf(f, " %d", (int)r);
  std::fprintf(f, "\ngroups");
  for (auto &g : groups) std::fprintf(f, " %d %d", g.first, g.second);
  std::fprintf(f, "\ntable");
  for (uint32_t r : table) std::fprintf(f, " %u %u", r >> 28, r & 0x0fffffffu);
  std::fprintf(f, "\n");
}

int main(int argc, char **argv) {
  if (argc != 3) return 2;
  FILE *in = std::fopen(argv[1], "rb");
  if (!in) return 3;
  int S = 0, R = 0;
  if (std::fread(&S, 4, 1, in) != 1 || std::fread(&R, 4, 1, in) != 1) return 4;
  std::vector<chem_reaction> rx(R > 0 ? R : 1);
  if (R > 0 && std::fread(rx.data(), sizeof(chem_reaction), R, in) != (size_t)R) return 5;
  std::fclose(in);
  Mechanism m;
  std::string msg;
  if (int rc = compile_mechanism(S, R, rx.data(), m, msg)) {
    std::printf("compile failed %d %s\n", rc, msg.c_str());
    return 1;
  }
  FILE *f = std::fopen(argv[2], "w");
  if (!f) return 6;
  dump(f, "f", m.f_prog);
  dump(f, "m", m.m_prog);
  dump(f, "lu", m.lu_prog);
  dump(f, "nudot", m.nudot_prog);
  dump(f, "jt", m.jt_prog);
  dump(f, "fwd", m.fwd_prog);
  dump(f, "bwd", m.bwd_prog);
  dump(f, "fwdT", m.fwdT_prog);
  dump(f, "bwdT", m.bwdT_prog);
  std::fclose(f);
  return 0;
}
