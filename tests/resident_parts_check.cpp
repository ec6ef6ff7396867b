// Host check of the resident kernel's parts (mesh_build.cpp,
// build_resident_parts): every cell is owned by exactly one part, every face
// slot of every cell is written by exactly one record side, every index lies
// inside its part, halo cells carry their owner's publication number, and
// both sides and the geometry of each record are the mesh's. Reads a mesh
// (int64 V, int64 T, V x 2 doubles, T x 3 int32) from argv[1], the cell order
// from argv[2], the number of parts from argv[3]; prints "ok <parts>
// <records>" or the first failure, and exits non-zero on one.
#include <cstdio>
#include <cstdlib>
#include <map>
#include <vector>

#include "../paper_1807_00672_gb300/csrc/mesh_build.h"

#define NEED(cond, what)                    \
  do {                                      \
    if (!(cond)) {                          \
      std::printf("part %d: %s\n", b, what); \
      return 1;                             \
    }                                       \
  } while (0)

int main(int argc, char** argv) {
  if (argc < 4) return 2;
  FILE* f = std::fopen(argv[1], "rb");
  if (!f) return 2;
  int64_t V = 0, T = 0;
  if (std::fread(&V, 8, 1, f) != 1 || std::fread(&T, 8, 1, f) != 1) return 2;
  std::vector<double> xy(2 * V);
  std::vector<int32_t> tri(3 * T);
  if (std::fread(xy.data(), 8, 2 * V, f) != (size_t)(2 * V) ||
      std::fread(tri.data(), 4, 3 * T, f) != (size_t)(3 * T))
    return 2;
  std::fclose(f);
  const int order = std::atoi(argv[2]), parts = std::atoi(argv[3]);
  swe::HostMesh m;
  if (swe::build_host_mesh(xy.data(), V, tri.data(), T, order, 0, false, m, false, true) != 0) return 3;
  swe::ResidentParts p;
  if (!swe::build_resident_parts(m, xy.data(), tri.data(), order == 1, parts, p)) return 3;
  int b = -1;
  NEED((int)p.cell0.size() == parts + 1 && (int)p.cells.size() == T, "part or cell count");
  std::vector<int32_t> owner(T, -1), pub_of(T, -1), pub_cell(p.npub, -1);
  for (b = 0; b < parts; ++b) {
    NEED(p.cell0[b + 1] > p.cell0[b] && p.cell0[b + 1] - p.cell0[b] <= p.cell_cap, "cells of the part");
    for (int32_t q = p.cell0[b]; q < p.cell0[b + 1]; ++q) {
      const int32_t i = p.cells[q];
      NEED(i >= 0 && i < T && owner[i] < 0, "a cell out of range or owned twice");
      owner[i] = b;
      pub_of[i] = p.pub[q];
      if (p.pub[q] >= 0) {
        NEED(p.pub[q] < p.npub && pub_cell[p.pub[q]] < 0, "a publication number used twice");
        pub_cell[p.pub[q]] = i;
      }
    }
  }
  std::vector<int> written(3 * T, 0);  // face slots of every cell
  const swe::HostEdges& ed = m.edges;
  for (b = 0; b < parts; ++b) {
    const int32_t nc = p.cell0[b + 1] - p.cell0[b], nh = p.halo0[b + 1] - p.halo0[b];
    NEED(nh <= p.halo_cap && p.rec0[b + 1] - p.rec0[b] <= p.rec_cap, "caps");
    std::map<int32_t, int> seen;
    for (int32_t q = p.halo0[b]; q < p.halo0[b + 1]; ++q) {
      NEED(owner[p.halo[q]] != b && !seen[p.halo[q]]++, "an own or repeated halo cell");
      NEED(p.halo_pub[q] >= 0 && pub_cell[p.halo_pub[q]] == p.halo[q], "halo publication number");
    }
    for (int32_t r = p.rec0[b]; r < p.rec0[b + 1]; ++r) {
      const uint32_t code[2] = {p.side[r] >> 16, p.side[r] & 0xffffu};
      int64_t cell[2] = {-1, -1};
      int face[2] = {-1, -1};
      for (int s = 0; s < 2; ++s) {
        if (s == 1 && code[s] == 0xffffu) continue;  // wall
        const int k = code[s] >> 14, idx = code[s] & 0x3fff;
        NEED(idx < (k == 3 ? nh : nc), "a side index out of range");
        cell[s] = k == 3 ? p.halo[p.halo0[b] + idx] : p.cells[p.cell0[b] + idx];
        face[s] = k;
        if (k < 3) NEED(written[3 * cell[s] + k]++ == 0, "a face slot written twice");
      }
      NEED(face[0] != 3 || face[1] != 3, "a record without an own cell");
      const int s = face[0] < 3 ? 0 : 1;
      const int32_t e = ed.of_half[3 * (int64_t)m.perm[cell[s]] + face[s]];
      NEED(ed.cL[e] == m.perm[cell[0]], "side A is not the edge's left cell");
      NEED(ed.cR[e] == (cell[1] < 0 ? -1 : m.perm[cell[1]]), "side B is not the edge's right cell");
      NEED(p.nx[r] == ed.nx[e] && p.ny[r] == ed.ny[e] && p.len[r] == ed.len[e], "geometry");
    }
  }
  b = -1;
  for (int64_t k = 0; k < 3 * T; ++k) NEED(written[k] == 1, "a face slot that no record writes");
  std::printf("ok %d %d\n", parts, (int)p.side.size());
  return 0;
}
