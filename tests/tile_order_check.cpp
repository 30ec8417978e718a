// Checks that the tile plan of the tiled barotropic sub-cycle (csrc/tiles.cu)
// sums every copy of an edge or a cell in one order: term j of a local edge
// (cell) is term j of its global edge (cell), or the dummy where that lies
// outside the patch.  Usage: tile_order_check <mesh dir> <patches>.
#include <cstdio>
#include <cstdlib>
#include <string>
#include <vector>

#include "../paper_2105_13484_gb300/csrc/tiles.h"

using namespace sse;

template <class T> static std::vector<T> rd(const std::string &f, size_t n) {
    std::vector<T> v(n);
    FILE *fp = fopen(f.c_str(), "rb");
    if (!fp || fread(v.data(), sizeof(T), n, fp) != n) exit(2);
    fclose(fp);
    return v;
}

int main(int argc, char **argv) {
    if (argc != 3) return 2;
    const std::string d = argv[1];
    HostMesh hm;
    FILE *fp = fopen((d + "/hdr.txt").c_str(), "r");
    if (!fp || fscanf(fp, "%d %d %d %d", &hm.C, &hm.E, &hm.maxE, &hm.maxE2) != 4) return 2;
    fclose(fp);
    const int C = hm.C, E = hm.E, mE = hm.maxE, mE2 = hm.maxE2, P = atoi(argv[2]);
    const auto coe = rd<int>(d + "/coe.bin", 2 * (size_t)E);
    for (int e = 0; e < E; e++) { hm.c1.push_back(coe[2 * e]); hm.c2.push_back(coe[2 * e + 1]); }
    hm.neoc = rd<int>(d + "/neoc.bin", C);
    hm.eoc = rd<int>(d + "/eoc.bin", (size_t)C * mE);
    hm.neoe = rd<int>(d + "/neoe.bin", E);
    hm.eoe = rd<int>(d + "/eoe.bin", (size_t)E * mE2);
    hm.cfc.assign((size_t)E * mE2, 1.0);
    hm.divc.assign((size_t)C * mE, 1.0);
    hm.invdc.assign(E, 1.0); hm.H.assign(C, 1.0);
    TilePlan plan;
    if (!build_tile_plan(hm, P, 3, plan)) { printf("no plan\n"); return 1; }
    long moved = 0, copies = 0;
    for (const TilePatch &t : plan.patches) {
        auto ordered = [&](int n, const int16_t *idx, const int *gl) {
            for (int j = 0; j < n; j++)
                if (idx[j] != t.ne && t.edge_gid[idx[j]] != gl[j]) return false;
            return true;
        };
        for (int l = 0; l < t.ne; l++, copies++)
            moved += !ordered(t.n2[l], &t.eoe[(size_t)l * mE2], &hm.eoe[(size_t)t.edge_gid[l] * mE2]);
        for (int l = 0; l < t.nc; l++, copies++)
            moved += !ordered(t.nce[l], &t.ce[(size_t)l * mE], &hm.eoc[(size_t)t.cell_gid[l] * mE]);
    }
    if (moved) { printf("%ld of %ld copies in another order\n", moved, copies); return 1; }
    printf("ok\n");
    return 0;
}
