// Host-side check of the row gather's shared-memory layout (tests/test_layout_cpu.py).
//
// For every precision, mode (assembly, time step, nodal outputs), number of
// lanes per row H, longest row and number of walk bytes, the layout that the
// launches carve (gather_smem with group_slots' W) has its regions in order
// and without overlap; every region starts on a 16-byte boundary and a warp's
// slice is a multiple of 32 bytes, so that the next warp's FP64 vectors are
// aligned; the H accumulator planes are whole 16-byte blocks inside their region;
// the staged entries (4 T each, row t's in CSR order or from t * (W + 1) on) and
// the next group's column indices past them lie in the bytes of nb0 and nb1;
// the copied walk words and the row bounds and diagonal positions lie in
// theirs; and one warp's slice fits a block.  So does the layout of a batch,
// which takes the maxima of its meshes.  Prints one summary line; exit code 0
// when every case holds.
#include <algorithm>
#include <cstdio>

#include "../paper_2111_05651_gb300/csrc/nsi_internal.cuh"

int main() {
  long cases = 0, bad = 0;
  for (int prec : {NSI_FP64, NSI_MIXED_F32_ACC64, NSI_MIXED_F32_ACC32})
    for (int mode : {nsi::ASSEMBLE, nsi::STEP, nsi::NODAL})
      for (int H : {1, 2, 4})
        for (int slots = 1; slots < nsi::STAR_MAX_ROW; ++slots)
          for (int S : {0, 1, 7, 100, 4095, 32 / H * (255 * H + H)}) {
            const int W = nsi::group_slots(prec, H, slots);
            const nsi::GatherSmem g = nsi::gather_smem(prec, mode, H, W, S);
            ++cases;
            auto check = [&](bool ok, const char* what) {
              if (!ok && bad++ < 10)
                std::printf("FAIL %s (precision %d, mode %d, H %d, slots %d, S %d)\n", what, prec, mode, H, slots, S);
            };
            const size_t T = prec == NSI_FP64 ? 8 : 4, R = 32 / H, N = R * W, L = R * (W + 1);
            // FP64 assembly: two planes of T[2]; mixed: one of T[4]; time step one T
            const size_t ab = mode == nsi::ASSEMBLE ? 4 * T : mode == nsi::STEP ? T : 0;
            check(W >= slots && W <= std::max(slots, prec == NSI_FP64 ? 3 : 5),
                  "slots of the longest row, and no more than the staging needs");
            check((size_t)g.R == R && g.N() == N && (size_t)g.L == L && (size_t)g.tb == T && (size_t)g.ab == ab,
                  "sizes");
            check(g.nb1() % 16 == 0 && g.acc() % 16 == 0 && g.plane() % 16 == 0 && g.walk() % 16 == 0 &&
                      g.info() % 16 == 0 && g.cols() % 16 == 0,
                  "16-byte boundaries");
            check(g.total() % 32 == 0, "a slice of a multiple of 32 bytes");
            check(4 * T * N <= g.nb1() && g.nb1() + 2 * T * N <= g.acc() && g.acc() + H * ab * N <= g.walk(),
                  "nb0, nb1 and the planes in order without overlap");
            check(g.plane() == ab * N, "a plane holds every slot");
            check(g.walk() + 4 * ((size_t)(S + 3 + 3) / 4) <= g.info(), "the walk bytes from any offset, in whole words");
            check(R % 4 == 0 && g.info() + 2 * 4 * (R + 1) + R <= g.total(), "row bounds and diagonal positions");
            check(4 * T * L <= g.cols() && g.cols() + 4 * L <= g.acc(), "staging and column indices in nb0 and nb1");
            check((R - 1) * (W + 1) + W + 1 <= L, "the last row's place in the staging");
            check(g.total() <= (size_t)nsi::SMEM_MAX, "one warp's slice in a block");
            for (int other : {1, 14, 31}) {  // a batch with a mesh of rows of other lengths
              const nsi::GatherSmem b =
                  nsi::gather_smem(prec, mode, H, std::max(W, nsi::group_slots(prec, H, other)), std::max(S, 500));
              check(b.group_fits() && b.L >= g.L && b.W >= g.W && b.total() <= (size_t)nsi::SMEM_MAX, "batch maxima");
            }
          }
  std::printf("cases=%ld failures=%ld\n", cases, bad);
  return bad == 0 ? 0 : 1;
}
