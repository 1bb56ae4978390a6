"""Scratch that one part of the library reserves and another fills
(csrc/size_rules.h), compiled with the host C++ compiler: whatever batches a
call is cut into, every batch fits what was reserved for the first."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2009_12663_gb300", "csrc")


def run(tmp_path, body, head=""):
    src = tmp_path / "rules.cpp"
    src.write_text("#include <cstdio>\n#include <initializer_list>\n#include \"resident_plan.h\"\n#include \"size_rules.h\"\n"
                   "using namespace resident;\nusing namespace sizes;\n" + head + "int main() {\n  int bad = 0;\n" + body + "  return bad != 0;\n}\n")
    exe = str(tmp_path / "rules")
    subprocess.check_call(["g++", "-std=c++17", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", exe])
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_strain_sums_of_every_batch_fit_the_buffer_of_the_first(tmp_path):
    run(tmp_path, r"""
  for (int nex : {1, 5, 12, 57, 81, 126, 160, 253, 340})
    for (int nez : {1, 3, 6, 21, 46, 60, 70})
      for (int nt : {2, 15, 16, 40, 500, 800, 1333, 3000})
        for (int nshot = 1; nshot <= 24; ++nshot)
          for (int most = 1; most <= nshot; ++most) {
            const int last = last_batch(nshot, most);
            const long long ne = (long long)nex * nez;
            if (last < 1 || last > most || (nshot - last) % most || integral_bytes(ne, nt, last) > integral_bytes(ne, nt, most)) {
              std::printf("%d x %d, nt %d: %d shots by %d\n", nex, nez, nt, nshot, most);
              ++bad;
            }
          }
""")


# an SM of 228 KB shared memory (1 KB a CTA taken by the system), 152 of them; registers let
# at least the CTAs of the launch bounds in, and shared memory decides here
PLAN = r"""
struct Plan { Tile t; int per_launch; };
static int slots(int NT, bool adj, size_t smem) {
  if (smem > 227 * 1024 - 64) return 0;
  return 152 * (int)std::min<size_t>(228 * 1024 / (smem + 1024), 2048 / (NT + corr_threads(NT, adj)));
}
// receivers along the surface: those of a tile, on five nodes each
static Plan plan(int nex, int nez, bool adj, int shots, int nrec = 8) {
  auto all = [&](int NT, size_t smem, int &nsm) { nsm = 152; return slots(NT, adj, smem); };
  auto launch = [&](const Tile &t) {
    const int rec = (nrec * t.TX + nex - 1) / nex;
    const size_t smem = smem_bytes(t.NT, adj, t.TX, t.TZ, t.ntx, t.ntz, true, adj ? 4 * t.TX + 1 : 8, adj ? 5 * rec : 8, adj ? 0 : rec);
    return slots(t.NT, adj, smem) / (t.ntx * t.ntz);
  };
  const Tile t = best_tile(nex, nez, true, adj, shots, all, [&](const Tile &c) { return launch(c) >= 1; });
  return {t, t.NT ? launch(t) : 0};
}
"""


def test_exchange_of_every_batch_fits_what_both_batch_sizes_reserve(tmp_path):
    """Forward runs: the last batch has a plan of its own, which may take more
    shots a launch than the first batch's (the grid holds such calls), so both
    count in what is reserved."""
    run(tmp_path, r"""
  int wider = 0;
  for (auto [nex, nez] : {std::pair{5, 3}, {40, 20}, {57, 46}, {106, 40}, {110, 37}, {253, 24}, {280, 10}, {340, 70}})
    for (int spl : {1, 8, 24})
      for (int nshot : {1, 5, 13, 24, 37, 43, 44, 61}) {
        const Plan all = plan(nex, nez, false, nshot);
        if (all.per_launch < 1) continue;
        const int most = std::min(nshot, std::max(all.per_launch, spl)), last = last_batch(nshot, most);
        const long long nodes = (4LL * nez + 1) * (4 * nex + 4);
        size_t reserved = 0, first = 0;
        for (int B : {most, last}) {
          const Plan p = plan(nex, nez, false, B);
          reserved = std::max(reserved, exchange_bytes(p.t.ntx * p.t.ntz, B, p.per_launch, nodes));
          if (B == most) first = reserved;
        }
        for (int i0 = 0; i0 < nshot; i0 += most) {
          const int B = std::min(most, nshot - i0);
          const Plan p = plan(nex, nez, false, B);
          for (int s0 = 0; s0 < B; s0 += p.per_launch) {      // the launches of a batch, 32 bytes a node and shot
            const size_t used = p.t.ntx * p.t.ntz > 1 ? 32 * (size_t)std::min(p.per_launch, B - s0) * nodes : 0;
            if (used > reserved) { std::printf("%d x %d, %d shots by %d\n", nex, nez, nshot, most); ++bad; }
            if (used > first) ++wider;
          }
        }
      }
  if (!wider) { std::printf("no last batch needs more than the first\n"); ++bad; }
""", "#include <utility>\n" + PLAN)


def test_partials_of_unet_products_fit_the_scratch(tmp_path):
    """Every 3x3 layer's forward product and weight gradient over the networks
    the library accepts, alone and in batches: partials within the scratch, which
    some layers' weight gradients do not fit even alone."""
    run(tmp_path, r"""
  const long long cap = 32LL << 20;
  int wide = 0;
  for (int levels = 1; levels <= 6; ++levels)
    for (int base : {8, 32, 64, 96})
      for (int unit : {1, 2, 8})                               // coarsest level of unit x 8 unit pixels
        for (int samples : {1, 2, 5, 64}) {
          auto check = [&](int M, int N, int K, bool accumulate) {
            int splits = 0;
            const int kchunk = split_chunk(M, N, K, cap, &splits);
            const long long outputs = (long long)M * N;
            const int fit = gemm_samples(outputs, splits, samples, accumulate, cap);
            if (accumulate && outputs > cap) ++wide;
            if (fit < 1 || fit > samples || kchunk % kGemmBK || (long long)kchunk * splits < K) ++bad;
            for (int b0 = 0; b0 < samples; b0 += fit) {
              const int nb = std::min(fit, samples - b0);
              if (gemm_partial(splits, nb, accumulate) ? nb * splits * outputs > cap : accumulate && nb > 1) {
                std::printf("levels %d base %d: %d x %d over %d, %d samples\n", levels, base, M, N, K, nb);
                ++bad;
              }
            }
          };
          for (int l = 0; l < levels; ++l) {
            const int ch = base << l, below = l ? ch / 2 : 5, px = (unit << (levels - 1 - l)) * ((8 * unit) << (levels - 1 - l));
            for (int cin : {below, ch, 3 * ch}) {              // encoder, second convolutions, decoder
              const int kcp = (9 * cin + 7) / 8 * 8;
              check(ch, px, kcp, false);
              check(ch, kcp, px, true);
            }
          }
        }
  if (!wide) { std::printf("no layer is wider than the scratch\n"); ++bad; }
""")


def test_less_is_reserved_when_memory_is_short(tmp_path):
    """Choices in order until one fits; what a failed one took is given back first;
    other errors end the search."""
    run(tmp_path, r"""
  for (int room = 0; room <= 40; ++room) {
    int held = 0, released = 0;
    auto reserve = [&](int want) {                   // in pieces of three, like a call's buffers
      for (int got = 0; got < want; got += 3, held += 3)
        if (held + 3 > room) return -2;
      return 0;
    };
    const int rc = first_that_fits(std::initializer_list<int>{36, 12, 3}, -2, reserve, [&] { held = 0; ++released; });
    const int want = room >= 36 ? 36 : room >= 12 ? 12 : 3;
    if (rc != (room >= 3 ? 0 : -2) || (rc == 0 && held != want) || released != (want == 36 ? 0 : want == 12 ? 1 : 2)) ++bad;
  }
  int asked = 0;
  if (first_that_fits(std::initializer_list<int>{2, 1}, -2, [&](int) { ++asked; return -1; }, [] {}) != -1 || asked != 1) ++bad;
""")


def test_whether_a_mesh_is_resident_does_not_depend_on_the_shots(tmp_path):
    """Some shots choose a tile that many receivers' lists do not fit: another one
    takes its place."""
    run(tmp_path, r"""
  int fit = 0, not_fit = 0;
  for (auto [nex, nez] : {std::pair{12, 6}, {46, 42}, {60, 30}, {110, 37}, {340, 70}, {700, 80}})
    for (bool adj : {false, true})
      for (int nrec : {10, 1000, 2000, 3000, 12000, 100000}) {
        const bool one = plan(nex, nez, adj, 1, nrec).per_launch >= 1;
        (one ? fit : not_fit)++;
        for (int shots = 2; shots <= 40; ++shots)
          if ((plan(nex, nez, adj, shots, nrec).per_launch >= 1) != one) {
            std::printf("%d x %d, %d receivers, %d shots\n", nex, nez, nrec, shots);
            ++bad;
          }
      }
  if (!fit || !not_fit) ++bad;
""", "#include <utility>\n" + PLAN)
