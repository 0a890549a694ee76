"""The launch rules of csrc/launch_rules.hpp, compiled by the host compiler (no GPU, no CUDA header)."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2010_14132_gb300", "csrc")


def _run(tmp_path, body):
    """Compile a main() around body, run it, return the lines it prints."""
    cxx = shutil.which("g++") or pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "rules.cpp", tmp_path / "rules"
    src.write_text('#include <cstdio>\n#include <initializer_list>\n#include "launch_rules.hpp"\nusing namespace pgb;\nint main() {\n' + body + "}\n")
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()


def test_warp_masks_name_existing_lanes_only(tmp_path):
    """Blocks of the column kernels (16 to 128 threads), and blocks whose last warp is partly filled."""
    lines = _run(tmp_path, """
  for (int n : {16, 20, 32, 48, 64, 100, 128})
    for (int t = 0; t < n; ++t) printf("%d %d %d %u\\n", n, t, warp_lanes(t, n), warp_mask(t, n));
""")
    assert len(lines) == 16 + 20 + 32 + 48 + 64 + 100 + 128
    for line in lines:
        n, t, lanes, mask = map(int, line.split())
        exists = [32 * (t // 32) + b < n for b in range(32)]
        assert lanes == sum(exists)
        assert mask == sum(1 << b for b in range(32) if exists[b]), line


def test_kernel_grants_are_kept_per_device(tmp_path):
    """A shared memory limit is raised on each device once, never lowered, and asked for again only above it; the CTAs per
    SM are those of the device and of the size launched; errors come back and leave no grant behind."""
    lines = _run(tmp_path, """
  KernelGrants g;
  int k1, k2, n = -1;
  auto ask = [&](int device, const void* kernel, size_t smem, int threads, int fail = 0) {
    size_t allowed = 0;
    int counted = 0;
    const int e = g.get(device, kernel, smem, threads, [&](size_t b) { allowed = b; return fail; },
                        [&](int* out) { ++counted; *out = 100 * device + (int)(smem / 1024); return 0; }, &n);
    printf("%d %zu %d %d\\n", e, allowed, counted, n);
  };
  ask(0, &k1, 65536, 0);
  ask(0, &k1, 65536, 0);
  ask(1, &k1, 65536, 0);     // the second device has not been asked
  ask(1, &k1, 65536, 0);
  ask(0, &k2, 65536, 0);
  ask(0, &k1, 32768, 0);     // below the limit
  ask(0, &k1, 131072, 0);
  ask(0, &k1, 65536, 256);   // CTAs per SM, of each size and device
  ask(0, &k1, 65536, 256);
  ask(0, &k1, 131072, 256);
  ask(0, &k1, 65536, 256);
  ask(1, &k1, 65536, 256);
  ask(1, &k1, 131072, 256, 7);   // refused
  ask(1, &k1, 131072, 256);
""")
    assert [tuple(map(int, line.split())) for line in lines] == [
        (0, 65536, 0, 0), (0, 0, 0, 0), (0, 65536, 0, 0), (0, 0, 0, 0), (0, 65536, 0, 0), (0, 0, 0, 0), (0, 131072, 0, 0),
        (0, 0, 1, 64), (0, 0, 0, 64), (0, 0, 1, 128), (0, 0, 0, 64), (0, 0, 1, 164),
        (7, 131072, 0, 164), (0, 131072, 1, 228)]


def test_launchers_keep_no_grants_of_their_own():
    """Every remembered cudaFuncSetAttribute goes through the per-device table; the other launchers set it each time."""
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        if "cudaFuncSetAttribute" in text and name != "kernel_grants.cuh":
            assert "unordered_map" not in text and "static size_t" not in text, name


def test_level_chunks_of_the_tiled_pass_have_all_their_blocks(tmp_path):
    """Slots for the blocks of one launch over all levels (or for the larger count of another pass) are enough for every
    chunk: each launches all groups of rows that are resident at once, and the slots in use never pass their number."""
    lines = _run(tmp_path, """
  const int resident = 608;
  for (int per_level : {1, 3, 32, 128, 700})
    for (int nz : {2, 37, 48, 128})
      for (int spare : {0, 100})
        for (int chunk : {1, 5, 19, 128}) {
          const int lc = chunk < nz ? chunk : nz;
          const int slots = tile_pass_blocks((long long)per_level * nz, resident, 1 << 30) + spare;
          int used = 0;
          for (int l0 = 0; l0 < nz; l0 += lc) {
            const long long groups = (long long)per_level * (l0 + lc < nz ? lc : nz - l0);
            const int n = tile_pass_blocks(groups, resident, slots);
            used += added_slots(used, n);
            printf("%lld %d %d %d\\n", groups, n, used, slots);
          }
        }
""")
    assert len(lines) > 1000
    for line in lines:
        groups, n, used, slots = map(int, line.split())
        assert n == min(groups, 608) and n <= used <= slots


def test_fp64_column_form_by_the_device(tmp_path):
    """Values a lane for the least FP64 work of the busiest of four units an SM, on devices of several sizes (also one whose
    SM count could not be told)."""
    sizes = [(nx // 2 + 1, ny) for nx in (4, 16, 32, 54, 64, 128, 256, 512, 1024, 4096) for ny in (4, 27, 32, 81, 128, 512, 4096)]
    lines = _run(tmp_path, "".join(
        f'  for (int sms : {{0, 1, 76, 148, 152}}) printf("%d %d\\n", sms, fp64_column_values({(ny // 2 + 1) * nxh}ll, {ny * nxh}ll, sms));\n'
        for nxh, ny in sizes))
    assert len(lines) == 5 * len(sizes)
    seen = set()
    for i, line in enumerate(lines):
        nxh, ny = sizes[i // 5]
        sms, values = map(int, line.split())
        warps = lambda lanes: -(-lanes // 16)  # noqa: E731
        cost = {v: -(-warps(lanes) // max(1, 4 * sms)) * per_level
                for v, lanes, per_level in ((4, (ny // 2 + 1) * nxh, 19), (2, ny * nxh, 13), (1, 2 * ny * nxh, 10))}
        assert values == min((4, 2, 1), key=lambda v: cost[v]), (nxh, ny, sms)
        seen.add((sms, values))
    assert {(76, 1), (76, 4), (152, 1), (152, 2), (152, 4)} <= seen


def test_no_launcher_counts_the_sms_of_one_device():
    for name in sorted(os.listdir(CSRC)):
        for n, line in enumerate(open(os.path.join(CSRC, name))):
            code = line.split("//")[0]
            assert not re.search(r"\b(152|304|608|607)\b", code), f"{name}:{n + 1}"
