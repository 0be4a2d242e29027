"""Host-side parts of the CUDA encoder back end that need no GPU: small programs over csrc/encoder_core.hpp."""
import os
import re
import subprocess

import numpy as np
import pytest

import paper_2609_34185_b200 as ep

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _program(tmp_path, body):
    """Compiles `body` as the main function of a program and returns a function that runs it on numbers."""
    src, exe = tmp_path / "p.cpp", tmp_path / "p"
    src.write_text('#include "encoder_core.hpp"\n#include <algorithm>\n#include <cmath>\n#include <cstdio>\n#include <cstdlib>\nusing namespace ep;\n'
                   "int main(int argc, char **argv) {\n" + body + "\nreturn 0;\n}\n")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2609_34185_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    return lambda *a: subprocess.run([str(exe)] + [repr(v) for v in a], check=True, capture_output=True, text=True).stdout.split()


def disjoint_cosets():
    """All zero but two blocks, one on integer and one on half-integer coordinates, far apart: at the fine end of the
    search the two cosets' tables do not meet (-3873 .. and 3872)."""
    W = np.zeros((600, 120), np.float32)
    W[0, 8:16] = -1.0
    W[1, 8:16] = 1.0
    W[1, 0] = 0.04
    return W


def test_coder_entries_hold_cosets_that_do_not_meet(tmp_path):
    run = _program(tmp_path, """
        Model m;
        for (int t = 0; t < EP_NUM_TABLES; ++t) { m.t[t].lo = atoi(argv[1 + t]); m.t[t].n.resize(atoi(argv[18 + t])); }
        const CoderLayout L = coder_layout(m);
        bool inside = true;
        for (int k = 1; k < 9; ++k)
            for (int c = 0; c < 2; ++c) {
                const Table &tb = m.t[table_id(c, k)];
                const int64_t at = int64_t(L.first[k]) + tb.lo - L.lo[k], next = k < 8 ? L.first[k + 1] : L.size;
                if (tb.K()) inside = inside && at >= L.first[k] && at + tb.K() <= next;
            }
        printf("%u %u %d\\n", L.entries(), kCoderEntries, int(inside));""")
    info = ep.encode(disjoint_cosets(), 8.0).info
    assert sum(info.table_K) <= 40960                        # a stream that the device encoder takes
    entries, room, inside = map(int, run(*info.table_min, *info.table_K))
    assert 2 * 40960 + 2 < entries <= room and inside        # more than two entries per symbol of any such stream
    # the widest there can be: a value at either end of what the passes count, in every field
    entries, room, inside = map(int, run(0, *[-4096] * 8, *[4095] * 8, 2, *[1] * 16))
    assert entries == room and inside
    # a tensor with one coset only, and tables that share a range
    assert run(0, *[-3] * 8, *[0] * 8, 1, *[7] * 8, *[0] * 8)[0] == str(2 * 8 * 7 + 2)
    assert run(0, *[-3] * 8, *[-2] * 8, 2, *[7] * 16)[0] == str(2 * 8 * 8 + 2)


def test_encode_that_fails_leaves_no_copy_under_way(tmp_path):
    # the page-locked buffer of the counts goes back to the process when the call ends: nothing may be on its way into it
    exe, csrc = str(tmp_path / "fake_device"), os.path.join(ROOT, "paper_2609_34185_b200", "csrc")
    nvcc = os.environ.get("NVCC") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-O0", "-std=c++17", "-cudart", "none", "-Xcompiler", "-pthread",
                    "-I", os.path.join(ROOT, "include"), "-I", csrc, "-o", exe, os.path.join(ROOT, "tests", "fake_device.cpp")]
                   + [os.path.join(csrc, f) for f in ("encode_gpu.cu", "encoder.cpp", "stream.cpp")], check=True)
    run = lambda buffers: subprocess.run([exe, str(buffers)], check=True, capture_output=True, text=True).stdout.split()
    assert run(2) == ["0", "0"]
    assert run(0) == ["-6", "0"]          # no memory for the counts
    assert run(1) == ["-6", "0"]          # none for the blob: the tile coder and its copies are queued by then


def test_next_scale_error_covers_another_log2_and_exp2(tmp_path):
    # run_encode's secant step with log2 and exp2 two units in the last place off, in every combination, over moves from
    # neighbouring scales to whole doublings
    run = _program(tmp_path, """
        auto ulps = [](double v, int n) { for (; n > 0; --n) v = std::nextafter(v, 1e9); for (; n < 0; ++n) v = std::nextafter(v, -1e9); return v; };
        uint64_t st = 7;
        auto rnd = [&] { st = st * 6364136223846793005ull + 1442695040888963407ull; return double(st >> 11) / 9007199254740992.0; };
        double worst = 0.0, neighbours = 0.0, ordinary = 0.0;
        for (int i = 0; i < 20000; ++i) {
            const float s = float(std::exp2(-9.0 + 12.0 * rnd()));
            const bool next_to = i % 2 == 0;
            const float before = next_to ? std::nextafter(s, rnd() < 0.5 ? 0.0f : 9.0f) : float(double(s) * std::exp2((rnd() < 0.5 ? -1 : 1) * std::exp2(-12.0 * rnd())));
            const double a = std::log2(double(s)), p = std::log2(double(before)), target = 0.08 * (rnd() - 0.5), slope = 0.4 + 4.0 * rnd();
            const double gained = -slope * (a - p);                            // the rates differ by this: a slope inside and outside the clamps
            auto move = [&](int da, int dp, int de, double *per_out) {
                double per = -gained / (ulps(a, da) - ulps(p, dp));
                if (!(per >= 0.5)) per = 0.5;
                if (per > 4.0) per = 4.0;
                if (per_out) *per_out = per;
                return ulps(std::exp2(ulps(a, da) + target / per), de);
            };
            double per;
            const double here = move(0, 0, 0, &per), bound = next_scale_error(a, p, true, target, per);
            (next_to ? neighbours : ordinary) = std::max(next_to ? neighbours : ordinary, bound);
            for (int da = -2; da <= 2; ++da)
                for (int dp = -2; dp <= 2; ++dp)
                    for (int de = -2; de <= 2; ++de) worst = std::max(worst, std::fabs(move(da, dp, de, nullptr) / here - 1.0) / bound);
        }
        printf("%g %g %g\\n", worst, neighbours, ordinary);""")
    worst, neighbours, ordinary = map(float, run())
    assert 0.1 < worst <= 1.0                  # covered, and not by orders of magnitude too much
    assert neighbours > 1e-10 > ordinary       # no fixed 1e-10 covers neighbouring scales


def test_payload_room_fits_the_blob(tmp_path):
    # the blob is laid out before its words are counted: the room must not refuse a blob that is within 32-bit offsets, and a
    # blob of the returned size always is
    run = _program(tmp_path, """printf("%llu", (unsigned long long)payload_room(atof(argv[1]), atoll(argv[2]), atoll(argv[3]), atoll(argv[4])));""")
    room = lambda words, tiles, area, before: int(run(16.0 * words, tiles, area, before)[0])
    tiles, before = 1 << 20, (1 << 20) * 132 + 500_000
    for size in (1 << 20, 1 << 28, (1 << 32) - 4_000_000, (1 << 32) - 3):
        words = (size - before) // 2
        if words < 0:
            continue
        got = room(words, tiles, 1 << 36, before)
        assert words <= got and before + 2 * got < 1 << 32
    assert room(1 << 40, 10, 1 << 41, 1000) == 0                      # hopeless
    assert room(1500, 3, 2000, 1000) == 1501 + 24 + 256           # an ordinary tensor: 0.1 % and a little per tile
    assert room(1000, 3, 1010, 1000) == 1010                          # never more than the area holds


def test_kernels_that_come_up_early_read_by_ordinary_loads():
    # what the predecessor of such a kernel writes must not be declared read-only in it: the load may then move above the wait
    text = open(os.path.join(ROOT, "paper_2609_34185_b200", "csrc", "encode_gpu.cu")).read()
    kernels = {re.search(r"(\w+)\(", k.split(")", 1)[1] if k.startswith(" __launch_bounds__") else k).group(1): k
               for k in re.split(r"__global__ void", text)[1:]}
    chained = {name: k.split("\n}\n")[0] for name, k in kernels.items() if "chained_start();" in k.split("\n}\n")[0]}
    assert {"encode_entries_kernel", "tile_encode_kernel", "compact_kernel"} <= set(chained)
    assert set(re.findall(r"launch_chained\((\w+_kernel)", text)) <= set(chained)
    for name, k in chained.items():
        assert not re.search(r"__restrict__|__ldg\(|\.nc\.", k), name


def test_a_late_cta_takes_no_part_in_the_next_pass(tmp_path):
    # a CTA of a search pass that has no share of it may read the number of scales after the pass's last CTA has stored the next pass's
    run = _program(tmp_path, """
        int wrong = 0, spare = 0;
        for (uint32_t grid : {15u, 16u, 132u, 148u, 160u})
            for (uint32_t n_blocks : {1u, 256u, 3000u, 65536u, 1u << 20})
                for (uint32_t pass = 1; pass < 6; ++pass)
                    for (uint32_t n = 1; n <= 15; ++n) {
                        const uint32_t word = scales_word(pass, n);
                        if (scales_of(word, pass) != n) ++wrong;               // what the others read
                        for (uint32_t later = pass + 1; later < 8; ++later)
                            for (uint32_t m = 0; m <= 15; ++m) {
                                // (0: the search has ended; and no later pass counts the scales of an earlier one)
                                if (scales_of(word, later)) ++wrong;
                                const uint32_t seen = scales_of(scales_word(later, m), pass);
                                for (uint32_t cta = 0; cta < grid; ++cta) {
                                    if (pass_share(grid, cta, n, n_blocks).scale < n) continue;
                                    ++spare;
                                    if (seen && pass_share(grid, cta, seen, n_blocks).scale < seen) ++wrong;
                                }
                            }
                    }
        printf("%d %d\\n", wrong, spare > 0);""")
    assert run() == ["0", "1"]


def test_every_scale_of_a_pass_is_counted_whole_on_any_number_of_sms(tmp_path):
    run = _program(tmp_path, """
        int wrong = 0;
        for (uint32_t sms = 1; sms <= 160; ++sms)
            for (uint32_t n_blocks : {1u, 255u, 257u, 4000u, 1u << 18, (1u << 31) - 1u})
                for (uint32_t n = 1; n <= kMostScales; ++n) {
                    std::vector<std::vector<int>> seen(n);
                    for (uint32_t cta = 0; cta < pass_grid(sms); ++cta) {
                        const PassShare s = pass_share(pass_grid(sms), cta, n, n_blocks);
                        if (s.scale >= n) continue;
                        seen[s.scale].resize(s.ctas);
                        if (s.part < s.ctas) ++seen[s.scale][s.part]; else ++wrong;
                    }
                    for (const auto &parts : seen) {
                        if (parts.empty()) ++wrong;
                        for (int times : parts) wrong += times != 1;
                    }
                }
        printf("%d\\n", wrong);""")
    assert run() == ["0"]


@pytest.fixture(scope="module")
def search_program(tmp_path_factory):
    tmp = tmp_path_factory.mktemp("search_state")
    exe, csrc, obj = str(tmp / "search_state"), os.path.join(ROOT, "paper_2609_34185_b200", "csrc"), str(tmp / "fake_device.o")
    nvcc = os.environ.get("NVCC") or "/usr/local/cuda/bin/nvcc"
    flags = ["-gencode", "arch=compute_100a,code=sm_100a", "-O0", "-std=c++17", "-Xcompiler", "-pthread", "-I", os.path.join(ROOT, "include"), "-I", csrc]
    subprocess.run([nvcc, "-c", "-Dmain=fake_main", "-DcudaLaunchKernelExC=fake_launch", *flags, "-o", obj, os.path.join(ROOT, "tests", "fake_device.cpp")], check=True)
    subprocess.run([nvcc, "-cudart", "none", *flags, "-o", exe, os.path.join(ROOT, "tests", "search_state.cu"), obj]
                   + [os.path.join(csrc, f) for f in ("encoder.cpp", "stream.cpp")], check=True)
    return lambda *a: subprocess.run([exe] + [str(v) for v in a], check=True, capture_output=True, text=True).stdout.split()


def test_a_search_that_has_not_ended_is_left_to_the_host(search_program):
    run = search_program
    assert run(0, 0)[:3] == ["0", "1", "1"]
    assert run(1, 0)[:3] == ["0", "0", "0"]   # steps not taken: the scale is not the bisection's


def test_frequencies_that_did_not_come_are_not_compared(search_program):
    # the launches end without the report: state and counts are fetched, the frequencies in the page-locked buffer are those of an earlier call
    assert search_program(0, 1)[:3] == ["0", "1", "1"]


def test_a_report_that_takes_long_does_not_keep_the_core(search_program):
    # earlier work on the stream, for instance: after a few milliseconds the thread waits as the process has its threads wait
    assert int(search_program(0, 0)[3]) < 25
