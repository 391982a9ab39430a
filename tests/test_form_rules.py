"""The rules that choose a plan's kernel form, called on the host: a small program is compiled against
the library's internal header and prints their answers."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1710_08576_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


def answers(tmp_path, body):
    """The integers that a program with the given main body prints."""
    src, exe = tmp_path / "rules.cpp", tmp_path / "rules"
    src.write_text('#include <cstdio>\n#include <cuda_runtime.h>\n#include "rfi.h"\n#include "internal.h"\n#include "plan_impl.h"\nusing namespace rfi;\n'
                   "int main() {\n" + body + "\nreturn 0;\n}\n")
    subprocess.check_call(["g++", "-std=c++17", "-I" + CSRC, "-I" + os.path.join(ROOT, "include"),
                           "-I" + os.path.join(CUDA, "include"), str(src), "-o", str(exe)])
    return [int(v) for v in subprocess.check_output([str(exe)], text=True).split()]


PLANS = [  # (bits, noise, mom, [(streams, window)], whether the any-window form is the faster one)
    (8, 0, 0, [(60, 1001)], True), (8, 1, 0, [(60, 50001)], True), (12, 1, 0, [(60, 1001)], True),
    (8, 0, 0, [(60, 1600)], True), (8, 0, 0, [(60, 3200)], True), (8, 0, 0, [(60, 4000)], True), (8, 0, 0, [(60, 4800)], False), (8, 0, 0, [(60, 8000)], False),
    (8, 1, 0, [(60, 4800)], True), (8, 1, 0, [(60, 8000)], False), (8, 0, 0, [(60, 10000)], False),
    (8, 0, 0, [(60, 4096)], False), (8, 0, 0, [(60, 16384)], False), (12, 0, 0, [(60, 1600)], False),
    (8, 0, 0, [(10, 3200), (50, 4096)], False), (8, 0, 0, [(10, 3200), (50, 16384)], False),
    (8, 0, 0, [(8, 1000), (52, 16384)], True), (8, 0, 0, [(1, 16385), (59, 16384)], False),
    (8, 0, 1, [(10, 1600), (50, 512)], False), (8, 0, 1, [(60, 1600)], True), (8, 0, 1, [(60, 4800)], True), (8, 0, 1, [(60, 8000)], False),
    (8, 0, 1, [(4, 1001), (56, 4096)], True), (8, 0, 1, [(4, 1001), (56, 16384)], True),
]


@pytest.mark.parametrize("i", range(len(PLANS)))
def test_the_any_window_form_where_it_is_the_faster_one(tmp_path, i):
    bits, noise, mom, streams, want = PLANS[i]
    gains = answers(tmp_path, "".join('printf("%%lld\\n", (long long)any_form_gain(%d, %d, %d, %d, 1 << 22));' %
                                      (bits, noise, mom, W) for _, W in streams))
    assert (sum(n * g for (n, _), g in zip(streams, gains)) > 0) == want, gains


def test_tuned_shapes_are_kept_apart(tmp_path):
    """A short stream's length and the caller's constraints are in the key of a tuned shape; whole
    windows are, and nothing else of a longer stream."""
    keys = ["tune_key(8, 0, {100}, {65536}, nullptr)", "tune_key(8, 0, {60000}, {65536}, nullptr)",
            "tune_key(8, 0, {70000}, {65536}, nullptr)", "tune_key(8, 0, {70001}, {65536}, nullptr)",
            "tune_key(8, 0, {70000}, {65536}, &none)", "tune_key(8, 0, {70000}, {65536}, &two)"]
    got = answers(tmp_path, "rfi_launch_shape none{}, two{};\ntwo.stages = 2;\nstd::string k[] = {" + ", ".join(keys) + "};\n" +
                  "for (int i = 0; i < 6; ++i) for (int j = 0; j < 6; ++j) printf(\"%d\\n\", k[i] == k[j]);")
    same = {(2, 3), (2, 4), (3, 4)}
    assert got == [int(i == j or (min(i, j), max(i, j)) in same) for i in range(6) for j in range(6)]


def test_cached_shapes_have_to_hold_the_windows(tmp_path):
    """A cached shape whose stage is smaller than the plan's largest window, or that no tuner wrote, is
    not taken."""
    shapes = [("8, 2, 3, 512, 1, 1, 1, 1", 65536, 0), ("8, 2, 1, 65536, 1, 1, 1, 1", 65536, 1), ("8, 2, 1, 65537, 1, 1, 1, 1", 65536, 0),
              ("8, 9, 1, 65536, 1, 1, 1, 1", 65536, 0), ("8, 2, 0, 65536, 1, 1, 1, 1", 65536, 0), ("5, 2, 1, 65536, 1, 1, 1, 1", 65536, 0),
              ("8, 2, 1, 65536, 1, 3, 1, 1", 65536, 0), ("16, 1, 2, 1024, 2, 4, 1, 2", 128, 1)]
    got = answers(tmp_path, "".join('printf("%%d\\n", (int)tuned_shape_fits(Shape{%s}, %d));' % s[:2] for s in shapes))
    assert got == [s[2] for s in shapes]


def test_tiles_of_small_plans(tmp_path):
    """Tiles are halved while all of them run at once; a large plan, a stage size of the caller's, and
    windows that are a tile each keep theirs. Median of MAD: at most the apply pass' 32."""
    plans = [  # (windows of each stream, their length, stage, caller's stage, mom) -> windows per tile
        ([256], [4096], 16384, 0, 0, [1]), ([1024], [4096], 16384, 0, 0, [4]), ([256], [4096], 16384, 1, 0, [4]),
        ([256], [1024], 16384, 0, 0, [1]), ([1024], [1024], 16384, 0, 0, [4]), ([4096], [512], 16384, 0, 0, [16]),
        ([64], [16384], 16384, 0, 0, [1]), ([32, 300], [8192, 1024], 16384, 0, 0, [1, 1]), ([100000], [16], 16384, 0, 1, [32]),
    ]
    body = "".join("for (auto v : windows_per_tile(8, 0, %d, %d, {%s}, {%s}, %d, 456)) printf(\"%%lld\\n\", (long long)v);\n" %
                   (mom, whole, ", ".join(map(str, n)), ", ".join(map(str, W)), stage) for n, W, stage, whole, mom, _ in plans)
    assert answers(tmp_path, body) == sum((p[-1] for p in plans), [])


def test_plans_of_many_tiles(tmp_path):
    """Twelve tiles a CTA and more come from the cursor, fewer round robin."""
    got = answers(tmp_path, "".join('printf("%%d\\n", (int)many_tiles(%d, 456));' % n for n in (1, 456 * 9, 456 * 12 - 1, 456 * 12, 456 * 40)))
    assert got == [0, 0, 0, 1, 1]


def test_copies_share_passes_where_that_is_the_faster_way(tmp_path):
    """Multiples of the variants -> one pass per multiple: not for variants with a multiple each, nor where
    the shared ones are too few to pay for the others."""
    cases = [([3], 0), ([3, 3], 1), ([3, 5], 0), ([3] * 4 + [5] * 4, 1), ([1, 2, 3, 4, 5, 6, 7, 8], 0), ([3, 3, 5, 5, 7, 7, 9, 9], 1),
             ([3, 3, 5], 0), ([3, 5, 3, 5, 2, 3, 5, 9], 1), ([3, 3, 3, 5, 6, 7], 0)]
    body = "".join("{ int64_t k[] = {%s}; printf(\"%%d\\n\", (int)copies_share(%d, [&](int v) { return k[v]; })); }\n" %
                   (", ".join(map(str, k)), len(k)) for k, _ in cases)
    assert answers(tmp_path, body) == [w for _, w in cases]


def test_consumers_agree_on_a_timeout_at_their_first_barrier():
    """Every barrier of the joint consumers' loop between the bounded wait for a stage and the window passes
    carries a vote: at a plain one, a thread whose wait timed out would be taken for one that is
    there, and its vote would be lost."""
    text = open(os.path.join(CSRC, "kernels_impl.cuh")).read()
    loop = text[text.index("bool dirty = false;"):text.index("// the group's flagged total")]
    assert "named_bar_or(" in loop and "named_bar(" not in loop
