"""The rules by which a call takes one kernel or another, held against what both sides took on a B200 (us, the same process and minute)."""
import subprocess

import pytest

from paper_2510_04147_b200 import build


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    """rule(expressions): their values, as the host code has them."""
    folder = tmp_path_factory.mktemp("routes")

    def values(expressions):
        (folder / "r.cpp").write_text('#include "routes.h"\n#include <cstdio>\nusing namespace ssd;\nint main() {\n' +
                                      "".join(f'std::printf("%d\\n", (int)({e}));\n' for e in expressions) + "}\n")
        r = subprocess.run(["g++", "-std=c++17", "-I", build.CSRC, "-o", str(folder / "r"), str(folder / "r.cpp")], capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
        return [int(x) for x in subprocess.run([str(folder / "r")], capture_output=True, text=True, check=True).stdout.split()]
    return values


def within(took, best):
    return took <= 1.05 * best + 0.5          # what runs of one side differ by


# (vocabulary, d, rows): skinny, dense; LM head and merge kernel, behind other layers
LM_HEAD = {
    (512, 256, 192): (15.4, 14.5), (2048, 256, 192): (15.8, 15.0), (2048, 256, 256): (18.7, 15.0), (2048, 256, 512): (19.1, 15.8),
    (8192, 256, 256): (19.2, 15.4), (2048, 512, 192): (16.7, 16.3), (2048, 512, 256): (19.7, 16.7), (2048, 512, 512): (20.6, 17.4),
    (24576, 256, 192): (21.2, 25.4), (65536, 256, 192): (41.2, 50.1), (100352, 256, 192): (58.2, 66.9), (128256, 256, 256): (93.5, 79.8),
    (16384, 512, 192): (18.3, 22.3), (32000, 512, 192): (28.7, 33.2), (65536, 512, 256): (60.2, 52.3), (128256, 512, 512): (180.1, 125.7),
    (512, 1024, 192): (18.3, 30.9), (2048, 1024, 224): (21.4, 27.1), (16384, 1024, 512): (35.1, 39.5), (24576, 1024, 192): (28.5, 39.8),
    (32000, 1024, 256): (38.6, 42.1), (50304, 1024, 256): (63.8, 55.0), (65536, 1024, 192): (59.0, 64.8), (65536, 1024, 448): (111.4, 81.1),
    (2048, 2048, 192): (22.0, 28.4), (16384, 2048, 192): (26.5, 32.9), (50304, 2048, 192): (75.3, 60.0), (128256, 2048, 192): (147.6, 131.8),
    (2048, 4096, 192): (30.3, 39.4), (8192, 4096, 416): (36.3, 41.4), (16384, 4096, 192): (40.2, 44.6), (50304, 4096, 192): (126.4, 93.2),
    (128256, 4096, 192): (245.7, 214.2), (128256, 4096, 512): (479.3, 399.4), (126464, 4096, 161): (223.0, 211.0), (152064, 3584, 256): (288.0, 252.0),
}


def test_lm_head_takes_no_slower_kernel(rule):
    took = rule([f"lm_head_dense({v}, {k}, {r})" for v, k, r in LM_HEAD])
    for (case, times), dense in zip(LM_HEAD.items(), took):
        assert within(times[dense], times[0]), (case, dense)
    assert within(sum(t[d] for t, d in zip(LM_HEAD.values(), took)), sum(min(t) for t in LM_HEAD.values()))


# (gate|up features, d, rows): without, with the evenly shared kernel
GATE_UP = {
    (1408, 256, 192): (7.5, 5.3), (1408, 256, 256): (6.5, 5.4), (11264, 2048, 192): (15.4, 13.4), (24576, 4096, 192): (47.2, 39.3),
    (28672, 4096, 192): (50.2, 46.5), (37888, 4096, 192): (57.2, 57.4), (37888, 4096, 256): (58.4, 60.8), (38912, 4096, 192): (88.1, 67.9),
    (38912, 4096, 256): (81.2, 72.9), (45056, 4096, 192): (91.3, 73.5), (45056, 4096, 256): (80.1, 78.3), (49152, 4096, 192): (95.9, 80.2),
    (49152, 2048, 192): (52.4, 42.4), (51200, 4096, 192): (100.7, 81.5), (53248, 4096, 192): (102.6, 88.2), (53248, 4096, 256): (85.6, 90.0),
    (57344, 4096, 192): (105.9, 96.3), (57344, 4096, 256): (112.3, 100.8), (65536, 4096, 192): (112.2, 105.1), (65536, 4096, 256): (114.5, 109.1),
    (67584, 4096, 176): (99.9, 104.2), (67584, 2048, 256): (53.8, 58.1), (75776, 4096, 192): (121.0, 120.5), (75776, 4096, 256): (117.4, 124.9),
    (76800, 4096, 192): (154.7, 125.1), (76800, 4096, 256): (146.0, 133.9), (79872, 4096, 192): (151.8, 131.1), (90112, 2048, 192): (86.1, 73.3),
    (90112, 2048, 256): (67.3, 74.4),
}


def test_gate_up_takes_no_slower_kernel(rule):
    took = rule([f"gemm_wave_gains({n}, {int(r > 240)})" for n, _, r in GATE_UP])
    for (case, times), even in zip(GATE_UP.items(), took):
        assert within(times[even], times[0]), (case, even)
    assert within(sum(t[e] for t, e in zip(GATE_UP.values(), took)), sum(min(t) for t in GATE_UP.values()))


def test_units_of_the_widths_that_test_gpu_even_takes(rule):
    pads = (256, 9664, 18944, 19456, 28672, 37888, 60032)          # gates, in whole weight tiles
    got = rule([f"wave_share(2 * {f}).{what}" for f in pads for what in ("turns", "couples")])
    assert list(zip(got[::2], got[1::2])) == [(1, 16), (1, 136), (1, 256), (2, 136), (2, 200), (2, 256), (4, 208)]


# (parts, key tiles, query tiles x heads x sequences, rows of a query tile): by the CTAs that share the parts
ATTENTION = {
    (2, 2, 32, 128): {1: 13.2, 2: 10.1},
    (2, 17, 160, 128): {1: 79.0, 2: 67.5},
    (3, 3, 48, 128): {1: 17.3, 3: 21.3},
    (4, 5, 32, 32): {1: 12.9, 2: 11.2, 4: 9.2},
    (4, 5, 64, 128): {1: 19.3, 2: 18.4, 4: 22.9},
    (8, 17, 16, 128): {1: 43.2, 4: 23.1, 8: 28.0},
    (8, 9, 16, 32): {1: 18.3, 4: 11.8, 8: 17.0},
    (8, 33, 16, 128): {1: 72.5, 4: 31.8, 8: 36.4},
    (7, 7, 24, 128): {1: 26.9, 7: 22.9},
    (2, 2, 4, 64): {1: 9.6, 2: 8.6},
    (2, 3, 48, 128): {1: 14.9, 2: 11.9},
    (2, 17, 180, 128): {1: 86.4, 2: 70.3},
    (2, 2, 40, 128): {1: 13.7, 2: 9.9},
    (4, 33, 160, 128): {1: 144.7, 2: 129.9, 4: 121.2},
    (7, 7, 16, 128): {1: 25.2, 7: 20.7},
    (4, 4, 160, 128): {1: 34.1, 2: 44.7, 4: 51.5},
    (4, 4, 28, 128): {1: 18.1, 2: 16.4, 4: 12.1},
    (8, 33, 16, 128): {1: 71.7, 4: 30.0, 8: 34.6},
    (3, 3, 48, 64): {1: 11.5, 3: 16.9},
    (5, 5, 32, 128): {1: 19.5, 5: 21.3},
}


def test_attention_takes_no_slower_cluster(rule):
    took = rule([f"attn_pipe_ctas({p}, {t}, {w}, {q})" for p, t, w, q in ATTENTION])
    for (case, times), ctas in zip(ATTENTION.items(), took):
        assert within(times[ctas], min(times.values())), (case, ctas)


def test_attention_has_whole_clusters_of_its_parts(rule):
    sizes = [(p, t, w, q) for p in range(2, 9) for t in (p, 2 * p + 1, 257) for w in (1, 33, 149, 4096) for q in (32, 64, 128)]
    for (parts, *_), ctas in zip(sizes, rule(["attn_pipe_ctas(%d, %d, %d, %d)" % s for s in sizes])):
        assert ctas in (1, parts, parts / 2)


# (tiles, splits, K blocks, row blocks, rows of one, CTAs of the kernel in front): single tiles, pairs
RESIDUAL = {
    (2, 4, 8, 1, 128, 8): (8.1, 8.7),
    (4, 4, 16, 1, 256, 16): (11.7, 12.2),
    (8, 4, 16, 1, 128, 16): (8.5, 9.1),
    (8, 4, 8, 2, 144, 16): (8.9, 9.6),
    (12, 4, 24, 1, 128, 24): (8.6, 9.4),
    (16, 4, 16, 1, 128, 16): (8.2, 8.9),
    (16, 4, 16, 2, 144, 32): (10.2, 20.1),
    (16, 4, 24, 2, 192, 48): (12.1, 22.3),
    (20, 4, 32, 1, 160, 32): (11.2, 10.8),
    (20, 4, 96, 2, 176, 192): (30.1, 24.0),
    (24, 4, 64, 1, 256, 64): (18.3, 18.4),
    (24, 4, 128, 1, 160, 128): (19.8, 18.6),
    (24, 4, 192, 2, 144, 384): (34.0, 31.0),
    (28, 4, 64, 2, 160, 128): (21.9, 20.8),
    (28, 4, 296, 1, 128, 296): (30.0, 29.1),
    (28, 4, 296, 2, 176, 592): (64.8, 47.1),
    (28, 4, 296, 2, 224, 592): (74.0, 63.1),
    (32, 4, 32, 2, 144, 64): (17.1, 22.5),
    (32, 4, 96, 2, 160, 192): (25.5, 37.5),
    (32, 4, 128, 2, 176, 256): (36.2, 29.0),
    (32, 4, 192, 2, 144, 384): (36.0, 33.2),
    (32, 4, 192, 2, 192, 384): (48.6, 41.6),
    (32, 4, 224, 2, 192, 448): (55.0, 70.9), (32, 4, 224, 2, 144, 448): (39.8, 42.6), (32, 4, 256, 2, 176, 512): (60.5, 58.0),
    (32, 4, 240, 2, 144, 480): (42.9, 52.1), (32, 4, 272, 2, 192, 544): (65.5, 54.4), (32, 4, 352, 2, 144, 704): (58.0, 51.8), (32, 4, 384, 2, 160, 768): (63.1, 92.7),
    (32, 4, 296, 2, 160, 592): (53.5, 48.1),
}


def test_residual_tiles_are_paired_where_that_is_no_slower(rule):
    took = rule(["residual_pairs(%d, %d, %d, %d, %d, %d)" % c for c in RESIDUAL])
    for (case, times), pairs in zip(RESIDUAL.items(), took):
        assert within(times[pairs], times[0]), (case, pairs)
    assert within(sum(t[p] for t, p in zip(RESIDUAL.values(), took)), sum(min(t) for t in RESIDUAL.values()))
