"""Host-side rules that choose a form of the greedy loop, compiled from the library's own headers."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    """A program that reads one question per line and answers it."""
    from paper_2211_00839_b200 import build
    out = str(tmp_path_factory.mktemp("rules") / "rules")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(os.path.dirname(os.path.dirname(build._nvcc())), "include"),
                    "-I", os.path.join(ROOT, "include"), "-I", build.CSRC, os.path.join(ROOT, "tests", "dispatch_rules.cpp"), "-o", out], check=True)

    def ask(questions):
        text = "\n".join(" ".join(map(str, q)) for q in questions) + "\n"
        answers = subprocess.run([out], input=text, capture_output=True, text=True, check=True).stdout.splitlines()
        assert len(answers) == len(questions)
        return [tuple(map(int, a.split())) for a in answers]
    return ask


def test_graph_cut_values_fit_the_packed_word(rules):
    """f(A) of int8 features reaches M^2 / 4 * 2^14 * d; the packed word holds what lies below 2^55."""
    sizes = [1, 2, 5000, 8191, 8192, 8193, 12000, 16384, 23170, 23171, 30000, 32767, 32768, 65535]
    widths = [1, 16, 64, 512, 2048, 4096, 8191, 8192, 16384, 57883, 65535, 129089, 131071]
    questions = [("cut_values", M, d) for M in sizes for d in widths]
    for (_, M, d), (fits,) in zip(questions, rules(questions)):
        assert fits == (M * M // 4 * 16384 * d < 1 << 55), (M, d)
        if fits and M <= 32768:
            # and the gains fit the 48 bits of a key: within three times the largest sum of a row, either way
            assert 6 * M * 16384 * d + 1 < 1 << 48, (M, d)


B200 = (148, 232448)        # SMs, bytes of shared memory a CTA can ask for


def test_graph_cut_in_step_covers_every_column(rules):
    """Whatever the sizes and the largest cluster that the GPU can place (none at all on a slice of a few SMs)."""
    import random
    rng = random.Random(5)
    log = lambda lo, hi: int(round(lo * (hi / lo) ** rng.random()))      # noqa: E731
    questions = [("cut_plan", *rng.choice([B200, B200, (16, 232448), (1, 232448), (132, 101376)]), rng.choice([1, 2, 4, 8, 16]), log(1, 2000), log(1, 65535),
                  log(1, 131071), log(1, 200)) for _ in range(20000)]
    taken = 0
    for (_, sms, shared, most, L, M, d, W), (C, K, warps, columns, smem) in zip(questions, rules(questions)):
        if C == 0:
            continue
        taken += 1
        assert C in (1, 2, 4, 8, 16) and C <= most and K in (1, 2, 3, 4, 8) and 1 <= warps <= 8
        assert C * columns >= M and columns % 32 == 0 and warps * 32 * K >= columns and smem == W * columns * 8 <= shared - 8192
        assert M * M // 4 * 16384 * d < 1 << 55 and W <= 128
    assert taken > 2000


def test_graph_cut_in_step_without_large_clusters(rules):
    """A class that wants a cluster of 16 takes the largest there is, and another form where its gains do not fit that."""
    ask = lambda most, M, W: rules([("cut_plan", *B200, most, 1, M, 64, W)])[0][0]      # noqa: E731
    assert [ask(m, 6000, 12) for m in (16, 8, 4, 2, 1)] == [16, 8, 4, 0, 0]
    assert [ask(m, 1300, 8) for m in (16, 8, 4, 2, 1)] == [8, 8, 4, 2, 1]


def test_shapes_compared_on_the_gpu_take_what_they_name(rules):
    """The graph cut in step: every number of columns per thread, alone and in clusters."""
    from test_gpu_cut_lockstep import SHAPES
    got = rules([("cut_plan", *B200, 16, L + 1, M, 16, W) for L, M, W, _, _ in SHAPES])
    assert [(C, K) for C, K, *_ in got] == [(C, K) for *_, C, K in SHAPES]
    assert {K for *_, K in SHAPES} == {1, 3, 4, 8}          # (two: a class of 6000 into 12 blocks, beside them)


def test_graph_cut_in_step_where_it_is_the_faster_form(rules):
    """Either side of the choice as measured (ms on a B200): in step against clusters of C CTAs, or against a CTA per class."""
    uneven = lambda L, M: [M] + [round(M * (l + 0.5) / L) for l in range(L - 1)]       # noqa: E731
    faster, slower = [
        ("clusters", 8, 8, 16, [5000] * 10),        # 7.2, 8.7
        ("clusters", 8, 4, 33, [2500] * 30),        # 3.6, 5.1
        ("clusters", 8, 1, 148, [700] * 200),       # 1.2, 2.9
        ("chain", 100, 0, 0, [3000] * 2),           # 3.0, 11.7
        ("chain", 65, 0, 0, [770, 5]),
    ], [
        ("clusters", 7, 2, 74, [1941] * 70),        # 4.8, 3.8
        ("clusters", 6, 2, 74, [609] * 67),         # 0.90, 0.85
        ("clusters", 6, 4, 33, uneven(83, 1051)),   # 2.5, 1.6
        ("clusters", 9, 4, 33, uneven(86, 1068)),   # 2.5, 2.1
        ("chain", 111, 0, 0, [1383] * 208),         # 20.7, 7.4
        ("chain", 124, 0, 0, [2955] * 92),          # 46.4, 20.4
        ("chain", 107, 0, 0, uneven(183, 1633)),    # 10.8, 8.8
    ]
    got = rules([("cut_cycles", W, max(C, 1), max(at, 1), len(sizes), *sizes) for _, W, C, at, sizes in faster + slower])
    for k, ((other, *_, sizes), (steps, clusters, chain)) in enumerate(zip(faster + slower, got)):
        assert steps > 0
        assert (steps <= (clusters if other == "clusters" else chain)) == (k < len(faster)), (other, sizes[0], len(sizes))


def test_finish_time_of_uneven_classes(rules):
    """Largest first on the machine that is free first: two clusters take 9 + 2 and 7 + 6, costs by the number of samples alone."""
    (_, two, _), (_, one, _) = rules([("cut_cycles", 1, 1 << 20, 2, 4, 9, 7, 6, 2), ("cut_cycles", 1, 1 << 20, 1, 4, 9, 7, 6, 2)])
    assert two == 13 * 1200 and one == 24 * 1200
