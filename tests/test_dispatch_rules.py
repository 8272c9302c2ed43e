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
