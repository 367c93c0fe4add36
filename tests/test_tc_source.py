"""The split-BF16 kernel's whole-warp roles: their barrier answers are voted on by the warp before anything
depends on them, because warp-collective (.sync.aligned) tensor-memory instructions follow."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_barrier_answers_are_voted_on():
    src = open(os.path.join(ROOT, "paper_2412_02246_gb300", "csrc", "triple_tc.cu")).read()
    body = src[src.index("k_triple_tc(TcParams G"):]
    body = re.sub(r"//[^\n]*", "", body[:body.index("\n}\n")])
    loader = body[body.index("if (warp == 0) {\n"):body.index("else if (warp <= NISS)")]
    rest = body.replace(loader, "")
    # one lane loads; every other wait goes through a vote
    assert re.findall(r"mbar_wait\(", rest) and all(
        rest[:m.start()].rstrip().endswith("__all_sync(FULL,") for m in re.finditer(r"mbar_wait\(", rest))
    # answers of the non-blocking tests are read through a vote only
    answers = set(re.findall(r"(\w+) = [^;]*mbar_test\(", rest))
    assert answers
    for a in answers:
        uses = [m for m in re.finditer(rf"\b{a}\b", rest)
                if not re.match(rf"{a} = ", rest[m.start():])]
        assert uses and all(rest[:m.start()].endswith("__all_sync(FULL, ") for m in uses), a
