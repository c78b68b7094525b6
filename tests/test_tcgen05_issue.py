"""tcgen05.commit tracks only the MMAs of the thread that executes it, so a kernel whose MMAs are issued by the lane that
elect_one() picks has to commit from that lane too, its last commit (before TMEM is freed) included. Checked on the
source text: an MMA that a commit misses shows only after a timeout, as TMEM freed while the tensor core still writes it."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_01718_gb300", "csrc")
ISSUE = re.compile(r"\b(?:mma_bf16|mma_e4m3|mma_commit)\s*(?:<[^<>;()]*>)?\s*\(")


def _elected(text, at):
    """Whether the call at offset `at` is under an `if (elect_one())`: its own statement, or a block around it."""
    if "elect_one()" in re.split(r"[;{}]", text[:at])[-1]:
        return True
    depth = 0
    for i in range(at - 1, -1, -1):
        if text[i] == "}":
            depth += 1
        elif text[i] == "{":
            depth -= 1
            if depth < 0:   # the head of an enclosing block
                depth = 0
                if "elect_one()" in re.split(r"[;{}]", text[:i])[-1]:
                    return True
    return False


def test_every_mma_and_commit_is_issued_by_the_elected_lane():
    calls = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in ISSUE.finditer(text):
            if re.search(r"\bvoid\s+$", text[:m.start()]):   # the definition
                continue
            line = text.count("\n", 0, m.start()) + 1
            assert _elected(text, m.start()), f"{os.path.basename(path)}:{line}: not under elect_one()"
            calls += 1
    assert calls >= 8   # both tensor-core kernels: the MMA, two commits per use of it and the drain
