"""What the kernels' sources have to keep to and no run shows."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_04214_b200", "csrc")


def code_lines(name):
    """The lines of a source without their comments, empty ones left out."""
    text = re.sub(r"/\*.*?\*/", "", open(os.path.join(CSRC, name)).read(), flags=re.S)
    lines = (re.sub(r"//.*", "", line).strip() for line in text.splitlines())
    return [line for line in lines if line]


def test_warps_are_whole_at_every_named_barrier():
    """A named barrier is an .aligned instruction: undefined unless all lanes of a warp execute it together, which nothing promises
    behind a lane's own wait or branch.  So each call of the helpers stands right behind a __syncwarp()."""
    calls = 0
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh")):
            continue
        lines = code_lines(name)
        for before, line in zip(lines, lines[1:]):
            if re.search(r"\bnamed_barrier_(and|sync)\(", line) and "__device__" not in line:
                calls += 1
                assert before == "__syncwarp();", (name, line)
    assert calls > 0
