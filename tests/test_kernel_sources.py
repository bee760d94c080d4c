"""What the kernels' sources have to keep to and no run shows."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2511_04214_b200", "csrc")


def code_lines(name):
    """The lines of a source without their comments, empty ones left out."""
    text = re.sub(r"/\*.*?\*/", "", open(os.path.join(CSRC, name)).read(), flags=re.S)
    lines = (re.sub(r"//.*", "", line).strip() for line in text.splitlines())
    return [line for line in lines if line]


def test_no_barrier_by_hand():
    """bar.sync and its kin are .aligned instructions: undefined unless all lanes of a warp execute them together, which nothing
    promises behind a lane's own wait or branch.  The threads of a block meet at __syncthreads(), before which the compiler joins
    them."""
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh")):
            for line in code_lines(name):
                assert not re.search(r"\bbar(rier)?\.(cta\.)?(sync|red|arrive)\b", line), (name, line)
