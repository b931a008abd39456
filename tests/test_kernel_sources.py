"""Rules of the kernel sources that no run on a GPU shows reliably."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2401_16757_gb300", "csrc")
WEIGHTS = {"W", "g", "table"}  # parameters that hold weights (g: RMSNorm gains; table: the embedding's)


def _kernels():
    """(file, head, body) of every kernel that starts before the launch ahead of it has ended."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"__global__", text):
            start = text.index("{", m.end())
            end = text.index("\n}", start)
            if "pdl_wait()" in text[start:end]:
                yield os.path.basename(path), text[m.end():start], text[start:end]


def test_outputs_of_an_overlapped_launch_are_not_read_as_read_only():
    """A read-only load (ld.global.nc) is for memory that nothing writes while the kernel runs, and may be moved across
    the wait for the launch before, which is still writing this kernel's inputs when it starts."""
    seen = 0
    for name, head, body in _kernels():
        seen += 1
        assert "__ldg(" not in body, (name, head)
        params = re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", head)
        assert set(params) <= WEIGHTS, (name, params)
    assert seen >= 18


def test_rotation_releases_the_attention_after_its_wait():
    """The attention kernels read the position and older cache rows before their own wait: what they overlap, the
    rotation launched right before them, lets them start only once everything ahead of it has ended."""
    bodies = [body for _, head, body in _kernels() if "rope_append_kernel" in head]
    assert len(bodies) == 1
    assert 0 <= bodies[0].index("pdl_wait()") < bodies[0].index("pdl_launch_dependents()")
    assert not re.search(r"\breturn\b", bodies[0][:bodies[0].index("pdl_launch_dependents()")])
    text = open(os.path.join(CSRC, "k_decoder.cu")).read()
    launch = text[text.index("int launch_attention("):]
    between = launch[launch.index("rope_append_kernel<T, 1, 1>"):launch.index("attention_split_kernel<T>, static_cast")]
    assert between.count("launch_pdl(") == 0 and between.count("launch_attention_tc(") == 1
