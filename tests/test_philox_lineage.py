"""What the transport keeps of a lineage instead of it, over counters and keys of
random and extreme words: all four words of every draw equal Philox4x32-10 of the
counter, also after a particle record kept two of the three words, and the
lineage itself (the parent's, from which a secondary's is made) comes back."""
import os
import subprocess

from paper_1101_1245_gb300 import build as b

HERE = os.path.dirname(os.path.abspath(__file__))


def test_draws_and_lineage_of_any_counter(tmp_path):
    exe = str(tmp_path / "philox_lineage")
    subprocess.run([b.nvcc(), "-std=c++17", "-O2", *b.ARCH, "-I", b.INCLUDE, "-I", b.CSRC, "-o", exe,
                    os.path.join(HERE, "philox_lineage.cu")], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.startswith("0 of ")
