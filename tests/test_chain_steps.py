"""Steps of a Metropolis chain near the end of the history range: a call may
advance up to 2^32 - 1 histories over up to 2^24 chains, where the count of
steps has to be rounded up without leaving 32 bits.  Host arithmetic, no GPU."""
import os
import subprocess

from paper_1107_3355_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))


def test_steps_and_tiles_at_the_end_of_the_range(tmp_path):
    exe = str(tmp_path / "chain_steps_host")
    subprocess.check_call([B.nvcc(), *B.ARCH, "-std=c++17", "-I", B.INCLUDE, "-I", B.CSRC,
                           os.path.join(HERE, "cuda", "chain_steps_host.cu"), "-o", exe])
    top = 2 ** 32 - 1
    cases = [(n, c, 56) for c in (1, 2, 31, 4096, 2 ** 24 - 1, 2 ** 24)
             for n in (1, c - 1, c, c + 1, 56 * c, top // 300 * 299, top - c, top - c + 1, top - 1, top)
             if 0 < n <= top]
    # batch 299 of 300 of the largest calculation starts here, with the most chains
    cases.append((4280650738, 2 ** 24, 56))
    out = subprocess.run([exe], input="".join("%d %d %d\n" % c for c in cases), capture_output=True, text=True,
                         check=True).stdout.split("\n")
    for (n, c, tile), line in zip(cases, out):
        steps = -(-n // c)
        assert line == "%d %d" % (steps, -(-steps // tile)), (n, c)
    assert len(out) == len(cases) + 1
