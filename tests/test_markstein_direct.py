"""The square root of the device generator as it is (one Markstein correction
of the reciprocal-square-root approximation, without refining the seed first):
the IEEE result on every radicand from the correctly rounded seed, and off for
three of them from a seed one ulp away (tests/host/markstein_direct.c).  So the
steps alone do not prove the device's roots whatever its approximation gives;
test_gpu_box_muller_all.py, which runs every radicand on the device, does."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def test_roots_from_the_rounded_seed_and_its_neighbours(orc, tmp_path):
    exe = str(tmp_path / "markstein_direct")
    src = os.path.join(HERE, "host", "markstein_direct.c")
    subprocess.run(["gcc", "-O2", "-std=c11", "-ffp-contract=off", "-fno-fast-math",
                    "-frounding-math", src, orc.build(), "-o", exe, "-lm"], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, check=True)
    words = r.stdout.split()
    assert int(words[2]) == 0, r.stdout
    assert int(words[4]) == 3, r.stdout
