"""The word-sized prime's arithmetic as the kernels compile it, built for the host: ranges and residues."""
import os
import random
import subprocess

HOST = os.path.join(os.path.dirname(os.path.abspath(__file__)), "host")
CSRC = os.path.join(os.path.dirname(os.path.dirname(HOST)), "paper_1809_07592_gb300", "csrc")


def test_products_butterflies_and_canonical_values(tmp_path):
    exe = str(tmp_path / "residues")
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", HOST, "-I", CSRC, os.path.join(HOST, "residues.cpp"), "-o", exe], check=True)
    q = 7 * 2**26 + 1
    rng = random.Random(3)
    ends = [0, 1, q - 1, q, q + 1, 2 * q - 1, 2 * q, 3 * q, 4 * q - 1]  # lazy residues, [0, 4q)
    rows = [(a, b, w) for a in ends for b in ends for w in (0, 1, 2, q // 2, q - 2, q - 1)]
    rows += [(rng.randrange(4 * q), rng.randrange(4 * q), rng.randrange(q)) for _ in range(20000)]
    out = subprocess.run([exe], input="\n".join("%d %d %d" % r for r in rows), check=True, capture_output=True, text=True,
                         timeout=120).stdout.split("\n")
    got_q, lg, root = map(int, out[0].split())
    assert (got_q, lg) == (q, 26) and pow(root, 32, q) == 1 and pow(root, 16, q) == q - 1
    for (a, b, w), line in zip(rows, out[1:]):
        bw, aw, add, sub, add1, sub1, canon, back, quot = map(int, line.split())
        assert bw < 2 * q and aw < 2 * q and (bw - b * w) % q == 0 and (aw - a * w) % q == 0
        assert max(add, sub, add1, sub1) < 4 * q
        assert (add - a - b * w) % q == (sub - a + b * w) % q == (add1 - a - b) % q == (sub1 - a + b) % q == 0
        assert canon == back == a % q and quot == (canon << 32) // q
