"""The word-sized exact transform: its prime's properties (CPU) and the length rule that selects it (GPU)."""
import numpy as np
import pytest

Q = 7 * 2**26 + 1


def test_prime_covers_every_count_and_length():
    """q is prime (trial division), exceeds the largest count 2^27, has roots of order 2^26, and 3 generates."""
    assert all(Q % d for d in range(2, int(Q**0.5) + 1))
    assert Q > 2**27 and (Q - 1) % 2**26 == 0 and 4 * Q < 2**32
    assert all(pow(3, (Q - 1) // p, Q) != 1 for p in (2, 7))  # q - 1 = 7 * 2^26


def test_lazy_butterfly_ranges():
    """The butterfly's bounds at the ends of its ranges: products below 2q, sums and differences below 4q."""
    rng = np.random.default_rng(1)
    w = np.concatenate([[0, 1, Q - 1], rng.integers(0, Q, 2000)]).astype(object)
    b = np.concatenate([[0, 1, Q, 2 * Q - 1, 4 * Q - 1, 2**32 - 1], rng.integers(0, 2**32, 2000)]).astype(object)
    for x in w[:64]:
        wq = (int(x) << 32) // Q
        t = np.array([(int(y) * int(x) - (int(y) * wq >> 32) * Q) % 2**32 for y in b], dtype=object)
        assert all(0 <= v < 2 * Q for v in t) and all((v - int(x) * int(y)) % Q == 0 for v, y in zip(t, b))
    a, t = 4 * Q - 1, 2 * Q - 1
    a1 = min(a, (a - 2 * Q) % 2**32)
    assert a1 < 2 * Q and a1 + t < 4 * Q and 0 <= a1 - t + 2 * Q < 4 * Q


@pytest.mark.gpu
@pytest.mark.parametrize("need", [2**25 + 1, 2**26, 2**26 + 1])
def test_lengths_around_the_rule_agree_with_fp64(need):
    """Whole outputs at the last length of the word-sized prime and the first of the 64-bit one, two keys each."""
    import torch

    import paper_1809_07592_gb300 as pa
    m = 2**20 + 3
    n = need - m + 1
    g = torch.Generator(device="cuda").manual_seed(need)
    words = lambda *s: torch.randint(-(1 << 63), (1 << 63) - 1, s, generator=g, device="cuda", dtype=torch.int64)
    keys, seed = words(2, (n + 127) // 128 * 2), words((need + 127) // 128 * 2)
    outs = []
    for dtype in (pa.PA_NTT64, pa.PA_FP64):
        plan = pa.Plan(n, m, dtype)
        plan.set_seed(seed)
        out = torch.zeros((2, (m + 127) // 128 * 2), dtype=torch.int64, device="cuda")
        outs.append(plan.hash(keys, out).clone())
        torch.cuda.synchronize()
        plan.close()
    assert torch.equal(outs[0], outs[1])
