"""What vla_backward asks for in scratch memory, as include/vla.h states it (no GPU: a size query)."""
import random

import paper_2605_11196_b200 as vla


def _token_level(B, H, T, d):
    """Seven vectors, a word per token, the key sum per 16 tokens, two matrices and a vector per unit, progress words."""
    r = lambda n: (n + 255) // 256 * 256
    u = B * H
    return 7 * r(4 * u * T * d) + r(4 * u * T) + 2 * r(4 * u * d * d) + r(4 * u * d) + r(4 * u * ((T + 15) // 16) * d) + r(4 * (u + 1)) + 256


def test_workspace_stays_below_its_bound():
    rng = random.Random(5)
    shapes = [(8, 16, 2048, 128), (1, 512, 8192, 128), (8, 16, 65536, 128), (16, 16, 65536, 128), (1, 128, 16384, 128), (1, 4096, 4096, 64)]
    for _ in range(300):
        T = int(2 ** rng.uniform(0, 17))
        shapes.append((int(2 ** rng.uniform(0, 7)), int(2 ** rng.uniform(0, 9)), T, rng.choice((16, 32, 64, 128))))
    for B, H, T, d in shapes:
        one = vla.backward_workspace_bytes(1, 1, T, d)
        got = vla.backward_workspace_bytes(B, H, T, d)
        assert got >= _token_level(B, H, T, d)
        assert got <= max(4 << 30, _token_level(B, H, T, d), one) + 8 * B * H + 1024, (B, H, T, d, got)   # (a few words per unit)
