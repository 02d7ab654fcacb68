"""The constant pairs of the per-path kernels (csrc/fast/path_pairs.inc) against the oracle's coupling tensors."""
import os
import re

import numpy as np

from oracle import cg


def test_both_orders_of_every_path_are_the_oracle_tensor(repo_root):
    text = open(os.path.join(repo_root, "paper_2609_35099_b200", "csrc", "fast", "path_pairs.inc")).read()
    triples = [tuple(map(int, t)) for t in re.findall(r"X\((\d), (\d), (\d)\)", text)]
    want = [(a, b, c) for a in range(4) for b in range(4) for c in range(abs(a - b), min(a + b, 3) + 1)]
    assert triples == want
    for l1, l2, L in triples:
        ref = np.asarray(cg.real_cg_block(l1, l2, L), dtype=np.float64)
        assert ref.shape == (2 * L + 1, 2 * l1 + 1, 2 * l2 + 1)
        for side in (0, 1):
            body = re.search(rf"#define E3J_PATH_BY{side}_{l1}{l2}{L}\(B, P1, P2, E\) (.*)", text).group(1)
            got, row = np.zeros_like(ref), None
            for op, args in re.findall(r"(B|P1|P2|E)\(([^)]*)\)", body):
                a = [float(v) for v in args.split(",")]
                if op == "B":
                    row = int(a[0])
                elif op == "E":
                    assert row == int(a[0])
                else:
                    for i, c in zip(a[1::2], a[2::2]):
                        m0, m1 = (row, int(a[0])) if side == 0 else (int(a[0]), row)
                        assert got[m0, m1, int(i)] == 0
                        got[m0, m1, int(i)] = c
            np.testing.assert_allclose(got, ref, rtol=0, atol=1e-14)
