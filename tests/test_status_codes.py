"""The second word of the status block says which kernel and role gave up: no two places record the same number."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_00916_b200", "csrc")


def read(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


def test_no_two_places_record_the_same_timeout():
    kinds = read("common.cuh")
    kinds = re.search(r"enum GemmKind \{(.*?)GEMM_KINDS", kinds, re.S).group(1).count("GEMM_")
    assert kinds >= 8
    seen = {}
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh")):
            for i, (base, kind) in enumerate(re.findall(r"record_status\([^,]*, DEV_TIMEOUT, (\d+)( \+ KIND)?\)", read(name))):
                for code in range(int(base), int(base) + (kinds if kind else 1)):
                    assert code not in seen, f"{code}: {name} and {seen[code]}"
                    seen[code] = f"{name}, place {i}"
    assert len(seen) >= 9 * kinds + 3
