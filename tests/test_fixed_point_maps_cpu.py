"""Host checks of the FP64 form's shared-memory lines (restated from fft_core.cuh and
fixed_point.cuh): padding every 8 values, addresses of a pass as a base plus compile-time offsets,
and stores that meet no bank twice in a quarter-warp."""

import pytest

SIZES = (4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 128, 256, 512, 1024)


def pad(p):
    return p + (p >> 3)


def plans(L):
    three = L % 3 == 0
    a = (L // 3 if three else L).bit_length() - 1
    n8 = a // 3 - 1 if a % 3 == 1 and a > 1 and L != 16 else a // 3
    rest = a - 3 * n8
    default = [8] * n8 + {0: [], 1: [2], 2: [4], 4: [4, 4]}[rest] + [3] * three
    odd = ([2] if a == 1 else [8]) if a % 2 else []
    n4 = (0 if a == 1 else (a - 3) // 2) if a % 2 else a // 2
    return default, [3] * three + [4] * n4 + odd


@pytest.mark.parametrize("L", SIZES)
def test_passes_address_the_line_once_by_base_and_offset(L):
    for radices in plans(L):
        ns, size = 1, 1
        for r in radices:
            size *= r
        assert size == L
        for R in radices:
            nb = L // R
            reads, writes = set(), set()
            for j in range(nb):
                base = (j // ns) * ns * R + j % ns
                for r in range(R):
                    reads.add(j + r * nb)
                    writes.add(base + r * ns)
                    if L & (L - 1) == 0:
                        assert pad(j + r * nb) == pad(j) + pad(r * nb)
                        assert pad(base + r * ns) == pad(base) + pad(r * ns)
            assert reads == writes == set(range(L))
            ns *= R


@pytest.mark.parametrize("L", [64, 128, 256, 512, 1024])
def test_first_pass_stores_meet_no_bank_twice(L):
    # eight 16-byte values cover all the banks; a quarter-warp is eight lanes, at element stride 1
    # (x lines) and at the odd strides of the y and z tiles
    for stride in (1, 5, 9, 13, 25, 49):
        for j0 in range(0, L // 8, 8):
            for r in range(8):
                assert len({pad(8 * j + r) * stride % 8 for j in range(j0, j0 + 8)}) == 8
