"""Which fixed observation layouts solve with several particles per CTA: a
CTA of P particles keeps their right-hand sides (n doubles each) in shared
memory, so a layout too large for that must take a warp per particle,
whatever the number of particles (no GPU needed)."""
import pytest

from paper_1910_01031_gb300 import iewpf

SMEM_MAX = 227 * 1024        # dynamic shared memory of a CTA at most


# 3064, 6140: the last that fit 8 and 4 particles; 6144: the last with its right-hand side in the shared memory
# of a warp; 29056: the last of a wave estimate of 1 by shared memory; then the largest 32-bit layouts
@pytest.mark.parametrize("n", [2, 512, 3042, 3064, 3066, 6128, 6140, 6142, 6144, 6146, 29054, 29056, 29058, 29060, 65534])
@pytest.mark.parametrize("sms", [1, 132, 152])
def test_a_group_is_chosen_only_where_its_vectors_fit(n, sms):
    for ne in (1, 3, 4, 40, 100, 152, 608, 1000, 5000, 65535):
        P = iewpf.solve_group(n, ne, sms)
        assert P in (1, 4, 8)
        if P > 1:
            assert 8 * n * P < SMEM_MAX, (n, ne, sms, P)


def test_large_layouts_and_the_benchmark_layout():
    for ne in (1, 10, 1000):
        assert iewpf.solve_group(2 * 14529, ne) == 1
    # 1521 coupled moorings: one wave of 8 particles per CTA at 1000, 4 at 100
    assert iewpf.solve_group(3042, 1000) == 8
    assert iewpf.solve_group(3042, 100) == 4


def test_arguments_are_checked():
    for bad in ((0, 1, 1), (2, 0, 1), (2, 1, 0)):
        with pytest.raises(iewpf.IewpfError):
            iewpf.solve_group(*bad)
