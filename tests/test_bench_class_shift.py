"""The class shift that bench.py reports: the library's rule (EPI_TC_AUTO), from
the largest counts of a genotype-0 or -1 row, on both sides of 2^24."""
from types import SimpleNamespace

import numpy as np
import pytest

import bench


@pytest.mark.parametrize("c1,c0,shift", [(1, 0, 1), (3, 1, 2), (4094, 4094, 12), (4095, 4094, 12), (4096, 4094, 0),
                                         (4095, 4095, 0), (2047, 4095, 13), (2048, 4095, 0), (3, 8190, 13)])
def test_class_shift(c1, c0, shift):
    # one SNP: c1 cases and c0 controls of genotype 1, the others of genotype 2
    m1, m0 = c1 + 3, c0 + 5
    geno = np.full((1, m1 + m0), 2, np.uint8)
    geno[0, :c1] = 1
    geno[0, m1:m1 + c0] = 1
    pheno = (np.arange(m1 + m0) < m1).astype(np.uint8)
    assert bench.class_shift(SimpleNamespace(geno=geno, pheno=pheno)) == shift
    assert (c1 * (1 << shift) + c0 < 1 << 24) if shift else c1 * (1 << (c0 + 1).bit_length()) + c0 >= 1 << 24
