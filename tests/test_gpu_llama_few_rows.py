"""Decoder layers of few rows, whose RMSNorm is part of the QKV product: sizes on both sides of the rule, rows that are not multiples of the
product's 16, several sequences, partial rotary embedding."""
import pytest

from tests.test_gpu_llama import case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,S,hidden,rot", [(1, 17, 256, 32), (2, 20, 512, 0), (3, 11, 1024, 64), (1, 40, 256, 0), (1, 41, 256, 0), (2, 32, 3072, 32),
                                            (5, 13, 3072, 0)])
def test_layer(B, S, hidden, rot):
    case(710, B, S, hidden, hidden // 128, 1, rotary_dim=rot)
