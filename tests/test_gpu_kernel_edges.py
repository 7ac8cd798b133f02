"""The hot kernels at the edges of their layouts: pixel panels and column
blocks of the FP32 Gram."""
import numpy as np
import pytest
import torch

from paper_2509_05464_gb300 import build as fqbuild
from paper_2509_05464_gb300 import fq

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    fqbuild.build()
    fq.lib()


# products of a sum of 2 P terms in binary32, any order: within gamma_2P of
# the sum of magnitudes
@pytest.mark.parametrize("F", [2, 3, 4, 5, 31, 100, 130, 201, 260])
@pytest.mark.parametrize("P,dt", [(1, "f32"), (15, "f32"), (33, "f32"), (1000, "f32"), (5003, "f32"), (1000, "bf16")])
def test_gram_panels(F, P, dt):
    g = torch.Generator(device="cuda").manual_seed(F * 1000 + P)
    S = torch.randn((P, F, 2), generator=g, device="cuda").to(torch.float32 if dt == "f32" else torch.bfloat16)
    G = torch.view_as_complex(fq.fq_casorati_gram(S).double().contiguous())
    s = torch.view_as_complex(S.double().contiguous())
    mag = (S.double().abs().sum(2)).mT @ S.double().abs().sum(2)
    err = (G - s.mH @ s).abs()
    assert bool((err <= 2.0 ** -24 * (2 * P + 16) * mag).all())
