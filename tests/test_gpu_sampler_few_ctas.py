"""The one-launch sampler where its CTAs are few: at 32 CTAs of 16 vocabulary tiles every CTA
reads all keys itself, one tile more takes the leaders' exchange."""
import pytest

from tests.test_gpu_sampler_groups import test_sampler_edges as _edges

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,B,V,rc,temperature", [
    (16, 3, 16384, 64, 1.0),    # 32 CTAs, two groups of requests
    (9, 3, 16400, 32, 0.0),     # 33 CTAs: leaders
    (7, 4, 1024, 64, 0.7),      # a tile a CTA
    (16, 2, 224, 32, 1.0),      # seven CTAs write the tokens of groups of eight
])
@pytest.mark.parametrize("noalloc", [False, True])
def test_sampler_few_ctas(C, B, V, rc, temperature, noalloc):
    _edges(C, B, V, rc, temperature, noalloc)
