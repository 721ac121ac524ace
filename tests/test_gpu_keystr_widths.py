"""pk_key_strings at the row widths whose characters a warp encodes together
(multiples of 64 bytes) and at their neighbours, with prefixes that end inside
and on a 4-byte word, rows that leave a partial warp and a partial tile, and
more tiles than fit the GPU at once, so that both of a CTA's tiles are filled
and reused.  Bit-exact against the oracle."""
import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()
    if not torch.cuda.is_available():
        pytest.skip("no GPU")


@pytest.mark.parametrize("width,plen", [(22, 0), (23, 1), (63, 41), (64, 0), (64, 42), (65, 7), (128, 53), (192, 170),
                                        (255, 233), (256, 0), (256, 127), (256, 234)])
@pytest.mark.parametrize("n", [1, 31, 33, 257, 1023, 500001])
def test_rows_bit_exact(width, plen, n):
    from paper_2609_38706_gb300 import pk
    rng = np.random.default_rng(width * 1000 + plen + n)
    keys = rng.integers(0, 256, (n, 32), dtype=np.uint8)
    prefix = bytes(rng.integers(1, 256, plen, dtype=np.uint8))
    buf = torch.full((n * width + 32,), 0xA5, dtype=torch.uint8, device="cuda")
    pk.pk_key_strings(torch.from_numpy(keys).cuda(), prefix, width, buf, n=n)
    got = buf.cpu().numpy()
    assert np.array_equal(got[:n * width].reshape(n, width), O.key_strings(keys, prefix, width))
    assert (got[n * width:] == 0xA5).all()
