"""Admission counts the record blocks that a request's packets own (CPU)."""
import pytest

from paper_1309_3458_gb300 import serving as S
from tests.test_serving_host import _req, _server

BLOCK = 5184 + 4 + 8 + 16  # words of a block, count, owner, list entry


@pytest.mark.parametrize("size,packets", [(1, 1), (1000, 250), (9728, 2432), (9729, 2433), (19455, 2432),
                                          (19456, 2432), (38912, 2432), (77824, 2432), (200000, 6250),
                                          (1000001, 31251)])
def test_first_blocks_of_a_request(size, packets):
    """Packets of 4 to 32 queries, as many as fill 152 SMs with 16 each."""
    srv = _server()
    want = 2 * packets * BLOCK
    got = S.first_record_bytes(size, srv.sms)
    assert want <= got <= 1.5 * want
    r = _req(0, size)
    assert srv.estimate(r) >= want + 16 * r.est_pairs + size * 72
