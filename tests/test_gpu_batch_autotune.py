"""The autotuner of batches keeps the work list that pic_batch_init made where no list
of its own is faster: a single run of 200,000 markers, which that list spreads over 49
blocks of one trip, took lists of three trips and more."""
import pytest

from paper_2411_09605_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2411_09605_gb300 import build
    build.build()


def test_the_first_list_stays_where_it_is_fastest():
    from paper_2411_09605_gb300 import pic
    b = pic.Batch([W.two_stream(n=200_000, nc=128, seed=1)])
    try:
        b.step(40)
        blocks = pic.pic_batch_info(b.b)[1]
        assert pic.pic_batch_autotune(b.b, 40) in (4, 8, 16)
        assert pic.pic_batch_info(b.b)[1] == blocks
        b.step(1)
        assert pic.pic_batch_autotune(b.b, 40) in (4, 8, 16)   # the remembered choice
        assert pic.pic_batch_info(b.b)[1] == blocks
    finally:
        b.close()
