"""The element operator's dispatch over orders, precisions and element counts, with a fake CUDA runtime
(tests/fake_dispatch.cpp): the form that sem_axl_chosen names launches a kernel, and sem_ax and sem_axl
say so when they have none for an order instead of launching nothing."""
from fake_util import run_driver


def test_every_order_launches_or_says_so(tmp_path):
    run_driver("fake_dispatch.cpp", tmp_path)
