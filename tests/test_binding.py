"""The C module that marshals the hot calls, without a GPU: a C function that only waits stands in for the library's."""
import ctypes
import threading
import time

import pytest

from paper_2601_13143_b200 import build, fastav


@pytest.fixture(scope="module")
def native():
    build.build_binding()
    return fastav._native()


@pytest.mark.parametrize("name,count", [("prune", 23), ("select_mask", 9), ("compact", 15)])
def test_other_threads_run_during_a_call(native, name, count):
    """usleep takes the params pointer for its microseconds; a thread that counts meanwhile has to get on."""
    usleep = ctypes.cast(ctypes.CDLL(None).usleep, ctypes.c_void_p).value
    done, steps = threading.Event(), []

    def count_up():
        while not done.is_set():
            steps.append(time.perf_counter())
            time.sleep(0.001)

    other = threading.Thread(target=count_up)
    other.start()
    try:
        while not steps:
            time.sleep(0.001)
        start = time.perf_counter()
        assert getattr(native, name)(usleep, 300_000, *[None] * (count - 3), 0) == 0
        end = time.perf_counter()
    finally:
        done.set()
        other.join()
    assert end - start > 0.25
    assert sum(start + 0.05 < t < end - 0.05 for t in steps) >= 5


def test_params_may_be_of_a_derived_type():
    class Named(fastav.fastav_params):
        pass

    params = Named()
    assert fastav._params(params) == ctypes.addressof(params)
    with pytest.raises(TypeError):
        fastav._params(None)
