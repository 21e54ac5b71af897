"""Kernel attributes are set once per device, and no thread launches a kernel before that has happened: a second
thread that asks for the same kernel waits until the first one's setter has returned.  Host code only; the setter
here is a slow one of the test's own."""

import ctypes
import threading
import time

SET = ctypes.CFUNCTYPE(None, ctypes.c_void_p)
NAME = "_ZN4cola14once_on_deviceEPKvPFvS1_E"   # void cola::once_on_device(const void*, void (*)(const void*))


def test_second_thread_waits_for_the_first_setter():
    from paper_1507_05329_gb300 import build
    build.build()
    lib = ctypes.CDLL(build.LIB_PATH)
    once = getattr(lib, NAME)
    once.argtypes, once.restype = [ctypes.c_void_p, SET], None
    calls, began, done, early = [], threading.Event(), threading.Event(), []

    @SET
    def setter(key):
        calls.append(key)
        began.set()
        time.sleep(0.3)
        done.set()

    mark = ctypes.create_string_buffer(1)
    key = ctypes.addressof(mark)

    def second():
        began.wait(5)
        once(key, setter)
        early.append(not done.is_set())

    threads = [threading.Thread(target=once, args=(key, setter))] + [threading.Thread(target=second) for _ in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join(10)
    assert early == [False] * 3
    once(key, setter)
    assert calls == [key]
