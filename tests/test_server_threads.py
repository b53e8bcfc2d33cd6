"""The Python Server with one thread that submits and another that collects, on the CPU (a fake library).

A request may finish, and its ticket come out of wait_any, before the submitting thread has returned from
the library; the collecting thread's poll still finds its image's shape.  Unknown and retired tickets
raise KeyError, as ever."""
import ctypes
import threading

import numpy as np
import pytest

from paper_1603_09180_gb300 import thin


class FakeLib:
    """Finishes a request inside its submit call, and returns from it only when the result is being polled."""

    def __init__(self):
        self.finished = threading.Event()
        self.resume = threading.Event()
        self.code = thin.THIN_OK

    def thin_serve_create(self, budget, slots, cap, handle):
        return thin.THIN_OK

    def thin_serve_destroy(self, handle):
        return thin.THIN_OK

    def thin_serve_submit(self, handle, img, w, h, pitch, dtype, lam, ticket):
        if self.code == thin.THIN_OK:
            ctypes.cast(ticket, ctypes.POINTER(ctypes.c_uint64))[0] = 41
        self.finished.set()
        self.resume.wait(10)
        return self.code

    def thin_serve_poll(self, handle, ticket, out, pitch, done, stats):
        ctypes.cast(done, ctypes.POINTER(ctypes.c_int))[0] = 1
        return thin.THIN_OK


@pytest.fixture
def server(monkeypatch):
    lib = FakeLib()
    monkeypatch.setattr(thin, "load", lambda: lib)
    return thin.Server(1 << 20), lib


def test_poll_while_submit_returns(server):
    srv, lib = server
    got = []

    def collect():
        lib.finished.wait(10)
        threading.Timer(0.2, lib.resume.set).start()
        try:
            got.append(srv.poll(41))
        except KeyError as e:
            got.append(e)

    th = threading.Thread(target=collect)
    th.start()
    assert srv.submit(np.zeros((5, 7), np.uint16), 0) == 41
    th.join()
    done, img, _, rc = got[0]
    assert done and rc == thin.THIN_OK and img.shape == (5, 7) and img.dtype == np.uint16
    with pytest.raises(KeyError):
        srv.poll(41)


def test_refused_submit_leaves_no_ticket(server):
    srv, lib = server
    lib.code = thin.THIN_EAGAIN
    lib.resume.set()
    with pytest.raises(thin.ThinError):
        srv.submit(np.zeros((5, 7), np.uint8), 0)
    with pytest.raises(KeyError):
        srv.poll(0)
    assert not srv.shapes
