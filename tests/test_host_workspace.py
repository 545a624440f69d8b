"""A workspace whose start would make a call's own accesses misaligned is
refused on the host, before anything is enqueued."""
import ctypes as C

import pytest

import hdof_inputs as hi

pytest.importorskip("torch")


@pytest.fixture(scope="module")
def H():
    from paper_2210_04981_gb300 import build as b
    b.build()
    import paper_2210_04981_gb300.hdof as H
    H.load()
    return H


@pytest.mark.parametrize("call,offsets", [("reference", (1, 4, 8)), ("trace", (1, 4)), ("hits", (2, 4)),
                                          ("mask_coc", (1, 2)), ("spec", (4, 8))])
def test_misaligned_workspace_is_refused(H, call, offsets):
    lib, ptr = H.load(), C.c_void_p(1 << 20)
    cam, lens = H.camera(hi.Camera(width=64, height=48)), H.lens(hi.Lens())
    p = H.params(hi.Params(mask_coc=1, blades=6 if call == "spec" else 0))
    g = H.hdof_gbuf(64, 48, 0, 0, ptr, ptr, ptr, ptr)
    n = 1 << 30
    for off in offsets:
        ws = C.c_void_p((1 << 30) + off)
        rc = {
            "reference": lambda: lib.hdof_reference_rt(ptr, C.byref(cam), C.byref(lens), C.byref(p), 1, None, ptr, ws, n,
                                                       None),
            "trace": lambda: lib.hdof_trace(ptr, C.byref(cam), C.byref(lens), C.byref(p), ptr, None, ptr, None, None,
                                            None, ws, n, None, None),
            "hits": lambda: lib.hdof_trace_hits(ptr, C.byref(cam), C.byref(p), ptr, ws, n, ptr, None, None),
            "mask_coc": lambda: lib.hdof_mask_coc(C.byref(g), None, C.byref(cam), C.byref(lens), C.byref(p), ptr, ptr,
                                                  ws, n, None),
            "spec": lambda: lib.hdof_postfilter_spec(C.byref(g), C.byref(cam), C.byref(lens), C.byref(p), ptr, ws, n,
                                                     None),
        }[call]()
        buf = C.create_string_buffer(256)
        lib.hdof_last_error(buf, 256)
        assert rc == -1 and b"multiple of 16 bytes" in buf.value, (call, off, rc, buf.value)
