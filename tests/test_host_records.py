"""The record converters of the binding copy and normalise whatever they are
given, C records among them; a record with unset lights is refused."""
import ctypes as C

import pytest

import hdof_inputs as hi

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def H():
    from paper_2210_04981_gb300 import build as b
    b.build()
    import paper_2210_04981_gb300.hdof as H
    H.load()
    return H


def test_params_of_a_record(H):
    p = H.params(hi.Params())
    assert p.n_lights < 4
    with pytest.raises(ZeroDivisionError):
        H.params(p)
    with pytest.raises(ZeroDivisionError):
        H.hdof_workspace_bytes(64, 48, p)
    for k in range(4):  # four lights that are not of unit length
        p.light_dir[k][:] = [3.0, 0.0, -4.0 - k]
        p.light_E[k] = 0.5
    q = H.params(p)
    assert q is not p and q.n_lights == 4
    for k in range(4):
        assert abs(sum(x * x for x in q.light_dir[k]) - 1.0) < 1e-6 and q.light_dir[k][2] < 0.0
    assert [x for x in p.light_dir[0]] == [3.0, 0.0, -4.0]  # the caller's record is left alone


def test_camera_and_lens_of_a_record_are_copies(H):
    for make, src in ((H.camera, hi.Camera(width=64, height=48)), (H.lens, hi.Lens())):
        a = make(src)
        b = make(a)
        assert b is not a and bytes(b) == bytes(a) and C.addressof(b) != C.addressof(a)


def test_calls_take_gbuffers_not_records(H):
    g = H.hdof_gbuf(64, 48, 0, 0, None, None, None, None)
    with pytest.raises(AttributeError):
        H.hdof_postfilter(g, hi.Camera(width=64, height=48), hi.Lens(), hi.Params(), None, torch.zeros(4))
