"""What Pipeline.realize takes for its inputs and its stream, as the other calls
of the binding do.  The buffers are refused by the library before any CUDA call,
which shows that the arguments reached it."""

import ctypes

import pytest

import __graft_entry__
from paper_2012_07145_gb300 import hp, pipelines


@pytest.fixture(scope="module", autouse=True)
def built():
    __graft_entry__.build()


class SubBuffer(hp.Buffer):
    pass


def null(cls=hp.Buffer):
    return cls(None, hp.HP_F32, 1, 8, 8, 32, 256)


FIELDS = (None, hp.HP_F32, 1, 8, 8, 32, 256)


@pytest.mark.parametrize("inputs", [[null()], (null(),), {0: null()}.values(), [FIELDS], [null(SubBuffer)],
                                    (hp.Buffer * 1)(null())], ids=["list", "tuple", "view", "fields", "subclass", "array"])
@pytest.mark.parametrize("stream", [None, 0, 12345])
def test_accepted_forms_reach_the_library(inputs, stream):
    p = pipelines.stencil_chain(1, "binomial")
    with pytest.raises(hp.HPError) as e:
        p.realize(inputs, null(), stream)
    assert e.value.status == hp.HP_ERR_INVALID_ARG and "null data" in str(e.value)


@pytest.mark.parametrize("stream", [b"bytes", "text", ctypes.c_void_p(1)])
def test_streams_that_are_not_integers_are_refused(stream):
    p = pipelines.stencil_chain(1, "binomial")
    with pytest.raises(TypeError):
        p.realize([null()], null(), stream)
