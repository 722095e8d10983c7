"""What the binding makes of its arguments, without a GPU: every call below is answered on the host, by an argument error or
by the size of its workspace, before anything is launched (a workspace of 16 bytes is the last thing that is looked at)."""
import numpy as np
import pytest
import torch

import __graft_entry__ as entry
import paper_2509_10798_b200 as jq


@pytest.fixture(scope="module", autouse=True)
def built():
    entry.build()


class Tensor:
    """An address that is never followed, a shape, a size."""

    def __init__(self, address=0x1000, elements=1 << 40, shape=(2, 2048, 128), element_size=1):
        self.address, self.elements, self.shape, self.size = address, elements, shape, element_size

    def data_ptr(self):
        return self.address

    def numel(self):
        return self.elements

    def element_size(self):
        return self.size


class Stream:
    cuda_stream = 0


S = jq.shape(2, 8, 2048, 16, 256)
T, SMALL, STREAM = Tensor(), Tensor(elements=16), Stream()


def ragged(K=(T, T), V=(T, T), Q=(T, T), s=S, L=None, budget=None):
    jq.evict_ragged(K, V, Q, s, L, budget, T, T, T, SMALL, stream=STREAM)


def append(n_old, cache=(2, 4096, 128), new=(2, 48, 128)):
    jq.evict_append(Tensor(shape=cache), T, n_old, Tensor(shape=new), T, T, S, T, SMALL, stream=STREAM)


def code_of(call, *args, **kw):
    with pytest.raises(jq.JqError) as e:
        call(*args, **kw)
    return e.value.code


TAKEN = [dict(), dict(L=[5, 6, 7]), dict(budget=[5, 6, 7]), dict(L=np.array([5, 6])), dict(L=torch.tensor([5, 6])), dict(L=[5.5, 6.0]),
         dict(L=["5", "6"]), dict(L=range(5, 7)), dict(L={5: 1, 6: 1}), dict(K=torch.zeros(2, 8), V=torch.zeros(2, 8), Q=torch.zeros(2, 8)),
         dict(K={1: T, 2: T}.values())]


@pytest.mark.parametrize("kw", TAKEN, ids=lambda kw: ",".join("%s:%s" % (k, type(v).__name__) for k, v in kw.items()) or "plain")
def test_ragged_arguments_that_are_taken(kw):
    """Any sequence of tensors and of whatever int() takes, the lengths and budgets longer than the units if need be."""
    assert code_of(ragged, **kw) == jq.JQ_ERR_WORKSPACE


def test_ragged_arguments_that_are_refused():
    for kw in (dict(V=[T]), dict(Q=[T]), dict(V=[]), dict(K=[], V=[], Q=[]), dict(L=[5, 0])):
        assert code_of(ragged, **kw) == jq.JQ_ERR_INVALID_ARG
    assert code_of(jq.evict_layers, [T, T], [T], [T, T], S, T, T, T, SMALL, stream=STREAM) == jq.JQ_ERR_INVALID_ARG
    for kw, error in ((dict(V=[T] * 3), IndexError), (dict(K=[T, None]), AttributeError), (dict(L=[5]), ValueError), (dict(L=[5, None]), TypeError),
                      (dict(L=iter([5, 6])), TypeError), (dict(K=iter([T, T])), TypeError)):
        with pytest.raises(error):
            ragged(**kw)


@pytest.mark.parametrize("n_old", [2000, 2000.0, 2000.7, "2000", np.int64(2000), np.float32(2000), torch.tensor(2000), torch.tensor(2000.0)],
                         ids=lambda v: type(v).__name__)
def test_append_takes_what_int_takes(n_old):
    assert code_of(append, n_old) == jq.JQ_ERR_WORKSPACE
    assert code_of(append, n_old, cache=(2, 4096.0, 128), new=(2, 48.0, 128)) == jq.JQ_ERR_WORKSPACE
    with pytest.raises(TypeError):
        append(None)


@pytest.mark.parametrize("s", [bytes(S), np.frombuffer(bytes(S), np.int32), (2, 8, 4, 2048, 128, 16, 256, 7), None], ids=lambda s: type(s).__name__)
def test_a_shape_is_a_JqShape(s):
    for call in (lambda: ragged(s=s), lambda: jq.evict_layer(T, T, T, s, T, T, T, SMALL, stream=STREAM), lambda: jq.select_topk(T, s, T, SMALL, stream=STREAM)):
        with pytest.raises(TypeError):
            call()


def test_a_workspace_counts_as_many_bytes_as_it_has_elements():
    wide = Tensor(elements=jq.workspace_bytes(S) // 4 + 1, element_size=4)
    for call in (lambda: jq.score(T, T, S, T, wide, stream=STREAM), lambda: jq.select_topk(T, S, T, wide, stream=STREAM),
                 lambda: jq.evict_layer(T, T, T, S, T, T, T, wide, stream=STREAM), lambda: jq.evict_layer_windowed(T, T, T, T, S, T, T, T, wide, stream=STREAM)):
        assert code_of(call) == jq.JQ_ERR_WORKSPACE


def test_null_pointers_are_the_librarys_to_reject():
    assert code_of(jq.evict_layer, None, T, T, S, T, T, T, SMALL, stream=STREAM) == jq.JQ_ERR_INVALID_ARG
    assert code_of(jq.decode_attention, T, T, Tensor(shape=(8, 128)), None, T, stream=STREAM) == jq.JQ_ERR_INVALID_ARG
    assert code_of(jq.evict_layer_host, T, T, T, S, T, T, T, SMALL, stream=STREAM) == jq.JQ_ERR_WORKSPACE
    with pytest.raises(AttributeError):
        jq.evict_layer(T, T, T, S, T, T, T, None, stream=STREAM)
    with pytest.raises(AttributeError):
        jq.evict_layer(T, T, T, S, T, T, T, SMALL, stream=7)
