"""Which stream and device the library's temporaries come from when torch's
allocator serves them, with the CUDA calls replaced by records of them."""
import contextlib
import types

import pytest

import paper_2506_06805_gb300 as P

torch = pytest.importorskip("torch")


class Stream:
    def __init__(self, handle, device=0):
        self.cuda_stream, self.device_index = handle, device

    def __eq__(self, other):
        return (self.cuda_stream, self.device_index) == (other.cuda_stream, other.device_index)


class Tensor:
    def __init__(self, *shape):
        self.shape = shape

    def data_ptr(self):
        return 4096


@pytest.fixture
def cuda(monkeypatch):
    st = types.SimpleNamespace(device=0, stream=Stream(7), hooks=None, lib_stream=None, blocks=[])

    @contextlib.contextmanager
    def on(stream):
        before, st.stream = st.stream, stream
        yield
        st.stream = before

    def alloc(n, device=None, stream=None):
        st.blocks.append((st.device if device is None else device, st.stream.cuda_stream))
        return 1 << 20

    c = torch.cuda
    for name, f in {"is_available": lambda: True, "current_device": lambda: st.device,
                    "current_stream": lambda device=None: st.stream, "stream": on,
                    "caching_allocator_alloc": alloc,
                    "caching_allocator_delete": lambda p: None}.items():
        monkeypatch.setattr(c, name, f)

    def set_allocator(a, f, u):
        st.hooks = a, f
        return 0

    def set_stream(s):
        st.lib_stream = s
        return 0

    def zgemm(*a):
        st.hooks[1](st.hooks[0](64, None), None)
        return 0

    fake = types.SimpleNamespace(cc_set_default_allocator=set_allocator, cc_set_default_stream=set_stream,
                                 cc_zgemm_dev=zgemm)
    monkeypatch.setattr(P, "lib", lambda: fake)
    monkeypatch.setattr(P, "_TORCH_HOOKS", None)
    monkeypatch.setattr(P, "_TORCH_STREAM", None, raising=False)
    return st


def test_zgemm_temporaries_come_from_the_stream_it_works_on(cuda):
    P.use_torch_memory()
    A = Tensor(4, 4)
    P.zgemm_dev(A, A, A)
    other = Stream(9)
    cuda.stream = other
    P.zgemm_dev(A, A, A)
    assert cuda.lib_stream == 7
    assert cuda.blocks == [(0, 7), (0, 7)]
    assert cuda.stream is other


def test_temporaries_come_from_the_device_of_the_call(cuda):
    P.use_torch_memory()
    cuda.device, cuda.stream = 1, Stream(0, 1)
    A = Tensor(4, 4)
    P.zgemm_dev(A, A, A)
    assert cuda.blocks == [(1, 0)]
