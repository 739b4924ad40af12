"""Publishes from host memory against the same blob on the device: page-locked blobs up to 512 KB, which the publish kernel reads itself (at an
odd offset, up to the last byte of an allocation of exactly their size, registered afterwards), larger ones and pageable memory, which are
copied first.  Which of the two a publish does is read off the graph that it is captured into."""
import ctypes as C

import numpy as np
import pytest

from parity_util import blob_for, fields_for

pytestmark = pytest.mark.gpu


def _cudart():
    import torch  # noqa: F401  (loads the runtime)
    rt = C.CDLL("libcudart.so.12")
    rt.cudaHostAlloc.argtypes = [C.POINTER(C.c_void_p), C.c_size_t, C.c_uint]
    rt.cudaFreeHost.argtypes = [C.c_void_p]
    rt.cudaHostRegister.argtypes = [C.c_void_p, C.c_size_t, C.c_uint]
    rt.cudaHostUnregister.argtypes = [C.c_void_p]
    rt.cudaGraphGetNodes.argtypes = [C.c_void_p, C.POINTER(C.c_void_p), C.POINTER(C.c_size_t)]
    rt.cudaGraphNodeGetType.argtypes = [C.c_void_p, C.POINTER(C.c_int)]
    return rt


class _Sources:
    """One blob in several kinds of host memory."""

    def __init__(self, rt, blob):
        import torch
        self.rt, n = rt, blob.size * 4
        self.exact = C.c_void_p()
        assert rt.cudaHostAlloc(C.byref(self.exact), n, 0) == 0
        C.memmove(self.exact, blob.ctypes.data, n)
        self.shifted = torch.empty(blob.size + 1, dtype=torch.float32).pin_memory()
        self.shifted[1:] = torch.from_numpy(blob)
        raw = np.empty(n + 8192, np.uint8)                       # whole pages around the blob, registered where they lie
        start = (-raw.ctypes.data) % 4096
        self.registered = raw[start:start + -(-n // 4096) * 4096]
        self.raw = raw
        assert rt.cudaHostRegister(self.registered.ctypes.data, self.registered.size, 0) == 0
        C.memmove(self.registered.ctypes.data, blob.ctypes.data, n)
        self.pageable = blob.copy()
        self.addresses = {"exact": self.exact.value, "shifted": self.shifted.data_ptr() + 4, "registered": self.registered.ctypes.data,
                          "pageable": self.pageable.ctypes.data}

    def close(self):
        assert self.rt.cudaFreeHost(self.exact) == 0
        assert self.rt.cudaHostUnregister(self.registered.ctypes.data) == 0


@pytest.fixture
def sources():
    import torch
    made = []

    def make(blob):
        made.append(_Sources(_cudart(), blob))
        return made[-1]
    yield make
    torch.cuda.synchronize()
    for s in made:
        s.close()


@pytest.mark.parametrize("kind,D,A,H,wd", [(0, 4, 2, 61, 0), (1, 6, 3, 128, 0), (0, 4, 2, 256, 2), (2, 64, 8, 256, 1), (2, 128, 16, 512, 1)])
def test_same_outputs_from_every_memory(kind, D, A, H, wd):
    import torch
    from paper_2502_20190_b200 import binding
    N = 200
    f = fields_for(env_kind=kind, n_envs=N, obs_dim=D, n_actions=A, hidden=H, weight_dtype=wd, epsilon=0.1, seed=3, replay_capacity=N * 8,
                   minibatch=64, staleness_bound=8, warmup=0, target_sync_interval=1000, gamma=0.99, huber_delta=1.0)
    blob = torch.from_numpy(blob_for(f, 5))
    n = blob.numel()
    pinned = torch.empty(n + 1, dtype=torch.float32).pin_memory()
    pinned[1:] = blob
    whole = blob.clone().pin_memory()
    outs = []
    for b, on_device in ((blob.cuda(), 1), (whole, 0), (pinned[1:], 0), (blob, 0)):
        ctx = binding.Context(**f)
        assert binding.tj_publish_weights(ctx.h, b.data_ptr(), n * 4, on_device)[0] == 0
        out = torch.empty((N, A), dtype=torch.float32, device="cuda")
        ctx.actor_step(1, out)
        torch.cuda.synchronize()
        outs.append(out.cpu().numpy().view(np.uint32))
    assert all(np.array_equal(outs[0], o) for o in outs[1:])


def test_the_kernel_reads_what_the_memory_holds_when_it_runs():
    """Publishes of one page-locked buffer, rewritten between them once the stream has drained."""
    import torch
    from paper_2502_20190_b200 import binding
    N = 64
    f = fields_for(env_kind=0, n_envs=N, obs_dim=4, n_actions=2, hidden=64, weight_dtype=0, epsilon=0.0, seed=4, replay_capacity=N * 8, minibatch=16,
                   staleness_bound=8, warmup=0, target_sync_interval=1000, gamma=0.99, huber_delta=1.0)
    a, b = binding.Context(**f), binding.Context(**f)
    buf = torch.from_numpy(blob_for(f, 1)).pin_memory()
    for v in range(1, 5):
        buf.copy_(torch.from_numpy(blob_for(f, v)))
        assert binding.tj_publish_weights(a.h, buf.data_ptr(), buf.numel() * 4, 0)[0] == 0
        b.publish_weights(buf.cuda())
        oa, ob = (torch.empty((N, 2), dtype=torch.float32, device="cuda") for _ in range(2))
        a.actor_step(1, oa)
        b.actor_step(1, ob)
        torch.cuda.synchronize()
        assert torch.equal(oa.view(torch.int32), ob.view(torch.int32))


@pytest.mark.parametrize("kind,D,A,H,wd", [(0, 4, 2, 61, 0), (1, 6, 3, 128, 0), (0, 4, 2, 256, 2), (0, 4, 2, 354, 0), (0, 4, 2, 360, 0),
                                           (2, 64, 8, 256, 1), (2, 128, 16, 512, 1)])
def test_page_locked_blobs_are_read_where_they_lie(sources, kind, D, A, H, wd):
    import torch
    from paper_2502_20190_b200 import binding
    N = 200
    f = fields_for(env_kind=kind, n_envs=N, obs_dim=D, n_actions=A, hidden=H, weight_dtype=wd, epsilon=0.1, seed=3, replay_capacity=N * 8,
                   minibatch=64, staleness_bound=8, warmup=0, target_sync_interval=1000, gamma=0.99, huber_delta=1.0)
    blob, rt = blob_for(f, 5), _cudart()
    s = sources(blob)
    stream, outs = torch.cuda.Stream(), {}
    with torch.cuda.stream(stream):
        for name, address in s.addresses.items():
            ctx = binding.Context(**f)
            ctx.publish_weights(blob_for(f, 1))                  # the first publish also fills the target network
            stream.synchronize()
            if name == "pageable":                               # a copy from such memory cannot be captured
                assert binding.tj_publish_weights(ctx.h, address, blob.size * 4, 0)[0] == 0
            else:
                g = torch.cuda.CUDAGraph(keep_graph=True)
                with torch.cuda.graph(g, stream=stream):
                    assert binding.tj_publish_weights(ctx.h, address, blob.size * 4, 0)[0] == 0
                n, kind_of, nodes = C.c_size_t(16), C.c_int(), (C.c_void_p * 16)()
                assert rt.cudaGraphGetNodes(g.raw_cuda_graph(), nodes, C.byref(n)) == 0
                kinds = []
                for node in nodes[:n.value]:
                    assert rt.cudaGraphNodeGetType(node, C.byref(kind_of)) == 0
                    kinds.append(kind_of.value)                  # 0: kernel, 1: copy
                assert sorted(kinds) == ([0] if blob.size * 4 <= 512 * 1024 else [0, 1]), (name, kinds)
                g.replay()
            out = torch.empty((N, A), dtype=torch.float32, device="cuda")
            ctx.actor_step(1, out)
            stream.synchronize()
            outs[name] = out.cpu().numpy().view(np.uint32)
        ctx = binding.Context(**f)
        ctx.publish_weights(blob_for(f, 1))
        ctx.publish_weights(torch.from_numpy(blob).cuda())
        ctx.actor_step(1, out)
        stream.synchronize()
        for name, o in outs.items():
            assert np.array_equal(out.cpu().numpy().view(np.uint32), o), name
