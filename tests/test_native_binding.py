"""The Python extension that takes the common forms of the calls (csrc/py_fast.cpp)."""
import threading

import pytest
import torch

import synth


def lak():
    import paper_1409_0669_gb300 as m
    return m


@pytest.mark.gpu
def test_threads_of_one_stream_while_the_workspace_grows():
    """One thread's inner products while another one on the same stream grows the kept
    workspace and takes the memory of the smaller one for tensors of its own: the sums
    stay right and the tensors keep their contents.  (A call that did not hold its
    workspace would launch on memory that has another owner by then.)"""
    m = lak()
    assert m._fast is not None
    x, y = synth.normal(4096, 1, "f32").cuda(), synth.normal(4096, 2, "f32").cuda()
    want = m.vec_dot(x, y).item()
    big = torch.zeros(4 << 20, device="cuda")
    least = m.vec_dot_workspace(4096, "f32")
    dev = torch.cuda.current_device()
    torch.cuda.synchronize()
    for _ in range(30):
        side = torch.cuda.Stream()
        m._workspaces.pop((dev, side.cuda_stream), None)
        with torch.cuda.stream(side):               # start from the least workspace
            m._fast.keep_workspace(dev, side.cuda_stream,
                                   torch.zeros(least, dtype=torch.uint8, device="cuda"))
            outs = torch.zeros(300, device="cuda")
        start = threading.Barrier(2)
        junk, errors = [], []

        def sums():
            try:
                with torch.cuda.stream(side):
                    start.wait()
                    for i in range(300):
                        m.vec_dot(x, y, out=outs[i:i + 1])
            except Exception as e:
                errors.append(e)

        def grow():
            try:
                with torch.cuda.stream(side):
                    start.wait()
                    for k in range(10, 23):
                        n = 1 << k
                        m.vec_dot(big[:n], big[:n])
                        junk.append(torch.full((least,), 7, dtype=torch.uint8, device="cuda"))
            except Exception as e:
                errors.append(e)

        threads = [threading.Thread(target=f) for f in (sums, grow)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        side.synchronize()
        assert not errors, errors
        assert (outs == want).all()
        assert all((j == 7).all() for j in junk)
