"""The Python extension that takes the common forms of the calls (csrc/py_fast.cpp): it is
there, gives the bits of the Python path, and returns None without side effects for every
form that it leaves to that path."""
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


# ---- both paths --------------------------------------------------------------------

STORAGES = ["f32", "f64", "bf16", "f16"]


def vecs(storage, n, k=3):
    return [synth.uniform(n, 10 + i, storage).cuda() for i in range(k)]


def acc(storage):
    return torch.float64 if storage == "f64" else torch.float32


def csr(storage, m=700, n=500):
    g = torch.Generator().manual_seed(4)
    lens = torch.randint(0, 30, (m,), generator=g)
    rp = torch.zeros(m + 1, dtype=torch.int32)
    rp[1:] = torch.cumsum(lens, 0)
    ci = torch.randint(0, n, (int(rp[-1]),), generator=g, dtype=torch.int32)
    return (rp.cuda(), ci.cuda(), synth.normal(int(rp[-1]), 5, storage).cuda(),
            synth.uniform(n, 6, storage).cuda(), synth.uniform(m, 7, storage).cuda())


def matrix(storage, shape):
    return synth.normal(shape, 8, storage).cuda()


def calls(m, storage):
    """(name, function of the extension, arguments for it, the public call) of every form;
    each call makes its own output operands."""
    n = 5003
    x, y, z = vecs(storage, n)
    one = lambda: torch.zeros(1, dtype=acc(storage), device="cuda")
    f = m._fast
    yield "copy", lambda: f.vec_copy(x.clone(), y), lambda: m.vec_copy(x.clone(), y)
    yield "axpy", lambda: f.vec_axpy(x.clone(), y, z, 0.25), lambda: m.vec_axpy(x.clone(), y, z, 0.25)
    yield "axpby", lambda: f.vec_axpby(x.clone(), 2, y, 0.5, z), lambda: m.vec_axpby(x.clone(), 2, y, 0.5, z)
    yield "dot", lambda: f.vec_dot(x, y, None, False), lambda: m.vec_dot(x, y)
    yield "dot out", lambda: f.vec_dot(x, y, one(), False), lambda: m.vec_dot(x, y, out=one())
    yield "norm2", lambda: f.vec_axpy_norm2(x.clone(), y, z, 0.5, None), \
        lambda: m.vec_axpy_norm2(x.clone(), y, z, 0.5)
    if storage != "f64":
        yield "dot compensated", lambda: f.vec_dot_compensated(x, y, None), \
            lambda: m.vec_dot_compensated(x, y)
    for name, A in (("row", matrix(storage, (70, 301))), ("row padded", matrix(storage, (70, 310))[:, :301]),
                    ("column", matrix(storage, (301, 70)).t()), ("one row", matrix(storage, (1, 301))),
                    ("one row of a larger", matrix(storage, (9, 301))[4:5]),
                    ("one column", matrix(storage, (70, 1))), ("a column", matrix(storage, (70, 9))[:, 3:4]),
                    ("few long rows", matrix(storage, (5, 150_000))),
                    ("few long columns", matrix(storage, (150_000, 5)).t())):
        u, v, w = (vecs(storage, k, 1)[0] for k in (A.shape[1], A.shape[0], A.shape[0]))
        yield f"gemv {name}", lambda A=A, u=u: f.dense_gemv(A, u, None, 1.0, 0.0, False), \
            lambda A=A, u=u: m.dense_gemv(A, u)
        yield f"gemv {name} into y", lambda A=A, u=u, w=w: f.dense_gemv(A, u, w.clone(), 0.5, 2.0, False), \
            lambda A=A, u=u, w=w: m.dense_gemv(A, u, w.clone(), alpha=0.5, beta=2.0)
        yield f"gemv {name} transposed", lambda A=A, v=v: f.dense_gemv(A, v, None, 1.0, 0.0, True), \
            lambda A=A, v=v: m.dense_gemv_trans(A, v)
    rp, ci, val, cx, cy = csr(storage)
    yield "spmv", lambda: f.csr_spmv(rp, ci, val, cx, None, None), lambda: m.csr_spmv(rp, ci, val, cx)
    yield "spmv into y", lambda: f.csr_spmv(rp, ci, val, cx, torch.empty_like(cy), 500), \
        lambda: m.csr_spmv(rp, ci, val, cx, torch.empty_like(cy), n_cols=500)
    yield "sampled outer", lambda: f.csr_sampled_outer(rp, ci, cy, cx), \
        lambda: m.csr_sampled_outer(rp, ci, cy, cx)
    yield "outer", lambda: f.dense_outer(x[:70], y[:301]), lambda: m.dense_outer(x[:70], y[:301])
    scale = torch.full((1,), 0.75, dtype=acc(storage), device="cuda")
    yield "scale", lambda: f.vec_scale_dev(x, scale), lambda: m.vec_scale_dev(x, scale)
    yield "scale, 0-d", lambda: f.vec_scale_dev(x, scale[0]), lambda: m.vec_scale_dev(x, scale[0])


@pytest.mark.gpu
@pytest.mark.parametrize("storage", STORAGES)
def test_same_bits_as_the_python_path(storage, monkeypatch):
    m = lak()
    assert m._fast is not None and m._fast.torch_version == torch.__version__
    fast = m._fast
    made = list(calls(m, storage))
    monkeypatch.setattr(m, "_fast", None)
    slow = [(name, call()) for name, _, call in made]
    monkeypatch.setattr(m, "_fast", fast)
    here = (torch.cuda.current_device(), torch.cuda.current_stream().cuda_stream)
    fast.keep_workspace(*here, m._workspaces[here])              # grown meanwhile
    for (name, direct, public), (_, want) in zip(made, slow):
        got = direct()
        assert got is not None, f"{name}: the extension left it to the Python path"
        for r in (got, public()):
            assert r.dtype == want.dtype and r.shape == want.shape and r.is_contiguous(), name
            assert torch.equal(r, want), name


@pytest.mark.gpu
def test_a_scalar_result():
    m = lak()
    x, y, _ = vecs("f32", 1000)
    m.vec_dot(x, y)
    s = m._fast.vec_dot(x, y, None, True)
    assert s.dim() == 0 and s.item() == m.vec_dot(x, y).item()


class Sub(torch.Tensor):
    pass


@pytest.mark.gpu
def test_refused_forms_leave_no_trace():
    """Each refused form returns None and changes nothing; the public call then takes it or
    raises as the Python path does."""
    m, f = lak(), lak()._fast
    n = 1000
    x, y, z = vecs("f32", n)
    m.vec_dot(x, y), m.vec_axpy_norm2(x.clone(), y, z, 0.5)          # a workspace is there
    keep = x.clone()
    other = {"a subclass": y.as_subclass(Sub), "strided": vecs("f32", 2 * n, 1)[0][::2],
             "expanded": y[:1].expand(n), "2-D": y.view(10, 100), "another type": y.double(),
             "an integer type": y.int(), "on the host": y.cpu(), "shorter": y[:-1], "empty": y[:0],
             "complex": y.to(torch.complex64), "its imaginary part, conjugated": torch.view_as_real(
                 torch.randn(n, dtype=torch.complex64, device="cuda")).select(1, 1),
             "a negative view": torch.randn(n, dtype=torch.complex64, device="cuda").conj().imag,
             "not a tensor": [0.0] * n, "None": None}
    assert other["a negative view"].is_neg()
    A = matrix("f32", (40, n))
    rp, ci, val, cx, _ = csr("f32")
    for what, b in other.items():
        assert f.vec_copy(x, b) is None and f.vec_copy(b, x) is None, what
        assert f.vec_axpy(x, b, z, 0.5) is None and f.vec_axpy(x, y, b, 0.5) is None, what
        assert f.vec_axpby(x, 1.0, b, 1.0, z) is None, what
        assert f.vec_dot(x, b, None, False) is None and f.vec_dot(b, y, None, True) is None, what
        assert f.vec_dot_compensated(x, b, None) is None, what
        assert f.vec_axpy_norm2(x, b, z, 0.5, None) is None, what
        assert f.dense_gemv(A, b, None, 1.0, 0.0, False) is None, what
        assert f.csr_spmv(rp, ci, val, b, None, None) is None or what == "shorter", what
        if what not in ("shorter", "another type"):
            assert f.dense_outer(x, b) is None and f.vec_scale_dev(b, x[:1]) is None, what
    assert torch.equal(x, keep)
    # results and coefficients
    assert f.vec_dot(x, y, torch.zeros(1, dtype=torch.float64, device="cuda"), False) is None
    assert f.vec_axpy(x, y, z, "half") is None and f.vec_axpy(x, y, z, 1j) is None
    assert f.vec_scale_dev(x, torch.zeros(1, dtype=torch.float64, device="cuda")) is None
    assert f.dense_gemv(A, x, None, 1.0, 1.0, False) is None          # beta without y
    assert f.dense_gemv(A, x, x[:39], 1.0, 0.0, False) is None
    assert f.dense_gemv(A[:, ::2], x[:500], None, 1.0, 0.0, False) is None
    assert f.dense_gemv(A[0].expand(40, n), x, None, 1.0, 0.0, False) is None
    assert f.csr_spmv(rp.long(), ci, val, cx, None, None) is None
    assert f.csr_spmv(rp, ci[:-1], val, cx, None, None) is None
    assert f.csr_spmv(rp, ci, val, cx, None, "500") is None
    assert f.vec_copy(x) is None and f.vec_copy(x, y, z) is None      # another number of arguments
    assert torch.equal(x, keep)
    # the Python path takes or refuses them
    assert torch.equal(m.vec_copy(x.clone(), other["a subclass"]), y)
    for call in (lambda: m.vec_copy(x, other["strided"]), lambda: m.vec_dot(x, other["shorter"]),
                 lambda: m.vec_axpy(x, y, other["on the host"], 0.5),
                 lambda: m.dense_gemv(A, other["2-D"]), lambda: m.dense_gemv(A, x, beta=1.0, y=x[:39])):
        with pytest.raises((ValueError, TypeError)):
            call()
    assert torch.equal(x, keep)


@pytest.mark.gpu
def test_vmap_levels_and_workspaces_are_left_to_the_python_path():
    m, f = lak(), lak()._fast
    x, y, _ = vecs("f32", 1000)
    seen = []
    torch.func.vmap(lambda a: (seen.append(f.vec_dot(a, y, None, False)), a)[1])(x.view(1, 1000))
    assert seen == [None]
    # no workspace yet, or one too small: None, and the public call makes it
    side = torch.cuda.Stream()
    dev = torch.cuda.current_device()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        m._workspaces.pop((dev, side.cuda_stream), None)
        f.keep_workspace(dev, side.cuda_stream, torch.zeros(256, dtype=torch.uint8, device="cuda"))
        assert f.vec_dot(x, y, None, False) is None
        want = m.vec_dot(x, y)
        got = f.vec_dot(x, y, None, False)
        assert torch.equal(got, want)
    side.synchronize()
    with pytest.raises(TypeError):
        f.keep_workspace(dev, 0, None)
