"""Work space of the operator and the network, whatever was called before."""
import numpy as np
import pytest

from gpu_common import lib, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", [0, 1])
@pytest.mark.parametrize("R", [1, 5])
def test_right_hand_side_before_assembly(kernel, R):
    # ibem_rhs needs no assembly and sizes the work vectors before there are coupling matrices
    import torch
    ibem = lib()
    hs = [ibem.ibem_create(ibem.sphere_patches(), ibem.make_params(1, 2, q_cheb=4, eta=1.6, kernel=kernel,
                                                                   kappa=3.0 if kernel else 0.0)) for _ in range(2)]
    info = ibem.ibem_get_info(hs[0])
    tail = (2,) if kernel else ()
    g = torch.from_numpy(np.random.default_rng(1600).normal(size=(R, info.n_quad_points) + tail)).cuda()
    x = torch.from_numpy(np.random.default_rng(1601).normal(size=(R, info.ndof) + tail)).cuda()
    b = [torch.full_like(x, np.nan) for _ in hs]
    y = [torch.full_like(x, np.nan) for _ in hs]
    ibem.ibem_rhs(hs[0], g, R, b[0])
    for h, out in zip(hs, y):
        ibem.ibem_assemble(h)
        ibem.ibem_matvec(h, x, out, R)
    ibem.ibem_rhs(hs[1], g, R, b[1])
    torch.cuda.synchronize()
    for a in (b, y):
        assert rel_err(a[0].cpu().numpy(), a[1].cpu().numpy()) < 1e-13
    for h in hs:
        ibem.ibem_destroy(h)


@pytest.mark.parametrize("first", ["rhs", "fp32"])
def test_application_recorded_after_another_call_of_its_width(first):
    # the stored Helmholtz coupling's work space is sized with the rest: after any call of as
    # many vectors an FP64 application allocates nothing, so it can be recorded (thread-local
    # capture fails on an allocation)
    import torch
    ibem = lib()
    stream = torch.cuda.Stream()
    prm = ibem.make_params(1, 2, q_cheb=5, eta=1.6, kernel=1, kappa=3.0)
    hs = [ibem.ibem_create(ibem.sphere_patches(), prm, stream) for _ in range(2)]
    info = ibem.ibem_get_info(hs[0])
    rng = np.random.default_rng(1602)
    x = torch.from_numpy(rng.normal(size=(3, info.ndof, 2))).cuda()
    g = torch.from_numpy(rng.normal(size=(3, info.n_quad_points, 2))).cuda()
    ref, y = torch.full_like(x, np.nan), torch.full_like(x, np.nan)
    torch.cuda.synchronize()
    for h in hs:
        ibem.ibem_assemble(h)
    ibem.ibem_matvec(hs[0], x, ref, 3)             # loads every kernel
    if first == "rhs":
        ibem.ibem_rhs(hs[1], g, 3, y)
    else:
        ibem.ibem_matvec(hs[1], x, y, 3, ibem.IBEM_FP32)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
        ibem.ibem_matvec(hs[1], x, y, 3)
    y.fill_(float("nan"))
    torch.cuda.synchronize()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, ref)
    del graph
    for h in hs:
        ibem.ibem_destroy(h)


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_network_after_a_refused_allocation(precision):
    # the activations of 65535 images of 4096 x 4096 (hundreds of TB) cannot be allocated; the
    # call fails before it touches its images, and neither the network nor a handle finds
    # the old buffers' sizes or the old error afterwards
    import ctypes
    import torch
    ibem = lib()
    prec = ibem.IBEM_FP32 if precision == "fp32" else ibem.IBEM_BF16
    c = ibem.ibem_cnn_create(8, seed=3)
    h = ibem.ibem_create(ibem.sphere_patches(), ibem.make_params(1, 2, q_cheb=4, eta=1.6))
    ibem.ibem_assemble(h)
    v = torch.from_numpy(np.random.default_rng(1604).normal(size=(1, ibem.ibem_get_info(h).ndof))).cuda()
    x = torch.from_numpy(np.random.default_rng(1603).normal(size=(3, 2, 20, 24)).astype(np.float32)).cuda()
    out, mv = [torch.full_like(x, np.nan) for _ in range(2)], [torch.full_like(v, np.nan) for _ in range(2)]
    for k in range(2):
        ibem.ibem_matvec(h, v, mv[k], 1)
        ibem.ibem_cnn_forward(c, x, out[k], prec)
        torch.cuda.synchronize()
        if k == 0:
            p = ctypes.c_void_p(x.data_ptr())
            status = ibem._lib.ibem_cnn_forward(c, p, 65535, 4096, 4096, p, prec)
            assert ibem._lib.ibem_status_string(status) == b"IBEM_ERR_OOM"
    assert torch.equal(out[0], out[1]) and torch.equal(mv[0], mv[1])
    ibem.ibem_destroy(h)
    ibem.ibem_cnn_destroy(c)


def test_handle_after_a_refused_batch():
    # vectors of 256 right-hand sides for each of 8000 instances (some 700 GB) cannot be
    # allocated; the handle's next application does not find the old error
    import torch
    ibem = lib()
    h = ibem.ibem_create(ibem.sphere_patches(), ibem.make_params(2, 4, q_cheb=4, eta=1.6))
    ibem.ibem_assemble(h)
    v = torch.from_numpy(np.random.default_rng(1605).normal(size=(1, ibem.ibem_get_info(h).ndof))).cuda()
    y = [torch.full_like(v, np.nan) for _ in range(2)]
    ibem.ibem_matvec(h, v, y[0], 1)
    with pytest.raises(ibem.IbemError) as e:
        ibem.ibem_batch_create([h] * 8000, [256] * 8000)
    assert e.value.status == "IBEM_ERR_OOM"
    ibem.ibem_matvec(h, v, y[1], 1)
    torch.cuda.synchronize()
    assert torch.equal(y[0], y[1])
    ibem.ibem_destroy(h)
