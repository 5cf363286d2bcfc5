"""Helpers shared by the GPU parity tests (no method arithmetic)."""
import numpy as np
import torch


def to_np(t: torch.Tensor) -> np.ndarray:
    """Exact float64 copy of a (bf16 / fp32) tensor on the host."""
    return t.detach().to(torch.float32).cpu().numpy().astype(np.float64)


def rel_fro(got, want) -> float:
    got = np.asarray(got, dtype=np.float64)
    want = np.asarray(want, dtype=np.float64)
    return float(np.linalg.norm(got - want) / max(np.linalg.norm(want), 1e-300))


def worst_row_error(got, want) -> float:
    """Largest relative error of a single row (a vector along the last axis) among the rows whose
    reference norm is at least the median row norm of the tensor: the companion of a whole-tensor
    Frobenius bound, which one badly wrong row in a few thousand would pass."""
    got = np.asarray(got, dtype=np.float64)
    want = np.asarray(want, dtype=np.float64)
    err = np.linalg.norm(got - want, axis=-1)
    ref = np.linalg.norm(want, axis=-1)
    sel = ref >= np.median(ref)
    if not sel.any() or ref[sel].max() == 0.0:
        return 0.0
    sel &= ref > 0
    return float((err[sel] / ref[sel]).max())


def followed_by_torch(f, x, y):
    """Yields (name, f(y)) as each of torch's ways of following a function of a tensor gives it: recorded on `x` and played on
    `y`, traced symbolically, or run under a mode."""
    from torch._subclasses.fake_tensor import FakeTensorMode
    from torch.fx.experimental.proxy_tensor import make_fx
    yield "trace", torch.jit.trace(lambda a: f(a), (x,), check_trace=False)(y)
    yield "make_fx", make_fx(lambda a: f(a))(x)(y)
    yield "compile", torch.compile(lambda a: f(a), backend="eager", fullgraph=True)(y)
    with FakeTensorMode(allow_non_fake_inputs=False) as mode:
        fake = f(mode.from_tensor(y))
    want = f(y)
    assert type(fake).__name__ == "FakeTensor" and fake.shape == want.shape and fake.dtype == want.dtype
    seen = []

    class Mode(torch.overrides.TorchFunctionMode):
        def __torch_function__(self, func, types, args=(), kwargs=None):
            seen.append(func)
            return func(*args, **(kwargs or {}))
    with Mode():
        got = f(y)
    assert len(seen) > 1 and any("zeros" in str(s) or "cat" in str(s) for s in seen)
    yield "function mode", got


def _kernel_nodes(f):
    """(node, parameters) of the kernels that f() launches, from a graph that captures the call."""
    from cuda.bindings import driver
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        f()
    graph = driver.CUgraph(g.raw_cuda_graph())
    _, _, count = driver.cuGraphGetNodes(graph, 0)
    _, nodes, _ = driver.cuGraphGetNodes(graph, count)
    for node in nodes[:count]:
        if _got(driver.cuGraphNodeGetType(node)) == driver.CUgraphNodeType.CU_GRAPH_NODE_TYPE_KERNEL:
            yield node, _got(driver.cuGraphKernelNodeGetParams(node))


def _got(result):
    from cuda.bindings import driver
    assert result[0] == driver.CUresult.CUDA_SUCCESS, result[0]
    return result[1]


def launched(f):
    """[(kernel's mangled name, (grid x, y, z))] of the kernels that f() launches."""
    from cuda.bindings import driver
    return [(_got(driver.cuFuncGetName(p.func)).decode(), (p.gridDimX, p.gridDimY, p.gridDimZ)) for _, p in _kernel_nodes(f)]


def clusters(f):
    """[(kernel's mangled name, CTAs of a cluster)] of the kernels that f() launches (1: launched without clusters)."""
    from cuda.bindings import driver
    attr = driver.CUlaunchAttributeID.CU_LAUNCH_ATTRIBUTE_CLUSTER_DIMENSION
    found = []
    for node, p in _kernel_nodes(f):
        dim = _got(driver.cuGraphKernelNodeGetAttribute(node, attr)).clusterDim
        found.append((_got(driver.cuFuncGetName(p.func)).decode(), max(dim.x, 1) * max(dim.y, 1) * max(dim.z, 1)))
    return found
