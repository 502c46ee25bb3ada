"""The allocation-free predictor call against the same sums in 64 bits: widths around its blocks of four hidden units and
256 threads, the widest hidden layer, and inputs that do not start on 16 bytes (the path without wide loads)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,hid,nmax,shift", [
    (1, 1, 1, 0), (7, 5, 3, 0), (64, 8, 1, 0), (256, 128, 8, 1), (2048, 504, 8, 0), (2056, 512, 15, 0),
    (4096, 520, 10, 0), (4096, 512, 10, 1), (4104, 4096, 15, 0), (33, 4095, 2, 0)])
def test_static_predictor_sums(d, hid, nmax, shift):
    from paper_2412_18910_b200 import ada_ldlp_eval_static
    g = torch.Generator("cuda").manual_seed(d + hid)

    def make(*dims, std, dtype=torch.bfloat16):
        n = 1
        for x in dims:
            n *= x
        flat = torch.empty(n + shift, device="cuda").normal_(0.0, std, generator=g).to(dtype)
        return flat[shift:].view(*dims)

    w1, b1 = make(hid, 2 * d, std=0.05), make(hid, std=0.05)
    w2, b2 = make(nmax, hid, std=0.05), make(nmax, std=0.05)
    e, f = make(d, std=1.0), make(d, std=1.0, dtype=torch.float32)
    n, z = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.zeros(nmax, device="cuda")
    assert ada_ldlp_eval_static(w1, b1, w2, b2, e, f, n, z, stream=torch.cuda.current_stream()) == 0
    x = torch.cat([e.double(), f.double()])
    h = torch.relu(w1.double() @ x + b1.double())
    ref = w2.double() @ h + b2.double()
    # 32-bit sums of K terms in any order: at most K 2^-24 of the sum of their sizes, in both layers
    size1 = w1.double().abs() @ x.abs() + b1.double().abs()
    bound = (2 * d + hid + 4) * 2.0 ** -24 * (w2.double().abs() @ size1 + b2.double().abs())
    assert bool(((z.double() - ref).abs() <= bound).all()), float((z.double() - ref).abs().max())
    assert int(n) == int(torch.argmax(z)) + 1


def test_static_predictor_calls_in_a_row():
    """Calls behind one another on a stream without a wait between them, each with its own weights, inputs and outputs: grids of one
    block, partly filled last blocks, the widest hidden layer and pointers off 16 bytes, in changing order.  They share the hidden
    activations' array, and calls of as many blocks a count."""
    from paper_2412_18910_b200 import ada_ldlp_eval_static
    g = torch.Generator("cuda").manual_seed(3)
    d, calls = 264, []
    for i in range(60):
        hid, nmax, shift = (1, 5, 130, 512, 4096, 129, 510)[(i * i + i // 7) % 7], 1 + i % 15, i % 3 == 2

        def make(*dims, std, dtype=torch.bfloat16):
            n = 1
            for x in dims:
                n *= x
            flat = torch.empty(n + shift, device="cuda").normal_(0.0, std, generator=g).to(dtype)
            return flat[int(shift):].view(*dims)

        calls.append((make(hid, 2 * d, std=0.05), make(hid, std=0.05), make(nmax, hid, std=0.05), make(nmax, std=0.05), make(d, std=1.0),
                      make(d, std=1.0, dtype=torch.float32), torch.zeros(1, dtype=torch.int32, device="cuda"),
                      torch.full((nmax,), float("nan"), device="cuda")))
    for _ in range(3):
        for c in calls:
            assert ada_ldlp_eval_static(*c, stream=torch.cuda.current_stream()) == 0
    for w1, b1, w2, b2, e, f, n, z in calls:
        x = torch.cat([e.double(), f.double()])
        ref = w2.double() @ torch.relu(w1.double() @ x + b1.double()) + b2.double()
        # 32-bit sums in any order, as above
        bound = (2 * d + len(b1) + 4) * 2.0 ** -24 * (w2.double().abs() @ (w1.double().abs() @ x.abs() + b1.double().abs()) + b2.double().abs())
        assert bool(((z.double() - ref).abs() <= bound).all()), len(b1)
        assert int(n) == int(torch.argmax(z)) + 1


def test_static_predictor_is_ordered_behind_everything():
    """Captured between two other kernels: the call's dependencies are full ones.  (Behind a programmatic one it could start, and finish,
    before kernels that the kernel before it did not wait for.)"""
    from cuda.bindings import runtime as rt
    from paper_2412_18910_b200 import ada_ldlp_eval_static
    d, hid, nmax = 64, 32, 4
    bf = dict(dtype=torch.bfloat16, device="cuda")
    args = (torch.zeros(hid, 2 * d, **bf), torch.zeros(hid, **bf), torch.zeros(nmax, hid, **bf), torch.zeros(nmax, **bf), torch.zeros(d, **bf),
            torch.zeros(d, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda"))
    other = torch.zeros(8, device="cuda")
    assert ada_ldlp_eval_static(*args, stream=torch.cuda.current_stream()) == 0   # (the first call looks the array up)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(graph):
        other.add_(1)
        assert ada_ldlp_eval_static(*args, stream=torch.cuda.current_stream()) == 0
        other.add_(1)
    raw = rt.cudaGraph_t(init_value=graph.raw_cuda_graph())
    err, roots, count = rt.cudaGraphGetRootNodes(raw, 4)
    assert err == rt.cudaError_t.cudaSuccess and count == 1     # (the first other kernel)
    err, _, count = rt.cudaGraphNodeGetDependentNodes(roots[0], 4)
    assert err == rt.cudaError_t.cudaSuccess and count == 1     # cudaErrorLossyQuery: there is an edge that is not a full dependency
