"""GPU checks of the dense <-> level copies at the sizes where their column and row blocks end:
values come back exactly, FP32 and FP64 transfers agree, and a level uploaded through single
accesses (a misaligned device buffer) steps like one uploaded through vectors, so the ghost images
are the same."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1), (3, 2), (4, 4), (31, 5), (32, 33), (127, 3), (1023, 9), (1024, 6), (1030, 5), (5, 4, 3), (36, 7, 5),
          (130, 2, 9)]


@pytest.fixture(scope="module")
def mm():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2505_17057_gb300 import mmfd
    return mmfd


def solver(mm, n, storage):
    d = len(n)
    return mm.Solver(mm.make_desc("NSE", "D2Q9" if d == 2 else "D3Q19", 2, list(n), 1.0, [1.0] * d, storage=storage,
                                  a=(1.0, 0.0, 0.0), abar=(1.0, 0.0, 0.0), ref=[1.0] + [0.0] * d))


def device(v, dtype, shift):
    """v on the device, `shift` elements off the allocation's alignment."""
    import torch
    flat = torch.empty(v.size + shift, dtype=dtype, device="cuda")
    flat[shift:].copy_(torch.from_numpy(np.ascontiguousarray(v).ravel()).to(dtype))
    return flat[shift:].view(v.shape)


@pytest.mark.parametrize("n", SHAPES)
@pytest.mark.parametrize("storage", ["fp64", "fp32", "bf16"])
def test_copies(mm, n, storage):
    import torch
    rng = np.random.default_rng(n[0] * 97 + n[1])
    shape = tuple(reversed(n))
    vals = [(1.0 + 0.01 * rng.standard_normal(shape)).astype(np.float32)]
    vals += [(0.03 * rng.standard_normal(shape)).astype(np.float32) for _ in n]
    stored = []
    for f, v in enumerate(vals):
        ref = 1.0 if f == 0 else 0.0
        if storage == "fp64":
            stored.append(v.astype(np.float64))
            continue
        off = v.astype(np.float64) - ref                     # exact in FP64
        q = torch.from_numpy(np.atleast_1d(off)).to(torch.float32)
        if storage == "bf16":
            q = q.to(torch.bfloat16)
        stored.append(ref + q.to(torch.float64).numpy().reshape(shape))
    stepped = []
    for dtype, shift in [(torch.float32, 0), (torch.float32, 1), (torch.float64, 0), (torch.float64, 1)]:
        s = solver(mm, n, storage)
        try:
            s.set_fields([device(v, dtype, shift) for v in vals])
            for got, want in zip(s.fields(0), stored):       # host, FP64
                assert np.array_equal(got, want)
            for back, np_t in ((torch.float32, np.float32), (torch.float64, np.float64)):
                outs = [device(np.zeros(shape), back, shift) for _ in vals]
                mm.mmfd_fields(s.h, 0, [o.data_ptr() for o in outs], mm.MMFD_DEVICE,
                               mm.MMFD_DT_F32 if back == torch.float32 else mm.MMFD_DT_F64)
                torch.cuda.synchronize()
                for o, want in zip(outs, stored):
                    assert np.array_equal(o.cpu().numpy(), want.astype(np_t))
            s.step(2)
            stepped.append(s.fields(0))
        finally:
            s.close()
    for other in stepped[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(stepped[0], other))
