"""Read-outs into a device buffer whose allocation ends before the values: refused
on the host, before any kernel runs."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
SIZE = 64 << 20


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1407_1810_gb300 import build

    build.build()


def _ahead(addr):
    base, size = C.c_uint64(), C.c_size_t()
    rc = C.CDLL("libcuda.so.1").cuMemGetAddressRange_v2(C.byref(base), C.byref(size), C.c_uint64(addr))
    return 0 if rc else base.value + size.value - addr


@pytest.fixture()
def allocate():
    """Device allocations of the runtime's own; freed after the test."""
    import torch

    torch.cuda.init()
    lib = C.CDLL(next(line.split()[-1] for line in open("/proc/self/maps") if "libcudart" in line))
    held = []

    def one():
        q = C.c_void_p()
        assert lib.cudaMalloc(C.byref(q), C.c_size_t(SIZE)) == 0
        held.append(q)
        return q.value

    yield one
    torch.cuda.synchronize()
    for q in held:
        assert lib.cudaFree(q) == 0


@pytest.mark.parametrize("call", ["fields", "total", "flux", "charge", "luminosity"])
def test_short_device_buffer(call, allocate):
    import torch

    from paper_1407_1810_gb300 import picsar as P

    L = P.lib()
    s = P.Simulation(P.make_desc(nr=12, nth=20, r_min=1.0, r_max=3.0, r_map="log", th_map="linear", dt=0.004, n_filt=1,
                                 vacuum="monopole", b0=2.0, precision="fp32", pusher="vay"),
                     stream=torch.cuda.current_stream().cuda_stream)
    s.load(*(np.full(4, v) for v in (3.5, 4.25, 0.1, 0.2, 0.3, 1.0)))
    s.step(2)

    def ask(p, n):
        p, n = C.c_void_p(p) if p is not None else None, C.byref(n)
        if call in ("fields", "total"):
            return L.pic_get_fields(s.h, int(call == "total"), p, n, P.PIC_MEM_DEVICE)
        if call == "charge":
            return L.pic_get_charge(s.h, 1, p, n, P.PIC_MEM_DEVICE)
        return getattr(L, "pic_get_" + call)(s.h, p, n, P.PIC_MEM_DEVICE)

    n = C.c_int64()
    assert ask(None, n) == P.PIC_OK
    blocks = [allocate() for _ in range(8)]
    block = next((b for b in blocks if not _ahead(b + SIZE)), None)
    if block is None:
        pytest.skip("an allocation follows each of the buffers")
    for short in (8, 8 * (n.value - 1)):  # one value too short, room for one
        assert ask(block + SIZE - (8 * n.value - short), n) == P.PIC_ECUDA
    out = torch.full((n.value + 1,), -7.0, dtype=torch.float64, device="cuda")
    assert ask(out.data_ptr(), n) == P.PIC_OK
    assert ask(block + SIZE - 8 * n.value, n) == P.PIC_OK  # to the last byte of it
    ref = {"fields": s.fields, "total": lambda: s.fields(total=True), "flux": s.flux,
           "charge": lambda: s.charge(filtered=True), "luminosity": s.luminosity}[call]()
    assert np.array_equal(out[:-1].cpu().numpy(), ref.ravel()) and out[-1] == -7.0
