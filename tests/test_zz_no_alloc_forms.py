"""The forms of the no-allocation potential: every x length, both precisions, and a single-precision state eight bytes
behind the address that bulk copies can start at (another chain of kernels), against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["fp64", "fp32", "fp32 off by 8 bytes"])
@pytest.mark.parametrize("n", [(32, 512), (64, 32, 128), (128, 64, 32), (256, 32, 32), (512, 64), (32, 256, 32)])
def test_noalloc_forms(n, form):
    torch = pytest.importorskip("torch")
    from paper_1601_04640_gb300 import build as gbuild
    from paper_1601_04640_gb300 import dgpe, synth
    gbuild.build()
    dim, fp64, off = len(n), form == "fp64", int(form.endswith("bytes"))
    h = (0.2, 0.25, 0.3)[:dim]
    ctype, rtype = (torch.complex128, torch.float64) if fp64 else (torch.complex64, torch.float32)
    psi = synth.gaussian_state(n, h, (1.0, 0.8, 1.2)[:dim], 0.05, 9)
    buf = torch.empty(psi.size + 2, dtype=ctype, device="cuda")[off:off + psi.size]
    buf.copy_(torch.from_numpy(psi).to(ctype).reshape(-1))
    phi = torch.full((psi.size,), float("nan"), dtype=rtype, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    dgpe.dgpe_dipolar_potential_noalloc(buf.data_ptr(), phi.data_ptr(), fp64, dim, n, h, stream=stream)
    got = phi.double().cpu().numpy().reshape(psi.shape)
    held = buf.cpu().numpy().astype(np.complex128).reshape(psi.shape)
    op = oracle.Params(dim=dim, n=n, h=h, nu=(0,) * dim, kernel="dipolar3d" if dim == 3 else "quasi2d", qd=0.5)
    ref = oracle.dipolar_potential(op, np.abs(held) ** 2)
    e = np.max(np.abs(got - ref)) / np.max(np.abs(ref))
    print(n, form, "rel max", e)
    # two transforms of log2 N layers, a handful of roundings each, against the largest value
    assert e < 8 * np.log2(psi.size) * (2.0 ** -53 if fp64 else 2.0 ** -24)
