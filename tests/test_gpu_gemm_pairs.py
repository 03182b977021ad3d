"""The product on CTA pairs (K >= 2048, M and N multiples of 256, at least 76 tiles
of 128 x 256) and its neighbours in the dispatch: the ring's wrap (32 and 33 chunks
of K over 6 stages), a K one chunk short, an odd count of row tiles, the N below,
and K loops of one to four chunks (rings of as many stages)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_1911_13255_gb300 as pkg  # noqa: E402


@pytest.mark.parametrize("M,N,K", [(9728, 256, 2048), (9728, 256, 2112), (9728, 256, 1984), (9856, 256, 2048),
                                   (4864, 512, 2432), (9728, 128, 2048), (19200, 256, 64), (19200, 256, 128),
                                   (9728, 512, 192), (384, 48, 256)])
@pytest.mark.parametrize("bias", [False, True])
def test_products_around_the_pair_dispatch(M, N, K, bias):
    g = torch.Generator().manual_seed(M + 3 * N + 7 * K)
    A = torch.randn(M, K, generator=g).to(torch.bfloat16).cuda()
    B = torch.randn(N, K, generator=g).to(torch.bfloat16).cuda()
    b = torch.randn(N, generator=g).cuda() if bias else None
    C = torch.full((M, N), float("nan"), device="cuda")
    pkg.gemm_bf16(A, B, b, out=C)
    torch.cuda.synchronize()
    ref = A.double() @ B.double().T
    if bias:
        ref = ref + b.double()
    # FP32 accumulation over K: about sqrt(K) roundings of 2^-24 relative, per
    # 128 x 128 block so that a block in the wrong place cannot hide
    tol = 4.0 * np.sqrt(K) * 2.0 ** -24
    d, r = (C.double() - ref).pow(2), ref.pow(2)
    if N % 128 == 0:
        d, r = (t.view(M // 128, 128, N // 128, 128).sum((1, 3)) for t in (d, r))
    else:
        d, r = d.sum(), r.sum()
    assert bool(((d / r).sqrt() < tol).all()), float((d / r).sqrt().max())
    assert pkg.tc_status(reset=True) == 0
