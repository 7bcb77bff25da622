"""A plan reserves the buffers its kernels use: what an exact-layer-block (strip) plan, a
banded one and a single subdomain hold beside the factors, the basis and the vectors."""
import pytest

from paper_1102_3137_gb300 import dyson as D


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_1102_3137_gb300 import build
    build.build()
    return D.load()


def need(L, p, K, k, mixed, layer, block=1):
    """Bytes of the buffers of a 2D plan, from their shapes."""
    Lx, Ly = L
    h = -(-(Ly - p + 1) // p)
    W = (h + 3) & ~3
    N, nsub, ifc, A = Lx * Ly, Lx * W, (p - 1) * Lx, Lx
    ndd, c = p * nsub + ifc, 8 if mixed else 16
    slots = K * block
    b = N * 8 + K * 8 + K * N * 16 + block * N * 8 + ndd * 4                 # inputs, index map
    b += K * p * nsub * W * (c + (16 if mixed else 0))                       # factors
    b += K * ndd * 16 * (2 + k + block) + slots * ndd * 16                   # diag B, sum, basis, u
    b += slots * p * nsub * c + slots * p * 2 * A * 16 + slots * 7 * ifc * 16   # rows, boundary, interface
    b += K * (k + block) * 2 * block * 16 + K * (8 + 32 + 4) + K * N * 16 + slots * p * 8
    if mixed:
        b += slots * ndd * 16 * 2 + K * ndd * 16                             # w, residual; H_ii
        if block == 1 and k <= 64:
            b += K * (k + 1) ** 2 * 16                                       # Gram matrix
    if layer:
        b += K * p * 2 * A * A * 8 + K * (p - 1) * A * A * c + K * p * 4 * nsub * 8
    elif p > 1:
        b += K * ifc * 3 * 16 + 2 * K * p * nsub * 16
    return b


@pytest.mark.parametrize("L,p,K,k,block", [((512, 512), 16, 32, 16, 1), ((101, 101), 4, 63, 16, 1), ((128, 128), 4, 16, 16, 2),
                                           ((128, 128), 4, 16, 80, 1)])
@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("layer", [False, True])
def test_strip_plan_holds_what_it_uses(L, p, K, k, block, mixed, layer):
    g = D.make_geometry(L, p=p, k_max=k, max_freqs=K, block_size=block,
                        precision=D.DYSON_MIXED if mixed else D.DYSON_FP64,
                        precond=D.DYSON_PRECOND_LAYER if layer else D.DYSON_PRECOND_BANDED)
    b = need(L, p, K, k, mixed, layer, block)
    assert b <= D.dyson_plan_footprint(g) <= b + 33 * 256                    # each buffer starts on 256 bytes
