"""Calls with more query and key tiles than SMs, so that a CTA takes several of them one after the other: tiles with one step and
with several, with none at all between others, a last tile that is ragged, outputs that are aligned to 16 bytes only."""
import numpy as np
import pytest

from paper_2410_09397_b200 import inputs
from tests import helpers as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("det", [0, 1])
@pytest.mark.parametrize("heads,n,mask_kind", [(500, 72, inputs.MASK_NONE), (330, 264, inputs.MASK_NONE), (331, 200, inputs.MASK_CAUSAL),
                                               (130, 520, inputs.MASK_CAUSAL), (320, 131, inputs.MASK_CAUSAL), (310, 259, inputs.MASK_NONE)])
def test_no_lists(heads, n, mask_kind, d, det):
    from paper_2410_09397_b200 import binding as B
    errs = H.run_case(1, heads, n, d, "bf16", mask_kind, seed=71, cfg=B.Cfg(deterministic=det), check_bwd_only=False)
    H.assert_within(errs, "bf16")


def _holes(nb):
    """Block rows and columns that keep nothing beside full ones, and single blocks."""
    keep = np.zeros((1, nb, nb), dtype=np.uint8)
    keep[0, 1::3, 1::2] = 1
    keep[0, nb - 1, :] = 1
    keep[0, 0, nb // 2] = 1
    return keep


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("det", [0, 1])
@pytest.mark.parametrize("block", [32, 64, 128, 256])
@pytest.mark.parametrize("mask_kind", [inputs.MASK_BLOCK_SPARSE, inputs.MASK_BLOCK_SPARSE_CAUSAL])
def test_lists_with_empty_rows_and_columns(block, mask_kind, d, det):
    from paper_2410_09397_b200 import binding as B
    n = 904
    errs = H.run_case(1, 60, n, d, "bf16", mask_kind, seed=72, block=block, bmask=_holes((n + block - 1) // block),
                      cfg=B.Cfg(deterministic=det), check_bwd_only=False)
    H.assert_within(errs, "bf16")


@pytest.mark.parametrize("n", [8, 136, 1000, 1160, 4104])
@pytest.mark.parametrize("mask_heads", [1, 2])
def test_row_lists_of_element_masks(n, mask_heads):
    """At most one tile of work a CTA.  Tiles with a single entry, in their first and last row and column, and rows of tiles without any."""
    keep = np.zeros((mask_heads, n, n), dtype=np.uint8)
    for h in range(mask_heads):
        keep[h, 0, n - 1] = keep[h, n - 1, h] = keep[h, n // 2, n // 2] = 1
        if n > 256:
            keep[h, 255, 127] = keep[h, 255, 128] = 1
            keep[h, n - 8, ::300] = 1
    errs = H.run_case(1, 2, n, 64, "bf16", inputs.MASK_ELEMENT, seed=75, bmask=keep, check_bwd_only=False)
    H.assert_within({name: errs[name] for name in ("O", "LSE", "dV")}, "bf16")     # a row with one key has a dS of zero: nothing to relate an error to


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("block", [64, 128])
@pytest.mark.parametrize("mask_kind", [inputs.MASK_BLOCK_SPARSE, inputs.MASK_BLOCK_SPARSE_CAUSAL])
def test_lists_at_a_length_with_two_terms(block, mask_kind, d):
    n = 901
    errs = H.run_case(1, 60, n, d, "bf16", mask_kind, seed=76, block=block, bmask=_holes((n + block - 1) // block), check_bwd_only=False)
    H.assert_within(errs, "bf16")


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("det", [0, 1])
@pytest.mark.parametrize("heads,n,mask_heads", [(200, 392, 1), (90, 1160, 1), (90, 392, 90)])
def test_element_masks(heads, n, mask_heads, d, det):
    """Several tiles of a CTA whose lists and keep words differ: few keys a row but at least two, tiles that keep none at all."""
    from paper_2410_09397_b200 import binding as B
    rng = np.random.default_rng(77)
    keep = (rng.random((mask_heads, n, n)) < 8 / n).astype(np.uint8)
    keep[:, :, 128:256] = 0
    rows = np.arange(n)
    keep[:, rows, rows % 100] = keep[:, rows, n - 1 - rows % 70] = 1
    errs = H.run_case(1, heads, n, d, "bf16", inputs.MASK_ELEMENT, seed=77, bmask=keep, cfg=B.Cfg(deterministic=det), check_bwd_only=False)
    H.assert_within(errs, "bf16")


@pytest.mark.parametrize("heads,n,mask_kind", [(300, 72, inputs.MASK_NONE), (90, 328, inputs.MASK_CAUSAL)])
def test_wide_heads(heads, n, mask_kind):
    errs = H.run_case(1, heads, n, 256, "bf16", mask_kind, seed=73, check_bwd_only=False)
    H.assert_within(errs, "bf16")


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("det", [0, 1])
def test_outputs_aligned_to_16_bytes(d, det):
    """The same call into outputs that begin 16 bytes behind a multiple of 32: results that repeat are the same bit for bit, dQ
    from atomics within its rounding."""
    import torch
    import paper_2410_09397_b200 as attn
    g = torch.Generator("cuda").manual_seed(74)
    shape = (1, 160, 264, d)
    q, k, v, do = (torch.randn(shape, device="cuda", dtype=torch.bfloat16, generator=g) for _ in range(4))
    cfg, mask = attn.Cfg(deterministic=det), attn.Mask(kind=attn.ATTN_MASK_CAUSAL)

    def like(off):
        return torch.full((q.numel() + 8,), 7.0, device="cuda", dtype=torch.bfloat16)[off:off + q.numel()].view(shape)

    def step(off):
        out = [like(off) for _ in range(4)]
        lse = torch.empty(shape[:3], device="cuda")
        attn.attn_fwd(q, k, v, out[0], lse, mask=mask, cfg=cfg)
        attn.attn_bwd(q, k, v, out[0], do, lse, *out[1:], mask=mask, cfg=cfg)
        return out
    a, b = step(0), step(8)
    assert a[0].data_ptr() % 32 == 0 and b[0].data_ptr() % 32 == 16
    for i, (x, y) in enumerate(zip(a, b)):
        if i == 1 and not det:
            assert (x.float() - y.float()).abs().max() <= 2 ** -7 * x.float().abs().max()    # one bf16 rounding
        else:
            assert torch.equal(x, y), i
