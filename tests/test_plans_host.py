"""Which kernel entry calls at the limits of the dispatch rules take (no GPU): the GPU tests that
run these calls then reach the entries they mean to."""
import pytest

from tests import plans


@pytest.mark.parametrize("dtype,T,H,off,res,plain", plans.NORM_LIMITS)
def test_norm_entries(dtype, T, H, off, res, plain):
    assert plans.norm(True, dtype, H, T, off) == res
    assert plans.norm(False, dtype, H, T, off) == plain


@pytest.mark.parametrize("T,Hq,Hkv,D,qk,entry", plans.ROPE_LIMITS)
def test_rope_entries(T, Hq, Hkv, D, qk, entry):
    assert plans.rope(T, Hq, Hkv, D, qk) == entry


def test_chain_entries():
    got = [plans.chain(qk, H, Hq, I, T, pdl, inplace) for H, Hq, I, qk, T, pdl, inplace, _ in plans.CHAIN_LIMITS]
    assert got == [c[-1] for c in plans.CHAIN_LIMITS]
