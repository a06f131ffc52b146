"""The append's split of nodes over CTAs and its rounding, bit for bit against the fp64 oracle.

The kernel rotates in pairs of fp32 values and decides each bf16 rounding from them, falling back to fp64 where
they cannot; the values below reach every branch: cancellation between the two products, signed zeros, values
whose products are not exact in fp32, and magnitudes near the top of the range.
"""
import numpy as np
import pytest
import torch

from oracle import oracle
from paper_2604_26412_gb300 import kvshot
from paper_2604_26412_gb300 import workloads as wl

pytestmark = pytest.mark.gpu
D = wl.HEAD_DIM


def _values(rng, shape):
    """bf16 bits: N(0, 1), with heads of equal partners, zeros of both signs, tiny and huge values."""
    x = rng.standard_normal(shape).astype(np.float32)
    heads = x.reshape(-1, D)
    for i, h in enumerate(heads):
        kind = i % 7
        if kind == 1:
            h[D // 2:] = h[:D // 2]
        elif kind == 2:
            h[rng.random(D) < 0.5] = 0.0
            h[::3] *= -1
        elif kind == 3:
            h *= np.float32(2.0) ** rng.integers(-140, -50, D).astype(np.float32)
        elif kind == 4:
            h *= np.float32(2.0) ** rng.integers(90, 124, D).astype(np.float32)
        elif kind == 5:
            h[:D // 2] *= np.float32(2.0) ** rng.integers(-30, 0, D // 2).astype(np.float32)
    return wl.bf16_bits(torch.from_numpy(x).to(torch.bfloat16))


# One node split over CTAs (with fewer heads than CTAs too), the last node counts with a split, one and two nodes per
# CTA, an odd one left over; positions that repeat and change inside a CTA's nodes, small, at 2^31 - 1 and between.
@pytest.mark.parametrize("caches,n_new,hq,hkv,base", [
    (1, 1, 32, 8, 1e6), (1, 1, 1, 1, 1e6), (2, 64, 4, 2, 1e4), (16, 16, 8, 4, 1e6), (3, 171, 2, 1, 1e6),
    (5, 205, 2, 2, 500.0), (1, 1031, 1, 1, 1e6), (3, 5, 4, 4, 1.0)])
def test_append_is_bit_exact(caches, n_new, hq, hkv, base):
    rng = np.random.default_rng(caches * 1000 + n_new)
    q, k, v = (_values(rng, (caches, n_new, h, D)) for h in (hq, hkv, hkv))
    pos = rng.choice(np.array([0, 1, 5, 4096, 32771, 10 ** 6, 2 ** 31 - 1]), (caches, n_new)).astype(np.int32)
    pos = np.repeat(pos, 2, axis=1)[:, :n_new] if n_new > 4 else pos
    n_max = n_new + 3
    dev = lambda b: wl.bits_to_bf16(b).cuda()  # noqa: E731
    qd, kd, vd = dev(q), dev(k), dev(v)
    dk = torch.full((caches, hkv, n_max, D), 7.0, dtype=torch.bfloat16, device="cuda")
    dv = dk.clone()
    q_out = torch.empty_like(qd)
    desc = kvshot.make_desc(num_caches=caches, num_seqs=caches, hq=hq, hkv=hkv, n_nodes=0, n_query=0, n_max=n_max,
                            max_seq_len=0)
    pos_d = torch.from_numpy(np.ascontiguousarray(pos)).cuda()
    kvshot.draft_append(desc, qd, kd, vd, pos_d, 2, n_new, base, dk, dv, q_out)
    rk, rv = (np.full((caches, hkv, n_max, D), wl.bf16_bits(torch.tensor([7.0], dtype=torch.bfloat16))[0], np.uint16)
              for _ in range(2))
    od = oracle.make_desc(num_caches=caches, num_seqs=caches, hq=hq, hkv=hkv, head_dim=D, n_nodes=0, n_query=0,
                          n_max=n_max, tree=False, l_cap=1)
    rq = oracle.append(od, q, k, v, np.ascontiguousarray(pos), 2, n_new, base, rk, rv)
    torch.cuda.synchronize()
    assert np.array_equal(wl.bf16_bits(q_out), rq)
    assert np.array_equal(wl.bf16_bits(dk), rk) and np.array_equal(wl.bf16_bits(dv), rv)
    kvshot.draft_append(desc, qd, kd, vd, pos_d, 2, n_new, base, dk, dv, qd)  # in place
    assert np.array_equal(wl.bf16_bits(qd), rq)


def test_angles_beyond_the_fast_reduction_still_rotate():
    # rope_base below 1 makes angles up to 1e38, past the range of the kernel's own reduction; their phase depends on
    # the last bit of the frequency, but every pair keeps its norm (three bf16 roundings: 2^-8 relative).
    g = torch.Generator().manual_seed(3)
    q = torch.randn((2, 3, 4, D), generator=g).to(torch.bfloat16).cuda()
    pos = torch.tensor([[0, 1, 77], [4096, 10 ** 6, 2 ** 31 - 1]], dtype=torch.int32, device="cuda")
    dk, dv = (torch.zeros((2, 4, 8, D), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    out = torch.empty_like(q)
    desc = kvshot.make_desc(num_caches=2, num_seqs=2, hq=4, hkv=4, n_nodes=0, n_query=0, n_max=8, max_seq_len=0)
    kvshot.draft_append(desc, q, q, q, pos, 0, 3, 1e-30, dk, dv, out)
    a, b = q.double(), out.double()
    before, after = (torch.hypot(x[..., :D // 2], x[..., D // 2:]) for x in (a, b))
    assert torch.allclose(before, after, rtol=2.0 ** -7, atol=0)
    assert torch.equal(out[0, 0], q[0, 0])  # position 0 is the identity
    assert torch.equal(dk[:, :, :3], out.transpose(1, 2))
