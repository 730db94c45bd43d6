"""The gate-up kernels at the edges of their ranges.  The weight-streaming one
(calls of at most 160 tokens, 224 where each CTA has an SM and half the SMs or
more have one): one token, around the multiples of 16 that change the MMA's N,
the largest call it takes and the first one past it; the smallest K and
feature counts, K around the length of each ring, and CTAs that share SMs,
called back to back.  The CTA-pair one: last rounds whole and in slices, many
rounds of little K.  Every element against the float64 oracle, and the rows
after the last token untouched."""
import numpy as np
import pytest
import torch

from oracle import mlp
from test_gpu_gateup import _check, _inputs, ppas  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1, 15, 16, 17, 33, 64, 65, 127, 128, 129, 145, 160, 161])
@pytest.mark.parametrize("H,I", [(64, 128), (1024, 384)])
def test_every_element_and_nothing_past_the_tokens(ppas, T, H, I):  # noqa: F811
    x, w = _inputs(T, H, I, seed=3 * T + H)
    wp = torch.empty_like(w)
    ppas.ppas_gateup_pack(w, wp, H, I)
    y = torch.full((T + 3, I), 7.0, dtype=torch.bfloat16, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    ppas.ppas_gateup_swiglu(x, wp, y, T, H, I, err)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    assert bool((y[T:] == 7.0).all())
    _check(y[:T].float().cpu().numpy(), mlp.gate_up(x.float().cpu().numpy(), w.float().cpu().numpy()),
           f"T={T} H={H} I={I}")


@pytest.mark.parametrize("T,H,I", [
    (1, 64 * 11, 128),      # the long ring (12 stages), one K block short of it
    (1, 64 * 12, 256),      # just its length
    (1, 64 * 25, 128),      # twice, and one
    (128, 64 * 6, 384),     # the long ring of 6 stages
    (128, 64 * 7, 384),
    (160, 64 * 7, 128),
    (224, 64 * 6, 4864),    # half the SMs stream: the long ring of 5 stages up to 224 tokens
    (193, 64 * 4, 9728),
    (225, 64 * 6, 4864),    # and CTA pairs past that
    (161, 64 * 6, 4736),    # fewer than half: CTA pairs past 160
    (50, 64 * 20, 9728),    # a CTA for each of 152 SMs: the long ring
    (50, 64 * 20, 9856),    # two CTAs more: the short one
])
def test_ring_lengths(ppas, T, H, I):  # noqa: F811
    """K around the length of the long ring, and both sides of the CTA count
    where the short one takes over."""
    test_every_element_and_nothing_past_the_tokens(ppas, T, H, I)


@pytest.mark.parametrize("T,H,I", [
    (225, 64, 128 * 40),    # 40 tiles: one round of whole tiles
    (200, 128, 128 * 30),   # 30 tiles: halves
    (256, 64, 128 * 19),    # 19 tiles: quarters
    (257, 192, 128),        # 2 tiles, the second of one token
    (513, 64, 128 * 27),    # 81 tiles: a round of whole tiles, then 5 in quarters
    (400, 64, 128 * 55),    # 110 tiles: whole, then 34 in halves
])
def test_pair_tiles_and_slices_of_the_last_round(ppas, T, H, I):  # noqa: F811
    """Calls of the CTA-pair kernel whose last round is whole, halved or
    quartered (on 76 pairs), ragged in tokens, K shorter than the ring; and
    the rows after the last token untouched."""
    x, w = _inputs(T, H, I, seed=T + I)
    wp = torch.empty_like(w)
    ppas.ppas_gateup_pack(w, wp, H, I)
    y = torch.full((T + 3, I), 7.0, dtype=torch.bfloat16, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    for _ in range(2):
        ppas.ppas_gateup_swiglu(x, wp, y, T, H, I, err)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    assert bool((y[T:] == 7.0).all())
    _check(y[:T].float().cpu().numpy(), mlp.gate_up(x.float().cpu().numpy(), w.float().cpu().numpy()),
           f"T={T} H={H} I={I}")


@pytest.mark.parametrize("T,H,I", [(4000, 64, 128 * 54), (2500, 512, 128 * 31)])
def test_many_rounds_of_short_tiles(ppas, T, H, I):  # noqa: F811
    """Many rounds of the CTA-pair kernel with little K: the epilogue sets the
    pace, and the next tile's MMAs wait for it to leave each accumulator."""
    x, w = _inputs(T, H, I, seed=T + H)
    wp = torch.empty_like(w)
    ppas.ppas_gateup_pack(w, wp, H, I)
    ys = [torch.full((T + 1, I), 7.0, dtype=torch.bfloat16, device="cuda") for _ in range(4)]
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    for y in ys:
        ppas.ppas_gateup_swiglu(x, wp, y, T, H, I, err)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    for y in ys:
        assert bool((y[T:] == 7.0).all()) and torch.equal(y, ys[0])
    _check(ys[0][:T].float().cpu().numpy(), mlp.gate_up(x.float().cpu().numpy(), w.float().cpu().numpy()),
           f"T={T} H={H} I={I}")


@pytest.mark.parametrize("T,H,I", [
    (160, 64 * 7, 11008),   # two CTAs on most SMs: all 512 TMEM columns, three stages, the epilogue over them
    (129, 64 * 4, 11008),
    (144, 64 * 3, 9856),    # just more CTAs than SMs, K as long as the ring
    (8, 2048, 11008),       # a decode iteration
    (64, 64 * 8, 20480),    # 320 CTAs: more than two for each SM
])
def test_shared_sms_back_to_back(ppas, T, H, I):  # noqa: F811
    """More CTAs than SMs, each call started while the one before still runs."""
    x, w = _inputs(T, H, I, seed=T + H + I)
    wp = torch.empty_like(w)
    ppas.ppas_gateup_pack(w, wp, H, I)
    ys = [torch.full((T + 3, I), 7.0, dtype=torch.bfloat16, device="cuda") for _ in range(6)]
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    for y in ys:
        ppas.ppas_gateup_swiglu(x, wp, y, T, H, I, err)
    torch.cuda.synchronize()
    assert int(err.item()) == 0
    for y in ys:
        assert bool((y[T:] == 7.0).all()) and torch.equal(y, ys[0])
    _check(ys[0][:T].float().cpu().numpy(), mlp.gate_up(x.float().cpu().numpy(), w.float().cpu().numpy()),
           f"T={T} H={H} I={I}")


def test_both_kernels_in_turn_on_one_stream(ppas):  # noqa: F811
    """Calls of 8, 160 and 300 tokens (rings of other depths, one and two CTAs
    an SM, CTA pairs) after one another without a wait equal the same calls
    with one."""
    H, I = 64 * 10, 11008
    x, w = _inputs(300, H, I, seed=5)
    wp = torch.empty_like(w)
    ppas.ppas_gateup_pack(w, wp, H, I)
    got = []
    for wait in (True, False):
        ys = []
        torch.cuda.synchronize()
        for T in (8, 160, 300) * 4:
            y = torch.full((T, I), 7.0, dtype=torch.bfloat16, device="cuda")
            ppas.ppas_gateup_swiglu(x[:T], wp, y, T, H, I)
            if wait:
                torch.cuda.synchronize()
            ys.append(y)
        torch.cuda.synchronize()
        got.append(ys)
    assert all(torch.equal(a, b) for a, b in zip(*got))
    _check(got[0][2].float().cpu().numpy(), mlp.gate_up(x.float().cpu().numpy(), w.float().cpu().numpy()), "300 tokens")


def test_back_to_back_calls_on_each_others_output(ppas):  # noqa: F811
    """Each call reads what the call before wrote (the kernel sets up while
    its predecessor still runs): a chain of calls equals the same chain with
    a wait after each."""
    T, H = 24, 256
    x, w = _inputs(T, H, H, seed=11)
    wp = torch.empty_like(w)
    ppas.ppas_gateup_pack(w, wp, H, H)
    got = []
    for wait in (True, False):
        a = x.clone()
        for _ in range(6):
            b = torch.empty_like(a)
            ppas.ppas_gateup_swiglu(a, wp, b, T, H, H)
            if wait:
                torch.cuda.synchronize()
            a = b
        torch.cuda.synchronize()
        got.append(a.float().cpu().numpy())
    assert np.array_equal(got[0], got[1])
