"""GPU parity of the packing over packet sizes.  Few large packets whose assembly takes just below or above 48 KB of shared memory, what a
kernel gets unasked (its static part counted): every size is the first call of a process of its own, since what an earlier call has
asked for stays allowed.  And sizes at the lines between a block and a warp for a packet."""
import multiprocessing as mp

import numpy as np
import pytest

from gpu_util import oracle_plan_encode, params_dict

pytestmark = pytest.mark.gpu

D = 100_003  # 17 bits of position


def packet_shared(packet_bytes, quantizer):
    """shared memory of a packet at work: its words and two more, with QSGD the squares of as many values as it may hold"""
    return (packet_bytes + 8 + 15) // 16 * 16 + (8 * ((8 * packet_bytes - 80) // 18) if quantizer else 0)


def sizes(quantizer):
    """packet sizes below, in and above the last 64 bytes of 48 KB"""
    fits = [b for b in range(9_000, 60_000, 4) if 48 * 1024 - 64 < packet_shared(b, quantizer) <= 48 * 1024]
    return sorted({fits[0] - 64, *fits[::max(1, len(fits) // 3)], fits[-1], fits[-1] + 4})


def first_call(packet_bytes, quantizer, results):
    from gpu_util import gpu_plan_encode
    try:
        x = np.random.default_rng(packet_bytes).laplace(0, 1e-3, D).astype(np.float32)
        pd = params_dict(D, 2 * 8 * packet_bytes, packet_bits=8 * packet_bytes, quantizer=quantizer, seed=3)
        status, _, out = gpu_plan_encode(x, pd)
        results.put((status, bool(np.array_equal(out, oracle_plan_encode(x, pd)[1]))))
    except Exception as e:  # what the call raised, for the assertion
        results.put((repr(e), False))


@pytest.mark.parametrize("quantizer,packet_bytes", [(q, b) for q in (0, 1) for b in sizes(q)])
def test_first_call_with_large_packets(quantizer, packet_bytes):
    ctx = mp.get_context("spawn")
    results = ctx.Queue()
    p = ctx.Process(target=first_call, args=(packet_bytes, quantizer, results))
    p.start()
    try:
        got = results.get(timeout=120)
    finally:
        p.join(timeout=60)
    assert got == (0, True)


SMS = 148


@pytest.mark.parametrize("quantizer,packet_bits,R,d", [
    (0, 1_824, 3, 8_000), (0, 1_888, 3, 8_000), (1, 736, 3, 8_000), (1, 768, 3, 8_000),              # 124 to 135, 46 to 49 records
    (0, 2_080, 9 * SMS, 200_003), (0, 2_528, 9 * SMS, 200_003), (0, 2_528, 9 * SMS + 1, 200_003),    # few and enough records
    (0, 35_968, 9 * SMS + 1, 6_000_001), (0, 36_000, 9 * SMS + 1, 6_000_001),                        # 4496 and 4500 bytes
    (0, 36_000, 13 * SMS, 6_000_001), (0, 36_000, 13 * SMS + 1, 6_000_001)])
def test_block_or_warp_for_a_packet(quantizer, packet_bits, R, d):
    from gpu_util import gpu_plan_encode
    x = np.random.default_rng(packet_bits + R).laplace(0, 1e-3, d).astype(np.float32)
    pd = params_dict(d, R * packet_bits, packet_bits=packet_bits, quantizer=quantizer, seed=4)
    status, _, out = gpu_plan_encode(x, pd)
    assert status == 0
    assert np.array_equal(out, oracle_plan_encode(x, pd)[1])
