"""CPU models of two parts of the tridiagonal eigensolver: the exchange of the
published values between the blocks (values that are their own flags, four
buffers in turn, unset two steps ahead) under random interleavings, and the
compact WY form of the back-transformation by block doubling against the
reflectors applied one by one."""
import random

import numpy as np
import pytest

BUFS = 4


@pytest.mark.parametrize("blocks,steps,seed", [(1, 9, 0), (2, 12, 1), (3, 40, 2), (7, 30, 3), (7, 30, 4)])
def test_no_block_reads_a_stale_value(blocks, steps, seed):
    """Block g at step t: read everyone's words of step t-1 (waiting while one is
    unset), unset its own word of step t+2's buffer, publish step t's.  Writes
    become visible to the others late and, between fences, in any order; the
    fence stands behind the unsetting, before the next publication."""
    rng = random.Random(seed)
    mem = [[None] * blocks for _ in range(BUFS)]         # what everyone sees
    pending = [[] for _ in range(blocks)]                # (slot, value) not yet visible
    unfenced = [[] for _ in range(blocks)]
    phase = [("read", 0, 0)] * blocks                    # (what, step, next word)
    done = 0
    for _ in range(2_000_000):
        g = rng.randrange(blocks)
        if (pending[g] or unfenced[g]) and rng.random() < 0.3:
            box = unfenced[g] if unfenced[g] and (rng.random() < 0.5 or not pending[g]) else pending[g]
            slot, v = box.pop(rng.randrange(len(box)))
            mem[slot][g] = v
            continue
        what, t, i = phase[g]
        if what == "read":
            if t == 0 or i == blocks:
                phase[g] = ("unset", t, 0)
                continue
            v = mem[(t - 1) % BUFS][i]
            if v is None:
                continue
            assert v == (t - 1, i), (g, t, i, v)
            phase[g] = ("read", t, i + 1)
        elif what == "unset":
            if t + 2 < steps:
                unfenced[g].append(((t + 2) % BUFS, None))
            # this step's value may pass this step's unsetting, not the last one's
            pending[g].append((t % BUFS, (t, g)))
            phase[g] = ("fence", t, 0)
        else:
            # the fence: the unset words are visible before the next publication
            if unfenced[g]:
                continue
            if t + 1 == steps:
                phase[g] = ("end", t, 0)
                done += 1
            else:
                phase[g] = ("read", t + 1, 0)
        if what == "end" or done == blocks:
            if done == blocks:
                break
    assert done == blocks


@pytest.mark.parametrize("n", [2, 63, 64, 65, 130, 200])
@pytest.mark.parametrize("zero", [False, True])
def test_compact_wy_by_block_doubling(n, zero):
    """Z = Y - P^H T (P Y) with T built from diagonal blocks of 64 and T12 = -(T G)
    T there, against the reflectors one by one: 1e-13 (n eps for n <= 200, twice
    over)."""
    rng = np.random.default_rng(n)
    m = n - 1
    V = np.tril(rng.standard_normal((n, m)) + 1j * rng.standard_normal((n, m)), -1)
    V[np.arange(1, n), np.arange(m)] = 1.0
    V[1:] = np.tril(V[1:])
    tau = 2.0 / np.sum(np.abs(V) ** 2, axis=0) * np.exp(1j * 0.0)
    if zero:
        tau[::3] = 0.0
    Y = np.linalg.qr(rng.standard_normal((n, n)))[0].astype(complex)
    want = Y.copy()
    for k in range(m - 1, -1, -1):
        want -= tau[k] * np.outer(V[:, k], V[:, k].conj() @ want)
    P = np.where(tau[:, None] != 0, V.conj().T, 0.0)
    P = np.vstack([P, np.zeros((1, n))])
    t1 = np.append(np.where(tau != 0, tau, 1.0), 1.0)
    G = P @ P.conj().T
    T = np.zeros((n, n), complex)
    for k0 in range(0, n, 64):
        k1 = min(k0 + 64, n)
        T[k0:k1, k0:k1] = np.linalg.inv(np.triu(G[k0:k1, k0:k1], 1) + np.diag(1.0 / t1[k0:k1]))
    w = 64
    while w < n:
        N = (T @ G) @ T
        for i in range(0, n, 2 * w):
            T[i:i + w, i + w:i + 2 * w] = -N[i:i + w, i + w:i + 2 * w]
        w *= 2
    got = Y - P.conj().T @ (T @ (P @ Y))
    assert np.max(np.abs(got - want)) < 1e-13
