"""Emulated division of planes at and above shared memory in blocks of one to eight
planes (the qubits below those of a and c), registers interleaved and unordered,
and blocks above a batch (nine complex128 qubits with three below).  Bit-exact
against the definition in torch."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _value(x, qubits):
    return sum(((x >> q) & 1) << j for j, q in enumerate(qubits))


def _placed(qubits, r):
    return sum(((r >> j) & 1) << q for j, q in enumerate(qubits))


def _run(lo, k, N):
    return list(range(lo + k * N, lo + (k + 1) * N))


def _mixed(n, N, lo, seed):
    p = [lo + int(v) for v in np.random.default_rng(seed).permutation(n - lo)]
    b = list(range(lo)) + p[2 * N:]
    return p[:N], b[:N], p[N:2 * N]


REGS = [(20, (_run(2, 2, 6), _run(2, 1, 6), _run(2, 0, 6))), (21, (_run(2, 2, 6), _run(2, 1, 6), _run(2, 0, 6))),
        (22, (_run(4, 2, 6), _run(4, 1, 6), _run(4, 0, 6))), (22, _mixed(22, 6, 3, 4)), (22, (_run(1, 2, 7), _run(1, 1, 7), _run(1, 0, 7))), (23, (_run(2, 2, 7), _run(2, 1, 7), _run(2, 0, 7))),
        (24, (_run(3, 2, 7), _run(3, 1, 7), _run(3, 0, 7))), (21, (_run(7, 1, 7), _run(0, 0, 7), _run(7, 0, 7))),
        (22, _mixed(22, 7, 2, 1)), (23, _mixed(23, 7, 3, 2)), (25, _mixed(25, 8, 3, 3)),
        (27, (_run(9, 1, 9), _run(0, 0, 9), _run(9, 0, 9)))]


@pytest.mark.parametrize("n,regs", REGS, ids=lambda v: str(v) if isinstance(v, int) else "")
@pytest.mark.parametrize("dtype", ["c128", "c64"])
def test_division_blocks(n, regs, dtype):
    import torch
    from paper_1604_06460_gb300 import qe
    qa, qb, qc = regs
    N = len(qa)
    with qe.State(n, dtype) as st:
        st.set_policy(qe.POLICY_EMULATE)
        st.init_random(n)
        torch.cuda.synchronize()
        before = st.tensor.view(-1, 2).clone()
        st.div(qa, qb, qc)
        torch.cuda.synchronize()
        after = st.tensor.view(-1, 2)
        for part in torch.arange(1 << n, device="cuda").split(1 << 24):
            a, b, c = _value(part, qa), _value(part, qb), _value(part, qc)
            rest = part & ~_placed(qa + qc, torch.full_like(part, -1))
            for i in range(N - 1, -1, -1):
                c = c ^ (((b != 0) & (a >= (b << i))).long() << i)
                a = torch.where(((c >> i) & 1) == 1, (a - (b << i)) & ((1 << N) - 1), a)
            assert torch.equal(after[rest | _placed(qa, a) | _placed(qc, c)], before[part])
