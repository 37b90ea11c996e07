"""The addresses a State hands to the library, on CPU tensors (the call reads
no data): the two buffers of a pair may be one tensor, as State makes them, a
view of a larger one, or two tensors of their own."""
import pytest

torch = pytest.importorskip("torch")
sk = pytest.importorskip("paper_2604_25876_gb300")

N = (6, 7, 8)


def state(phi, vel):
    st = sk.State.__new__(sk.State)
    st.lat, st.phi, st.vel = sk.Lattice(N, 0.25, 1.0, 32), phi, vel
    st.scratch = torch.zeros(512, dtype=torch.uint8)
    return st


def buffer(count, *lead):
    return torch.zeros(lead + (count,) + N + (4,))


@pytest.mark.parametrize("make", [lambda: buffer(2), lambda: buffer(5)[1:3], lambda: buffer(6)[::3],
                                  lambda: buffer(2, 3)[1], lambda: torch.nn.Parameter(buffer(2)),
                                  lambda: [buffer(1)[0], buffer(1)[0]],
                                  lambda: (buffer(4)[3], buffer(4)[0])])
def test_a_state_hands_over_the_addresses_of_both_buffers(make):
    phi, vel = make(), make()
    c = state(phi, vel).c()
    assert list(c.phi) == [phi[0].data_ptr(), phi[1].data_ptr()]
    assert list(c.vel) == [vel[0].data_ptr(), vel[1].data_ptr()]


def test_a_pair_of_one_buffer_is_refused():
    with pytest.raises(IndexError):
        state(buffer(1), buffer(2)).c()
    with pytest.raises(IndexError):
        state(buffer(2), [buffer(1)[0]]).c()
