"""The allocator hook for tests: what blocks a net holds, and what is in them."""

WIN_BYTES = 768        # header of a window block, rounded up
WIN_P0 = 0             # its words: first step of the last window opened
WIN_BAR = 6            # arrivals at the grid barrier


_hooks = []


class Blocks:
    """The allocator hook on PyTorch's: remembers the blocks' sizes, refuses
    what `refuse` says, and gives nothing back before the end, so that a stale
    pointer reads old values."""

    def __init__(self):
        self.live, self.gone, self.asked = {}, [], []
        self.refuse = lambda n: False

    def __enter__(self):
        from paper_1310_8478_gb300 import snn
        alloc, self.free = snn.torch_allocator()

        def take(n, stream):
            self.asked.append(n)
            if self.refuse(n):
                return 0
            p = alloc(n, stream)
            self.live[p] = n
            return p

        def give(p):
            self.gone.append(p)
            del self.live[p]
        snn.set_allocator(take, give)
        _hooks.append(snn._allocator_refs)             # of nets that a failed test leaves open
        return self

    def __exit__(self, *exc):
        from paper_1310_8478_gb300 import snn
        snn.set_allocator(None)
        for p in self.gone:
            self.free(p)

    def words(self, p):
        """Block p as a tensor of 32-bit words."""
        import torch

        class Block:
            __cuda_array_interface__ = dict(shape=(self.live[p] // 4,), typestr="<i4", data=(p, False), version=2)
        return torch.as_tensor(Block(), device="cuda")


def up(x):
    return (x + 255) & ~255


def window_block(blocks, n_neurons):
    """Of a net with a resident grid: header, histories, trains, spike bits of
    64 steps, second input."""
    size = WIN_BYTES + 2 * up(8 * n_neurons) + up(64 * 4 * ((n_neurons + 31) // 32)) + up(4 * n_neurons)
    found = [p for p, n in blocks.live.items() if n == size]
    assert len(found) == 1
    return found[0]
