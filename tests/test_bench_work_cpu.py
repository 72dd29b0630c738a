"""The benchmark's rooflines divide counted work by a pipe's rate, so a count must not exceed what
the kernels need on that pipe: a fraction above 1 would say that the pipe does more than it can."""
import bench

# measured on a GB300 at full occupancy: cycles per compression of a warp on an SM quarter, whose
# ALU pipe takes a warp instruction in two cycles
SHA_CYCLES, ALU_CYCLES = 2264, 2


def test_sha256_work_fits_the_time_of_a_compression():
    assert 0.9 < bench.ALU_PER_COMPRESSION * ALU_CYCLES / SHA_CYCLES <= 1.0


def test_aes_work_is_that_of_one_permute_and_one_read_a_lookup():
    lookups = 10 * 20                                  # 16 of the round, 4 of the key schedule
    other = 10 * 7 + 9 * 8 + 4 * (3 + 1) + 4 + 4       # key schedule, columns, last columns, two XORs of a block
    assert bench.AES_LOOKUPS == lookups
    assert bench.AES_INSTR == 2 * lookups + other
    # issue (four warp instructions a cycle) is a looser bound than the reads (one a cycle)
    assert bench.AES_INSTR / 4 < bench.AES_LOOKUPS
