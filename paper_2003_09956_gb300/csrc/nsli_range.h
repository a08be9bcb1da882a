// nsli_range.h -- does an allocation hold what a kernel is to read?  (also
// compiled for the host by the tests)
#pragma once

#include <cstddef>
#include <cstdint>

namespace nsli {

// Do `count` elements of `elem` bytes from address p on lie inside the
// allocation of `size` bytes at `base`?
constexpr bool range_covers(std::uintptr_t base, std::size_t size, std::uintptr_t p, std::size_t count,
                            std::size_t elem)
{
    return p >= base && p - base <= size && count <= (size - (p - base)) / elem;
}

}  // namespace nsli
