// Decisions of the host side that need no GPU: plain C++, so that a test can compile them alone.
#pragma once

namespace imrt {

// Where a caller's array lives.
enum class Memory { kHost, kDevice, kManaged };

// Whether kernels on device `dev` may read and write an array in place: managed memory and the device's own.
// Another GPU's memory is reached only by copies (peer access may be off, and a kernel's access would then
// fault), host memory likewise.
constexpr bool kernels_may_use(Memory where, int owner, int dev) {
    return where == Memory::kManaged || (where == Memory::kDevice && owner == dev);
}

}  // namespace imrt
