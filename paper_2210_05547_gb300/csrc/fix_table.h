// Generated by gen_fix_table.py: constants of the integer exponential and logarithm in
// fix64.cuh. Do not edit.
#pragma once

#define FIX_EXP_C72 0xb17217f7d1cf79acull   // ln2/256 in units of 2^-72
#define FIX_EXP_K19 193635250            // 256/ln2 in units of 2^-19, rounded down
#define FIX_LN2_58 0x02c5c85fdf473de7ull    // ln2 in units of 2^-58
// 2^(j/256), j = 0..255, in units of 2^-62
#define FIX_EXP_BODY \
    0x4000000000000000ull, 0x402c6be96af2fb58ull, 0x4058f6a7ecccd5b6ull, 0x4085a050ec0a036aull, \
    0x40b268f9de0183baull, 0x40df50b846ef302bull, 0x410c57a1b9fe12f6ull, 0x41397dcbd952c4a6ull, \
    0x4166c34c5615d0ecull, 0x41942838f07e22a3ull, 0x41c1aca777db771bull, 0x41ef50adcaa0d899ull, \
    0x421d1461d66f2023ull, 0x424af7d9981f7e98ull, 0x4278fb2b1bce0d15ull, 0x42a71e6c7ce464afull, \
    0x42d561b3e6243d8aull, 0x4303c51791b21550ull, 0x433248adc91fdd02ull, 0x4360ec8ce577ae44ull, \
    0x438fb0cb4f468808ull, 0x43be957f7ea712b6ull, 0x43ed9abffb4c6bc9ull, 0x441cc0a35c8cf8eaull, \
    0x444c0740496d4294ull, 0x447b6ead78aad636ull, 0x44aaf701b0c72feeull, 0x44daa053c812abd2ull, \
    0x450a6abaa4b77ecdull, 0x453a564d3cc4b723ull, 0x456a632296394492ull, 0x459a9151c70f0819ull, \
    0x45cae0f1f545eb73ull, 0x45fb521a56ef0042ull, 0x462be4e23237a6efull, 0x465c9960dd74bd4bull, \
    0x468d6fadbf2dd4f3ull, 0x46be67e04e28717cull, 0x46ef821011734e6bull, 0x4720be54a071ad01ull, \
    0x47521cc5a2e6a9e0ull, 0x47839d7ad1009a90ull, 0x47b5408bf36472e2ull, 0x47e70610e3393241ull, \
    0x4818ee218a3358eeull, 0x484af8d5e2a06536ull, 0x487d2645f7725895ull, 0x48af7689e44b44eaull, \
    0x48e1e9b9d588e19bull, 0x49147fee085028d6ull, 0x4947393eca98fcd6ull, 0x497a15c47b39d53eull, \
    0x49ad159789f37496ull, 0x49e038d0777ca5e0ull, 0x4a137f87d58e025bull, 0x4a46e9d646edbf6aull, \
    0x4a7a77d47f7b84b1ull, 0x4aae299b443c4a6bull, 0x4ae1ff436b663ff7ull, 0x4b15f8e5dc6cbab0ull, \
    0x4b4a169b900c2d00ull, 0x4b7e587d905625d1ull, 0x4bb2bea4f8bd5847ull, 0x4be7492af621abd6ull, \
    0x4c1bf828c6dc54b8ull, 0x4c50cbb7bacbf4cbull, 0x4c85c3f13360c4d5ull, 0x4cbae0eea3a8c63cull, \
    0x4cf022c9905bfd32ull, 0x4d25899b8fe8b365ull, 0x4d5b157e4a7fc325ull, 0x4d90c68b7a20eb1eull, \
    0x4dc69cdceaa72a9cull, 0x4dfc988c79d52661ull, 0x4e32b9b417619617ull, 0x4e69006dc503ba65ull, \
    0x4e9f6cd3967fdba8ull, 0x4ed5feffb1b3d155ull, 0x4f0cb70c4ea39210ull, 0x4f439513b785cc80ull, \
    0x4f7a993048d088d7ull, 0x4fb1c37c7145d328ull, 0x4fe91412b2006e83ull, 0x50208b0d9e8090dfull, \
    0x50582887dcb8a7e1ull, 0x508fec9c251a267cull, 0x50c7d76542a25b72ull, 0x50ffe8fe12e750c4ull, \
    0x513821818624b40cull, 0x5170810a9f48c7cfull, 0x51a907b474015dc9ull, 0x51e1b59a2cc8da3eull, \
    0x521a8ad704f3404full, 0x525387864abb4762ull, 0x528cabc35f4f799dull, 0x52c5f7a9b6df5b77ull, \
    0x52ff6b54d8a89c75ull, 0x533906e05f045106ull, 0x5372ca67f774358full, 0x53acb60762affaaeull, \
    0x53e6c9da74b29ab5ull, 0x542105fd14c7b869ull, 0x545b6a8b3d990704ull, 0x5495f7a0fd3bbb8eull, \
    0x54d0ad5a753e077cull, 0x550b8bd3dab49cbdull, 0x5546932976483b15ull, 0x5581c377a44346f0ull, \
    0x55bd1cdad49f699cull, 0x55f89f6f8b133af4ull, 0x56344b525f1ff495ull, 0x5670209ffc1f2e82ull, \
    0x56ac1f752150a563ull, 0x56e847eea1e80a49ull, 0x57249a29651adc07ull, 0x57611642662e4a33ull, \
    0x579dbc56b48521baull, 0x57da8c8373adc331ull, 0x581786e5db7022c2ull, 0x5854ab9b37dbd1e5ull, \
    0x5891fac0e95612c8ull, 0x58cf747464a7f584ull, 0x590d18d3330c7f1eull, 0x594ae7faf23eda52ull, \
    0x5988e20954889245ull, 0x59c7071c20cfd70cull, 0x5a05575132a5cc20ull, 0x5a43d2c67a54e0c0ull, \
    0x5a827999fcef3242ull, 0x5ac14be9d45cf869ull, 0x5b0049d42f6afbb6ull, 0x5b3f737751d915c8ull, \
    0x5b7ec8f19468bbc9ull, 0x5bbe4a6164eb92f4ull, 0x5bfdf7e546520f3eull, 0x5c3dd19bd0ba1c1aull, \
    0x5c7dd7a3b17dcf75ull, 0x5cbe0a1bab4226dfull, 0x5cfe69229605cef5ull, 0x5d3ef4d75f2ff504ull, \
    0x5d7fad59099f22feull, 0x5dc092c6adb825b8ull, 0x5e01a53f7974fd86ull, 0x5e42e4e2b073d935ull, \
    0x5e8451cfac061b5full, 0x5ec5ec25db3f6a41ull, 0x5f07b404c304c9f1ull, 0x5f49a98bfe1bc11cull, \
    0x5f8bccdb3d398841ull, 0x5fce1e124712437cull, 0x60109d50f86846d8ull, 0x60534ab7441b6546ull, \
    0x6096266533384a2bull, 0x60d9307ae507dd9aull, 0x611c69188f1eb339ull, 0x615fd05e7d6c83e4ull, \
    0x61a3666d124bb204ull, 0x61e72b64c690d8afull, 0x622b1f66299a6599ull, 0x626f4291e1603dd5ull, \
    0x62b39508aa836d6full, 0x62f816eb585de1edull, 0x633cc85ad5122fbdull, 0x6381a978219b628full, \
    0x63c6ba6455dcd8aeull, 0x640bfb40a0b22959ull, 0x64516c2e47ff1623ull, 0x64970d4ea8bf8766ull, \
    0x64dcdec3371793d1ull, 0x6522e0ad7e639312ull, 0x6569132f21483ba7ull, 0x65af7669d9c2cbe4ull, \
    0x65f60a7f79393e2eull, 0x663ccf91e88a8873ull, 0x6683c5c3281ee6e9ull, 0x66caed354ff83222ull, \
    0x6712460a8fc24072ull, 0x6759d0652ee352afull, 0x67a18c678c8c8c61ull, 0x67e97a341fca775bull, \
    0x683199ed779592caull, 0x6879ebb63ae2edc6ull, 0x68c26fb128b4cd63ull, 0x690b2601182b5e56ull, \
    0x69540ec8f895722dull, 0x699d2a2bd181482aull, 0x69e6784cc2cd61bdull, 0x6a2ff94f04b962b0ull, \
    0x6a79ad55e7f6fd10ull, 0x6ac39484d5bae8c5ull, 0x6b0daeff4fcde703ull, 0x6b57fce8f09dd17full, \
    0x6ba27e656b4eb57aull, 0x6bed33988bcbfab5ull, 0x6c381ca636d99642ull, 0x6c8339b26a25494eull, \
    0x6cce8ae13c57ebdbull, 0x6d1a1056dd26c382ull, 0x6d65ca379564e639ull, 0x6db1b8a7c714a92bull, \
    0x6dfddbcbed791babull, 0x6e4a33c89d278e49ull, 0x6e96c0c284192610ull, 0x6ee382de69bc7bf8ull, \
    0x6f307a412f074892ull, 0x6f7da70fce881bf9ull, 0x6fcb096f5c782210ull, 0x7018a18506ccf314ull, \
    0x70666f76154a7089ull, 0x70b47367e994ae92ull, 0x7102ad7fff41e9b4ull, 0x71511de3ebec8913ull, \
    0x719fc4b95f452d29ull, 0x71eea2262324cb0cull, 0x723db6501b9ed447ull, 0x728d015d47136b40ull, \
    0x72dc8373be41a454ull, 0x732c3cb9b459d38bull, 0x737c2d55770fe711ull, 0x73cc556d6eadce5full, \
    0x741cb5281e25ee34ull, 0x746d4cac2325a155ull, 0x74be1c203627c62bull, 0x750f23ab2a87593eull, \
    0x75606373ee921c97ull, 0x75b1dba18b9b4c20ull, 0x76038c5b260e5eeeull, 0x765575c7fd81d5a0ull, \
    0x76a7980f6cca15c2ull, 0x76f9f358ea0c5249ull, 0x774c87cc06d1812eull, 0x779f559070195e36ull, \
    0x77f25ccdee6d7ae6ull, 0x78459dac65f45bb5ull, 0x78991853d684a285ull, 0x78ecccec5bb84661ull, \
    0x7940bb9e2cffd89dull, 0x7994e4919db5d74eull, 0x79e947ef1d320d2dull, 0x7a3de5df36dcfeefull, \
    0x7a92be8a92436616ull, 0x7ae7d219f329b948ull, 0x7b3d20b6399fc237ull, 0x7b92aa886214411cull, \
    0x7be86fb985689ddcull, 0x7c3e7072d904a6ceull, 0x7c94acddaeea5d3aull, 0x7ceb252375c9cf9bull, \
    0x7d41d96db915019dull, 0x7d98c9e62113e1faull, 0x7deff6b672f84e24ull, 0x7e47600890f223deull, \
    0x7e9f06067a4360baull, 0x7ef6e8da4b544f9aull, 0x7f4f08ae3dc7c426ull, 0x7fa765aca88f6453ull
// per j = 0..127: inv_j = 1 / (1 + (j + 1/2) / 128) in units of 2^-64, -ln(inv_j) in units
// of 2^-58
#define FIX_LOG_BODY \
    {0xff00ff00ff00ff01ull, 0x0003fe0154562178ull}, \
    {0xfd08e5500fd08e55ull, 0x000bee23afc0853bull}, \
    {0xfb18856506ddaba6ull, 0x0013cea44346a575ull}, \
    {0xf92fb2211855a865ull, 0x001b9fc027af9198ull}, \
    {0xf74e3fc22c700f75ull, 0x002361b31247b300ull}, \
    {0xf57403d5d00f5740ull, 0x002b14b75f91c9a9ull}, \
    {0xf3a0d52cba872336ull, 0x0032b9061d91c7d7ull}, \
    {0xf1d48bcee0d399faull, 0x003a4ed715b616a4ull}, \
    {0xf00f00f00f00f00full, 0x0041d660d66391c5ull}, \
    {0xee500ee500ee500full, 0x00494fd8bc28505cull}, \
    {0xec979118f3fc4da2ull, 0x0050bb72fa991bc1ull}, \
    {0xeae56403ab95900full, 0x00581962a4dd430full}, \
    {0xe939651fe2d8d35cull, 0x005f69d9b5ec4b32ull}, \
    {0xe79372e225fe30d9ull, 0x0066ad091880ceb3ull}, \
    {0xe5f36cb00e5f36cbull, 0x006de320aec3b684ull}, \
    {0xe45932d7dc52100eull, 0x00750c4f59b2cd75ull}, \
    {0xe2c4a6886a4c2e10ull, 0x007c28c300458a9aull}, \
    {0xe135a9c97500e136ull, 0x008338a89652cb71ull}, \
    {0xdfac1f74346c575full, 0x008a3c2c233a1563ull}, \
    {0xde27eb2c41f3d9d1ull, 0x00913378c852d65cull}, \
    {0xdca8f158c7f91ab8ull, 0x00981eb8c723fe98ull}, \
    {0xdb2f171df7702919ull, 0x009efe158766314eull}, \
    {0xd9ba4256c0366e91ull, 0x00a5d1b79cd2af2bull}, \
    {0xd84a598ec9151f43ull, 0x00ac99c6ccc1042full}, \
    {0xd6df43fca482f00dull, 0x00b3566a13956a87ull}, \
    {0xd578e97c3f5fe551ull, 0x00ba07c7aa01bd26ull}, \
    {0xd4173289870ac52eull, 0x00c0ae050a1abf57ull}, \
    {0xd2ba083b445250abull, 0x00c74946f4436a05ull}, \
    {0xd161543e28e50274ull, 0x00cdd9b173efdc1bull}, \
    {0xd00d00d00d00d00dull, 0x00d45f67e44178c6ull}, \
    {0xcebcf8bb5b4169cbull, 0x00dada8cf47dad23ull}, \
    {0xcd712752a886d242ull, 0x00e14b42ac60c605ull}, \
    {0xcc29786c7607f99full, 0x00e7b1aa704e2ee2ull}, \
    {0xcae5d85f1bbd6c95ull, 0x00ee0de5055f63ebull}, \
    {0xc9a633fcd967300dull, 0x00f460129552d2ffull}, \
    {0xc86a78900c86a789ull, 0x00faa852b25bd9b8ull}, \
    {0xc73293d789b9f838ull, 0x0100e6c45ad501ccull}, \
    {0xc5fe740317f9d00cull, 0x01071b85fcd590d2ull}, \
    {0xc4ce07b00c4ce07bull, 0x010d46b579ab74b2ull}, \
    {0xc3a13de60495c773ull, 0x01136870293a8b06ull}, \
    {0xc2780613c0309e02ull, 0x011980d2dd4236f6ull}, \
    {0xc152500c152500c1ull, 0x011f8ff9e48a2f29ull}, \
    {0xc0300c0300c0300cull, 0x012596010df7639full}, \
    {0xbf112a8ad278e8ddull, 0x012b9303ab89d24aull}, \
    {0xbdf59c91700bdf5aull, 0x0131871c95441850ull}, \
    {0xbcdd535db1cc5b7bull, 0x013772662bfd85afull}, \
    {0xbbc8408cd63069a1ull, 0x013d54fa5c1f70f8ull}, \
    {0xbab656100bab6561ull, 0x01432ef2a04e813bull}, \
    {0xb9a7862a0ff46588ull, 0x0149006804009d0dull}, \
    {0xb89bc36ce3e0453aull, 0x014ec9732600269bull}, \
    {0xb79300b79300b793ull, 0x01548a2c3add262dull}, \
    {0xb68d31340e4307d8ull, 0x015a42ab0f4cfe1aull}, \
    {0xb58a485518d1e7e4ull, 0x015ff3070a793d3dull}, \
    {0xb48a39d44685fe97ull, 0x01659b57303e1f28ull}, \
    {0xb38cf9b00b38cf9bull, 0x016b3bb2235943d9ull}, \
    {0xb2927c29da5519cfull, 0x0170d42e2789235dull}, \
    {0xb19ab5c45606f00bull, 0x017664e1239dbcecull}, \
    {0xb0a59b418d749d53ull, 0x017bede0a37afbfaull}, \
    {0xafb321a1496fdf0eull, 0x01816f41da0d495bull}, \
    {0xaec33e1f671529a5ull, 0x0186e919a330ba01ull}, \
    {0xadd5e6323fd48a86ull, 0x018c5b7c858b48a8ull}, \
    {0xaceb0f891e6551bbull, 0x0191c67eb45a83d8ull}, \
    {0xac02b00ac02b00acull, 0x01972a3411351587ull}, \
    {0xab1cbdd3e2970f60ull, 0x019c86b02dc0862aull}, \
    {0xaa392f35dc17f00bull, 0x01a1dc064d5b9956ull}, \
    {0xa957fab5402a55ffull, 0x01a72a4966bd9ea1ull}, \
    {0xa87917088e262b6full, 0x01ac718c258b0e41ull}, \
    {0xa79c7b16ea64d422ull, 0x01b1b1e0ebdfc5b7ull}, \
    {0xa6c21df6e1625c80ull, 0x01b6eb59d3cf35daull}, \
    {0xa5e9f6ed347f0721ull, 0x01bc1e08b0dad0a4ull}, \
    {0xa513fd6bb00a5140ull, 0x01c149ff115f026bull}, \
    {0xa44029100a440291ull, 0x01c66f4e3ff6ff7eull}, \
    {0xa36e71a2cb033128ull, 0x01cb8e0744d7aca0ull}, \
    {0xa29ecf163bb6500aull, 0x01d0a63ae721e642ull}, \
    {0xa1d139855f7268eeull, 0x01d5b7f9ae2c683dull}, \
    {0xa105a932f2ca891full, 0x01dac353e2c59542ull}, \
    {0xa03c1688732b3032ull, 0x01dfc859906d5b54ull}, \
    {0x9f747a152d7836d0ull, 0x01e4c71a86877043ull}, \
    {0x9eaecc8d53ae2ddfull, 0x01e9bfa659861f56ull}, \
    {0x9deb06c9194aa416ull, 0x01eeb20c640ddf43ull}, \
    {0x9d2921c3d6411308ull, 0x01f39e5bc811e5bdull}, \
    {0x9c69169b30446dfaull, 0x01f884a36fe9ec23ull}, \
    {0x9baade8e4a2f6e10ull, 0x01fd64f20f61571dull}, \
    {0x9aee72fcf957c10full, 0x02023f5624bff143ull}, \
    {0x9a33cd67009a33cdull, 0x020713ddf9cc6768ull}, \
    {0x997ae76b50efd00aull, 0x020be297a4c8b381ull}, \
    {0x98c3bac74f5db00aull, 0x0210ab910968a1cbull}, \
    {0x980e4156201301c8ull, 0x02156ed7d9c29a38ull}, \
    {0x975a750ff68a58afull, 0x021a2c79973ad6fcull}, \
    {0x96a850096a850097ull, 0x021ee48393692faaull}, \
    {0x95f7cc72d1b887e9ull, 0x02239702f0f99f08ull}, \
    {0x9548e4979e0829fdull, 0x02284404a487a89eull}, \
    {0x949b92ddc02526e5ull, 0x022ceb957574c1c0ull}, \
    {0x93efd1c50e726b7cull, 0x02318dc1feb9e0c1ull}, \
    {0x93459be6b009345aull, 0x02362a96afb453deull}, \
    {0x929cebf48bbd90e5ull, 0x023ac21fccee0061ull}, \
    {0x91f5bcb8bb02d9cdull, 0x023f546970e12981ull}, \
    {0x9150091500915009ull, 0x0243e17f8cb7dd7cull}, \
    {0x90abcc0242af3009ull, 0x0248696de907267cull}, \
    {0x9009009009009009ull, 0x024cec4026861bfaull}, \
    {0x8f67a1e3fdc26178ull, 0x02516a01bec0f056ull}, \
    {0x8ec7ab397255e41dull, 0x0255e2be04c815a4ull}, \
    {0x8e2917e0e702c6cdull, 0x025a568025db93b5ull}, \
    {0x8d8be33f95d71590ull, 0x025ec5532a12a8c6ull}, \
    {0x8cf008cf008cf009ull, 0x02632f41f4ffcd44ull}, \
    {0x8c55841c815ed5caull, 0x0267945746513299ull}, \
    {0x8bbc50c8deb420c0ull, 0x026bf49dba6dd400ull}, \
    {0x8b246a87e19008b2ull, 0x0270501fcb0f2fd8ull}, \
    {0x8a8dcd1feeae465cull, 0x0274a6e7cfd7bf32ull}, \
    {0x89f87469a23920e0ull, 0x0278f8fffee640b9ull}, \
    {0x89645c4f6e055decull, 0x027d46726d65eb70ull}, \
    {0x88d180cd3a4133d7ull, 0x02818f49101b9d24ull}, \
    {0x883fddf00883fddfull, 0x0285d38dbbf017e6ull}, \
    {0x87af6fd5992d0d40ull, 0x028a134a2677614aull}, \
    {0x872032ac13008720ull, 0x028e4e87e67555a6ull}, \
    {0x869222b1acf1ce96ull, 0x02928550745f80efull}, \
    {0x86053c345a0b8473ull, 0x0296b7ad2adc4e72ull}, \
    {0x85797b917765ab89ull, 0x029ae5a7473fa009ull}, \
    {0x84eedd357c1b0085ull, 0x029f0f47ea04dd11ull}, \
    {0x84655d9bab2f1008ull, 0x02a33498174688cdull}, \
    {0x83dcf94dc7570ce1ull, 0x02a755a0b7336f95ull}, \
    {0x8355ace3c897db10ull, 0x02ab726a968179a8ull}, \
    {0x82cf750393ac3319ull, 0x02af8afe66de3211ull}, \
    {0x824a4e60b3262bc5ull, 0x02b39f64bf5d0fbfull}, \
    {0x81c635bc123fdf8eull, 0x02b7afa61ce38e64ull}, \
    {0x814327e3b94f462full, 0x02bbbbcae293246full}, \
    {0x80c121b28bd1ba98ull, 0x02bfc3db5a312312ull}, \
    {0x8040201008040201ull, 0x02c3c7dfb48c8cd3ull}
